"""The Gram-Schmidt passes on the double-float pair basis (mixed-precision
solves) at the vector lengths where their blocks change, and the first
coefficients of spaces too small for a long run."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from oracle import ldos
from oracle import superblock as osb
from workloads.superblock import Pair, Superblock, seeded_normal

LENGTHS = [(31, 1), (8, 4), (3, 11), (33, 31), (32, 32), (41, 25), (63, 65), (64, 64), (17, 241), (128, 129)]


def build(r, c, batch, seed=3):
    """One sector with symmetric block Hamiltonians on both sides and a symmetric coupling."""
    rng = np.random.default_rng(seed)

    def sym(n):
        a = rng.standard_normal((n, n)) / np.sqrt(n)
        return a + a.T

    pairs = [Pair(0, 0, 0, sym(r), None), Pair(1, 0, 0, None, sym(c)), Pair(2, 0, 0, sym(r), sym(c))]
    return Superblock(np.array([r]), np.array([c]), np.random.default_rng(9).standard_normal((batch, 3)), pairs)


@pytest.fixture(scope="module")
def gpu():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_0902_3185_gb300 import binding
    return binding


@pytest.mark.parametrize("r,c", LENGTHS[:3])
def test_first_coefficients_of_small_spaces(gpu, r, c):
    """D = 31, 32, 33, eight coefficients: float64 sums of at most 33 terms."""
    sb = build(r, c, 2)
    X = np.stack([seeded_normal(b, sb.dim) for b in range(2)])
    _, a, b, got = gpu.GpuSuperblock(sb).lanczos_coeffs(torch.from_numpy(X).cuda(), 8)
    for m in range(2):
        _, ra, rb = ldos.lanczos_coefficients(lambda v: osb.apply_H(sb, v, m), X[m], 8)
        assert got[m] == 8
        assert np.abs(a[m].cpu().numpy() - ra).max() <= 1e-10 * np.abs(ra).max()
        assert np.abs(b[m, :7].cpu().numpy() - rb[:7]).max() <= 1e-10 * np.abs(rb).max()


def gram_schmidt(product, x, n):
    """n Lanczos steps in float64, every vector orthogonalised twice against all earlier ones."""
    V = [x / x.norm(dim=1, keepdim=True)]
    a, b = [], []
    for j in range(n):
        w = product(V[j])
        a.append((w * V[j]).sum(dim=1))
        for _ in range(2):
            for v in V:
                w = w - (w * v).sum(dim=1, keepdim=True) * v
        b.append(w.norm(dim=1))
        V.append(w / b[-1][:, None])
    return torch.stack(a, 1), torch.stack(b, 1)


@pytest.mark.parametrize("r,c", LENGTHS)
def test_pair_basis(gpu, r, c):
    """Eight coefficients with the library's own mixed product.  The passes keep
    48 bits (1e-13 of the sums here), which eight steps amplify by the condition
    of the Krylov vectors; an input rounded the other way to float32 changes a
    coefficient by 6e-8 of one element's share.  1e-9 of the largest."""
    sb = build(r, c, 2)
    g = gpu.GpuSuperblock(sb)
    x = torch.from_numpy(np.stack([seeded_normal(b, sb.dim) for b in range(2)])).cuda()
    _, a, b, got = g.lanczos_coeffs(x, 8, prec="bf16x3")
    ra, rb = gram_schmidt(lambda v: g.apply_H(v.contiguous(), prec="bf16x3"), x, 8)
    assert list(got) == [8, 8]
    assert float((a - ra).abs().max()) <= 1e-9 * float(ra.abs().max())
    assert float((b - rb)[:, :7].abs().max()) <= 1e-9 * float(rb.abs().max())


def test_pair_basis_same_bits_in_short_and_long_batches(gpu):
    """D = 1025 is one chunk: 99 members take the short path, 100 the long one."""
    out = []
    for batch in (99, 100):
        sb = build(41, 25, 100)
        sb = sb.with_coeffs(sb.coeffs[:batch])
        x = torch.from_numpy(np.stack([seeded_normal(b, sb.dim) for b in range(batch)])).cuda()
        _, a, b, _ = gpu.GpuSuperblock(sb).lanczos_coeffs(x, 20, prec="bf16x3")
        out.append((a[:99].cpu().numpy(), b[:99].cpu().numpy()))
    assert np.array_equal(out[0][0], out[1][0]) and np.array_equal(out[0][1], out[1][1])
