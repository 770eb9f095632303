"""The Gram-Schmidt passes of short and long vectors: vector lengths around
the chunk and block edges against the oracle, and the same members run in a
batch just below and just above the length where the passes change their
blocks, which must not change a bit."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from oracle import ldos
from oracle import superblock as osb
from workloads.superblock import Pair, Superblock, seeded_normal


def build(r, c, batch, seed=3):
    """One sector with symmetric block Hamiltonians on both sides and a
    symmetric coupling; one coefficient row per member."""
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


@pytest.mark.parametrize("r,c", [(31, 1), (8, 4), (3, 11), (33, 31), (32, 32), (41, 25), (63, 65), (64, 64), (17, 241)])
def test_lengths(gpu, r, c):
    """D = 31, 32, 33, 1023, 1024, 1025, 4095, 4096, 4097."""
    sb = build(r, c, 2)
    n = min(24, sb.dim)
    X = np.stack([seeded_normal(b, sb.dim) for b in range(2)])
    norm2, a, b, got = gpu.GpuSuperblock(sb).lanczos_coeffs(torch.from_numpy(X).cuda(), n)
    for m in range(2):
        rn, ra, rb = ldos.lanczos_coefficients(lambda v: osb.apply_H(sb, v, m), X[m], n)
        assert got[m] == len(ra) and abs(float(norm2[m]) - rn) <= 1e-12 * rn
        k = min(len(ra), len(rb), 20)  # the last coefficients of an exhausted space are rounding
        if sb.dim > 2 * n:
            assert np.abs(a[m, :k].cpu().numpy() - ra[:k]).max() <= 1e-10 * np.abs(ra).max()
            assert np.abs(b[m, :k].cpu().numpy() - rb[:k]).max() <= 1e-10 * np.abs(rb).max()


def test_same_bits_in_short_and_long_batches(gpu):
    """D = 1025 is one chunk: 303 members take the short path, 304 the long one."""
    out = []
    for batch in (303, 304):
        sb = build(41, 25, 304)
        sb = sb.with_coeffs(sb.coeffs[:batch])
        x = torch.from_numpy(np.stack([seeded_normal(b, sb.dim) for b in range(batch)])).cuda()
        norm2, a, b, n = gpu.GpuSuperblock(sb).lanczos_coeffs(x, 30)
        out.append((a[:303].cpu().numpy(), b[:303].cpu().numpy()))
    assert np.array_equal(out[0][0], out[1][0]) and np.array_equal(out[0][1], out[1][1])
