"""dmrg_set_coeffs keeps its promises when the table is the one already set and
when a call fails: the stream is synchronised, and a retry after a failure
does all of the work that the failed call left undone."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from workloads.superblock import seeded_normal
from workloads.synthetic import random_sectored


@pytest.fixture
def gpu():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_0902_3185_gb300 import binding
    return binding


def test_the_same_table_synchronises_the_stream(gpu):
    sb = random_sectored(seed=2, n_sectors=3, dmin=4, dmax=20, batch=2)
    g = gpu.GpuSuperblock(sb)
    side = torch.cuda.Stream()
    with torch.cuda.stream(side):
        torch.cuda._sleep(200_000_000)  # about 0.1 s
        g.set_coeffs(sb.coeffs, stream=side)
        assert side.query()


def test_a_retry_after_a_failure_rebuilds_everything(gpu):
    sb = random_sectored(seed=4, n_sectors=4, dmin=20, dmax=60, batch=2, identity_terms=True)
    x = torch.from_numpy(np.stack([seeded_normal(b, sb.dim) for b in range(2)])).cuda()
    g = gpu.GpuSuperblock(sb)
    for prec in ("tf32", "bf16x3"):
        g.apply_H(x, prec=prec)
        for _ in range(2):  # the second solve captures its iterations
            g.lanczos_ground(x, tol=1e-3, max_iter=12, prec=prec, refine="none")
    c = np.tile(1.5 * sb.coeffs[:1], (2, 1))  # the same for both members: folded into the operand panels
    ref = gpu.GpuSuperblock(sb.with_coeffs(c))
    g.set_coeffs(c)
    c = -0.5 * c
    assert g.lib.dmrg_test_inject(g.h, 3) == 0
    with pytest.raises(gpu.DmrgError):
        g.set_coeffs(c)
    g.set_coeffs(c)
    ref.set_coeffs(c)
    for prec in ("fp64", "tf32", "bf16x3"):
        assert torch.equal(g.apply_H(x, prec=prec), ref.apply_H(x, prec=prec))
    for prec in ("tf32", "bf16x3"):
        a = g.lanczos_ground(x, tol=1e-3, max_iter=12, prec=prec, refine="none")
        b = ref.lanczos_ground(x, tol=1e-3, max_iter=12, prec=prec, refine="none")
        assert np.array_equal(a[0], b[0]) and torch.equal(a[1], b[1])


def test_has_coeffs(gpu):
    sb = random_sectored(seed=4, n_sectors=3, dmin=20, dmax=40, batch=2, identity_terms=True)
    g = gpu.GpuSuperblock(sb)
    x = torch.from_numpy(np.stack([seeded_normal(b, sb.dim) for b in range(2)])).cuda()
    c = np.array(sb.coeffs)
    assert g.has_coeffs(c) and not g.has_coeffs(c[:1]) and not g.has_coeffs(-c)
    g.set_coeffs(-c)
    assert g.has_coeffs(-c) and not g.has_coeffs(c)
    d = np.tile(2.0 * c[:1], (2, 1))  # folded into the operand panels, whose build fails
    g.apply_H(x, prec="bf16x3")
    assert g.lib.dmrg_test_inject(g.h, 3) == 0
    with pytest.raises(gpu.DmrgError):
        g.set_coeffs(d)
    assert not g.has_coeffs(d) and not g.has_coeffs(-c)
    g.set_coeffs(d)
    assert g.has_coeffs(d)


def test_autograd_with_changing_couplings(gpu):
    """Two graphs on one superblock: each backward uses the couplings of its own forward."""
    sb = random_sectored(seed=6, n_sectors=3, dmin=5, dmax=30, batch=2)
    g = gpu.GpuSuperblock(sb)
    x = torch.from_numpy(np.stack([seeded_normal(b, sb.dim) for b in range(2)])).cuda().requires_grad_(True)
    cot = torch.from_numpy(np.stack([seeded_normal(9 + b, sb.dim) for b in range(2)])).cuda()
    cs = [torch.tensor(sb.coeffs * f, device="cuda", requires_grad=True) for f in (1.0, -0.5)]
    ys = [gpu.apply_H(x, c, g) for c in cs]
    for y, c in zip(ys, cs):
        dx, dc = torch.autograd.grad(y, (x, c), cot)
        ref = gpu.GpuSuperblock(sb.with_coeffs(c.detach().cpu().numpy()))
        assert torch.equal(y.detach(), ref.apply_H(x.detach()))
        want = ref.apply_H_backward(x.detach(), cot)
        assert torch.equal(dx, want[0]) and torch.equal(dc, want[1])
