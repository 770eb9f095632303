"""The stopping test of the device Lanczos: its float32 estimate must neither
stop a member above its tolerance nor keep it running past it, from one-step
Krylov spaces to lengths beyond a warp, at tolerances from coarse to near
rounding."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from oracle import lanczos as olz
from oracle import superblock as osb
from workloads.grown import grown_hubbard_superblock
from workloads.superblock import seeded_normal


@pytest.fixture(scope="module")
def case():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_0902_3185_gb300 import binding
    sb = grown_hubbard_superblock(12, "ladder", 5, 5, m=60, cut=6, U_values=[2.0, 5.0, 9.0])
    X = np.stack([seeded_normal(70 + b, sb.dim) for b in range(sb.batch)])
    return sb, binding.GpuSuperblock(sb), X, torch.from_numpy(X).cuda()


@pytest.mark.parametrize("check_every", [1, 5])
@pytest.mark.parametrize("tol", [1e-2, 1e-4, 0.99e-5, 1e-8, 1e-13])
def test_stops_at_the_tolerance(case, tol, check_every):
    """Residual beta_j |s_j| within the tolerance, and no more steps than the
    oracle needs for half of it (the float32 test of tol >= 1e-5 asks for
    half) plus one check interval and one step of rounding."""
    sb, g, X, x = case
    e0, psi, infos, st = g.lanczos_ground(x, tol=tol, max_iter=400, check_every=check_every)
    assert st == 0, infos
    psi = psi.cpu().numpy()
    for b in range(sb.batch):
        r = osb.apply_H(sb, psi[b], b) - e0[b] * psi[b]
        # the float64 residual of the returned vector: the tolerance, and the rounding of H psi
        assert np.linalg.norm(r) <= tol * max(1.0, abs(e0[b])) * (1 + 1e-6) + 1e-13 * np.abs(sb.coeffs[b]).sum()
        ref = olz.lanczos_ground(lambda v: osb.apply_H(sb, v, b), X[b], tol=0.5 * tol, max_iter=400)
        assert infos[b]["iters"] <= ref.iters + check_every + 1, (tol, b, infos[b]["iters"], ref.iters)


@pytest.mark.parametrize("max_iter", [1, 2, 3, 31, 32, 33])
def test_cap(case, max_iter):
    """At the cap the member ends with its float64 Ritz value: the lowest
    eigenvalue of the oracle's tridiagonal matrix of that length."""
    sb, g, X, x = case
    e0, _, infos, st = g.lanczos_ground(x, tol=1e-13, max_iter=max_iter)
    assert st == 4
    for b in range(sb.batch):
        ref = olz.lanczos_ground(lambda v: osb.apply_H(sb, v, b), X[b], tol=1e-13, max_iter=max_iter)
        assert infos[b]["iters"] == max_iter and infos[b]["status"] == 4
        assert abs(e0[b] - ref.e0) <= 1e-11 * max(1.0, abs(ref.e0))
