"""The cluster eigensolver's tournament: sizes around the block counts, odd
sizes (a player without a partner), one, few and many pairs per block, and
matrices of different sizes in one launch, against LAPACK."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def matrix(n, seed):
    """A random spectrum of both signs with a multiple and a zero eigenvalue."""
    rng = np.random.default_rng(seed)
    q, _ = np.linalg.qr(rng.standard_normal((n, n)))
    w = rng.standard_normal(n)
    w[n // 2:n // 2 + 3] = 0.25
    w[0] = 0.0
    M = (q * w) @ q.T
    return 0.5 * (M + M.T)


@pytest.mark.parametrize("sizes", [[33], [34, 35, 3, 1, 2], [63, 64, 65], [66, 5, 40], [95, 96, 97, 110],
                                   [111, 112, 113, 127, 128, 129], [224, 225, 33, 447]])
def test_against_lapack(sizes):
    """w to 1e-12 |M| sqrt(n), V orthogonal to 1e-12 sqrt(n), residual to 1e-11 |M| sqrt(n)."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_0902_3185_gb300 import binding
    mats = [matrix(n, 11 + n) for n in sizes]
    out = binding.sym_eig_batched([torch.from_numpy(M).cuda() for M in mats])
    for M, (w, V) in zip(mats, out):
        w, V = w.cpu().numpy(), V.cpu().numpy()
        n = M.shape[0]
        scale = max(np.abs(np.linalg.eigvalsh(M)).max(), 1e-300)
        assert np.all(np.diff(w) <= 0)
        assert np.abs(w - np.sort(np.linalg.eigvalsh(M))[::-1]).max() <= 1e-12 * scale * np.sqrt(n), n
        assert np.abs(V.T @ V - np.eye(n)).max() <= 1e-12 * np.sqrt(n), n
        assert np.abs(M @ V - V * w[None, :]).max() <= 1e-11 * scale * np.sqrt(n), n
