"""The per-term sums of the dot partials: terms with one and with several
segments in an output, terms with hundreds of outputs (more runs than a block
reads at once), terms that no pair has, in both directions and arithmetics."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from oracle import superblock as osb
from workloads.superblock import Pair, Superblock, seeded_normal

TOL = 1e-12  # of max|dots|: float64 sums of O(1000) products, double-float at 2^-46 per term


@pytest.mark.parametrize("sectors,batch", [(3, 1), (300, 2), (600, 1)])
def test_term_dots(sectors, batch):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_0902_3185_gb300 import binding
    rng = np.random.default_rng(sectors)
    r, c = rng.integers(1, 6, sectors), rng.integers(1, 6, sectors)
    r[:2], c[:2] = 40, 33
    pairs = []
    for s in range(sectors):
        # term 0: every sector; 1: identity on the left; 3: several pairs write the same output; 2: none
        pairs.append(Pair(0, s, s, rng.standard_normal((r[s], r[s])), rng.standard_normal((c[s], c[s]))))
        pairs.append(Pair(1, s, s, None, rng.standard_normal((c[s], c[s]))))
        for d in (1, 2):
            so = (s + d) % sectors if d == 1 else 0
            pairs.append(Pair(3, so, s, rng.standard_normal((r[so], r[s])), rng.standard_normal((c[so], c[s]))))
    sb = Superblock(r, c, rng.standard_normal((batch, 4)), pairs)
    g = binding.GpuSuperblock(sb)
    X = np.stack([seeded_normal(b, sb.dim) for b in range(batch)])
    G = np.stack([seeded_normal(50 + b, sb.dim) for b in range(batch)])
    x, gg = torch.from_numpy(X).cuda(), torch.from_numpy(G).cuda()
    ref = np.stack([osb.term_products(sb, X[b], X[b]) for b in range(batch)])
    for prec in ("fp64", "df64"):
        y, dots = g.apply_H_term_dots(x, prec=prec)
        assert np.abs(dots.cpu().numpy() - ref).max() <= TOL * np.abs(ref).max()
        again = g.apply_H_term_dots(x, prec=prec)[1]
        assert torch.equal(dots, again)
        for b in range(batch):
            want = osb.apply_H(sb, X[b], b)
            assert np.abs(y[b].cpu().numpy() - want).max() <= TOL * np.abs(want).max()
    dc = g.apply_H_backward(x, gg)[1].cpu().numpy()
    want = np.stack([osb.term_products(sb, G[b], X[b]) for b in range(batch)])
    assert np.abs(dc - want).max() <= TOL * np.abs(want).max()
