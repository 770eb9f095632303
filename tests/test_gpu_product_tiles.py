"""The CUDA-core product's tiles: lists cut into 8 x 8 and into 16 x 16 tiles,
sector widths around the tile edges, K remainders of every chunk, more
segments per output than the kernel keeps in shared memory, and both groups
of segments present, missing or alone, in every arithmetic and direction."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from oracle import grad as ograd
from oracle import superblock as osb
from workloads.superblock import Pair, Superblock, seeded_normal

TOL = 1e-12  # of max|y|: float64 sums of O(1000) terms, double-float at 2^-46 per term


def build(dims, n_terms, batch, sides, coeffs=None, seed=5):
    """Neighbouring sectors coupled both ways; `sides` picks which identity
    sides the diagonal terms have ("A", "B", "AB" or none)."""
    rng = np.random.default_rng(seed)
    r, c = np.array([d[0] for d in dims]), np.array([d[1] for d in dims])
    pairs = []
    for k in range(n_terms):
        for s in range(len(dims)):
            so = (s + k) % len(dims)
            pairs.append(Pair(k, so, s, rng.standard_normal((r[so], r[s])) / np.sqrt(r[s]),
                              rng.standard_normal((c[so], c[s])) / np.sqrt(c[s])))
    n = n_terms
    for side in sides:
        for s in range(len(dims)):
            if side == "B":
                pairs.append(Pair(n, s, s, rng.standard_normal((r[s], r[s])), None))
            else:
                pairs.append(Pair(n, s, s, None, rng.standard_normal((c[s], c[s]))))
        n += 1
    co = rng.standard_normal((batch, n)) if coeffs is None else np.resize(np.asarray(coeffs, dtype=float), (batch, n))
    return Superblock(r, c, co, pairs)


CASES = {
    # few tiles; more than 32 segments per output; coefficients +-1 and others
    "many_segments": lambda: build([(3, 5), (8, 7), (1, 17)], 45, 2, "AB", coeffs=[1.0, -1.0, 0.3]),
    # widths one below, at and above the tile edges and the K chunk
    "edges": lambda: build([(7, 9), (8, 15), (9, 16), (15, 17), (16, 8), (17, 31), (33, 1)], 3, 3, "AB"),
    # many tiles: 16 x 16 shapes with remainders on both sides
    "wide": lambda: build([(130, 257), (255, 100), (16, 300), (300, 40)], 2, 1, "A"),
    "wide_batch": lambda: build([(70, 90), (89, 61), (33, 120)], 3, 5, "B"),
    # outputs with only one group of segments
    "only_right": lambda: build([(20, 40), (24, 33)], 0, 2, "A"),
    "only_left": lambda: build([(40, 20), (33, 24)], 0, 2, "B"),
}


@pytest.mark.parametrize("name", sorted(CASES))
def test_product_tiles(name):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_0902_3185_gb300 import binding
    sb = CASES[name]()
    g = binding.GpuSuperblock(sb)
    X = np.stack([seeded_normal(b, sb.dim) for b in range(sb.batch)])
    G = np.stack([seeded_normal(50 + b, sb.dim) for b in range(sb.batch)])
    x, gg = torch.from_numpy(X).cuda(), torch.from_numpy(G).cuda()

    def close(got, ref):
        assert np.abs(got - ref).max() <= TOL * np.abs(ref).max()

    ref = [osb.apply_H(sb, X[b], b) for b in range(sb.batch)]
    dots = [osb.term_products(sb, X[b], X[b]) for b in range(sb.batch)]
    for prec in ("fp64", "df64"):
        y = g.apply_H(x, prec=prec).cpu().numpy()
        acc = gg.clone()
        g.apply_H(x, y=acc, accumulate=True, prec=prec)
        yt, dt = g.apply_H_term_dots(x, prec=prec)
        for b in range(sb.batch):
            close(y[b], ref[b])
            close(acc[b].cpu().numpy(), G[b] + ref[b])
            close(yt[b].cpu().numpy(), ref[b])
            close(dt[b].cpu().numpy(), dots[b])
    dpsi, dc = g.apply_H_backward(x, gg)
    for b in range(sb.batch):
        close(dpsi[b].cpu().numpy(), osb.apply_HT(sb, G[b], b))
        close(dc[b].cpu().numpy(), ograd.apply_H_backward(sb, X[b], G[b], b)[1])
