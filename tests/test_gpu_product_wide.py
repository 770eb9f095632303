"""The product's 24-wide tiles, taken by lists of many outputs: every element is
the same chain of operations in any tile, so a member's product is bit for bit
that of a superblock of its own, whose list is cut into 8 x 8 tiles.  Widths
around the multiples of 8, 16 and 24, K remainders, both groups of segments."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from oracle import superblock as osb
from workloads.superblock import seeded_normal
from workloads.synthetic import random_sectored

TOL = 1e-12  # of max|y|: float64 sums of O(1000) terms, double-float at 2^-46 per term


@pytest.mark.parametrize("dmin,dmax,batch", [(23, 25, 1500), (20, 75, 250), (95, 130, 60)])
def test_wide_lists(dmin, dmax, batch):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_0902_3185_gb300 import binding
    sb = random_sectored(seed=dmax, n_sectors=4, dmin=dmin, dmax=dmax, deltas=(0, 1, -1), batch=batch,
                         identity_terms=True)
    coeffs = np.array(sb.coeffs)
    coeffs[::3, 0], coeffs[1::3, 0] = 1.0, -1.0
    sb = sb.with_coeffs(coeffs)
    g = binding.GpuSuperblock(sb)
    x = torch.from_numpy(np.stack([seeded_normal(b, sb.dim) for b in range(batch)])).cuda()
    acc = torch.from_numpy(np.stack([seeded_normal(900 + b, sb.dim) for b in range(batch)])).cuda()
    for prec in ("fp64", "df64"):
        y = g.apply_H(x, prec=prec)
        ya = g.apply_H(x, y=acc.clone(), accumulate=True, prec=prec)
        yt = g.apply_H_backward(x, acc, want_dc=False)[0]
        for b in (0, 1, batch // 2, batch - 1):
            one = binding.GpuSuperblock(sb.with_coeffs(coeffs[b:b + 1]))
            xb, ab = x[b:b + 1].contiguous(), acc[b:b + 1].contiguous()
            assert torch.equal(one.apply_H(xb, prec=prec)[0], y[b])
            assert torch.equal(one.apply_H(xb, y=ab.clone(), accumulate=True, prec=prec)[0], ya[b])
            assert torch.equal(one.apply_H_backward(xb, ab, want_dc=False)[0][0], yt[b])
            ref = osb.apply_H(sb, x[b].cpu().numpy(), b)
            assert np.abs(y[b].cpu().numpy() - ref).max() <= TOL * np.abs(ref).max()
