"""The two groups of a sector's segments (those that end with an operator on
the right, those with one on the left) are summed by chains of their own in
every arithmetic, and their values added in float64: the product of a
superblock is, bit for bit, the sum of the products of its two halves.  One
chain over both groups would carry the first group's rounding through the
second (double-float: 1.4 times the error on a real superblock)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from workloads.superblock import Superblock, seeded_normal
from workloads.synthetic import random_sectored


def ends_on_the_right(sb, p):
    """Whether the pair's last product has its operator on the right (B)."""
    if p.A is None or p.B is None:
        return p.A is None
    ro, ri, co, ci = (int(v) for v in (sb.r[p.s_out], sb.r[p.s_in], sb.c[p.s_out], sb.c[p.s_in]))
    return ro * ri * ci + ro * ci * co <= ri * ci * co + ro * ri * co  # (A Psi) B^T is the cheaper order


# sector widths below and above every tile edge; one member and several
@pytest.mark.parametrize("dmin,dmax,batch", [(1, 20, 3), (9, 90, 2), (100, 300, 1), (200, 330, 4)])
@pytest.mark.parametrize("prec", ["fp64", "df64"])
def test_groups_are_summed_apart(dmin, dmax, batch, prec):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_0902_3185_gb300 import binding
    sb = random_sectored(seed=dmax, n_sectors=5, dmin=dmin, dmax=dmax, deltas=(0, 1, -1, 2), batch=batch,
                         identity_terms=True)
    x = torch.from_numpy(np.stack([seeded_normal(b, sb.dim) for b in range(batch)])).cuda()
    acc = torch.from_numpy(np.stack([seeded_normal(90 + b, sb.dim) for b in range(batch)])).cuda()

    def product(pairs, y=None):
        g = binding.GpuSuperblock(Superblock(sb.r, sb.c, sb.coeffs, pairs, sb.term_names))
        return g.apply_H(x, y=y, accumulate=y is not None, prec=prec)

    right = [p for p in sb.pairs if ends_on_the_right(sb, p)]
    left = [p for p in sb.pairs if not ends_on_the_right(sb, p)]
    assert right and left
    assert torch.equal(product(sb.pairs), product(right) + product(left))
    assert torch.equal(product(sb.pairs, acc.clone()), (acc + product(right)) + product(left))
