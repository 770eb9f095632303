"""The tensor-core product where its tiles are split along N and dealt to the
SMs by their modelled length: widths around the 16-column steps and the 32
column limit of a part, one long chain of segments among short ones, and a
batch whose rows fill several tiles, against the oracle."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from oracle import superblock as osb
from workloads.superblock import Pair, Superblock, seeded_normal

# operand rounding (a few units of TF32's 2^-11, of the split pair's 2^-16) and
# the FP32 sums, of the product of the absolute values
GAMMA = {"tf32": 8 * 2.0 ** -11 + 1e-5, "bf16x3": 8 * 2.0 ** -16 + 2e-6}


def build(r, c, batch, seed=5):
    """Sector 0 (r x c) takes twelve two-sided products and a one-sided one of
    each kind; sector 1 (9 x 17) takes one."""
    rng = np.random.default_rng(seed)

    def sym(n):
        a = rng.standard_normal((n, n)) / np.sqrt(n)
        return a + a.T

    pairs = [Pair(t, 0, 0, sym(r), sym(c)) for t in range(12)]
    pairs += [Pair(12, 0, 0, sym(r), None), Pair(13, 0, 0, None, sym(c)), Pair(13, 1, 1, sym(9), sym(17))]
    return Superblock(np.array([r, 9]), np.array([c, 17]), rng.standard_normal((batch, 14)), pairs)


@pytest.mark.parametrize("prec", ["bf16x3", "tf32"])
@pytest.mark.parametrize("r,c,batch", [(5, 31, 1), (31, 33, 1), (33, 48, 2), (40, 64, 1), (65, 96, 1), (120, 128, 2),
                                       (128, 130, 1), (300, 257, 1), (257, 300, 1), (24, 72, 16)])
def test_widths(r, c, batch, prec):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_0902_3185_gb300.binding import GpuSuperblock
    sb = build(r, c, batch)
    asb = Superblock(sb.r, sb.c, np.abs(sb.coeffs),
                     [Pair(p.term, p.s_out, p.s_in, None if p.A is None else np.abs(p.A),
                           None if p.B is None else np.abs(p.B)) for p in sb.pairs])
    X = np.stack([seeded_normal(b, sb.dim) for b in range(batch)])
    y = GpuSuperblock(sb).apply_H(torch.from_numpy(X).cuda(), prec=prec).cpu().numpy()
    for b in range(batch):
        bound = osb.apply_H(asb, np.abs(X[b]), b)
        assert np.all(np.abs(y[b] - osb.apply_H(sb, X[b], b)) <= GAMMA[prec] * bound)
