"""A matrix gives the same eigenpairs, bit for bit, whether the list it is in
sends it to a thread-block cluster of 16 (alone), of 8 or to one block (among
many)."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [33, 48, 64, 65, 79, 110, 111, 130, 207])
def test_alone_and_among_many(n):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_0902_3185_gb300 import binding
    g = torch.Generator("cuda").manual_seed(n)
    m = torch.randn(150 if n <= 110 else 21, n, n, dtype=torch.float64, device="cuda", generator=g)
    mats = [x.contiguous() for x in m + m.transpose(1, 2)]
    many = binding.sym_eig_batched(mats)
    for i in (0, len(mats) // 2, len(mats) - 1):
        w, v = binding.sym_eig_batched([mats[i]])[0]
        assert torch.equal(w, many[i][0]) and torch.equal(v, many[i][1])
