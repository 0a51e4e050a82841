"""FP32 sums of vectors a little longer than one block's 2,048 elements: blocks' sums meet in
FP64.  Two products in different blocks, 2^24 and 1, add up to 2^24 + 1, which FP32 cannot
hold.  Exact: the first pass's coefficient is rounded to 2^24 for the update, which
leaves 1 - 2^24, so the second pass returns -(2^24 - 1) and the coefficients add up to 2 (to 1
if the 1 were lost in the first sum)."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [2049, 3001, 4096])
@pytest.mark.parametrize("near,far", [(0, 1024), (0, 1536), (3, 2047)])
def test_fp32_dots_of_two_blocks(n, near, far):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1508_04596_gb300 import nc
    gp = nc.Problem(nc.make_params(2, 2, 2, 0.5, 1e3, 0.71), nc.cavity_bcs())
    V, w = (torch.zeros(n, dtype=torch.float32, device="cuda") for _ in range(2))
    V[near] = V[far] = 1.0
    w[near], w[far] = 2.0 ** 24, 1.0
    assert gp.arnoldi_orth(V, w, 1, n)[0] == 2.0
