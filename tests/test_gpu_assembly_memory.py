"""The FP32 assembly of a context that finds no room for its linearisation store: the 40 element
products with unit directions, against the matrix-free products (tolerance 1e-5 relative L2, as
test_gpu_assembly_rows.py), and bit by bit the same once there is room again."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims", [(5, 7, 6), (1, 4, 9), (33, 2, 3)])
def test_fp32_assembly_without_its_store(dims):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1508_04596_gb300 import nc
    gp = nc.Problem(nc.make_params(*dims, 1.0 / dims[0], 1e4, 0.71), nc.quarter_bcs(*dims))
    rng = np.random.default_rng(sum(dims))
    dev = lambda a: torch.tensor(a, dtype=torch.float32, device="cuda")  # noqa: E731
    x = gp.impose_dirichlet(dev(rng.standard_normal(gp.ndof)))
    gam, v = dev(rng.uniform(0, 1, gp.E)), dev(rng.standard_normal(gp.ndof))
    torch.cuda.empty_cache()
    hold = torch.empty(torch.cuda.mem_get_info()[0] - (6 << 30), dtype=torch.uint8, device="cuda")
    try:
        S = gp.assemble(x, gam)
    finally:
        del hold
        torch.cuda.empty_cache()
    for tr, f in ((False, gp.jvp), (True, gp.jtvp)):
        ref = f(x, gam, v).double()
        assert (gp.stencil_apply(S, v, transpose=tr).double() - ref).norm() <= 1e-5 * ref.norm()
    assert torch.equal(S, gp.assemble(x, gam))
