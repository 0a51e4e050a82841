"""The stencil assembled from element rows against the matrix-free products, for a tilted
gravity (all three buoyancy columns), a heat source, thin grids and both precisions.

Tolerance: FP64 1e-13 relative L2 (both sides sum about 10^3 products per row in FP64), FP32 1e-5
(the same in FP32; no rounding of inputs in between, both take the same FP32 arrays).
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_1508_04596_gb300 import synth  # noqa: E402


@pytest.mark.parametrize("dims", [(5, 7, 6), (1, 4, 9), (33, 2, 3), (12, 12, 12)])
@pytest.mark.parametrize("g_dir", [(0.3, -0.5, -0.8), (0.0, 0.0, -1.0), (0.0, 0.0, 0.0)])
@pytest.mark.parametrize("dt,tol", [(torch.float64, 1e-13), (torch.float32, 1e-5)])
def test_rows_match_products(dims, g_dir, dt, tol):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1508_04596_gb300 import nc
    nx, ny, nz = dims
    gp = nc.Problem(nc.make_params(nx, ny, nz, 1.0 / nx, 1e4, 0.71, g_dir=g_dir),
                    nc.quarter_bcs(nx, ny, nz))
    rng = np.random.default_rng(nx + ny)
    dev = lambda a: torch.tensor(a.ravel(), dtype=torch.float64, device="cuda")  # noqa: E731
    gp.set_source(dev(rng.uniform(0, 10, gp.E)))
    x = gp.impose_dirichlet(dev(synth.random_state(nx, ny, nz, 3, (0.5, 0.5, 0.5, 50.0, 1.0)))).to(dt)
    gam = dev(rng.uniform(0, 1, gp.E)).to(dt)
    S = gp.assemble(x, gam)
    assert torch.equal(S, gp.assemble(x, gam))
    for seed in range(2):
        v = dev(np.random.default_rng(seed).standard_normal(gp.ndof)).to(dt)
        for tr, f in ((False, gp.jvp), (True, gp.jtvp)):
            ref = f(x, gam, v).double()
            got = gp.stencil_apply(S, v, transpose=tr).double()
            assert (got - ref).norm() <= tol * ref.norm(), tr


def test_first_call_under_capture():
    """An FP32 assembly captured as a context's first one, replayed after an FP64 assembly."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1508_04596_gb300 import nc
    params, bcs = nc.make_params(12, 7, 9, 1.0 / 12, 1e4, 0.71), nc.cavity_bcs()
    gp, other = nc.Problem(params, bcs), nc.Problem(params, bcs)
    rng = np.random.default_rng(5)
    x = torch.tensor(rng.standard_normal(gp.ndof), dtype=torch.float32, device="cuda")
    gam = torch.tensor(rng.uniform(0, 1, gp.E), dtype=torch.float32, device="cuda")
    S = torch.zeros(675 * gp.Nn, dtype=torch.float32, device="cuda")
    other.assemble(x, gam)  # loads the kernels
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        gp.assemble(x, gam, S)
    gp.assemble(x.double(), gam.double())
    x.mul_(0.5)
    g.replay()
    torch.cuda.synchronize()
    assert torch.equal(S, other.assemble(x, gam))
