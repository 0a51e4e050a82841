"""The one-block FP32 smoother of small levels against the FP64 cycle's kernels.

A linear solve of one iteration gives the preconditioned residual up to a factor that both
precisions choose alike; the mixed solve's cycle smooths in one kernel on these grids, the FP64 one
by the general kernels.  Tolerance 1e-2: twelve FP32 products a level, each within 2e-4 of FP64, and
the small least-squares problems amplify by the conditioning of their six or eight columns (a few).
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_1508_04596_gb300 import synth  # noqa: E402


# one level without dense inverse (ragged; the largest; one layer), then two and three levels
@pytest.mark.parametrize("dims,levels", [((9, 7, 5), 1), ((8, 8, 8), 1), ((32, 16, 1), 1), ((1, 3, 70), 1),
                                         ((8, 8, 8), 2), ((6, 6, 6), 2), ((16, 8, 8), 3)])
@pytest.mark.parametrize("its", [1, 6, 8])
def test_one_cycle_matches_fp64(dims, levels, its):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1508_04596_gb300 import nc
    nx, ny, nz = dims
    gp = nc.Problem(nc.make_params(nx, ny, nz, 1.0 / nx, 1e3, 0.71, **synth.MATERIAL),
                    nc.cavity_bcs(nc.PATCH_FLUX, 1.0, (0.0, 1.0, 0.0, 1.0)))
    rng = np.random.default_rng(nx + nz + its)
    dev = lambda a: torch.tensor(a, dtype=torch.float64, device="cuda")  # noqa: E731
    gam = dev(rng.uniform(0.2, 1.0, gp.E))
    gp.set_source(dev(rng.uniform(0, 1, gp.E)))
    x = gp.impose_dirichlet(dev(synth.random_state(nx, ny, nz, 3, (0.5, 0.5, 0.5, 5.0, 1.0)).ravel()))
    d = dev(rng.standard_normal(gp.ndof))
    adj, new = [], []
    for mixed in (0, 1):
        o = nc.default_opts(mixed=mixed, mg_levels=levels, smooth_its=its, coarse_its=its, max_lin=1,
                            max_newton=1, ramp_steps=0, rtol_adjoint=1e-30, rtol_lin=1e-30)
        adj.append(gp.adjoint_solve(x, gam, d, opts=o, check=False)[0])
        xn = x.clone()
        gp.newton_solve(gam, xn, o, check=False)
        new.append((xn - x) / (xn - x).norm())  # the line search may scale the step
    for a, b in (adj, new):
        assert torch.isfinite(b).all() and a.norm() > 0
        assert (a - b).norm() <= 1e-2 * a.norm()
