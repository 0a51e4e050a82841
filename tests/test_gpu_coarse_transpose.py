"""The stored transpose of the coarsest level's inverse: with one level and a dense inverse the
cycle of the adjoint is exact, so one FGMRES iteration in FP64 solves J^T lambda = rhs to the
rounding of the inverse: n eps cond(J) = 450 * 1.1e-16 * 4e6 = 2e-7 of the right-hand side.
135 to 450 unknowns, all inverted on the host."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_1508_04596_gb300 import synth  # noqa: E402


@pytest.mark.parametrize("dims", [(2, 2, 2), (3, 3, 3), (5, 3, 2), (4, 4, 2), (4, 2, 5)])
def test_transposed_inverse(dims):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1508_04596_gb300 import nc
    gp = nc.Problem(nc.make_params(*dims, 1.0 / max(dims), 1e3, 0.71, **synth.MATERIAL),
                    nc.cavity_bcs(nc.PATCH_FLUX, 1.0, (0.0, 1.0, 0.0, 1.0)))
    rng = np.random.default_rng(sum(dims))
    dev = lambda a: torch.tensor(a, dtype=torch.float64, device="cuda")  # noqa: E731
    gam = dev(rng.uniform(0.2, 1.0, gp.E))
    x = gp.impose_dirichlet(dev(0.1 * rng.standard_normal(gp.ndof)))
    rhs = gp.jtvp(x, gam, dev(rng.standard_normal(gp.ndof)))
    lam, info = gp.adjoint_solve(x, gam, rhs, opts=nc.default_opts(mixed=0, mg_levels=1, max_lin=1, max_newton=1,
                                                                   rtol_adjoint=1e-30), check=False)
    assert ((gp.jtvp(x, gam, lam) - rhs).norm() <= 2e-7 * rhs.norm()).item()
