"""The dense inverse of the coarsest level, on the host (small systems) and on the device, through
a hierarchy of that one level: the V-cycle is then the exact inverse and an FGMRES solve takes
one iteration per linear solve, two at most for the FP32 rounding of the inverse in mixed solves.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_1508_04596_gb300 import synth  # noqa: E402


# 5 (nx+1)(ny+1)(nz+1) unknowns: 320, 400 (host), 500, 560, 750, 1000
@pytest.mark.parametrize("dims", [(3, 3, 3), (3, 3, 4), (3, 4, 4), (3, 3, 6), (4, 4, 5), (7, 4, 4)])
@pytest.mark.parametrize("mixed", [0, 1])
def test_one_level_solves_directly(dims, mixed):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1508_04596_gb300 import nc
    nx, ny, nz = dims
    gp = nc.Problem(nc.make_params(nx, ny, nz, 1.0 / nx, 1e3, 0.71, **synth.MATERIAL),
                    nc.cavity_bcs(nc.PATCH_FLUX, 1.0, (0.0, 1.0, 0.0, 1.0)))
    rng = np.random.default_rng(nx + nz)
    gam = torch.tensor(rng.uniform(0.2, 1.0, gp.E), dtype=torch.float64, device="cuda")
    x = torch.zeros(gp.ndof, dtype=torch.float64, device="cuda")
    opts = nc.default_opts(mixed=mixed, mg_levels=1, rtol_lin=1e-8 if not mixed else 1e-4)
    _, info = gp.newton_solve(gam, x, opts)
    per = 1 if not mixed else 2
    assert info["status"] == "NC_OK" and info["lin_its_total"] <= per * info["newton_its"], info
    phi, dphi = gp.objective(x)
    lam, ainfo = gp.adjoint_solve(x, gam, -dphi, opts=opts)
    assert ainfo["status"] == "NC_OK" and ainfo["lin_its_total"] <= (per + 1) * max(1, ainfo["newton_its"])
    r = gp.jtvp(x, gam, lam) + dphi
    assert (r.norm() <= 1e-9 * dphi.norm()).item()


def test_singular_coarse_operator_is_reported():
    """A design of NaN makes the device elimination find no pivot: an error, no hang."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1508_04596_gb300 import nc
    gp = nc.Problem(nc.make_params(4, 4, 5, 0.25, 1e3, 0.71), nc.cavity_bcs(nc.PATCH_FLUX, 1.0))
    gam = torch.full((gp.E,), float("nan"), dtype=torch.float64, device="cuda")
    x = torch.zeros(gp.ndof, dtype=torch.float64, device="cuda")
    d = torch.ones(gp.ndof, dtype=torch.float64, device="cuda")
    with pytest.raises(nc.NCError) as e:
        gp.adjoint_solve(x, gam, d, opts=nc.default_opts(mixed=0, mg_levels=1))
    assert e.value.status == 4
