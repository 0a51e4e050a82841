"""nc_filter at the edges of its node tiles and plane marches (node counts one below, at
and one above a tile, one element across, many planes), for radii from 0 (the mass matrix alone)
to 6 elements, against the oracle's sparse direct solve.

Tolerance 1e-12: CG stops at a relative residual of 1e-13 and the Jacobi-scaled system has a
condition number below 10 for these radii in the directions that matter (mass-dominated); the
mean over the nodes averages the rest.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from oracle import filter as F  # noqa: E402
from oracle import grid as G  # noqa: E402


@pytest.mark.parametrize("nx,ny,nz", [(30, 6, 3), (31, 7, 4), (32, 8, 2), (33, 15, 1), (63, 1, 17),
                                      (1, 16, 40), (2, 1, 90), (65, 9, 9)])
@pytest.mark.parametrize("rad", [0.0, 2.5, 6.0])
def test_filter_tiles(nx, ny, nz, rad):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1508_04596_gb300 import nc
    h = 1.0 / nx
    g = G.Grid(nx, ny, nz, h)
    gp = nc.Problem(nc.make_params(nx, ny, nz, h, 1e3, 0.71), nc.cavity_bcs())
    rho = np.random.default_rng(nx + 7 * ny + 11 * nz).uniform(0.0, 1.0, g.E)
    got = gp.filter(torch.tensor(rho, dtype=torch.float64, device="cuda"), radius=rad * h)
    ref = F.apply_filter(g, rho, rad * h)
    assert np.linalg.norm(got.cpu().numpy() - ref) <= 1e-12 * np.linalg.norm(ref)
