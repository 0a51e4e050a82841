"""The partitions that a grid gets, restated here so that the sizes reach the kernels they are
meant for: runs of 5 and 6 rows of the marching kernels in either precision, single rows with a
warp per chunk in FP32, and the largest grids that the one-block smoother takes at one, six and
eight steps.

Tolerances: products as in test_gpu_march.py (FP64 1e-12, FP32 2e-4, relative L2); the smoother's
cycle 1e-2 against the FP64 cycle as in test_gpu_block_smoother.py."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_1508_04596_gb300 import synth  # noqa: E402
from tests.helpers import oracle_problem, random_bc_state, sampled_rows  # noqa: E402

TOL = {torch.float64: 1e-12, torch.float32: 2e-4}


@pytest.fixture(scope="module")
def nc():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1508_04596_gb300 import nc as ncmod
    return ncmod


def march_rows(dims, fp64):
    """Rows of a run, and whether four warps share a chunk (the rule of march_plan)."""
    nx, ny, nz = dims
    slots, extra = (608, 0.05) if fp64 else (8 * 152, 0.6)
    stride = 32 if 32 % (nx + 1) == 0 else 31
    up = lambda a, b: -(-a // b)  # noqa: E731
    faces, room = (nx + 1) * nz, 40 * 32 * up(nx * ny * nz, 32)
    single = up(faces * ny, stride)

    def cost(rc, warps):
        turns = up(warps, slots)
        return (rc + extra) * (1.12 if fp64 and turns == 1 else turns)

    best, least = 1, cost(1, single)
    for rc in range(2, min(24, ny) + 1):
        warps = up(faces, stride) * up(ny, rc)
        if cost(rc, warps) < least and warps * (rc + 1) * 320 <= room:
            best, least = rc, cost(rc, warps)
    return best, best == 1 and single <= (304 if fp64 else 750)


@pytest.mark.parametrize("dims,dt,rows", [((20, 37, 220), torch.float64, 5), ((40, 23, 220), torch.float64, 6),
                                          ((20, 23, 300), torch.float32, 5), ((20, 26, 300), torch.float32, 6),
                                          ((29, 28, 28), torch.float32, 1)])
def test_runs_of_rows(nc, dims, dt, rows):
    assert march_rows(dims, dt == torch.float64) == (rows, False)
    nx, ny, nz = dims
    prob, _ = oracle_problem(nx, ny, nz, 1.0 / nx, 1e4, 0.71, patch_mode="flux")
    p = nc.make_params(nx, ny, nz, 1.0 / nx, 1e4, 0.71, alpha_max=1e4, q_alpha=1.0, q_f=1.0, Ck=0.1)
    gp = nc.Problem(p, nc.cavity_bcs(nc.PATCH_FLUX, 1.0))
    rng = np.random.default_rng(rows)
    gam, x, v = rng.uniform(0, 1, gp.E), random_bc_state(prob, 6), rng.standard_normal((5, gp.Nn))
    vi = np.where(prob.dmask, 0.0, v)
    pick = list(rng.integers(0, gp.Nn, 20))
    for j in (1, rows - 1, rows, rows + 1, 2 * rows, ny - 2, ny - 1):
        for face in (31, 62, 31 * 20, 31 * 77, 31 * 150 + 30):  # chunk ends
            i, k = face % (nx + 1), face // (nx + 1)
            if 0 < i < nx and 0 < k < nz:
                pick.append(i + (nx + 1) * (j + (ny + 1) * k))
    nodes = np.unique(pick)
    dev = lambda a: torch.tensor(np.ascontiguousarray(a).ravel(), dtype=dt, device="cuda")  # noqa: E731
    X, Ga, V = dev(x), dev(gam), dev(v)
    outs = [("jvp", gp.jvp(X, Ga, V)), ("jtvp", gp.jtvp(X, Ga, V))]
    if dt == torch.float64:
        gp.linearize(X, Ga)
        outs += [("jvp", gp.jvp_lin(V)), ("jtvp", gp.jtvp_lin(V))]
    for kind, got in outs:
        ref = sampled_rows(prob.g, prob.prm, x, gam, vi, nodes, kind)
        ref = np.where(prob.dmask[:, nodes], v[:, nodes], ref)
        got = got.double().cpu().numpy().reshape(5, -1)[:, nodes]
        assert np.linalg.norm(got - ref) <= TOL[dt] * np.linalg.norm(ref), kind


def block_takes(dims, its):
    """Whether the one-block smoother takes a level (the rule of smooth_block)."""
    E, Nn = np.prod(dims), np.prod([n + 1 for n in dims])
    return its <= 8 and E <= 512 and 4 * ((its + 4) * 5 * Nn + 40 * E) <= 227 * 1024 - 1168


@pytest.mark.parametrize("dims,its", [((16, 16, 2), 1), ((32, 16, 1), 1), ((8, 8, 8), 6), ((13, 12, 3), 6),
                                      ((8, 8, 7), 8), ((16, 16, 1), 8), ((1, 3, 70), 8),
                                      ((8, 5, 12), 7), ((1, 262, 1), 5)])
def test_block_smoother_largest_grids(nc, dims, its):
    assert block_takes(dims, its)
    nx, ny, nz = dims
    gp = nc.Problem(nc.make_params(nx, ny, nz, 1.0 / nx, 1e3, 0.71, **synth.MATERIAL),
                    nc.cavity_bcs(nc.PATCH_FLUX, 1.0, (0.0, 1.0, 0.0, 1.0)))
    rng = np.random.default_rng(nx + nz + its)
    dev = lambda a: torch.tensor(a, dtype=torch.float64, device="cuda")  # noqa: E731
    gam = dev(rng.uniform(0.2, 1.0, gp.E))
    x = gp.impose_dirichlet(dev(synth.random_state(nx, ny, nz, 3, (0.5, 0.5, 0.5, 5.0, 1.0)).ravel()))
    d = dev(rng.standard_normal(gp.ndof))
    a, b = (gp.adjoint_solve(x, gam, d, check=False, opts=nc.default_opts(
        mixed=m, mg_levels=1, smooth_its=its, coarse_its=its, max_lin=1, max_newton=1, rtol_adjoint=1e-30,
        rtol_lin=1e-30))[0] for m in (0, 1))
    assert torch.isfinite(b).all() and a.norm() > 0 and (a - b).norm() <= 1e-2 * a.norm()
