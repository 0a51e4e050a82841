"""The marching element kernels at the edges of their partition, against the oracle: chunks of 31
and 32 faces (element counts across of 1, 2, 3, 7, 30 to 33, 62), single rows and runs of several
rows with a partial last run, one element in a direction; and non-finite values, which must
reach the rows of their own elements and no others.

Tolerances as in the parity tests: FP64 1e-12 (relative L2; about 10^3 roundings per row), FP32
2e-4 (inputs rounded to 6e-8, up to two orders of cancellation).
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from tests.helpers import oracle_problem, random_bc_state, sampled_rows  # noqa: E402

TOL = {torch.float64: 1e-12, torch.float32: 2e-4}


@pytest.fixture(scope="module")
def nc():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1508_04596_gb300 import nc as ncmod
    return ncmod


def rel(a, b):
    return float(np.linalg.norm(a - b) / np.linalg.norm(b))


def gpu_problem(nc, nx, ny, nz, patch="flux"):
    p = nc.make_params(nx, ny, nz, 1.0 / nx, 1e4, 0.71, alpha_max=1e4, q_alpha=1.0, q_f=1.0, Ck=0.1)
    return nc.Problem(p, nc.cavity_bcs(nc.PATCH_FLUX if patch == "flux" else nc.PATCH_DIRICHLET, 1.0))


def dev(a, dt=torch.float64):
    return torch.tensor(np.ascontiguousarray(a).ravel(), dtype=dt, device="cuda")


@pytest.mark.parametrize("dims", [(1, 1, 5), (1, 9, 2), (2, 3, 11), (3, 4, 9), (7, 5, 4), (30, 2, 3),
                                  (31, 3, 2), (32, 2, 2), (33, 1, 3), (62, 2, 1), (15, 1, 8)])
def test_small_grids(nc, dims):
    prob, _ = oracle_problem(*dims, 1.0 / dims[0], 1e4, 0.71, patch_mode="flux")
    gp = gpu_problem(nc, *dims)
    rng = np.random.default_rng(sum(dims))
    gam = rng.uniform(0, 1, gp.E)
    x = random_bc_state(prob, 5)
    v = rng.standard_normal(gp.ndof)
    J = prob.jacobian(x, gam)
    R = prob.residual(x, gam).ravel()
    for dt in (torch.float64, torch.float32):
        X, Ga, V = dev(x, dt), dev(gam, dt), dev(v, dt)
        for got, ref in ((gp.residual(X, Ga), R), (gp.jvp(X, Ga, V), J @ v), (gp.jtvp(X, Ga, V), J.T @ v)):
            assert rel(got.double().cpu().numpy(), ref) <= TOL[dt], (dims, dt)
    gp.linearize(dev(x), dev(gam))
    assert rel(gp.jvp_lin(dev(v)).cpu().numpy(), J @ v) <= 1e-12
    assert rel(gp.jtvp_lin(dev(v)).cpu().numpy(), J.T @ v) <= 1e-12


# runs of several rows (5 and 6 here), the last one shorter; single rows, a warp per chunk (the
# smaller grids of this file share a chunk between four warps)
@pytest.mark.parametrize("dims,runs", [((40, 19, 220), 5), ((20, 27, 300), 6),
                                       ((32, 30, 31), 1), ((24, 24, 24), 1)])
@pytest.mark.parametrize("dt", [torch.float64, torch.float32])
def test_runs_of_rows(nc, dims, runs, dt):
    nx, ny, nz = dims
    prob, _ = oracle_problem(nx, ny, nz, 1.0 / nx, 1e4, 0.71, patch_mode="flux")
    g, prm = prob.g, prob.prm
    gp = gpu_problem(nc, nx, ny, nz)
    rng = np.random.default_rng(7)
    gam = rng.uniform(0, 1, gp.E)
    x = random_bc_state(prob, 6)
    v = rng.standard_normal((5, gp.Nn))
    vi = np.where(prob.dmask, 0.0, v)
    pick = []
    for j in (1, runs - 1, runs, runs + 1, 2 * runs, ny - 2, ny - 1):
        for face in (31, 62, 31 * 20, 31 * 40, 31 * 77, 31 * 150 + 30):  # chunk ends
            i, k = face % (nx + 1), face // (nx + 1)
            if 0 < i < nx and 0 < k < nz:
                pick.append(i + (nx + 1) * (j + (ny + 1) * k))
    nodes = np.unique(np.array(pick + list(rng.integers(0, gp.Nn, 20))))
    X, Ga, V = dev(x, dt), dev(gam, dt), dev(v, dt)
    outs = [("jvp", gp.jvp(X, Ga, V)), ("jtvp", gp.jtvp(X, Ga, V))]
    if dt == torch.float64:
        gp.linearize(X, Ga)
        outs += [("jvp", gp.jvp_lin(V)), ("jtvp", gp.jtvp_lin(V))]
    for kind, got in outs:
        ref = sampled_rows(g, prm, x, gam, vi, nodes, kind)
        ref = np.where(prob.dmask[:, nodes], v[:, nodes], ref)
        assert rel(got.double().cpu().numpy().reshape(5, -1)[:, nodes], ref) <= TOL[dt], kind


def touched(nx, ny, nz, n):
    """Nodes of the elements around node n."""
    i, j, k = n % (nx + 1), (n // (nx + 1)) % (ny + 1), n // ((nx + 1) * (ny + 1))
    m = np.zeros((nz + 1, ny + 1, nx + 1), bool)
    m[max(k - 1, 0):k + 2, max(j - 1, 0):j + 2, max(i - 1, 0):i + 2] = True
    return m.ravel()


@pytest.mark.parametrize("dims", [(31, 4, 5), (6, 5, 7), (1, 3, 20)])
@pytest.mark.parametrize("dt", [torch.float64, torch.float32])
def test_non_finite_values_stay_local(nc, dims, dt):
    """A NaN at one node (in x, or in v) leaves every row outside its elements finite and
    equal to the result without it."""
    nx, ny, nz = dims
    prob, _ = oracle_problem(nx, ny, nz, 1.0 / nx, 1e4, 0.71)
    gp = gpu_problem(nc, nx, ny, nz, "dirichlet")
    rng = np.random.default_rng(3)
    gam = dev(rng.uniform(0, 1, gp.E), dt)
    x, v = dev(random_bc_state(prob, 8), dt), dev(rng.standard_normal(gp.ndof), dt)
    sy = (nx + 1) * (ny + 1)
    for n in (nx + (nx + 1) * 1 + sy * 1, 0 + (nx + 1) * 2 + sy * 2, nx // 2 + (nx + 1) + sy * 3):
        m = touched(nx, ny, nz, n)
        for f in range(5):
            for which in ("x", "v"):
                a, b = x.clone(), v.clone()
                (a if which == "x" else b)[f * gp.Nn + n] = float("nan")
                for op in (gp.jvp, gp.jtvp):
                    ref = op(x, gam, v).cpu().numpy().reshape(5, -1)[:, ~m]
                    got = op(a, gam, b).cpu().numpy().reshape(5, -1)[:, ~m]
                    assert np.array_equal(got, ref), (n, f, which)
                if which == "x":
                    ref = gp.residual(x, gam).cpu().numpy().reshape(5, -1)[:, ~m]
                    got = gp.residual(a, gam).cpu().numpy().reshape(5, -1)[:, ~m]
                    assert np.array_equal(got, ref), (n, f)
