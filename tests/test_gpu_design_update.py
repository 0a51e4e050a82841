"""nc_mma_update's device-side multiplier search and compacted workspace, and the volume
reduction, against the oracle at the sizes where their partition changes: one variable, one
tile of 256 more or less, the largest grid of one tile per block (608 tiles) and one variable
beyond it; multipliers from 1e-6 to 1e6; no active mask, a sparse one and a single active
variable; and with the workspace refused (little device memory left).

Tolerance 1e-10: the iterate and multiplier come from a bracket a few units in the last place
wide; sums of up to 2e5 terms reorder at about 1e-14 and the multiplier amplifies that by the
relative slope of the constraint (below 100 here).
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

TOL = 1e-10


@pytest.fixture(scope="module")
def nc():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1508_04596_gb300 import nc as ncmod
    return ncmod


def problem(nc):
    return nc.Problem(nc.make_params(2, 2, 2, 0.5, 1e3, 0.71), nc.cavity_bcs())


def check(nc, gp, n, scale, mask, it, seed):
    from oracle import mma as M
    rng = np.random.default_rng(seed)
    x = rng.uniform(0.1, 0.9, n)
    xo1 = np.clip(x + 0.05 * rng.standard_normal(n), 0, 1)
    xo2 = np.clip(xo1 + 0.05 * rng.standard_normal(n), 0, 1)
    low, upp = xo1 - 0.3, xo1 + 0.3
    df0 = scale * rng.uniform(0.5, 1.5, n) / n
    df1 = -rng.uniform(0.5, 1.5, n) / n
    f1 = 0.02
    a = {"all": np.ones(n, bool), "some": rng.uniform(size=n) < 0.3,
         "one": np.arange(n) == n // 2}[mask]
    if mask == "some" and not a.any():
        a[0] = True
    if mask == "one":  # the one variable must be able to satisfy the constraint
        df1 = df1 * n
    dev = lambda t: torch.tensor(t, dtype=torch.float64, device="cuda")  # noqa: E731
    act = None if mask == "all" else torch.tensor(a.astype(np.uint8), device="cuda")
    g_o, dg_o = M.volume_constraint(x, a, 0.3)
    dg = torch.empty(n, dtype=torch.float64, device="cuda")
    assert gp.volume(dev(x), act, 0.3, grad=dg) == pytest.approx(g_o, rel=1e-12, abs=1e-12)
    assert np.allclose(dg.cpu().numpy(), dg_o, rtol=1e-14, atol=0)
    yo, Lo, Uo, lo = M.mma_step(it, x[a], xo1[a], xo2[a], low[a], upp[a], f1, df0[a], df1[a])
    X, X1, X2, L, U = (dev(t) for t in (x, xo1, xo2, low, upp))
    lam, chg = gp.mma_update(it, X, X1, X2, L, U, dev(df0), f1, dev(df1), active=act)
    X, X1, X2, L, U = (t.cpu().numpy() for t in (X, X1, X2, L, U))
    assert lam == pytest.approx(lo, rel=TOL)
    assert np.abs(X[a] - yo).max() <= TOL and np.array_equal(X[~a], x[~a])
    assert np.array_equal(X1, x) and np.array_equal(X2, xo1)
    assert np.abs(L[a] - Lo).max() <= 1e-14 and np.abs(U[a] - Uo).max() <= 1e-14
    assert np.array_equal(L[~a], low[~a]) and np.array_equal(U[~a], upp[~a])
    assert chg == pytest.approx(np.abs(yo - x[a]).max(), abs=TOL)


@pytest.mark.parametrize("n", [1, 255, 256, 257, 4096, 608 * 256, 608 * 256 + 1])
@pytest.mark.parametrize("mask", ["all", "some", "one"])
def test_mma_partition_edges(nc, n, mask):
    check(nc, problem(nc), n, 1.0, mask, 0 if n % 2 else 4, n)


@pytest.mark.parametrize("scale", [1e-6, 1e-2, 1e2, 1e6])
def test_mma_multiplier_range(nc, scale):
    check(nc, problem(nc), 3000, scale, "some", 3, 17)


def test_mma_without_workspace(nc):
    gp = problem(nc)
    torch.cuda.empty_cache()
    free = torch.cuda.mem_get_info()[0]
    hold = torch.empty(free - (6 << 30), dtype=torch.uint8, device="cuda")
    try:
        check(nc, gp, 70001, 1.0, "some", 4, 3)
    finally:
        del hold
        torch.cuda.empty_cache()
