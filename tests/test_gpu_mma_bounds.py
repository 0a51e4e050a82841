"""nc_mma_update beyond the ordinary: variables outside the box by more than the move limit,
whose two limits cross (the upper one holds).  Against the oracle; tolerance 1e-10 as in
test_gpu_design_update.py (a bracket a few units in the last place wide, sums of up to 3e3
terms, a relative slope of the constraint below 100)."""
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


def update(nc, x, df0, f1, df1, it=0):
    gp = nc.Problem(nc.make_params(2, 2, 2, 0.5, 1e3, 0.71), nc.cavity_bcs())
    dev = lambda t: torch.tensor(np.asarray(t, dtype=float), dtype=torch.float64, device="cuda")  # noqa: E731
    s = [dev(x) for _ in range(5)]
    lam, chg = gp.mma_update(it, *s, dev(df0), f1, dev(df1))
    return lam, chg, s[0].cpu().numpy()


@pytest.mark.parametrize("n", [300, 3000])
@pytest.mark.parametrize("side", ["above", "below"])
@pytest.mark.parametrize("sign", [1.0, -1.0])
def test_variables_outside_the_box(nc, n, side, sign):
    from oracle import mma as M
    rng = np.random.default_rng(n)
    x = rng.uniform(0.1, 0.9, n)
    out = rng.uniform(size=n) < 0.1
    x[out] = rng.uniform(1.25, 1.4, out.sum()) if side == "above" else rng.uniform(-0.4, -0.25, out.sum())
    df0 = sign * rng.uniform(0.5, 1.5, n) / n
    df1 = -sign * rng.uniform(0.5, 1.5, n) / n
    # the constraint value whose multiplier is near 1
    low, upp = x - 0.5, x + 0.5
    alpha, beta = M.bounds(x, low, upp, 0.0, 1.0, 0.2)
    assert (alpha[out] > beta[out]).all()
    p0, q0 = M.approx_coefficients(x, low, upp, df0, 1.0)
    p1, q1 = M.approx_coefficients(x, low, upp, df1, 1.0)
    y = M.y_of_lambda(1.0, low, upp, alpha, beta, p0, q0, p1, q1)
    f1 = -M.approx_value(0.0, x, y, low, upp, p1, q1)
    yo, _, _, lo = M.mma_step(0, x, x, x, x, x, f1, df0, df1)
    lam, chg, X = update(nc, x, df0, f1, df1)
    assert 0.9 < lo < 1.1 and lam == pytest.approx(lo, rel=TOL)
    assert np.abs(X - yo).max() <= TOL
    assert chg == pytest.approx(np.abs(yo - x).max(), abs=TOL)


def test_infinite_objective_gradient(nc):
    """An infinite entry of df0 sends its variable to the lower limit, whatever its sign; the
    others solve the subproblem with its (constant) term."""
    from oracle import mma as M
    rng = np.random.default_rng(8)
    n = 700
    x = rng.uniform(0.1, 0.9, n)
    df0, df1 = rng.uniform(0.5, 1.5, n) / n, -rng.uniform(0.5, 1.5, n) / n
    bad = np.arange(n) % 50 == 7
    low, upp = x - 0.5, x + 0.5
    alpha, _ = M.bounds(x, low, upp, 0.0, 1.0, 0.2)
    p1, q1 = M.approx_coefficients(x, low, upp, df1, 1.0)
    t = M.approx_value(0.0, x[bad], alpha[bad], low[bad], upp[bad], p1[bad], q1[bad])
    f = ~bad
    yo, _, _, lo = M.mma_step(0, x[f], x[f], x[f], x[f], x[f], 0.02 + t, df0[f], df1[f])
    assert 1e-3 < lo < 1e3
    df0[bad] = np.where(np.arange(bad.sum()) % 2, np.inf, -np.inf)
    lam, chg, X = update(nc, x, df0, 0.02, df1)
    assert lam == pytest.approx(lo, rel=TOL)
    assert np.abs(X[f] - yo).max() <= TOL and np.abs(X[bad] - alpha[bad]).max() <= 1e-15
    with pytest.raises(Exception):  # the constraint's gradient has no such limit
        update(nc, x, df1, 0.02, df0)


def test_constraint_sum_beyond_the_range(nc):
    """Finite terms whose sum with f1 overflows: violated for every multiplier."""
    lam, chg, X = update(nc, np.full(4, 0.5), np.full(4, 1.0), 1.2e308, np.full(4, -1e308))
    assert lam == 2.0 ** 200 and np.abs(X - 0.3).max() <= 1e-15


@pytest.mark.parametrize("n", [257, 70001, 608 * 256 * 2 + 77])
@pytest.mark.parametrize("share", [1.0, 0.4, 0.003])
def test_same_bits_without_the_workspace(nc, n, share):
    """The update does not depend on how much device memory is free: without the workspace it
    sums the same terms in the same order."""
    rng = np.random.default_rng(n)
    x = rng.uniform(0.1, 0.9, n)
    xo1 = np.clip(x + 0.05 * rng.standard_normal(n), 0, 1)
    xo2 = np.clip(xo1 + 0.05 * rng.standard_normal(n), 0, 1)
    df0, df1 = rng.uniform(0.5, 1.5, n) / n, -rng.uniform(0.5, 1.5, n) / (share * n)
    act = rng.uniform(size=n) < share
    act[n // 3] = True
    dev = lambda t: torch.tensor(t, dtype=torch.float64, device="cuda")  # noqa: E731
    mask = torch.tensor(act.astype(np.uint8), device="cuda")

    def run():
        gp = nc.Problem(nc.make_params(2, 2, 2, 0.5, 1e3, 0.71), nc.cavity_bcs())
        s = [dev(t) for t in (x, xo1, xo2, xo1 - 0.3, xo1 + 0.3)]
        lam, chg = gp.mma_update(4, *s, dev(df0), 0.02, dev(df1), active=mask)
        return [lam, chg] + [t.cpu() for t in s]

    with_ws = run()
    torch.cuda.empty_cache()
    hold = torch.empty(torch.cuda.mem_get_info()[0] - (6 << 30), dtype=torch.uint8, device="cuda")
    try:
        without = run()
    finally:
        del hold
        torch.cuda.empty_cache()
    assert with_ws[:2] == without[:2] and all(torch.equal(a, b) for a, b in zip(with_ws[2:], without[2:]))


@pytest.mark.parametrize("n", [1, 300, 608 * 256 * 3 + 5])
def test_volume_gradient_is_left_on_the_stream(nc, n):
    """The value is there when the call returns, the gradient in stream order; calls one after
    another on different designs do not disturb each other."""
    from oracle import mma as M
    rng = np.random.default_rng(n)
    gp = nc.Problem(nc.make_params(2, 2, 2, 0.5, 1e3, 0.71), nc.cavity_bcs())
    dev = lambda t: torch.tensor(t, dtype=torch.float64, device="cuda")  # noqa: E731
    xs = [rng.uniform(0, 1, n) for _ in range(3)]
    acts = [np.arange(n) % (k + 1) == 0 for k in range(3)]
    masks = [torch.tensor(a.astype(np.uint8), device="cuda") for a in acts]
    gam, grads = [dev(x) for x in xs], [torch.empty(n, dtype=torch.float64, device="cuda") for _ in xs]
    got = [gp.volume(g, m, 0.3, grad=d) for g, m, d in zip(gam, masks, grads)]
    for x, a, g, d in zip(xs, acts, got, grads):
        ref, dref = M.volume_constraint(x, a, 0.3)
        assert g == pytest.approx(ref, rel=1e-12, abs=1e-12)
        assert np.allclose(d.cpu().numpy(), dref, rtol=1e-14, atol=0)
    with pytest.raises(Exception):
        gp.volume(gam[0], torch.zeros_like(masks[0]), 0.3, grad=grads[0])


@pytest.mark.parametrize("n", [1, 300, 70001])
@pytest.mark.parametrize("slack", [0.5, 0.0])
def test_constraint_that_holds_without_a_multiplier(nc, n, slack):
    """The first evaluation ends the search: lambda = 0, the history shifted once."""
    from oracle import mma as M
    rng = np.random.default_rng(n)
    x = rng.uniform(0.1, 0.9, n)
    df0, df1 = -rng.uniform(0.5, 1.5, n) / n, -rng.uniform(0.5, 1.5, n) / n
    yo, _, _, lo = M.mma_step(0, x, x, x, x, x, -slack, df0, df1)
    assert lo == 0.0
    gp = nc.Problem(nc.make_params(2, 2, 2, 0.5, 1e3, 0.71), nc.cavity_bcs())
    dev = lambda t: torch.tensor(t, dtype=torch.float64, device="cuda")  # noqa: E731
    s = [dev(x), dev(x + 1), dev(x + 2), dev(x), dev(x)]
    lam, chg = gp.mma_update(0, *s, dev(df0), -slack, dev(df1))
    assert lam == 0.0 and chg == pytest.approx(np.abs(yo - x).max(), abs=TOL)
    assert np.abs(s[0].cpu().numpy() - yo).max() <= 1e-14
    assert np.array_equal(s[1].cpu().numpy(), x) and np.array_equal(s[2].cpu().numpy(), x + 1)
