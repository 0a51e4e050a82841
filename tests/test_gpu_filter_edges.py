"""nc_filter on fields that need no iteration (zero, not finite) or few (constant), between
ordinary ones: what a call leaves in the context's scratch does not reach the next."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def nc():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1508_04596_gb300 import nc as ncmod
    return ncmod


@pytest.mark.parametrize("n", [(1, 1, 1), (3, 5, 7), (24, 24, 24), (80, 60, 40)])
def test_fields_without_iterations(nc, n):
    h = 1.0 / max(n)
    make = lambda: nc.Problem(nc.make_params(*n, h, 1e3, 0.71), nc.cavity_bcs())  # noqa: E731
    gp = make()
    rho = torch.rand(gp.E, dtype=torch.float64, generator=torch.Generator().manual_seed(5)).cuda()
    want = make().filter(rho, 2.5 * h)
    zero, one, nan = torch.zeros_like(rho), torch.ones_like(rho), rho.clone()
    nan[gp.E // 2] = float("nan")
    inf = rho.clone()
    inf[0] = float("inf")
    for _ in range(2):
        assert torch.equal(gp.filter(zero, 2.5 * h, torch.full_like(rho, 7.0)), zero)
        assert torch.equal(gp.filter(rho, 2.5 * h), want)
        # preserved to the solve's 1e-13, here with a margin for the mean and the residual's norm
        assert float((gp.filter(one, 2.5 * h) - 1).abs().max()) <= 1e-11
        for bad in (nan, inf):
            out = torch.full_like(rho, 7.0)
            with pytest.raises(nc.NCError):
                gp.filter(bad, 2.5 * h, out)
            assert float(out.min()) == float(out.max()) == 7.0
        own = rho.clone()
        assert torch.equal(gp.filter(own, 2.5 * h, own), want)  # in place
        assert torch.equal(gp.filter(rho, 2.5 * h), want)
