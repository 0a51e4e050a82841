"""Prolongation of a state on grids on both sides of the size from which a thread takes a whole
node, against the three 1-D interpolations one after another (at most eight halves and sums a value:
1e-14 relative)."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims", [(4, 4, 8), (64, 66, 70), (70, 66, 70)])
def test_prolong_matches_interpolation(dims):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1508_04596_gb300 import nc
    gp = nc.Problem(nc.make_params(*dims, 1.0 / dims[0], 1e3, 0.71), nc.cavity_bcs())
    nx, ny, nz = dims
    g = torch.Generator(device="cuda").manual_seed(nx)
    c = torch.randn(5, nz // 2 + 1, ny // 2 + 1, nx // 2 + 1, generator=g, dtype=torch.float64, device="cuda")
    f = c
    for ax in (1, 2, 3):
        n = f.shape[ax]
        mid = 0.5 * (f.narrow(ax, 0, n - 1) + f.narrow(ax, 1, n - 1))
        shape = list(f.shape)
        shape[ax] = 2 * n - 1
        up = torch.empty(shape, dtype=f.dtype, device=f.device)
        idx = torch.arange(2 * n - 1, device=f.device)
        up.index_copy_(ax, idx[::2], f)
        up.index_copy_(ax, idx[1::2], mid)
        f = up
    ref = gp.impose_dirichlet(f.reshape(-1).clone())
    assert (gp.prolong(c.reshape(-1)) - ref).abs().max() <= 1e-14 * c.abs().max()
