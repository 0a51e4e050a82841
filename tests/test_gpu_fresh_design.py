"""Element operators whose design (and vectors) the kernel just ahead in the stream has written:
the operators may be launched while that kernel still runs and wait for it themselves.  Every
repetition writes another design and another direction with a kernel and calls the operator at
once; the result equals, bit by bit, that of the same call after a synchronisation.  Grids of the
four-warp and of the marching kernels."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

REPEATS = 8


@pytest.fixture(scope="module")
def nc():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1508_04596_gb300 import nc as ncmod
    return ncmod


@pytest.mark.parametrize("dims", [(8, 8, 8), (40, 33, 37), (96, 96, 96)])
@pytest.mark.parametrize("dtype", ["f64", "f32"])
def test_design_written_by_the_kernel_ahead(nc, dims, dtype):
    dt = torch.float64 if dtype == "f64" else torch.float32
    gp = nc.Problem(nc.make_params(*dims, 1.0 / max(dims), 1e3, 0.71), nc.cavity_bcs(nc.PATCH_FLUX, 1.0))
    gen = torch.Generator(device="cuda").manual_seed(3)
    rand = lambda n: torch.rand(n, dtype=torch.float64, device="cuda", generator=gen)  # noqa: E731
    x = (rand(gp.ndof) - 0.5).to(dt)
    designs, dirs = [rand(gp.E) for _ in range(REPEATS)], [rand(gp.ndof) - 0.5 for _ in range(REPEATS)]
    gam, v, out = torch.zeros(gp.E, dtype=dt, device="cuda"), torch.zeros_like(x), torch.empty_like(x)
    sens, store = torch.empty(gp.E, dtype=dt, device="cuda"), torch.empty_like(x)

    def write(k):  # the design last: its kernel is the one directly ahead
        v.copy_(dirs[k])
        if dtype == "f64":
            gp.design_map(designs[k], lo=0.1, hi=0.9, out=gam)
        else:
            gam.copy_(designs[k])

    def from_store():
        gp.linearize(x, gam)
        return gp.jtvp_lin(v, out=store)

    calls = [lambda: gp.residual(x, gam, out=out), lambda: gp.jvp(x, gam, v, out=out),
             lambda: gp.jtvp(x, gam, v, out=out)]
    if dtype == "f64":
        calls += [lambda: gp.sensitivity(x, gam, v, out=sens), from_store]
    for call in calls:
        want = []
        for k in range(REPEATS):
            write(k)
            torch.cuda.synchronize()
            want.append(call().clone())
        torch.cuda.synchronize()
        got = []
        for k in range(REPEATS):
            write(k)
            got.append(call().clone())
        torch.cuda.synchronize()
        assert all(torch.equal(a, b) for a, b in zip(got, want))
