"""Contexts of their own on threads of their own: mixed solves whose coarse levels are smoothed
by one block each (levels of 8^3, 4^3, 4x4x8 and 8x4x4 elements, with different amounts of
shared memory) run at the same time on two streams.  A context's results do not depend on what
other contexts do, and a solve is deterministic, so each equals the same solve alone, bit by
bit."""
import threading

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

GRIDS = [(16, 16, 16), (8, 8, 16), (16, 8, 8)]
REPEATS = 6


@pytest.fixture(scope="module")
def nc():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1508_04596_gb300 import nc as ncmod
    return ncmod


def solve(nc, gp, gam):
    x = torch.zeros(gp.ndof, dtype=torch.float64, device="cuda")
    gp.newton_solve(gam, x, nc.default_opts(max_newton=3, max_lin=20), check=False)
    _, g = gp.objective(x)
    lam, _ = gp.adjoint_solve(x, gam, g, opts=nc.default_opts(max_newton=2, max_lin=20), check=False)
    return x, lam


@pytest.mark.parametrize("pair", [(0, 1), (0, 2), (1, 2)])
def test_solves_on_two_threads(nc, pair):
    probs, gams, alone = [], [], []
    for t, i in enumerate(pair):
        n = GRIDS[i]
        probs.append(nc.Problem(nc.make_params(*n, 1.0 / max(n), 1e3, 0.71), nc.cavity_bcs(nc.PATCH_FLUX, 1.0)))
        g = torch.Generator(device="cuda").manual_seed(40 + t)
        gams.append(0.2 + 0.6 * torch.rand(probs[-1].E, dtype=torch.float64, device="cuda", generator=g))
        alone.append(solve(nc, probs[-1], gams[-1]))
    torch.cuda.synchronize()
    failed = []

    def work(t):
        try:
            with torch.cuda.stream(torch.cuda.Stream()):
                for _ in range(REPEATS):
                    x, lam = solve(nc, probs[t], gams[t])
                    torch.cuda.current_stream().synchronize()
                    if not (torch.equal(x, alone[t][0]) and torch.equal(lam, alone[t][1])):
                        failed.append(t)
        except Exception as e:  # noqa: BLE001
            failed.append(e)

    threads = [threading.Thread(target=work, args=(t,)) for t in range(2)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not failed
