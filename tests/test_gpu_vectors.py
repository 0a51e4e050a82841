"""The multi-dot behind nc_arnoldi_orth at every column count of its passes (one to seventeen) and
at lengths around its packets and blocks, aligned and unaligned columns, against the oracle's
two-pass Gram-Schmidt.

Tolerance as in the parity tests: 1e-12 in FP64, 1e-5 in FP32 (relative to the coefficient vector
and the unit vector; sums of up to 7e5 products in blocked order).
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from oracle import solve as S  # noqa: E402


@pytest.mark.parametrize("dt,tol", [(torch.float64, 1e-12), (torch.float32, 1e-5)])
@pytest.mark.parametrize("n,ld_pad,offset", [(7, 57, 0), (1023, 1, 0), (4096, 0, 1), (700001, 63, 0)])
def test_gram_schmidt_column_counts(dt, tol, n, ld_pad, offset):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1508_04596_gb300 import nc
    gp = nc.Problem(nc.make_params(2, 2, 2, 0.5, 1e3, 0.71), nc.cavity_bcs())
    ld = n + ld_pad
    rng = np.random.default_rng(n)
    kmax = min(17, n - 1)
    Q = np.linalg.qr(rng.standard_normal((n, kmax)))[0].T
    w0 = rng.standard_normal(n)
    for k in range(1, kmax + 1):
        buf = torch.zeros(offset + kmax * ld, dtype=dt, device="cuda")
        V = buf[offset:]
        V.view(kmax, ld)[:, :n] = torch.tensor(Q, dtype=dt, device="cuda")
        wb = torch.zeros(offset + n, dtype=dt, device="cuda")
        w = wb[offset:]
        w.copy_(torch.tensor(w0, dtype=dt, device="cuda"))
        Vr = V.view(kmax, ld)[:k, :n].double().cpu().numpy()
        wr = w.double().cpu().numpy()
        h = np.array(gp.arnoldi_orth(V, w, k, ld))
        ho, nuo, qo = S.gram_schmidt_twice(Vr, wr)
        scale = np.sqrt(np.linalg.norm(ho) ** 2 + nuo ** 2)
        assert np.linalg.norm(h[:k] - ho) <= tol * scale, k
        assert abs(h[k] - nuo) <= tol * scale, k
        assert np.linalg.norm(w.double().cpu().numpy() - qo) <= tol * scale / nuo, k
