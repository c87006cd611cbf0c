"""Real-data rows split in registers (real_pair.cuh): every row length that takes
it, with batches of one row, one row short of a tile and one row beyond a tile,
in all four directions against float64; values past the output stay untouched.

Bar: relative L2 error of every row <= 5e-7 * log2(N), the FP32 bound of the
complex transforms (one of length N/2 plus a split of a few roundings)."""
import numpy as np
import pytest
import torch

from paper_1707_07263_gb300 import api

pytestmark = pytest.mark.gpu
GUARD = 4096


def rel(got, ref):
    return np.sqrt((np.abs(got - ref) ** 2).sum(-1) / (np.abs(ref) ** 2).sum(-1)).max()


@pytest.mark.parametrize("extra", [None, -1, 1])
@pytest.mark.parametrize("lg", range(6, 16))
def test_every_direction(lg, extra):
    n, rows = 1 << lg, max(1, 4096 >> (lg - 1))
    batch = 1 if extra is None else max(2, rows + extra)
    m = n // 2
    g = np.random.default_rng(100 * lg + batch)
    x = g.standard_normal((batch, n)).astype(np.float32)
    X = (g.standard_normal((batch, m + 1)) + 1j * g.standard_normal((batch, m + 1))).astype(np.complex64)
    X.imag[:, [0, m]] = np.nan, np.inf   # these do not enter
    Xr = X.astype(np.complex128)
    Xr.imag[:, [0, m]] = 0
    fwd = np.fft.rfft(x.astype(np.float64))
    inv_adj = 2.0 / n * fwd
    inv_adj[:, [0, m]] /= 2
    # the adjoint of rfft: sum over the half spectrum only
    fwd_adj = np.fft.irfft(Xr * np.where((np.arange(m + 1) % m) == 0, 2.0, 1.0), n) * m
    p = api.Plan("r2c", (n,), batch)
    tol = 5e-7 * lg
    for src, dirs in ((x, ((api.FORWARD, fwd), (api.INVERSE | api.ADJOINT, inv_adj))),
                      (X, ((api.INVERSE, np.fft.irfft(Xr, n)), (api.FORWARD | api.ADJOINT, fwd_adj)))):
        a = torch.from_numpy(src).cuda()
        for d, ref in dirs:
            buf = torch.full((batch * ref.shape[1] + GUARD,), 7.0, device="cuda",
                             dtype=torch.complex64 if np.iscomplexobj(ref) else torch.float32)
            p.exec_ptr(a.data_ptr(), buf.data_ptr(), d)
            got = buf.cpu().numpy()
            assert (got[batch * ref.shape[1]:] == 7.0).all()
            assert rel(got[:batch * ref.shape[1]].reshape(ref.shape), ref) <= tol, (n, batch, d)
