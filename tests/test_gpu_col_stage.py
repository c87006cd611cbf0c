"""Column passes of 2^10 points staged in their exchange buffer, and the 2-D and
1-D splits around them, where they can go wrong: a single tile, fewer tiles
than CTAs, several tiles per CTA, in place, inputs that are only 8-byte aligned
(register path, same result), both directions, and images on both sides of the
128-column rule.  Against the oracle, bar 5e-7 * log2(points)."""
from __future__ import annotations


import numpy as np
import pytest
import torch

import oracle
from paper_1707_07263_gb300 import api, workloads

pytestmark = pytest.mark.gpu


def tol(n):
    return 5e-7 * np.log2(n)


def run(plan, x, d=0, inplace=False, shift=0):
    buf = torch.empty(x.size + 2, dtype=torch.complex64, device="cuda")
    xt = buf[shift:shift + x.size]
    xt.copy_(torch.from_numpy(x.reshape(-1)))
    out = xt if inplace else torch.empty(x.size, dtype=torch.complex64, device="cuda")
    plan.exec_ptr(xt.data_ptr(), out.data_ptr(), d)
    return out.cpu().numpy().reshape(x.shape)


@pytest.mark.parametrize("nx,batch", [(2, 1), (8, 1), (16, 3), (64, 45), (4096, 1)])
@pytest.mark.parametrize("d,inplace", [(0, False), (1, True)])
def test_images_of_1024_rows(nx, batch, d, inplace):
    x = workloads.cgauss(1024 * nx, batch, seed=36000 + nx).reshape(batch, 1024, nx)
    p = api.Plan("2d", (1024, nx), batch)
    y = run(p, x, d, inplace)
    z = run(p, x, d, False, shift=1)   # 8-byte aligned
    for b in sorted({0, batch // 2, batch - 1}):
        ref = oracle.fft2(x[b:b + 1].astype(np.complex128), d)[0]
        assert oracle.rel_l2(y[b], ref) <= tol(1024 * nx)
        assert oracle.rel_l2(z[b], ref) <= tol(1024 * nx)
    assert oracle.rel_l2(y, z) <= 1e-6


@pytest.mark.parametrize("ny,nx", [(2048, 128), (2048, 64), (4096, 256), (8192, 128), (16384, 128), (8192, 16)])
def test_tall_images(ny, nx):
    x = workloads.cgauss(ny * nx, 1, seed=36100 + nx).reshape(1, ny, nx)
    p = api.Plan("2d", (ny, nx), 1)
    ref = oracle.fft2(x.astype(np.complex128))
    for shift in (0, 1):
        assert oracle.rel_l2(run(p, x, shift=shift), ref) <= tol(ny * nx)
    assert oracle.rel_l2(run(p, x, inplace=True), ref) <= tol(ny * nx)


@pytest.mark.parametrize("lg,batch", [(20, 1), (20, 5), (21, 2), (22, 1)])
def test_two_passes(lg, batch):
    n = 1 << lg
    x = workloads.cgauss(n, batch, seed=36200 + lg)
    p = api.Plan("1d", (n,), batch)
    assert p.launches == 2
    y = run(p, x, 1)
    z = run(p, x, 1, shift=1)
    ref = oracle.fft(x[-1:].astype(np.complex128), oracle.INVERSE)
    assert oracle.rel_l2(y[-1:], ref) <= tol(n)
    assert oracle.rel_l2(z[-1:], ref) <= tol(n)
    assert oracle.rel_l2(y, z) <= 1e-6
