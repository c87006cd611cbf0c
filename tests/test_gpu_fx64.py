"""The FP64 tile kernel (64-bit integers with one exponent per transform) where
its route differs from plain FP64 arithmetic: neighbouring transforms of very
different scale, wide dynamic range inside one, impulses and constants,
subnormal and nearly overflowing rows, infinities and NaN, scales that are no
power of two, in place, one to five passes, two-pass lengths on both sides of
the dense twiddle table's limit.  Bar: 5e-15 * log2(n) + 2e-16 * sqrt(n), the
FP64 bar of every other test; the largest output bounds the error, so rows of
one scale are compared row by row."""
from __future__ import annotations

import numpy as np
import pytest
import torch

import oracle
import paper_1707_07263_gb300 as gb
from paper_1707_07263_gb300 import api, workloads

pytestmark = pytest.mark.gpu

LENGTHS = [2, 6, 7, 9, 64, 105, 1000, 2401, 4096, 6561, 7168]


def tol(n: int) -> float:
    return 5e-15 * max(1.0, np.log2(n)) + 2e-16 * np.sqrt(n)


def run(x, d=0, inplace=False):
    xt = torch.from_numpy(np.ascontiguousarray(x)).cuda()
    p = api.Plan("1d", (x.shape[-1],), x.shape[0], prec="fp64")
    return p(xt, out=xt if inplace else None, dir=d).cpu().numpy()


@pytest.mark.parametrize("n", LENGTHS)
@pytest.mark.parametrize("d", [0, 1])
def test_rows_of_different_scale(n, d):
    x = workloads.cgauss128(n, 7, seed=35000 + n)
    scale = np.array([1e-290, 1.0, 1e250, 0.0, 3e-20, 7e100, 1e-5])[:, None]
    y = run(x * scale, d, inplace=d == 1)
    ref = oracle.transform(x, d)
    for i, s in enumerate(scale[:, 0]):
        if s == 0:
            assert not y[i].any()
        else:
            assert oracle.rel_l2(y[i] / s, ref[i]) <= tol(n)


@pytest.mark.parametrize("n", LENGTHS)
def test_dynamic_range_impulse_constant(n):
    g = np.random.default_rng(35100 + n)
    x = np.zeros((4, n), complex)
    x[0] = (g.normal(size=n) + 1j * g.normal(size=n)) * np.exp(g.uniform(-300, 300, n))
    x[1, n // 3] = 1 - 2j
    x[2] = 1.5
    x[3] = np.arange(n) % 5 - 2
    y = run(x)
    assert oracle.rel_l2_rows(y, oracle.transform(x, 0)).max() <= tol(n)
    assert y[2, 0] == 1.5 * n


@pytest.mark.parametrize("n", [7, 64, 1000, 4096])
def test_ends_of_the_exponent_range(n):
    x = workloads.cgauss128(n, 1, seed=35200 + n)
    # subnormal inputs: multiples of 2^-1074, so the result is right to one of them a point
    q = np.round(x[0].real * 50) + 1j * np.round(x[0].imag * 50)
    y = run((q * 5e-324)[None])[0]
    ref = oracle.transform(q[None], 0)[0]
    got = y.real / 5e-324 + 1j * (y.imag / 5e-324)
    assert np.abs(got - ref).max() <= 1.0 + 1e-9
    # the transform of values near the largest number overflows only where the result does
    big = np.full((1, n), 1e308 / n, complex)
    y = run(big)[0]
    assert np.isfinite(y).all() and abs(y[0] / 1e308 - 1) <= tol(n)
    y = run(np.full((1, n), 1e308, complex))[0]
    assert np.isinf(y[0].real)


@pytest.mark.parametrize("n", LENGTHS)
@pytest.mark.parametrize("d", [0, 1])
@pytest.mark.parametrize("bad", [np.nan, np.inf])
def test_not_finite(n, d, bad):
    x = workloads.cgauss128(n, 5, seed=35300 + n)
    x[2, n // 2] = bad
    y = run(x, d, inplace=d == 1)
    assert not np.isfinite(y[2]).any()
    rows = [0, 1, 3, 4]
    assert oracle.rel_l2_rows(y[rows], oracle.transform(x[rows], d)).max() <= tol(n)


@pytest.mark.parametrize("ny,nx", [(6, 40), (100, 9), (1024, 6), (4096, 3), (7000, 2)])
def test_columns(ny, nx):
    x = workloads.cgauss128(ny * nx, 1, seed=35400 + ny).reshape(1, ny, nx)
    x[0, :, 1] *= 1e12   # a column of another scale in the same tile
    y = gb.fft2(torch.from_numpy(x).cuda()).cpu().numpy()
    assert oracle.rel_l2(y[0], oracle.fft2(x)[0]) <= tol(ny * nx)
    x[0, ny // 2, 0] = np.nan
    assert not np.isfinite(gb.fft2(torch.from_numpy(x).cuda()).cpu().numpy()).any()


@pytest.mark.parametrize("n", [7200, 1 << 13, 1 << 18, 1 << 19, 300000])
def test_two_passes(n):
    x = workloads.cgauss128(n, 2, seed=35500 + n % 1009)
    x[1] *= 1e-40
    y = run(x, 1)
    ks = np.unique(np.concatenate([np.arange(8), np.random.default_rng(6).integers(0, n, 40), [n - 1]]))
    ref = oracle.dft_bins(x, ks, oracle.INVERSE)
    assert oracle.rel_l2_rows(y[:, ks], ref).max() <= tol(n)
