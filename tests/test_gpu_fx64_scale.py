"""FP64 transforms hold every part of a result to FP64 arithmetic where inputs of
different scale meet (those go to FP64 arithmetic), keep the accuracy of 64-bit
integers where they do not, and treat each transform of a tile by itself.

Bars: tol(n), the FP64 bar of every other test, against the norm of the part
that is looked at.  For rows of one scale, 2e-16 of the row: an element is held
to 2^-57 of the row's largest value, at most 6 times the rms of a Gaussian row,
4.2e-17 of the rms a rounding; at most 16 roundings in four passes add in
squares to 1.7e-16, the conversion of the result to 53 bits adds 1.1e-16 at
most.  Two passes: sqrt(2) times that."""
from __future__ import annotations

import numpy as np
import pytest
import torch

import oracle
import paper_1707_07263_gb300 as gb
from paper_1707_07263_gb300 import api, workloads

pytestmark = pytest.mark.gpu


def tol(n: int) -> float:
    return 5e-15 * max(1.0, np.log2(n)) + 2e-16 * np.sqrt(n)


def run(x, d=0, inplace=False):
    xt = torch.from_numpy(np.ascontiguousarray(x)).cuda()
    p = api.Plan("1d", (x.shape[-1],), x.shape[0], prec="fp64")
    return p(xt, out=xt if inplace else None, dir=d).cpu().numpy()


def test_two_values():
    y = run(np.array([[1 + 1e-20j, 0], [1 + 1e-20j, 1], [1e-300 + 1j, -1j]]))
    assert (y == np.array([[1 + 1e-20j, 1 + 1e-20j], [2 + 1e-20j, 1e-20j], [1e-300, 1e-300 + 2j]])).all()


# 2^a 3^b: the sums of a constant cancel exactly in FP64
@pytest.mark.parametrize("n", [2, 3, 4, 6, 8, 9, 64, 576, 4096, 6561, 6912, 1 << 13, 1 << 16, 1 << 19])
@pytest.mark.parametrize("q", [1e-6, 1e-10, 1e-14, 1e-20])
def test_small_part_beside_a_constant(n, q):
    g = np.random.default_rng(41000 + n).normal(size=(2, n))
    for d in (0, 1):
        y = run(1 + 1j * q * g, d, inplace=d == 1)
        ref = 1j * q * oracle.transform(g + 0j, d) if n <= 8192 else 1j * q * (np.fft.ifft(g) if d else np.fft.fft(g))
        assert oracle.rel_l2_rows(y[:, 1:], ref[:, 1:]).max() <= tol(n)


@pytest.mark.parametrize("n", [2, 5, 7, 10, 105, 1000, 2401, 4096, 7168, 7200, 1 << 16])
@pytest.mark.parametrize("q", [1e-3, 1e-9, 1e-30, 1e-200])
def test_parts_of_different_scale(n, q):
    g = workloads.cgauss128(n, 3, seed=41100 + n)
    y = run(g.real + 1j * q * g.imag)
    norm = np.sqrt((g.imag ** 2).sum(1))
    assert (np.abs(y[:, 0].imag / q - g.imag.sum(1)) <= tol(n) * norm).all()
    y = run(q * g.real + 1j * g.imag)
    assert (np.abs(y[:, 0].real / q - g.real.sum(1)) <= tol(n) * norm).all()


@pytest.mark.parametrize("n", [64, 4096, 6912, 1 << 14])
def test_comb(n):
    g = workloads.cgauss128(n, 2, seed=41200 + n) * 1e-18
    x = g.copy()
    x[:, ::2] = 1 + 1j   # transforms to bins 0 and n/2 alone
    ref = oracle.transform(np.where(np.arange(n) % 2, g, 0), 0)
    keep = np.arange(n) % (n // 2) != 0
    assert oracle.rel_l2_rows(run(x)[:, keep], ref[:, keep]).max() <= tol(n)


@pytest.mark.parametrize("n", [8, 64, 105, 1000, 4096, 7168, 1 << 13])
@pytest.mark.parametrize("d", [0, 1])
def test_neighbours_do_not_change(n, d):
    """Bit for bit, whatever the other rows of a tile need."""
    rows = max(9, 3 * (5120 // n))
    x = workloads.cgauss128(n, rows, seed=41300 + n)
    y = run(x, d)
    odd = [(0, np.nan), (3, np.inf), (4, None), (rows - 1, np.nan)]
    z = x.copy()
    for i, v in odd:
        if v is None:
            z[i] = z[i].real + 1e-25j * z[i].imag
        else:
            z[i, n // 2] = v
    w = run(z, d, inplace=True)
    same = np.setdiff1d(np.arange(rows), [i for i, _ in odd])
    assert (w[same] == y[same]).all()
    assert not np.isfinite(w[[0, 3, rows - 1]]).any()
    assert oracle.rel_l2(w[4], oracle.transform(z[4:5], d)[0]) <= tol(n)


@pytest.mark.parametrize("ny,nx", [(12, 9), (96, 15), (1024, 7), (4096, 3), (7000, 5)])
def test_columns_of_different_scale(ny, nx):
    """A strided tile whose columns differ in scale, some zero and some not finite;
    the last tile of a row of columns is not full."""
    s = 10.0 ** ((np.arange(nx) * 2) % 5)
    s[nx // 2] = 0
    S = workloads.cgauss128(ny * nx, 1, seed=41400 + ny).reshape(ny, nx) * s
    x = np.fft.ifft(S, axis=1)   # its row transforms are S
    y = gb.fft2(torch.from_numpy(x[None]).cuda()).cpu().numpy()[0]
    ref = np.fft.fft(S.astype(np.clongdouble), axis=0)
    err = np.sqrt((np.abs(y - ref) ** 2).sum(0))
    norm = np.sqrt((np.abs(ref) ** 2).sum(0))
    worst = s.max() * np.sqrt(ny * ny)   # the row pass rounds against the largest column
    for c in range(nx):
        assert err[c] <= tol(ny * nx) * max(norm[c], worst), c
        if s[c] >= 10:   # and no column's exponent is another's
            assert err[c] <= 1e-9 * norm[c], c


@pytest.mark.parametrize("n,bar", [(8, 2e-16), (64, 2e-16), (105, 2e-16), (1000, 2e-16), (2401, 2e-16), (4096, 2e-16),
                                   (6561, 2e-16), (7168, 2e-16), (7200, 2.9e-16), (1 << 16, 2.9e-16)])
@pytest.mark.parametrize("kind", ["gauss", "uniform", "real", "offset"])
def test_accuracy_of_rows_of_one_scale(n, bar, kind):
    g = np.random.default_rng(41500 + n)
    x = workloads.cgauss128(n, 4, seed=41500 + n)
    if kind == "uniform":
        x = g.uniform(-1, 1, (4, n)) + 1j * g.uniform(-1, 1, (4, n))
    elif kind == "real":
        x = x.real + 0j
    elif kind == "offset":
        x = x + (3 - 2j)
    for d, f in ((0, np.fft.fft), (1, np.fft.ifft)):
        ref = f(x.astype(np.clongdouble))
        err = np.abs(run(x, d) - ref)
        assert np.sqrt((err ** 2).sum(1) / (np.abs(ref) ** 2).sum(1)).max() <= bar
