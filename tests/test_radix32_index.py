"""The radix-32 schedules of the 2^13 and 2^14 row kernels, forward and
remainder-last: the padded shared-memory index of every element that a
butterfly reads or writes is its first element's plus a constant (the kernels'
addressing), every pass touches each element once, and the chained passes give
the transform (against the DFT matrix at a small length of the same form)."""
from __future__ import annotations

import numpy as np
import pytest


def pidx(n):
    return n + (n >> 4)


def schedule(lg, rev, lgm=5):
    rem = [1 << (lg % lgm)] if lg % lgm else []
    full = [1 << lgm] * (lg // lgm)
    return full + rem if rev else rem + full


@pytest.mark.parametrize("lg", [13, 14])
@pytest.mark.parametrize("rev", [False, True])
def test_addresses(lg, rev):
    L, ns = 1 << lg, 1
    rad = schedule(lg, rev)
    assert np.prod(rad) == L
    for s, R in enumerate(rad):
        j = np.arange(L // R)
        if s > 0:   # exchange reads: j + r L/R
            d = np.arange(R)[:, None] * (L // R)
            assert (pidx(j + d) == pidx(j) + pidx(d)).all()
        if s + 1 < len(rad):   # exchange writes: base + q Ns
            base, q = (j // ns) * ns * R + j % ns, np.arange(R)[:, None] * ns
            assert (pidx(base + q) == pidx(base) + pidx(q)).all()
            assert np.unique(base + q).size == L
        ns *= R


@pytest.mark.parametrize("rad", [[8, 32], [32, 8], [4, 32, 32]])
def test_recurrence(rad):
    L = int(np.prod(rad))
    x = np.random.default_rng(3).normal(size=L) + 0j
    a, ns = x, 1
    for R in rad:
        j = np.arange(L // R)
        v = a[j + np.arange(R)[:, None] * (L // R)]
        v = v * np.exp(-2j * np.pi * np.arange(R)[:, None] * (j % ns) / (ns * R))
        V = np.exp(-2j * np.pi * np.outer(np.arange(R), np.arange(R)) / R) @ v
        b = np.empty(L, complex)
        b[(j // ns) * ns * R + j % ns + np.arange(R)[:, None] * ns] = V
        a, ns = b, ns * R
    assert np.allclose(a, np.fft.fft(x))
