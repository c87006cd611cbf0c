"""The FP32 mixed-radix tile kernel where its plans change: one to five passes,
the largest tile of the small and the large CTA, odd and even first radices
(unpadded and padded tiles), several transforms per CTA with a ragged last
tile, and, as columns of images, every width of a strided tile with columns
left over.  Against the oracle; bar 5e-7 * log2(points), as for every FP32
path."""
from __future__ import annotations

import numpy as np
import pytest
import torch

import oracle
from paper_1707_07263_gb300 import api, workloads

pytestmark = pytest.mark.gpu


def tol(n: int) -> float:
    return 5e-7 * max(1.0, np.log2(n))


@pytest.mark.parametrize("n", [3, 7, 9, 50, 192, 225, 486, 6300, 7203, 8748, 9600, 9604, 12005, 13122, 13440])
@pytest.mark.parametrize("batch,d", [(1, 0), (5, 1), (611, 0)])
def test_contiguous(n, batch, d):
    if batch > 100 and n > 1000:
        batch = 13
    x = workloads.cgauss(n, batch, seed=31000 + n + d)
    y = api.Plan("1d", (n,), batch)(torch.from_numpy(x).cuda(), dir=d).cpu().numpy()
    rows = sorted({0, batch // 2, batch - 1})
    ref = oracle.transform(x[rows].astype(np.complex128), d)
    assert oracle.rel_l2_rows(y[rows], ref).max() <= tol(n)
    # the other rows: Parseval and the first bin
    s = x.astype(np.complex128)
    scale = 1.0 if d == 0 else 1.0 / n
    assert np.allclose(y[:, 0], s.sum(1) * scale, rtol=0, atol=1e-5 * np.sqrt(n) * scale)
    assert np.allclose((np.abs(y.astype(np.complex128)) ** 2).sum(1), (np.abs(s) ** 2).sum(1) * n * scale * scale, rtol=1e-5)


@pytest.mark.parametrize("ny,nx", [(7, 35), (6, 45), (600, 20), (1029, 12), (2401, 9), (1200, 35), (4802, 5),
                                   (9604, 3), (12005, 3), (9600, 3)])
def test_columns(ny, nx):
    """nx columns of ny points: 16, 8, 4, 2 or 1 of them per CTA."""
    x = workloads.cgauss(ny * nx, 1, seed=32000 + ny).reshape(1, ny, nx)
    y = api.Plan("2d", (ny, nx), 1)(torch.from_numpy(x).cuda()).cpu().numpy()
    rows = oracle.transform(x[0].astype(np.complex128), 0)
    ref = np.stack([oracle.transform(np.ascontiguousarray(rows[:, c])[None], 0)[0] for c in range(nx)], 1)
    assert oracle.rel_l2(y[0], ref) <= tol(ny * nx)


@pytest.mark.parametrize("n", [14406, 18900, 1049760])
def test_two_passes(n):
    """Split lengths on both sides of the dense four-step table's limit (2^20),
    column counts that are no multiple of a tile's width; sampled bins."""
    x = workloads.cgauss(n, 2, seed=33000 + n % 1000)
    y = api.Plan("1d", (n,), 2)(torch.from_numpy(x).cuda()).cpu().numpy()
    ks = np.unique(np.concatenate([np.arange(8), np.random.default_rng(5).integers(0, n, 40), [n - 1]]))
    ref = oracle.dft_bins(x.astype(np.complex128), ks)
    assert oracle.rel_l2_rows(y[:, ks], ref).max() <= tol(n)
