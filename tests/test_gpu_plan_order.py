"""Plans that share a kernel run in any order: a plan made later with a smaller
tile must not lower the shared-memory limit that an earlier one needs."""
from __future__ import annotations

import numpy as np
import pytest
import torch

import oracle
from paper_1707_07263_gb300 import api, workloads

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("big,small", [(4096, 2048), (7000, 3500), (1 << 15, 1 << 13)])
def test_fp64_large_plan_after_small_plan(big, small):
    p = api.Plan("1d", (big,), 2, prec="fp64")
    q = api.Plan("1d", (small,), 2, prec="fp64")
    for n, plan in ((big, p), (small, q)):
        x = workloads.cgauss128(n, 2, seed=34000 + n % 97)
        y = plan(torch.from_numpy(x).cuda()).cpu().numpy()
        assert oracle.rel_l2_rows(y, oracle.transform(x, 0)).max() <= 5e-15 * np.log2(n) + 2e-16 * np.sqrt(n)
