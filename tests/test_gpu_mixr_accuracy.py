"""FP32 mixed-radix transforms are as accurate as the kernels of radices up to 16
that ran one pass per prime factor before them: relative L2 error over 2^22
Gaussian points against 64 bits, each bar that kernel's measured error on the same
input plus half a per cent."""
from __future__ import annotations

import pytest
import torch

from paper_1707_07263_gb300 import api

pytestmark = pytest.mark.gpu

BEFORE = {100: 9.5621e-08, 343: 1.1006e-07, 1000: 1.1786e-07, 1080: 1.1907e-07, 2187: 1.3971e-07, 2401: 1.3003e-07,
          3125: 1.3563e-07, 5000: 1.3749e-07, 5040: 1.3350e-07, 6561: 1.5087e-07, 7000: 1.3549e-07, 9000: 1.3691e-07,
          9375: 1.4546e-07, 12500: 1.4968e-07, 13720: 1.4032e-07, 14336: 1.4507e-07, 15000: 1.4526e-07,
          30000: 1.4918e-07, 100000: 1.6182e-07, 1000000: 1.7655e-07}


@pytest.mark.parametrize("n", BEFORE)
def test_no_less_accurate(n):
    g = torch.Generator(device="cuda").manual_seed(n)
    x = torch.randn(max(1, (1 << 22) // n), n, dtype=torch.complex64, device="cuda", generator=g)
    ref = torch.fft.fft(x.to(torch.complex128))
    y = api.Plan("1d", (n,), x.shape[0])(x).to(torch.complex128)
    assert float((y - ref).norm() / ref.norm()) <= 1.005 * BEFORE[n]
