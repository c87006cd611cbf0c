"""fft_exec_noalloc makes its twiddle tables on every call, so each launch counts:
the two passes, one stage table for each and the two levels of W_N."""
from __future__ import annotations

import ctypes

import pytest
import torch
from torch.profiler import ProfilerActivity, profile

from paper_1707_07263_gb300 import _lib

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("lg", [15, 18, 19, 20, 21, 22])
def test_launches_of_a_call(lg):
    lib = _lib.load()
    x = torch.randn(1 << lg, dtype=torch.complex64, device="cuda")
    y = torch.empty_like(x)
    s = ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)

    def call():
        assert lib.fft_exec_noalloc(1 << lg, 1, 0, ctypes.c_void_p(x.data_ptr()), ctypes.c_void_p(y.data_ptr()), s) == 0

    call()
    torch.cuda.synchronize()
    with profile(activities=[ProfilerActivity.CUDA]) as prof:
        call()
        torch.cuda.synchronize()
    names = [e.name for e in prof.events() if "gbfft" in e.name]
    if not names:
        pytest.skip("the profiler records no kernels here")
    assert len(names) <= 6, names
