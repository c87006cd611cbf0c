"""Views that conjugate or negate lazily (x.conj(), x.conj().imag, a gradient that
arrives as one): every entry point takes their values, not the memory under them."""
from __future__ import annotations

import pytest
import torch

import paper_1707_07263_gb300 as gb
from paper_1707_07263_gb300 import api

pytestmark = pytest.mark.gpu


def cx(*shape, dtype=torch.complex64):
    return torch.randn(*shape, dtype=dtype, device="cuda")


CALLS = [
    (gb.fft, lambda: cx(3, 64)),
    (gb.ifft, lambda: cx(3, 60)),
    (gb.fft, lambda: cx(3, 4096, dtype=torch.complex128)),
    (gb.fft2, lambda: cx(2, 16, 32)),
    (gb.ifft2, lambda: cx(12, 20)),
    (gb.irfft, lambda: cx(3, 33)),
    (lambda x: gb.range_compress(x, torch.linspace(1, 2, 64, device="cuda").to(torch.complex64)), lambda: cx(3, 64)),
    (lambda x: gb.fft_many(x, [64, 256, 16]), lambda: cx(336)),
    (lambda x: api.get_plan("1d", (64,), 3)(x), lambda: cx(3, 64)),
]


@pytest.mark.parametrize("i", range(len(CALLS)))
def test_conjugated_input_and_gradient(i):
    f, make = CALLS[i]
    x = make()
    v = x.conj()
    assert v.is_conj()
    assert torch.equal(f(v), f(v.resolve_conj()))
    if i + 1 < len(CALLS):
        grads = []
        for lazy in (True, False):
            t = x.clone().requires_grad_(True)
            y = f(t.conj())
            g = torch.linspace(1, 2, y.numel(), device="cuda").reshape(y.shape).to(y.dtype)
            g = (g * (1 + 2j)).conj() if y.is_complex() else g
            (gx,) = torch.autograd.grad(y, t, g if lazy else g.resolve_conj())
            grads.append(gx.resolve_conj())
        assert torch.equal(*grads)


def test_conjugated_filter():
    x, H = cx(3, 64), cx(64)
    assert torch.equal(gb.range_compress(x, H.conj()), gb.range_compress(x, H.conj().resolve_conj()))


def test_negated_real_rows():
    z = cx(3, 64)
    v = torch._neg_view(z.imag.contiguous())
    assert v.is_neg() and v.is_contiguous()
    assert torch.equal(gb.rfft(v), gb.rfft(v.resolve_neg()))
    assert torch.equal(gb.rfft(z.conj().imag), gb.rfft(-z.imag))


def test_conjugated_output_is_refused():
    p = api.get_plan("1d", (64,), 3)
    with pytest.raises(ValueError):
        p(cx(3, 64), out=torch.empty(3, 64, dtype=torch.complex64, device="cuda").conj())


def test_conjugated_host_buffers():
    x = torch.randn(4, 256, dtype=torch.complex64).pin_memory()
    ref = gb.fft_host(x.conj().resolve_conj())
    assert torch.equal(gb.fft_host(x.conj()), ref)
    pipe = api.HostPipeline(256, 4)
    out = torch.empty(4, 256, dtype=torch.complex64).pin_memory()
    pipe(x.conj(), out)
    torch.cuda.synchronize()
    assert torch.equal(out, ref)
    with pytest.raises(ValueError):
        pipe(x, torch.empty(4, 256, dtype=torch.complex64).pin_memory().conj())
