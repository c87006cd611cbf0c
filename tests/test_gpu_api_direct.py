"""Calls that need no gradient skip torch.autograd.Function: same values, and
everything that looks at the Function still meets it."""
from __future__ import annotations

import pytest
import torch
import torch.autograd.forward_ad as fwAD

import paper_1707_07263_gb300 as gb

pytestmark = pytest.mark.gpu


def cx(*shape):
    return torch.randn(*shape, dtype=torch.complex64, device="cuda")


CALLS = [
    (lambda x: gb.fft(x), lambda: cx(3, 64)),
    (lambda x: gb.ifft(x), lambda: cx(2, 3, 60)),
    (lambda x: gb.fft2(x), lambda: cx(2, 16, 32)),
    (lambda x: gb.ifft2(x), lambda: cx(12, 20)),
    (lambda x: gb.rfft(x), lambda: torch.randn(3, 64, device="cuda")),
    (lambda x: gb.irfft(x), lambda: cx(3, 33)),
    (lambda x: gb.range_compress(x, torch.ones(64, dtype=torch.complex64, device="cuda")), lambda: cx(3, 64)),
]


@pytest.mark.parametrize("i", range(len(CALLS)))
def test_same_values_with_and_without_gradient(i):
    f, make = CALLS[i]
    x = make()
    y = f(x)
    assert not y.requires_grad
    z = f(x.clone().requires_grad_(True))
    assert z.requires_grad and z.grad_fn is not None
    assert torch.equal(y, z.detach())
    with torch.no_grad():
        assert torch.equal(f(x.clone().requires_grad_(True)), y)
    assert torch.equal(f(torch.nn.Parameter(x)).detach(), y)
    t = x.transpose(0, 1).contiguous().transpose(0, 1)   # not contiguous
    assert torch.equal(f(t), y)
    s = torch.cuda.Stream()
    s.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(s):
        w = f(x)
    s.synchronize()
    assert torch.equal(w, y)


@pytest.mark.parametrize("i", range(len(CALLS)))
def test_forward_mode_and_vmap_are_refused(i):
    """The Functions define neither: silent answers without the tangent or
    over the wrong axis would be wrong."""
    f, make = CALLS[i]
    x = make()
    with fwAD.dual_level():
        with pytest.raises(Exception):
            f(fwAD.make_dual(x, torch.ones_like(x)))
    with pytest.raises(Exception):
        torch.func.vmap(f)(torch.stack([x, x]))
    with pytest.raises(Exception):
        torch.func.jvp(f, (x,), (torch.ones_like(x),))
    torch.cuda.synchronize()
