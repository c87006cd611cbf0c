"""One cached plan on several streams and from several host threads: every plan
kind that writes a workspace or work counters gives each call its own result, bit
for bit that of the call alone, with nothing but the library ordering the calls."""
from __future__ import annotations

import threading

import pytest
import torch

import paper_1707_07263_gb300 as gb

pytestmark = pytest.mark.gpu


def cx(*shape, dtype=torch.complex64):
    return torch.randn(*shape, dtype=dtype, device="cuda")


H = {}


def range_long(x):
    n = x.shape[-1]
    if n not in H:
        H[n] = cx(n)
    return gb.range_compress(x, H[n])


UNEVEN = [1 << (8 + i % 9) for i in range(200)]
SHORT = [1 << (4 + i % 9) for i in range(3000)]
CALLS = {
    "2^16": (gb.fft, lambda: cx(64, 1 << 16)),
    "2^20": (gb.ifft, lambda: cx(4, 1 << 20)),
    "2^23": (gb.fft, lambda: cx(1, 1 << 23)),
    "15000": (gb.fft, lambda: cx(200, 15000)),
    "fp64": (gb.fft, lambda: cx(16, 1 << 16, dtype=torch.complex128)),
    "rows 2^20": (gb.rfft, lambda: torch.randn(4, 1 << 20, device="cuda")),
    "to rows 2^18": (lambda x: gb.irfft(x), lambda: cx(16, (1 << 17) + 1)),
    "range 2^16": (range_long, lambda: cx(64, 1 << 16)),
    "4096 x 1024": (gb.fft2, lambda: cx(1, 4096, 1024)),
    "tc": (lambda x: gb.fft(x, prec="tc_fp16"), lambda: cx(64, 1 << 16)),
    "uneven": (lambda x: gb.fft_many(x, UNEVEN), lambda: cx(sum(UNEVEN))),
    "uneven short": (lambda x: gb.fft_many(x, SHORT), lambda: cx(sum(SHORT))),
}


@pytest.mark.parametrize("name", CALLS)
def test_streams(name):
    f, make = CALLS[name]
    xs = [make() for _ in range(4)]
    ref = [f(x) for x in xs]
    torch.cuda.synchronize()
    streams = [torch.cuda.Stream() for _ in xs]
    out = [[] for _ in xs]
    for _ in range(8):
        for i, (s, x) in enumerate(zip(streams, xs)):
            with torch.cuda.stream(s):
                out[i].append(f(x))
    torch.cuda.synchronize()
    for r, ys in zip(ref, out):
        for y in ys:
            assert torch.equal(y, r)


@pytest.mark.parametrize("name", ["2^16", "15000", "fp64", "uneven"])
def test_threads_on_one_stream(name):
    f, make = CALLS[name]
    xs = [make() for _ in range(4)]
    ref = [f(x) for x in xs]
    torch.cuda.synchronize()
    out = [[] for _ in xs]
    go = threading.Barrier(len(xs))

    def work(i):
        go.wait()
        for _ in range(40):
            out[i].append(f(xs[i]))
            if len(out[i]) > 4:
                out[i].pop(0)

    ts = [threading.Thread(target=work, args=(i,)) for i in range(len(xs))]
    for t in ts:
        t.start()
    for t in ts:
        t.join()
    torch.cuda.synchronize()
    for r, ys in zip(ref, out):
        for y in ys:
            assert torch.equal(y, r)


def test_captured_after_use_on_another_stream():
    x = cx(8, 1 << 16)
    ref = gb.fft(x)
    s = torch.cuda.Stream()
    s.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(s):
        gb.fft(x)
    torch.cuda.current_stream().wait_stream(s)
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        y = gb.fft(x)
    y.zero_()
    g.replay()
    assert torch.equal(y, ref)
    assert torch.equal(gb.fft(x), ref)


def test_explicit_stream_waits_for_what_the_call_makes():
    """A copy of a strided input and a fresh output are made on the current stream,
    which is still busy: the other stream's transform comes after them."""
    p = gb.Plan("1d", (4096,), 64)
    base = cx(4096, 64)
    x = base.t()
    ref = p(x)
    s = torch.cuda.Stream()
    torch.cuda.synchronize()
    for _ in range(3):
        torch.cuda._sleep(20_000_000)
        y = p(x, stream=s)
        s.synchronize()
        assert torch.equal(y, ref)
