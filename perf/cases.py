"""The work this library is used for, as cases to time and to compare.

A case is a plain dict; ``prepare`` makes what a program has in hand before
the call (inputs on the GPU from the seed, and the plan where a program keeps
one), ``run`` is one pass through the public entry points, ``exact`` is the
same result in 64 bits from torch.fft, ``work`` the bytes and operations the
result cannot do without.

Kinds:
  fft     complex rows, forward or inverse (float32 or float64 parts)
  fft2    complex images (rows, then columns)
  many    uneven packed lengths: the transform and the gradient (adjoint) pass
  real    real rows: the half spectrum and the gradient of the input
  irfft   half spectra back to real rows
  range   SAR range compression with one matched filter
"""
from __future__ import annotations

import math

import torch

import paper_1707_07263_gb300 as gb
from paper_1707_07263_gb300 import api

MAX_POINTS = 1 << 26   # complex float32 points of the largest case


def listed():
    return [
        # one range line by itself (interactive use): latency, launches and host work
        {"name": "line_4096", "kind": "fft", "n": 4096, "batch": 1, "inverse": False, "fp64": False},
        # an ordinary block of range lines
        {"name": "lines_4096", "kind": "fft", "n": 4096, "batch": 2048, "inverse": False, "fp64": False},
        # a whole scene of the longest lines one on-chip pass takes, back to the time domain
        {"name": "lines_16384", "kind": "fft", "n": 16384, "batch": 4096, "inverse": True, "fp64": False},
        # long lines (two passes), an ordinary block
        {"name": "lines_65536", "kind": "fft", "n": 65536, "batch": 512, "inverse": False, "fp64": False},
        # very long records, the largest 1-D batch of the benchmark
        {"name": "records_2p20", "kind": "fft", "n": 1 << 20, "batch": 64, "inverse": False, "fp64": False},
        # a full SAR image with bright scatterers
        {"name": "sar_8192", "kind": "fft2", "ny": 8192, "nx": 8192, "batch": 1, "inverse": False, "fp64": False},
        # uneven segments 2^8..2^16 of one acquisition, transform and gradient pass
        {"name": "uneven_4096", "kind": "many", "count": 4096},
        # real sensor rows in a training step: half spectrum and gradient
        {"name": "real_8192", "kind": "real", "n": 8192, "batch": 4096},
        # pulse compression of a block of range lines
        {"name": "range_8192", "kind": "range", "n": 8192, "batch": 4096},
        # a swath width that is not a power of two, an odd number of lines
        {"name": "swath_9000", "kind": "fft", "n": 9000, "batch": 3727, "inverse": False, "fp64": False},
        # a longer swath (two strided passes), inverse, an odd number of lines
        {"name": "swath_15000", "kind": "fft", "n": 15000, "batch": 1117, "inverse": True, "fp64": False},
        # double precision rows (reference processing of the same lines)
        {"name": "double_4096", "kind": "fft", "n": 4096, "batch": 4096, "inverse": False, "fp64": True},
    ]


# ---- drawn cases -------------------------------------------------------------
def _smooth(lo, hi):
    """Lengths 2^a 3^b 5^c 7^d in [lo, hi] that are not powers of two."""
    out = []
    a = 1
    while a <= hi:
        b = a
        while b <= hi:
            c = b
            while c <= hi:
                d = c
                while d <= hi:
                    if d >= lo and d & (d - 1):
                        out.append(d)
                    d *= 2
                c *= 3
            b *= 5
        a *= 7
    return sorted(out)


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _pick_smooth(rng, lo, hi):
    t = _log_int(rng, lo, hi)
    return min(_smooth(lo, hi), key=lambda v: abs(v - t))


def _batch(rng, n, lo_points, hi_points):
    hi_points = max(n, hi_points)
    return max(1, min(hi_points // n, _log_int(rng, max(lo_points, n), hi_points) // n))


def draw(rng):
    kind = rng.choice(["fft", "fft", "smooth", "smooth", "fft2", "many", "real", "irfft", "range", "double"])
    inverse = rng.random() < 0.5
    if kind == "fft":
        n = 1 << rng.randint(4, 22)
        return {"kind": "fft", "n": n, "batch": _batch(rng, n, 1 << 12, MAX_POINTS), "inverse": inverse, "fp64": False}
    if kind == "smooth":
        n = _pick_smooth(rng, 100, 200000)
        return {"kind": "fft", "n": n, "batch": _batch(rng, n, 1 << 14, MAX_POINTS // 2), "inverse": inverse,
                "fp64": False}
    if kind == "double":
        n = (1 << rng.randint(6, 20)) if rng.random() < 0.6 else _pick_smooth(rng, 100, 50000)
        return {"kind": "fft", "n": n, "batch": _batch(rng, n, 1 << 12, MAX_POINTS // 4), "inverse": inverse,
                "fp64": True}
    if kind == "fft2":
        if rng.random() < 0.6:
            ny, nx = 1 << rng.randint(6, 13), 1 << rng.randint(6, 13)
        else:
            ny, nx = _pick_smooth(rng, 100, 4000), _pick_smooth(rng, 100, 4000)
        return {"kind": "fft2", "ny": ny, "nx": nx, "batch": _batch(rng, ny * nx, 1 << 14, MAX_POINTS // 2),
                "inverse": inverse, "fp64": False}
    if kind == "many":
        return {"kind": "many", "count": _log_int(rng, 16, 4000)}
    n = 1 << rng.randint(6, 20)
    if kind == "range":
        n = 1 << rng.randint(8, 16)
        return {"kind": "range", "n": n, "batch": _batch(rng, n, 1 << 14, MAX_POINTS // 2)}
    return {"kind": kind, "n": n, "batch": _batch(rng, n, 1 << 14, MAX_POINTS)}


# ---- inputs --------------------------------------------------------------------
def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _cgauss(shape, g, dtype=torch.complex64):
    """Circular complex Gaussian CN(0, 1): receiver noise and speckle."""
    return torch.randn(shape, generator=g, device="cuda", dtype=dtype)


def _lengths(count, seed):
    """count lengths 2^8..2^16, the exponent uniform."""
    e = torch.randint(8, 17, (count,), generator=torch.Generator().manual_seed(int(seed)))
    return [1 << int(v) for v in e]


def _image(case, g):
    """Unit speckle with 64 bright point scatterers per image."""
    ny, nx, b = case["ny"], case["nx"], case["batch"]
    x = _cgauss((b, ny, nx), g)
    k = min(64, ny * nx)
    pix = torch.randint(0, ny * nx, (b, k), generator=g, device="cuda")
    ph = torch.rand((b, k), generator=g, device="cuda") * (2 * math.pi)
    x.view(b, -1).scatter_add_(1, pix, torch.polar(torch.full_like(ph, 100.0), ph))
    return x


def _range_lines(n, batch, g, bw=0.8, targets=8):
    """Echoes of a linear-FM pulse of n/4 samples at random circular delays in
    unit receiver noise."""
    p = n // 4
    t = torch.arange(n, device="cuda")
    x = _cgauss((batch, n), g)
    for _ in range(targets):
        d = torch.randint(0, n, (batch, 1), generator=g, device="cuda")
        amp = 1.0 + 9.0 * torch.rand((batch, 1), generator=g, device="cuda")
        ph = 2 * math.pi * torch.rand((batch, 1), generator=g, device="cuda")
        tau = (t - d) % n
        chirp = math.pi * bw / p * (tau.float() - p / 2.0) ** 2 + ph
        x += torch.polar(torch.where(tau < p, amp, 0.0 * amp), chirp)
    return x


def _range_filter(n, bw=0.8):
    """Matched filter of that pulse by stationary phase, natural frequency order."""
    p = n // 4
    k = torch.arange(n, device="cuda", dtype=torch.float64)
    f = torch.where(k < n / 2, k / n, k / n - 1.0)
    ph = math.pi * f * f * p / bw + math.pi * f * p
    H = torch.polar(torch.ones_like(ph), ph)
    H[f.abs() > bw / 2] = 0
    return H.to(torch.complex64)


def _inputs(case, seed):
    g = _gen(seed)
    k = case["kind"]
    if k == "fft":
        return {"x": _cgauss((case["batch"], case["n"]), g, torch.complex128 if case["fp64"] else torch.complex64)}
    if k == "fft2":
        return {"x": _image(case, g)}
    if k == "many":
        lengths = _lengths(case["count"], case["count"])   # the acquisition's layout: the same for every input
        total = sum(lengths)
        return {"lengths": lengths, "x": _cgauss((total,), g), "g": _cgauss((total,), g)}
    if k == "real":
        n, b = case["n"], case["batch"]
        return {"x": torch.randn((b, n), generator=g, device="cuda"), "g": _cgauss((b, n // 2 + 1), g)}
    if k == "irfft":
        return {"x": _cgauss((case["batch"], case["n"] // 2 + 1), g)}
    if k == "range":
        return {"x": _range_lines(case["n"], case["batch"], g), "H": _range_filter(case["n"])}
    raise ValueError(k)


def prepare(case, seed):
    st = dict(_inputs(case, seed), case=case)
    if case["kind"] == "many":
        # a program that runs the same layout again and again keeps its plan
        lengths = st.pop("lengths")
        st["plan"] = api.get_plan("many", (sum(lengths),), len(lengths), "fp32", st["x"].device, lengths=tuple(lengths))
    if case["kind"] == "real":
        st["x"].requires_grad_(True)
    return st


# ---- one pass --------------------------------------------------------------------
def run(st):
    case = st["case"]
    k = case["kind"]
    if k == "fft":
        return gb.ifft(st["x"]) if case["inverse"] else gb.fft(st["x"])
    if k == "fft2":
        return gb.ifft2(st["x"]) if case["inverse"] else gb.fft2(st["x"])
    if k == "many":
        return [st["plan"](st["x"]), st["plan"](st["g"], dir=api.ADJOINT)]
    if k == "real":
        y = gb.rfft(st["x"])
        (gx,) = torch.autograd.grad(y, st["x"], st["g"])
        return [y.detach(), gx]
    if k == "irfft":
        return gb.irfft(st["x"])
    return gb.range_compress(st["x"], st["H"])


# ---- 64-bit results ----------------------------------------------------------------
def exact(case, seed):
    st = _inputs(case, seed)
    k = case["kind"]
    x = st["x"]
    if k == "fft":
        x = x.to(torch.complex128)
        return torch.fft.ifft(x) if case["inverse"] else torch.fft.fft(x)
    if k == "fft2":
        x = x.to(torch.complex128)
        return torch.fft.ifft2(x) if case["inverse"] else torch.fft.fft2(x)
    if k == "many":
        y, gx = torch.empty_like(x, dtype=torch.complex128), torch.empty_like(x, dtype=torch.complex128)
        o = 0
        for n in st["lengths"]:
            y[o:o + n] = torch.fft.fft(x[o:o + n].to(torch.complex128))
            gx[o:o + n] = torch.fft.ifft(st["g"][o:o + n].to(torch.complex128), norm="forward")
            o += n
        return [y, gx]
    if k == "real":
        # the adjoint over the kept bins: the real part of the conjugate sum of g, zero-extended
        g = st["g"].to(torch.complex128)
        g = torch.cat([g, torch.zeros((g.shape[0], case["n"] // 2 - 1), dtype=g.dtype, device=g.device)], 1)
        return [torch.fft.rfft(x.double()), torch.fft.ifft(g, norm="forward").real.contiguous()]
    if k == "irfft":
        x = x.to(torch.complex128)
        x[:, 0].imag.zero_()
        x[:, -1].imag.zero_()
        return torch.fft.irfft(x, n=case["n"])
    return torch.fft.ifft(torch.fft.fft(x.to(torch.complex128)) * st["H"].to(torch.complex128))


# ---- what a pass cannot do without ---------------------------------------------------
def _flops(n, rows):
    return 5.0 * n * math.log2(n) * rows


def work(case):
    k = case["kind"]
    if k == "fft":
        n, b = case["n"], case["batch"]
        return {"bytes": (32 if case["fp64"] else 16) * n * b, "flops": _flops(n, b)}
    if k == "fft2":
        p = case["ny"] * case["nx"]
        return {"bytes": 16 * p * case["batch"], "flops": _flops(p, case["batch"])}
    if k == "many":
        lengths = _lengths(case["count"], case["count"])
        return {"bytes": 2 * 16 * sum(lengths), "flops": 2 * sum(_flops(n, 1) for n in lengths)}
    n, b = case["n"], case["batch"]
    if k == "range":
        return {"bytes": 16 * n * b + 8 * n, "flops": 2 * _flops(n, b) + 6.0 * n * b}
    one = (4 * n + 8 * (n // 2 + 1)) * b
    if k == "irfft":
        return {"bytes": one, "flops": 0.5 * _flops(n, b)}
    return {"bytes": 2 * one, "flops": _flops(n, b)}   # real: the transform and its adjoint
