"""The 64-bit fixed-point arithmetic of the FP64 transforms
(csrc/fx64_math.h, plain C++) against 128-bit integers and long double: rotations
and products within the units that they drop, on average exact, zero exactly
zero; factors right to the last bits of Q62; conversions from FP64 truncated at
their last unit and back rounded to nearest."""
from __future__ import annotations

import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PROGRAM = r"""
#include <cmath>
#include <cstdio>
#include <cstring>
#include <random>
#include "paper_1707_07263_gb300/csrc/fx64_math.h"
using namespace gbfft;
static double units(__int128 exact, long long got) { return (double)(((__int128)got << 64) - exact) / 18446744073709551616.0; }
int main() {
  std::mt19937_64 g(1);
  double worst = 0, worst_r = 0, mean = 0, trig = 0, from = 0, to = 0;
  const long double pi = 3.14159265358979323846264338327950288L;
  const int n = 400000;
  for (int it = 0; it < n; ++it) {
    const long long M = it % 2 ? 1 + it % 700 : 1 + (long long)(g() % (1 << 28)), m = (long long)(g() % M);
    const FxCosSin t = fx_cossin(m, M);
    // the angle in [0, pi/4] by exact integer symmetries, so that the reference is right to its last bit
    long long o = 8 * m / M, r = 8 * m - o * M;
    if (o & 1) r = M - r;
    const long double a = pi / 4 * ((long double)r / (long double)M);
    const long double ca = cosl(a), sa = sinl(a);
    const bool swap = o == 1 || o == 2 || o == 5 || o == 6;
    const long double c = (swap ? sa : ca) * (o >= 2 && o <= 5 ? -1 : 1), s = (swap ? ca : sa) * (o >= 4 ? -1 : 1);
    trig = std::fmax(trig, std::fmax(std::fabs((double)(c * 0x1p62L - t.c)), std::fabs((double)(s * 0x1p62L - t.s))));
    const Cq62 w{q62_split(t.c), q62_split(t.s)};
    const int b = 2 + (int)(g() % 60);
    long long x = (long long)(g() >> (64 - b)), y = (long long)(g() >> (64 - b));
    if (g() & 1) x = -x;
    if (g() & 1) y = -y;
    const __int128 wr = (__int128)w.r.h * 4294967296LL + w.r.l, wi = (__int128)w.i.h * 4294967296LL + w.i.l;
    const Fx p = fx_cmul(Fx{x, y}, w);
    const double d1 = units((__int128)x * wr - (__int128)y * wi, p.x), d2 = units((__int128)x * wi + (__int128)y * wr, p.y);
    worst = std::fmax(worst, std::fmax(std::fabs(d1), std::fabs(d2)));
    mean += d1 + d2;
    worst_r = std::fmax(worst_r, std::fabs(units((__int128)x * wr, fx_mulr(x, w.r))));
    // FP64 -> integer: truncated at the unit 2^(E - 1022 - F)
    const double v = std::ldexp((double)(long long)g(), (int)(g() % 200) - 100);
    long long bits;
    std::memcpy(&bits, &v, 8);
    const int E = (int)((bits >> 52) & 0x7ff) + (int)(g() % 40), F = 57 + (int)(g() % 4);
    const long long q = fx_from_bits<false>(bits, E, F);
    from = std::fmax(from, std::fabs(std::ldexp(v, 1022 + F - E) - (double)q) - std::ldexp(std::fabs((double)q), -53));
    if ((q < 0) != (v < 0) && q != 0) return 2;
    // integer -> FP64: to nearest
    const int ex = (int)(g() % 1900) - 1000;
    const long long ob = fx_to_bits(x, ex);
    double back;
    std::memcpy(&back, &ob, 8);
    const long double ref = std::ldexp((long double)x, ex);
    if (!fx_normal(ex) || (x == 0 && ob != 0)) return 3;
    if (x) to = std::fmax(to, std::fabs((double)(((long double)back - ref) / ref)) * 9007199254740992.0);
  }
  // zeros, subnormal rows, the largest headroom
  const Cq62 w{q62(0.3), q62(-0.9)};
  const Fx z = fx_cmul(Fx{0, 0}, w);
  if (z.x || z.y || fx_mulr(0, w.i) || fx_shr(0, 3)) return 4;
  if (fx_from_bits<true>(3, 1, 57) != 48 || fx_from_bits<true>((long long)0x8000000000000003ULL, 1, 57) != -48) return 5;
  for (int r = 2; r <= 16; ++r)
    if (std::ldexp(1.0, fx_headroom(r)) < r * std::sqrt(2.0)) return 6;
  std::printf("%g %g %g %g %g %g\n", worst, worst_r, std::fabs(mean) / (2 * n), trig, from, to);
  return 0;
}
"""


def test_fixed_point_arithmetic(tmp_path):
    src = tmp_path / "fx.cpp"
    src.write_text(PROGRAM)
    exe = tmp_path / "fx"
    r = subprocess.run(["g++", "-std=gnu++17", "-O2", "-I", ROOT, str(src), "-o", str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, (r.returncode, r.stdout)
    worst, worst_r, mean, trig, frm, to = map(float, r.stdout.split())
    # a rotation drops four floors (two of either sign, below 1 each) and two low
    # products (below 1/4 each); a real product two floors and one low product
    assert worst <= 2.5 and worst_r <= 1.25
    assert mean <= 0.01
    assert trig <= 2.0          # units of 2^-62
    assert frm <= 1.0           # truncation below one unit
    assert to <= 1.0 + 1e-9     # half an ulp, in units of 2^-53
