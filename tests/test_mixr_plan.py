"""The plan of the FP32 mixed-radix tile kernel (csrc/mixr_plan.h, plain C++)
for every 7-smooth length up to 14336, contiguous and strided, at batches of
one, a few and many: there is one, its radices multiply to the length, a
middle pass fits the registers that its kernel holds, and the tile fits shared
memory and its CTA."""
from __future__ import annotations

import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PROGRAM = r"""
#include <cstdio>
#include "paper_1707_07263_gb300/csrc/mixr_plan.h"
using namespace gbfft::mixr;
int main() {
  int lengths = 0, plans = 0;
  for (long long n = 2; n <= 14336; ++n) {
    long long m = n;
    for (int f : {2, 3, 5, 7})
      while (m % f == 0) m /= f;
    if (m != 1) continue;
    ++lengths;
    for (int mode = 0; mode < 3; ++mode)            // contiguous, strided, strided with contiguous input rows
      for (long long cols : {1LL, 2LL, 7LL, 16LL, 1000LL, 100000LL}) {
        Choice c;
        const bool st = mode > 0, rows = mode == 2;
        if (choose(c, n, cols, cols, st, rows)) return printf("no plan for %lld mode %d\n", n, mode), 1;
        ++plans;
        long long prod = 1;
        for (int s = 0; s < c.q.n; ++s) prod *= c.q.rad[s];
        const long long pts = c.C * n;
        const bool pad = needs_pad(c.q.rad[0], st, rows, c.C);
        bool ok = prod == n && c.q.n <= kMaxPasses && c.C >= 1 && c.C <= cols;
        ok = ok && c.T % 32 == 0 && c.T <= (c.big ? 512 : 384);
        ok = ok && (!st || ((c.C & (c.C - 1)) == 0 && c.C <= 16));
        ok = ok && (c.q.n == 1 || tile_bytes(n, c.C, st, rows, pad) <= 227 * 1024);
        for (int s = 1; s + 1 < c.q.n; ++s) {
          const int kp = c.big ? 32 : 25;
          const long long held = kp / c.q.rad[s] > 1 ? kp / c.q.rad[s] : 1;
          ok = ok && pts / c.q.rad[s] <= held * c.T;
        }
        // reciprocal divisions are exact while index * divisor < 2^32
        ok = ok && pts * n < (1LL << 32);
        if (!ok) return printf("bad plan for %lld mode %d cols %lld\n", n, mode, cols), 1;
      }
  }
  printf("%d %d\n", lengths, plans);
  return 0;
}
"""


def test_every_length_has_a_valid_plan(tmp_path):
    src = tmp_path / "plan.cpp"
    src.write_text(PROGRAM)
    exe = tmp_path / "plan"
    r = subprocess.run(["g++", "-std=c++17", "-O2", "-I", ROOT, str(src), "-o", str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stdout
    lengths, plans = map(int, r.stdout.split())
    assert lengths > 370 and plans == lengths * 18
