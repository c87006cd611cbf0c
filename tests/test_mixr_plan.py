"""The plans of the mixed-radix tile kernels (csrc/mixr_plan.h, plain C++) for
every 7-smooth length up to 14336 (FP32) and 7168 (FP64), contiguous and
strided, at batches of one, a few and many: there is one, its radices multiply
to the length, the passes that hold their points fit the registers of their
kernel, and the tile fits shared memory and its CTA."""
from __future__ import annotations

import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PROGRAM = r"""
#include <cstdio>
#include "paper_1707_07263_gb300/csrc/mixr_plan.h"
using namespace gbfft::mixr;
int check(const Family& f, long long most, bool held, int points, int points_big, int threads, int threads_big,
          int max_cols, int& plans) {
  int lengths = 0;
  for (long long n = 2; n <= most; ++n) {
    long long m = n;
    for (int p : {2, 3, 5, 7})
      while (m % p == 0) m /= p;
    if (m != 1) continue;
    ++lengths;
    for (int mode = 0; mode < 3; ++mode)            // contiguous, strided, strided with contiguous input rows
      for (long long cols : {1LL, 2LL, 7LL, 16LL, 1000LL, 100000LL}) {
        Choice c;
        const bool st = mode > 0, rows = mode == 2;
        if (choose(f, c, n, cols, cols, st, rows)) return printf("no plan for %lld mode %d\n", n, mode), -1;
        ++plans;
        long long prod = 1;
        for (int s = 0; s < c.q.n; ++s) prod *= c.q.rad[s];
        const long long pts = c.C * n;
        const bool pad = needs_pad(f, c.q.rad[0], st, rows, c.C);
        bool ok = prod == n && c.q.n <= kMaxPasses && c.C >= 1 && c.C <= cols;
        ok = ok && c.T % 32 == 0 && c.T <= (c.big ? threads_big : threads);
        ok = ok && (!st || ((c.C & (c.C - 1)) == 0 && c.C <= max_cols));
        ok = ok && (c.q.n == 1 || tile_bytes(f, n, c.C, st, rows, pad) + f.slot_bytes * c.q.n * c.C <= 227 * 1024);
        ok = ok && (c.q.n > 1 || n <= 7);
        for (int s = held ? 0 : 1; s + 1 < c.q.n; ++s) {
          const int kp = c.big ? points_big : points;
          const long long most_held = kp / c.q.rad[s] > 1 ? kp / c.q.rad[s] : 1;
          ok = ok && pts / c.q.rad[s] <= most_held * c.T;
        }
        // reciprocal divisions are exact while index * divisor < 2^32
        ok = ok && pts * n < (1LL << 32);
        if (!ok) return printf("bad plan for %lld mode %d cols %lld\n", n, mode, cols), -1;
      }
  }
  return lengths;
}
int main() {
  int plans = 0;
  const int a = check(family_f32(), 14336, false, 25, 32, 384, 512, 16, plans);
  const int b = check(family_fx(), 7168, true, 20, 20, 256, 512, 8, plans);
  if (a < 0 || b < 0) return 1;
  printf("%d %d %d\n", a, b, plans);
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
    a, b, plans = map(int, r.stdout.split())
    assert a > 370 and b > 300 and plans == (a + b) * 18
