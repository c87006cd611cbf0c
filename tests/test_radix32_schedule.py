"""The radix-32 schedules of the 2^10, 2^13 and 2^14 kernels and the schedules of
the paired real rows, read from the constexpr functions that the kernels and the
table generator share (compiled into a host program, no GPU): every pass touches
every element once, addresses are a base plus constants, tables lie inside their
allocation, and the passes chained with the factors that the tables hold give the
transform."""
from __future__ import annotations

import os
import shutil
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PROGRAM = r"""
#include <cstdio>
#include "real_pair.cuh"
#include "tile_registry.h"
using namespace gbfft;

template <int N>
void pads() {
  if constexpr (N >= 0) {
    pads<N - 1>();
    std::printf(" %d", pidx_c(N * 16 + 15));
  }
}

int main() {
  for (int lg = 1; lg <= 14; ++lg) {
    std::printf("T %d %d %d %d\n", lg, (int)stage_has_32(lg), stage_tw_size(lg), stage_table_size(lg));
    if (!stage_has_32(lg)) continue;
    for (int rev = 0; rev < 2; ++rev) {
      std::printf("S %d %d %d", lg, rev, stage_tw_size(lg, rev != 0, 5));
      for (int s = 0; s < radix_nst(lg, 5); ++s)
        std::printf(" %d:%d:%d", radix_lgr(lg, s, rev != 0, 5), radix_lgns(lg, s, rev != 0, 5), stage_tw_off(lg, s, rev != 0, 5));
      std::printf("\n");
    }
  }
  for (int lg = 5; lg <= 14; ++lg)
    for (int c2r = 0; c2r < 2; ++c2r) {
      if (!c2r && lg < 9) continue;
      std::printf("P %d %d", lg, c2r);
      for (int s = 0; s < pair_nst(lg); ++s) {
        const int r = pair_lgr(lg, c2r != 0, s), ns = pair_lgns(lg, c2r != 0, s);
        const int st = ns ? pair_tw_stage(lg, ns + r) : -1;
        std::printf(" %d:%d:%d:%d", r, ns, st, st < 0 ? 0 : radix_lgns(lg, st));
      }
      std::printf("\n");
    }
  using K = TileCfg<10, 8, true, true, 0, 5>;
  std::printf("K %d %d %d %d %d\n", K::P, K::T, K::SM_TILE, K::SM_EPI, K::SMEM_BYTES);
  std::printf("I");
  pads<63>();
  std::printf("\n");
  return 0;
}
"""


def pidx(n):
    return n + (n >> 4)


@pytest.fixture(scope="module")
def lines(tmp_path_factory):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    d = tmp_path_factory.mktemp("radix32")
    src, exe = d / "s.cu", d / "s"
    src.write_text(PROGRAM)
    subprocess.check_call([nvcc, "-std=c++17", "--expt-relaxed-constexpr", "-gencode", "arch=compute_103a,code=sm_103a",
                           "-I", os.path.join(ROOT, "paper_1707_07263_gb300", "csrc"), "-I", os.path.join(ROOT, "include"),
                           str(src), "-o", str(exe)])
    return subprocess.run([str(exe)], capture_output=True, text=True, check=True).stdout.splitlines()


def chained(x, passes, factor):
    """The Stockham passes (lgr, lgns) over x; factor(s, e, k) is the table's
    W^{2^e k} of pass s, the other powers are products of these."""
    L, a = x.size, x
    for s, (lgr, lgns) in enumerate(passes):
        R, Ns = 1 << lgr, 1 << lgns
        j = np.arange(L // R)
        k = j % Ns
        reads = j + np.arange(R)[:, None] * (L // R)
        writes = (j // Ns) * Ns * R + k + np.arange(R)[:, None] * Ns
        for idx, base, d in ((reads, j, np.arange(R)[:, None] * (L // R)),
                             (writes, (j // Ns) * Ns * R + k, np.arange(R)[:, None] * Ns)):
            assert np.array_equal(np.sort(idx, axis=None), np.arange(L))
            assert np.array_equal(pidx(base + d), pidx(base) + pidx(d))
        v = a[reads]
        if Ns > 1:
            w = [factor(s, e, k) for e in range(lgr)]
            for r in range(1, R):
                for e in range(lgr):
                    if r >> e & 1:
                        v[r] = v[r] * w[e]
        b = np.empty(L, complex)
        b[writes] = np.fft.fft(v, axis=0)
        a = b
    return a


def test_padding(lines):
    got = [int(v) for line in lines if line.startswith("I") for v in line.split()[1:]]
    assert got == [pidx(16 * i + 15) for i in range(64)]


def test_radix32_schedules(lines):
    tables = {int(f[1]): tuple(map(int, f[2:])) for f in (line.split() for line in lines) if f[0] == "T"}
    assert [lg for lg in tables if tables[lg][0]] == [10, 13, 14]
    seen = 0
    for f in (line.split() for line in lines):
        if f[0] != "S":
            continue
        lg, rev, size = map(int, f[1:4])
        p = [tuple(map(int, q.split(":"))) for q in f[4:]]
        want = [5] * (lg // 5)
        if lg % 5:
            want = want + [lg % 5] if rev else [lg % 5] + want
        assert [q[0] for q in p] == want
        table = np.zeros(size, complex)
        for lgr, lgns, off in p:   # the generator's rows
            if lgns:
                for e in range(lgr):
                    k = np.arange(1 << lgns)
                    lo = off + (e << lgns)
                    assert lo + k.size <= size and not table[lo:lo + k.size].any()
                    table[lo:lo + k.size] = np.exp(-2j * np.pi * ((k << e) / (1 << (lgns + lgr))))
        assert table.all()
        if not rev:   # beside the radix-16 table
            assert tables[lg][2] == tables[lg][1] + size
        x = np.random.default_rng(lg).normal(size=1 << lg) + 1j
        y = chained(x, [q[:2] for q in p], lambda s, e, k: table[p[s][2] + (e << p[s][1]) + k])
        assert np.allclose(y, np.fft.fft(x))
        seen += 1
    assert seen == 6


def test_paired_real_rows(lines):
    seen = 0
    for f in (line.split() for line in lines):
        if f[0] != "P":
            continue
        lg, c2r = map(int, f[1:3])
        p = [tuple(map(int, q.split(":"))) for q in f[3:]]
        assert all(1 <= q[0] <= 5 for q in p) and sum(q[0] for q in p) == lg
        assert p[0][0] <= (4 if c2r else 5)   # two butterflies, or one, of 32 points a thread
        if not c2r:
            assert p[-1][0] == 4

        def factor(s, e, k):
            lgr, lgns, st, lgnt = p[s]
            nt, mul = 1 << lgnt, 1 << (lgnt + 4 - lgr - lgns)
            assert lgr >= 4 and st > 0
            row, col = (3, 2 * k * mul) if e == 4 else (e, k * mul)
            assert col.max() < nt
            return np.exp(-2j * np.pi * (col << row) / (16 * nt))

        x = np.random.default_rng(lg).normal(size=1 << lg) + 1j
        assert np.allclose(chained(x, [q[:2] for q in p], factor), np.fft.fft(x))
        seen += 1
    assert seen == 10 + 6


def test_staged_columns(lines):
    p, t, tile, epi, smem = next(tuple(map(int, line.split()[1:])) for line in lines if line.startswith("K"))
    assert p == 32 and t * p == 8 << 10
    assert tile >= 8 << 10            # the copied box lies in the exchange tile
    assert epi == 8 * 32              # one step factor a column and output of a radix-32 butterfly
    assert smem == 8 * (tile + epi)
