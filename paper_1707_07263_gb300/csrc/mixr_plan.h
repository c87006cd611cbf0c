// mixr_plan.h -- the plan of one mixed-radix tile (FP32: mixr.cuh, FP64:
// fx64.cuh): the radix schedule, columns and threads per CTA of a
// sub-transform of any 7-smooth length, chosen by a cost model of its passes.  Plain C++17, so the host test
// suite can check every length's plan with g++.
#pragma once
#include <algorithm>
#include <cstddef>
#include <cstring>
#include <vector>

#include "../../include/gbfft.h"

namespace gbfft {
namespace mixr {

constexpr int kMaxPasses = 6;
constexpr size_t kSmemLimit = 227 * 1024, kSmemSm = 228 * 1024;

// What the two kernels differ in.
struct Family {
  int nradices, radices[16];   // ascending
  int threads[6], threads_big[6];   // CTA sizes of small and big tiles (0 ends the list)
  int points, points_big;      // points a thread may hold in a middle pass
  bool first_held;             // the first pass holds its points too
  long long max_tile, max_tile_big, big_from;   // tile points; big CTAs above big_from
  int regs, regs_big;
  int elem;                    // bytes of a tile element
  int max_cols;                // strided columns that fill 128 bytes
  int slot_bytes;              // per pass and column, beside the tile
  int extra_passes;            // schedules of this many passes over the fewest are tried too
  float (*pass_cost)(int r, bool first, bool last, bool pad);
  // tile_cost: idle threads of a last round, warps an SM should hold and the
  // cost of each that is missing, one or two CTAs an SM, threads per CTA
  float idle, warps, warp_cost, one_cta, two_ctas, thread_cost;
};

// FP32 instructions a point of the R-point DFT (additions, constant products)
inline float dft_cost(int r) {
  switch (r) {
    case 2: return 2.f;
    case 3: return 5.3f;
    case 4: return 4.f;
    case 5: return 8.f;
    case 7: return 13.f;
    case 8: return 6.5f;
    case 9: return 12.4f;
    case 10: return 11.6f;
    case 12: return 11.3f;
    case 14: return 16.7f;
    case 15: return 15.5f;
    case 16: return 10.5f;
    case 20: return 14.4f;
    case 21: return 20.6f;
    case 24: return 14.2f;
    default: return 18.6f;
  }
}
inline int log2_up(int r) {
  int e = 0;
  while ((1 << e) < r) ++e;
  return e;
}
// twiddles of a pass: loads and products of a basis w^(2^e), as they were when the
// weights below were fitted
inline float twiddle_cost(int r) {
  const int e = log2_up(r);
  return (2.f * e + 4.f * (r - 1 - e) + 4.f * (r - 1)) / r;
}

// The passes' arithmetic, index work and exchanges.  The weights (and those of
// tile_cost) are a fit to 9,000 measured (schedule, columns, threads) of 41
// lengths from 30 to 12288 on GB300: the pick was 0.7 % (at most 5 %) slower than
// the fastest measured.  With every twiddle from a table it is 1.8 % (at most 11 %)
// slower than the fastest of 6,605 measured at 44 lengths; weights fitted to those
// pick better there (0.7 %) but up to 30 % slower at lengths between, so these stay.
inline float pass_cost_f32(int r, bool first, bool last, bool pad) {
  float per = dft_cost(r) + 10.8f / (float)r + (pad ? 1.6f : 0.f);
  if (!first) per += 1.48f * twiddle_cost(r) + (r >= 15 ? 4.5f : 0.f) + (r >= 20 ? 4.f : 0.f);
  if (!first && !last) per += 4.5f;
  return per;
}
// The same for the 64-bit fixed-point passes: a fit to 6,700 measured
// (schedule, columns, threads) of 29 lengths from 60 to 7168 (the pick is 2 %
// slower than the fastest measured on average, at most 7 %).
inline float pass_cost_fx(int r, bool first, bool last, bool) {
  const float dft = r == 2 ? 3.5f : r == 3 ? 8.f : r == 4 ? 15.5f : r == 5 ? 27.2f : r == 7 ? 37.5f
                    : r == 8 ? 25.4f : r == 9 ? 36.3f : r == 10 ? 55.8f : r == 12 ? 33.f : r == 14 ? 56.9f
                    : r == 15 ? 52.9f : 27.6f;
  return dft + 184.f / (float)r + (first ? 52.7f : 46.5f * (float)(r - 1) / (float)r) + (last ? 62.9f : 0.f);
}

inline const Family& family_f32() {
  // up to 384 threads of 80 registers (two CTAs of 384, three of 256 or six of
  // 128 share an SM), 512 of 128 for big tiles
  static const Family f = {16,
                           {2, 3, 4, 5, 7, 8, 9, 10, 12, 14, 15, 16, 20, 21, 24, 25},
                           {96, 128, 192, 256, 320, 384},
                           {256, 320, 384, 448, 512, 0},
                           25, 32, false, 9600, 16384, 6144, 80, 128, 8, 16, 0, 0, pass_cost_f32,
                           0.22f, 24.f, 0.012f, 1.12f, 1.05f, 0.094f};
  return f;
}
inline const Family& family_fx() {
  static const Family f = {12,
                           {2, 3, 4, 5, 7, 8, 9, 10, 12, 14, 15, 16},
                           {64, 96, 128, 192, 256, 0},
                           {320, 384, 448, 512, 0, 0},
                           20, 20, true, 5120, 8192, 2048, 128, 128, 16, 8, 4, 1, pass_cost_fx,
                           1.37f, 16.f, 0.02f, 1.13f, 1.015f, 0.034f};
  return f;
}

struct Schedule {
  int n, rad[kMaxPasses];
};
struct Choice {
  Schedule q;
  int C, T;
  bool big;
  float cost;
};

inline bool needs_pad(const Family& f, int r0, bool strided, bool in_rows, int C) {
  if (r0 & 1) return false;
  return !strided || in_rows || C < f.max_cols;   // max_cols columns fill every bank whatever the row stride
}
inline size_t tile_bytes(const Family& f, long long N, int C, bool strided, bool in_rows, bool pad) {
  const long long rows = strided ? N : C * N;
  const long long padded = pad ? rows + ((rows - 1) >> 4) : rows;
  return (size_t)padded * (strided ? C + (in_rows ? 1 : 0) : 1) * (size_t)f.elem;
}

// Cost of a tile, in instructions a point, with part of what a pass's last,
// partly filled round leaves idle, and more where few warps share an SM.
inline float tile_cost(const Family& f, const Choice& c, long long N, size_t smem, bool pad) {
  const float P = (float)c.C * (float)N;
  float sum = 0;
  for (int s = 0; s < c.q.n; ++s) {
    const float nb = P / (float)c.q.rad[s];
    const float rounds = (float)(int)((nb + (float)c.T - 1.f) / (float)c.T);
    sum += f.pass_cost(c.q.rad[s], s == 0, s + 1 == c.q.n, pad) * (1.f + f.idle * (1.f - nb / (rounds * (float)c.T)));
  }
  const int regs = c.big ? f.regs_big : f.regs;
  int ctas = std::min<int>(65536 / (regs * c.T), (int)(kSmemSm / (smem + 1024)));
  ctas = std::max(1, std::min(ctas, 32));
  const float warps = (float)(ctas * c.T) / 32.f;
  if (warps < f.warps) sum *= 1.f + f.warp_cost * (f.warps - warps);
  sum *= ctas == 1 ? f.one_cta : ctas == 2 ? f.two_ctas : 1.f;
  return sum * (1.f + f.thread_cost * (float)c.T / 256.f);
}
// Cost of strided global runs of C of the ncols adjacent elements against
// aligned runs of 128 bytes: shorter runs, and runs that start inside a
// 32-byte sector or a 128-byte line.
inline float run_cost(const Family& f, int C, long long ncols) {
  const int b = C * f.elem;
  const float run = b >= 128 ? 0.f : b >= 64 ? 8.f : b >= 32 ? 15.f : b >= 16 ? 80.f : 200.f;
  const long long step = ncols * f.elem;
  return run + (step % 32 ? 10.f : step % 128 ? 2.f : 0.f);
}

// Every ordered factorisation of `rest` into npass register radices.
inline void factorisations(const Family& f, long long rest, int depth, int npass, Schedule& cur,
                           std::vector<Schedule>& out) {
  if (depth == npass) {
    if (rest == 1) out.push_back(cur);
    return;
  }
  long long most = 1;   // what the remaining passes can still cover
  for (int i = depth; i < npass; ++i) most *= f.radices[f.nradices - 1];
  if (rest > most) return;
  for (int i = 0; i < f.nradices; ++i) {
    const int r = f.radices[i];
    if (rest % r) continue;
    cur.rad[depth] = r;
    factorisations(f, rest / r, depth + 1, npass, cur, out);
  }
}

// The schedule, columns and threads per CTA of least cost for a sub-transform
// of length N with ncols columns a batch, `total` in all; FFT_ERR_UNSUPPORTED
// if there is none.  Fewest passes first (lengths above 7 take at least two: a single
// radix would read and write global memory at a stride of N).
inline int choose(const Family& f, Choice& best, long long N, long long ncols, long long total, bool strided,
                  bool in_rows) try {
  memset(&best, 0, sizeof(best));
  std::vector<Schedule> qs;
  int fewest = 0;
  for (int np = N > 7 ? 2 : 1; np <= kMaxPasses; ++np) {
    Schedule cur;
    memset(&cur, 0, sizeof(cur));
    cur.n = np;
    factorisations(f, N, 0, np, cur, qs);
    if (qs.empty()) continue;
    // columns per CTA.  Strided: the widest power of two that the tile holds, up
    // to 128 bytes.  Contiguous: tiles of 1500 points to the largest, fewer when
    // the batch would not give every SM a few CTAs.
    long long cmax = std::min(std::max(1LL, f.max_tile / N), std::max(1LL, ncols));
    long long cmin = 1;
    if (strided) {
      cmax = std::min<long long>(cmax, f.max_cols);
      while (cmin * 2 <= cmax) cmin *= 2;
    } else {
      cmax = std::min(cmax, std::max(1LL, total / (152 * 4)));
      cmin = std::min(cmax, std::max(1LL, (1500 + N - 1) / N));
    }
    for (long long C = cmin; C <= cmax; C += strided ? cmax : std::max(1LL, C / 8)) {
      for (int big = 0; big < 2; ++big) {
        if (big && C * N <= f.big_from) continue;
        if (C * N > (big ? f.max_tile_big : f.max_tile)) continue;
        for (int ti = 0; ti < 6; ++ti) {
          Choice c;
          c.C = (int)C;
          c.T = big ? f.threads_big[ti] : f.threads[ti];
          c.big = big != 0;
          if (c.T == 0) break;
          if (ti > 0 && C * N < 6LL * c.T) continue;
          for (const Schedule& q : qs) {
            bool fits = true;   // a middle pass holds its butterflies in registers
            for (int s = f.first_held ? 0 : 1; s + 1 < np; ++s)
              fits = fits && C * N / q.rad[s] <= (long long)std::max(1, (big ? f.points_big : f.points) / q.rad[s]) * c.T;
            if (!fits) continue;
            c.q = q;
            const bool pad = needs_pad(f, q.rad[0], strided, in_rows, c.C);
            const size_t smem =
                np > 1 ? tile_bytes(f, N, c.C, strided, in_rows, pad) + (size_t)(f.slot_bytes * np * c.C) : 0;
            if (smem > kSmemLimit) continue;
            c.cost = tile_cost(f, c, N, smem, pad);
            if (best.q.n == 0 || c.cost < best.cost) best = c;
          }
        }
      }
    }
    qs.clear();
    if (best.q.n && fewest == 0) fewest = np;
    if (fewest && np >= fewest + f.extra_passes) return FFT_OK;
  }
  return best.q.n ? FFT_OK : FFT_ERR_UNSUPPORTED;
} catch (...) {   // no exception leaves the C ABI
  return FFT_ERR_ALLOC;
}

// Modelled cost of a strided pass (to choose between splits of a longer
// length), negative if there is none.
inline float strided_cost(const Family& f, long long N, long long ncols, long long batches, bool in_rows) {
  Choice c;
  if (choose(f, c, N, ncols, ncols * batches, true, in_rows)) return -1.f;
  const long long tiles = (ncols + c.C - 1) / c.C;   // the last tile of a batch may be partly empty
  return c.cost * (float)(tiles * c.C) / (float)ncols + run_cost(f, c.C, ncols);
}

// N = n1 n2, both at most most: the column length n1 of the split with the
// least modelled cost of its column and row passes, 0 if there is none.
inline long long choose_split(const Family& f, long long N, long long batches, long long most) {
  long long b1 = 0;
  float best = 0;
  // factors within 8 : 1 of each other unless there are none
  for (int wide = 0; wide < 2 && b1 == 0; ++wide)
    for (long long d = 2; d * d <= N; ++d) {
      if (N % d || N / d > most || (!wide && N / d > 8 * d)) continue;
      for (const long long n1 : {d, N / d}) {
        const float ca = strided_cost(f, n1, N / n1, batches, false);
        const float cb = strided_cost(f, N / n1, n1, batches, true);
        if (ca < 0 || cb < 0) continue;
        if (b1 == 0 || ca + cb < best) {
          b1 = n1;
          best = ca + cb;
        }
      }
    }
  return b1;
}

}  // namespace mixr
}  // namespace gbfft
