// mixr_plan.h -- the plan of one FP32 mixed-radix tile (mixr.cuh): the radix
// schedule, columns and threads per CTA of a sub-transform of any 7-smooth
// length, chosen by a cost model of its passes.  Plain C++17, so the host test
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
constexpr int kRadices[] = {2, 3, 4, 5, 7, 8, 9, 10, 12, 14, 15, 16, 20, 21, 24, 25};
constexpr int kThreads[] = {96, 128, 192, 256, 320, 384};
constexpr int kThreadsBig[] = {256, 320, 384, 448, 512};
constexpr int kPoints = 25, kPointsBig = 32;          // middle-pass points a thread may hold
constexpr long long kMaxTile = 384 * kPoints;         // 9600 points
constexpr long long kMaxTileBig = 512 * kPointsBig;
constexpr size_t kSmemLimit = 227 * 1024, kSmemSm = 228 * 1024;

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
// twiddles of a pass: basis loads, products to build the other powers, R - 1 products
inline float twiddle_cost(int r) {
  const int e = log2_up(r);
  return (2.f * e + 4.f * (r - 1 - e) + 4.f * (r - 1)) / r;
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

inline bool needs_pad(int r0, bool strided, bool in_rows, int C) {
  if (r0 & 1) return false;
  return !strided || in_rows || C < 16;   // 16 columns fill every bank whatever the row stride
}
inline size_t tile_bytes(long long N, int C, bool strided, bool in_rows, bool pad) {
  const long long rows = strided ? N : C * N;
  const long long padded = pad ? rows + ((rows - 1) >> 4) : rows;
  return (size_t)padded * (strided ? C + (in_rows ? 1 : 0) : 1) * 8;
}

// Cost of a tile, in instructions a point: the passes' arithmetic, index work
// and exchanges, with part of what a pass's last, partly filled round leaves
// idle, and more where few warps share an SM.  The weights are a fit to 9,000
// measured (schedule, columns, threads) of 41 lengths from 30 to 12288 on
// GB300: the pick is 0.7 % (at most 5 %) slower than the fastest measured.
inline float tile_cost(const Choice& c, long long N, size_t smem, bool pad) {
  const float P = (float)c.C * (float)N;
  float sum = 0;
  for (int s = 0; s < c.q.n; ++s) {
    const int r = c.q.rad[s];
    const float nb = P / (float)r;
    const float rounds = (float)(int)((nb + (float)c.T - 1.f) / (float)c.T);
    float per = dft_cost(r) + 10.8f / (float)r + (pad ? 1.6f : 0.f);
    if (s > 0) per += 1.48f * twiddle_cost(r) + (r >= 15 ? 4.5f : 0.f) + (r >= 20 ? 4.f : 0.f);
    if (s > 0 && s + 1 < c.q.n) per += 4.5f;
    sum += per * (1.f + 0.22f * (1.f - nb / (rounds * (float)c.T)));
  }
  const int regs = c.big ? 128 : 80;
  int ctas = std::min<int>(65536 / (regs * c.T), (int)(kSmemSm / (smem + 1024)));
  ctas = std::max(1, std::min(ctas, 32));
  const float warps = (float)(ctas * c.T) / 32.f;
  if (warps < 24.f) sum *= 1.f + 0.012f * (24.f - warps);
  sum *= ctas == 1 ? 1.12f : ctas == 2 ? 1.05f : 1.f;
  return sum * (1.f + 0.094f * (float)c.T / 256.f);
}
// Cost of strided global runs of C of the ncols adjacent elements against
// aligned runs of 16 (128 bytes): shorter runs, and runs that start inside a
// 32-byte sector or a 128-byte line.
inline float run_cost(int C, long long ncols) {
  const float run = C >= 16 ? 0.f : C >= 8 ? 8.f : C >= 4 ? 15.f : C >= 2 ? 80.f : 200.f;
  return run + (ncols % 4 ? 10.f : ncols % 16 ? 2.f : 0.f);
}

// Every ordered factorisation of `rest` into npass register radices.
inline void factorisations(long long rest, int depth, int npass, Schedule& cur, std::vector<Schedule>& out) {
  if (depth == npass) {
    if (rest == 1) out.push_back(cur);
    return;
  }
  long long most = 1;   // what the remaining passes can still cover
  for (int i = depth; i < npass; ++i) most *= 25;
  if (rest > most) return;
  for (const int r : kRadices) {
    if (rest % r) continue;
    cur.rad[depth] = r;
    factorisations(rest / r, depth + 1, npass, cur, out);
  }
}

// The schedule, columns and threads per CTA of least cost for a sub-transform
// of length N with ncols columns a batch, `total` in all; FFT_ERR_UNSUPPORTED
// if there is none.  Fewest passes first (lengths above 7 take at least two: a single
// radix would read and write global memory at a stride of N).
inline int choose(Choice& best, long long N, long long ncols, long long total, bool strided, bool in_rows) try {
  memset(&best, 0, sizeof(best));
  std::vector<Schedule> qs;
  for (int np = N > 7 ? 2 : 1; np <= kMaxPasses; ++np) {
    Schedule cur;
    memset(&cur, 0, sizeof(cur));
    cur.n = np;
    factorisations(N, 0, np, cur, qs);
    if (qs.empty()) continue;
    // columns per CTA.  Strided: the widest power of two up to 16 that the tile
    // holds.  Contiguous: tiles of 1500 to 9600 points, fewer when the batch
    // would not give every SM a few CTAs.
    long long cmax = std::min(std::max(1LL, kMaxTile / N), std::max(1LL, ncols));
    long long cmin = 1;
    if (strided) {
      cmax = std::min(cmax, 16LL);
      while (cmin * 2 <= cmax) cmin *= 2;
    } else {
      cmax = std::min(cmax, std::max(1LL, total / (152 * 4)));
      cmin = std::min(cmax, std::max(1LL, (1500 + N - 1) / N));
    }
    for (long long C = cmin; C <= cmax; C += strided ? cmax : std::max(1LL, C / 8)) {
      for (int big = 0; big < 2; ++big) {
        if (big && C * N <= 6144) continue;
        if (C * N > (big ? kMaxTileBig : kMaxTile)) continue;
        for (int ti = 0; ti < (big ? 5 : 6); ++ti) {
          Choice c;
          c.C = (int)C;
          c.T = big ? kThreadsBig[ti] : kThreads[ti];
          c.big = big != 0;
          if (ti > 0 && C * N < 6LL * c.T) continue;
          for (const Schedule& q : qs) {
            bool fits = true;   // a middle pass holds its butterflies in registers
            for (int s = 1; s + 1 < np; ++s)
              fits = fits && C * N / q.rad[s] <= (long long)std::max(1, (big ? kPointsBig : kPoints) / q.rad[s]) * c.T;
            if (!fits) continue;
            c.q = q;
            const bool pad = needs_pad(q.rad[0], strided, in_rows, c.C);
            const size_t smem = np > 1 ? tile_bytes(N, c.C, strided, in_rows, pad) : 0;
            if (smem > kSmemLimit) continue;
            c.cost = tile_cost(c, N, smem, pad);
            if (best.q.n == 0 || c.cost < best.cost) best = c;
          }
        }
      }
    }
    if (best.q.n) return FFT_OK;
    qs.clear();
  }
  return FFT_ERR_UNSUPPORTED;
} catch (...) {   // no exception leaves the C ABI
  return FFT_ERR_ALLOC;
}

}  // namespace mixr
}  // namespace gbfft
