// real_pair.cuh -- real-data rows (N = 2L reals) with both halves of every
// split pair in one thread.
//
// A real-to-complex row is a length-L transform Z of the reals taken as complex
// pairs, then X[k] = E + W_N^k O and X[L-k] = conj(E - W_N^k O) from Z[k] and
// Z[L-k] (E = (Z[k] + conj Z[L-k]) / 2, O = (Z[k] - conj Z[L-k]) / 2i).  In the
// last pass, butterfly j (outputs j + q L/R) holds the partners of butterfly
// L/R - j, so a thread that runs both (32 points, 128 registers) splits in
// registers: no exchange beside those between the passes, one factor and one
// E and O per pair.  A complex-to-real row is the mirror image: the first pass
// (inputs j + r L/R) of butterflies j and L/R - j reads every X once and builds
// Z[n] = E + i O and Z[L-n] = conj(E) + i conj(O).  Butterflies 0 and L/2R are
// their own partners and share a thread.
//
// The exchanged split was bound by the shared-memory and L1 data paths (83 % busy
// at 2^13 reals: an exchange more in r2c, every X and factor read twice in c2r).
// 2^13 reals, 2^26 in all: r2c 101 -> 89 us, c2r 119 -> 91, where a copy takes 79;
// what is left is each row's own latency at 16 warps an SM.  Where the row lengths
// take this kernel: tile_inst_real.cu.
#pragma once
#include "tile_fft.cuh"

namespace gbfft {

// Schedule (log2 of the radices): r2c ends and c2r starts with radix 16 or, for
// c2r of few points, what radix 16 leaves; a 32-point remainder beside radix 16
// takes one pass (2^9 = 32 16, 2^13 = 32 16 16, 2^14 = 32 32 16).
__host__ __device__ constexpr int pair_nst(int lg) { return lg <= 9 ? 2 : 3; }
__host__ __device__ constexpr int pair_lgr(int lg, bool c2r, int s) {
  if (c2r) return lg <= 8 ? (s == 0 ? lg - 4 : 4) : lg == 9 ? (s == 0 ? 4 : 5)
                  : lg <= 12 ? (s == 0 ? lg - 8 : 4) : lg == 13 ? (s == 1 ? 5 : 4) : (s == 0 ? 4 : 5);
  return s == pair_nst(lg) - 1 ? 4 : lg <= 9 ? lg - 4 : lg <= 12 ? (s == 0 ? lg - 8 : 4) : lg == 13 ? (s == 0 ? 5 : 4) : 5;
}
__host__ __device__ constexpr int pair_lgns(int lg, bool c2r, int s) {
  return s == 0 ? 0 : pair_lgns(lg, c2r, s - 1) + pair_lgr(lg, c2r, s - 1);
}
// The radix-16 stage of the length's table (Ns = 2^lgns(st), rows W^{2^e k} with
// the period 16 Ns) that a pass reads at a step of `mul`: its period is mul times
// shorter, and W^{16 k} of a radix-32 pass is row 3 at twice the index.
__host__ __device__ constexpr int pair_tw_stage(int lg, int lgperiod) {
  int s = 0;
  while (radix_lgns(lg, s) + 4 < lgperiod) ++s;
  return s;
}

template <int LG, int C>
struct PairCfg {
  static constexpr int L = 1 << LG;
  static constexpr int T = C * L / 32;
  static constexpr int NST = pair_nst(LG);
  static constexpr int LP = TileCfg<LG, C, false, false>::LP;
  static constexpr int SMEM_BYTES = C * LP * 8;
};

template <int LG, bool C2R, int S>
__device__ __forceinline__ void pair_twiddle(float2* v, const TileArgs& a, int k) {
  constexpr int R = 1 << pair_lgr(LG, C2R, S), LGP = pair_lgns(LG, C2R, S) + pair_lgr(LG, C2R, S);
  constexpr int ST = pair_tw_stage(LG, LGP), NT = 1 << radix_lgns(LG, ST), MUL = 1 << (radix_lgns(LG, ST) + 4 - LGP);
  static_assert(R >= 16 && ST > 0 && radix_lgr(LG, ST) == 4, "a radix-16 stage with a table");
  apply_stage_twiddle<R>(v, a.tw + stage_tw_off(LG, ST), NT, k * MUL, 3 * NT + 2 * k * MUL);
}

// Pass S with the general mapping (butterflies tid + i T): a row's first pass
// from global memory, a middle pass, or (LASTG) the last one to global memory.
template <int LG, int C, bool C2R, int S, bool LASTG>
__device__ __forceinline__ void pair_pass(float2* sm, const TileArgs& a, const float2* gin, float2* gout,
                                          long long col0) {
  using Cfg = PairCfg<LG, C>;
  constexpr int LGR = pair_lgr(LG, C2R, S), R = 1 << LGR, LGNS = pair_lgns(LG, C2R, S), NS = 1 << LGNS;
  constexpr int NB = 32 / R, LR = Cfg::L / R;
  const int tid = threadIdx.x;
  float2 v[32];
#pragma unroll
  for (int i = 0; i < NB; ++i) {
    const int b = tid + i * Cfg::T, c = b / LR, j = b % LR;
    if constexpr (S == 0) {
      const bool ok = col0 + c < a.ncols;
      const float2* p = gin + c * a.in_sc + j;
#pragma unroll
      for (int r = 0; r < R; ++r) v[i * R + r] = ok ? __ldcs(p + r * LR) : make_float2(0.f, 0.f);
    } else {
      const float2* p = sm + c * Cfg::LP + pidx(j);
#pragma unroll
      for (int r = 0; r < R; ++r) v[i * R + r] = p[pidx_c(r * LR)];
    }
  }
  if constexpr (NS > 1) {
#pragma unroll
    for (int i = 0; i < NB; ++i)
      pair_twiddle<LG, C2R, S>(v + i * R, a, ((tid + i * Cfg::T) % LR) & (NS - 1));
  }
#pragma unroll
  for (int i = 0; i < NB; ++i) dft_fwd<R>(v + i * R);
  if constexpr (LASTG) {
#pragma unroll
    for (int i = 0; i < NB; ++i) {
      const int b = tid + i * Cfg::T, c = b / LR, j = b % LR;
      if (col0 + c < a.ncols) {
        float2* p = gout + c * a.out_sc + j;
#pragma unroll
        for (int q = 0; q < R; ++q) __stcs(p + q * NS, make_float2(v[i * R + q].x * a.sx, v[i * R + q].y * a.sy));
      }
    }
  } else {
    if constexpr (S > 0) __syncthreads();
#pragma unroll
    for (int i = 0; i < NB; ++i) {
      const int b = tid + i * Cfg::T, c = b / LR, j = b % LR;
      float2* p = sm + c * Cfg::LP + pidx(((j >> LGNS) << (LGNS + LGR)) + (j & (NS - 1)));
#pragma unroll
      for (int q = 0; q < R; ++q) p[pidx_c(q * NS)] = v[i * R + q];
    }
    __syncthreads();
  }
}

// Rows of L complex values in (in_sc), rows of X[0..L] out (out_sc); scale_out:
// X[1..L-1] times sx, X[0] and X[L] times sy.
template <int LG, int C>
__global__ void __launch_bounds__(PairCfg<LG, C>::T, 512 / PairCfg<LG, C>::T) pair_r2c_kernel(const TileArgs a) {
  using Cfg = PairCfg<LG, C>;
  extern __shared__ float2 smem[];
  const long long col0 = (long long)blockIdx.x * C;
  const float2* gin = a.in + (long long)blockIdx.x * a.in_gstride;
  float2* gout = a.out + (long long)blockIdx.x * a.out_gstride;
  pair_pass<LG, C, false, 0, false>(smem, a, gin, nullptr, col0);
  if constexpr (Cfg::NST == 3) pair_pass<LG, C, false, 1, false>(smem, a, nullptr, nullptr, col0);

  constexpr int S = Cfg::NST - 1, R = 16, NS = Cfg::L / R, TR = Cfg::L / 32;
  static_assert(pair_lgr(LG, false, S) == 4, "radix-16 last pass");
  const int c = threadIdx.x / TR, p = threadIdx.x % TR;
  const int j1 = p ? NS - p : NS / 2;
  float2 v0[R], v1[R];
  {
    const float2* s0 = smem + c * Cfg::LP + pidx(p);
    const float2* s1 = smem + c * Cfg::LP + pidx(j1);
#pragma unroll
    for (int r = 0; r < R; ++r) {
      v0[r] = s0[pidx_c(r * NS)];
      v1[r] = s1[pidx_c(r * NS)];
    }
  }
  pair_twiddle<LG, false, S>(v0, a, p);
  pair_twiddle<LG, false, S>(v1, a, j1);
  dft_fwd<R>(v0);
  dft_fwd<R>(v1);
  if (col0 + c >= a.ncols) return;
  float2* row = gout + c * a.out_sc;
  const float sx = a.scale_out ? a.sx : 1.f;
  if (p == 0) {
    const float sy = a.scale_out ? a.sy : 1.f;
    __stcs(row, make_float2((v0[0].x + v0[0].y) * sy, 0.f));
    __stcs(row + Cfg::L, make_float2((v0[0].x - v0[0].y) * sy, 0.f));
  }
  // Pair q is Z[k] and Z[L-k]: k = p + q NS with butterfly 1's output 15 - q; for
  // p = 0, pairs 1..8 lie in butterfly 0 (k = q NS) and the others in butterfly 1
  // (k = NS/2 + {0, 1..7} NS).
#pragma unroll
  for (int q = 0; q < R; ++q) {
    const int k = q * NS + (p ? p : q == 0 ? NS / 2 : q <= 8 ? 0 : NS / 2 - 8 * NS);
    const float2 zk = p || (q >= 1 && q <= 8) ? v0[q] : v1[q == 0 ? 0 : (q + 8) & 15];
    const float2 zm = p || q == 0 ? v1[15 - q] : q <= 8 ? v0[(16 - q) & 15] : v1[(23 - q) & 15];
    const float2 e = make_float2(0.5f * (zk.x + zm.x), 0.5f * (zk.y - zm.y));
    const float2 o = make_float2(0.5f * (zk.y + zm.y), -0.5f * (zk.x - zm.x));
    const float2 wo = cmul(__ldg(a.r_w + k), o);
    __stcs(row + k, make_float2((e.x + wo.x) * sx, (e.y + wo.y) * sx));
    __stcs(row + Cfg::L - k, make_float2((e.x - wo.x) * sx, (wo.y - e.y) * sx));
  }
}

// Rows of X[0..L] in (in_sc), rows of L complex values out (out_sc), times sx
// and sy (the transform runs on conj Z).
template <int LG, int C>
__global__ void __launch_bounds__(PairCfg<LG, C>::T, 512 / PairCfg<LG, C>::T) pair_c2r_kernel(const TileArgs a) {
  using Cfg = PairCfg<LG, C>;
  extern __shared__ float2 smem[];
  const long long col0 = (long long)blockIdx.x * C;
  const float2* gin = a.in + (long long)blockIdx.x * a.in_gstride;
  float2* gout = a.out + (long long)blockIdx.x * a.out_gstride;

  constexpr int R = 1 << pair_lgr(LG, true, 0), LR = Cfg::L / R, NP = 16 / R;   // pairs of butterflies a thread
#pragma unroll
  for (int i = 0; i < NP; ++i) {
    const int b = threadIdx.x + i * Cfg::T, c = b / (LR / 2), p = b % (LR / 2);
    const bool ok = col0 + c < a.ncols;
    const float2* row = gin + c * a.in_sc;
    // Pair r is X[n] and X[L-n]: n = p + r LR with butterfly 1's input R - 1 - r;
    // for p = 0, pairs 1..R/2 lie in butterfly 0 and the others in butterfly 1.
    float2 x1[R], x2[R], w[R];
#pragma unroll
    for (int r = 0; r < R; ++r) {
      const int n = r * LR + (p ? p : r == 0 ? LR / 2 : r <= R / 2 ? 0 : LR / 2 - (R / 2) * LR);
      x1[r] = ok ? __ldcs(row + n) : make_float2(0.f, 0.f);
      x2[r] = ok ? __ldcs(row + Cfg::L - n) : make_float2(0.f, 0.f);
      w[r] = __ldg(a.r_w + n);
    }
    float2 z0 = make_float2(0.f, 0.f);   // conj Z[0] (Im X[0] and Im X[L] do not enter)
    if (p == 0 && ok) {
      const float em = (float)(1 + a.r_end2), f = row[0].x * em, g = row[Cfg::L].x * em;
      z0 = make_float2(0.5f * (f + g), -0.5f * (f - g));
    }
#pragma unroll
    for (int r = 0; r < R; ++r) {
      const float2 e = make_float2(0.5f * (x1[r].x + x2[r].x), 0.5f * (x1[r].y - x2[r].y));
      const float2 d = make_float2(0.5f * (x1[r].x - x2[r].x), 0.5f * (x1[r].y + x2[r].y));
      const float2 o = cmul(d, make_float2(w[r].x, -w[r].y));
      x1[r] = make_float2(e.x - o.y, -(e.y + o.x));   // conj Z[n]
      x2[r] = make_float2(e.x + o.y, e.y - o.x);      // conj Z[L-n]
    }
    float2 v0[R], v1[R];
#pragma unroll
    for (int r = 0; r < R; ++r) {
      v0[r] = p || (r >= 1 && r <= R / 2) ? x1[r] : r == 0 ? z0 : x2[R - r];
      v1[r] = p || r == R - 1 ? x2[R - 1 - r] : r < R / 2 ? x1[r == 0 ? 0 : R / 2 + r] : x2[(R / 2 + R - 1 - r) % R];
    }
    dft_fwd<R>(v0);
    dft_fwd<R>(v1);
    // (Ns = 1: output q of butterfly j is element j R + q)
    const int j1 = p ? LR - p : LR / 2;
    float2* s0 = smem + c * Cfg::LP + pidx(p * R);
    float2* s1 = smem + c * Cfg::LP + pidx(j1 * R);
#pragma unroll
    for (int q = 0; q < R; ++q) {
      s0[q] = v0[q];
      s1[q] = v1[q];
    }
  }
  __syncthreads();
  if constexpr (Cfg::NST == 3) pair_pass<LG, C, true, 1, false>(smem, a, nullptr, nullptr, col0);
  pair_pass<LG, C, true, Cfg::NST - 1, true>(smem, a, nullptr, gout, col0);
}

}  // namespace gbfft
