// mixr.cuh -- the FP32 mixed-radix tile kernel: C sub-transforms of any
// 7-smooth length N on chip, radices chosen at plan time from the register
// radices {2,3,4,5,7,8,9,10,12,14,15,16,20,21,24,25}.
//
// Every pass is the Stockham recurrence of Sec. 2.1's split (natural order in
// and out): butterfly j of a pass with radix R and Ns = the product of the
// earlier radices
//   v[r] = a[j + r N/R] * W_{Ns R}^{r (j mod Ns)},  V = R-point DFT of v,
//   b[(j div Ns) Ns R + (j mod Ns) + q Ns] = V[q].
// What bounds it is instruction issue and the latency of the exchanges, not
// HBM, so the design keeps both down:
//   * few passes: a radix of up to 25 points is itself a Cooley-Tukey split in
//     registers, so almost every N <= 14336 takes two or three passes;
//   * one shared-memory buffer, not two: a middle pass holds all of a thread's
//     butterflies (at most K(R) of them) in registers between its reads and its
//     writes, so a tile costs 8 bytes a point and several CTAs share an SM;
//   * the first pass reads global memory and needs no twiddle, the last writes
//     global memory; each role is its own code, only the radix is switched on;
//   * every twiddle of a pass is an entry of a dense table of Ns columns
//     (coalesced: lanes hold consecutive k), right to half a unit.  Products of
//     up to four entries of a basis w^(2^e) are as many instructions but rounded
//     as often: the largest errors of the transform (9000 points: 1.41e-7 by
//     products, 1.34e-7 so, 1.37e-7 with the small radices before).  Two to a
//     16-byte load: against products 0.8 % more time on average over 130 lengths
//     (8-byte loads 1.6 %: 1000 107 us instead of 102, 9000 146 instead of 144), 5
//     at most (9720, whose tile leaves little L1).
// Measured on GB300 per 2^25 points, against one pass per prime factor or
// radix-16 block with two buffers (216 instructions a point and one CTA per SM
// at N = 9000): 100 173 -> 91 us, 1080 246 -> 114, 7000 340 -> 142, 9000 393 ->
// 144, 14336 362 -> 205; two passes: 15000 338 -> 207 (1117 of them: 175 -> 112),
// 10^6 427 -> 282; images of 1000^2 342 -> 252.  (One read and one write of 2^25 points take 79 us.)
// STR = false: contiguous transforms, element n of transform c at c N + n, in
// memory and in the tile.  STR = true: C = 2^csh columns, element n of column c
// at c cs + n ns in memory and n pitch + c in the tile, lanes along columns;
// when the input columns are contiguous rows (in_rows), the first pass takes
// lanes along the row instead, and an odd pitch keeps its writes apart.
// PAD adds one entry (row) every 16 for first passes of even radix, whose
// stride-R writes would share banks; odd radices need none.
#pragma once
#include <cuda_runtime.h>

#include "gbfft_internal.h"
#include "mixed_ct.cuh"

namespace gbfft {

// middle-pass butterflies a thread may hold: as many as fit KP points
template <int R, int KP>
struct MixrK {
  static constexpr int value = KP / R > 0 ? KP / R : 1;
};

// v[r] *= w^r: pairs (w^{2p+1}, w^{2p+2}) of column k at entry p Ns + k of
// 16-byte entries, then the last w^r of an even R at one of 8.
template <int R>
__device__ __forceinline__ void mixr_twiddles(float2* v, const float2* tw, int Ns, int k) {
  float2 w[R + 1];
  const float4* t = (const float4*)tw + k;
#pragma unroll
  for (int p = 0; p < (R - 1) / 2; ++p) {
    const float4 q = __ldg(t + p * Ns);
    w[2 * p + 1] = make_float2(q.x, q.y);
    w[2 * p + 2] = make_float2(q.z, q.w);
  }
  if constexpr (R % 2 == 0) w[R - 1] = __ldg(tw + (R - 2) * Ns + k);
#pragma unroll
  for (int r = 1; r < R; ++r) v[r] = cmul(v[r], w[r]);
}

template <bool STR, bool PAD>
struct MixrTile {
  const MixrArgs& a;
  float2* sm;
  const float2* gin;
  float2* gout;
  unsigned col0;   // first column of the tile (STR: of its batch)
  int valid;       // columns of the tile that exist

  // butterfly b -> (column, index j)
  __device__ __forceinline__ void split(int b, int s, int& c, int& j) const {
    if (STR && (s > 0 || !a.in_rows)) {
      c = b & ((1 << a.csh) - 1);
      j = b >> a.csh;
    } else {
      c = (int)fdiv((unsigned)b, a.nb_m[s]);
      j = b - c * (int)a.nb[s];
    }
  }
  // tile position of row n of column c
  __device__ __forceinline__ int at(int c, int n) const {
    if constexpr (STR)
      return msidx<PAD>(n) * a.pitch + c;
    else
      return msidx<PAD>(c * a.N + n);
  }

  template <int R>
  __device__ __forceinline__ void load_global(float2* v, int c, int j, int NB) const {
    const bool ok = c < valid;
    if constexpr (STR) {
      const unsigned o = (unsigned)c * a.in_cs + (unsigned)j * a.in_ns, st = (unsigned)NB * a.in_ns;
#pragma unroll
      for (int r = 0; r < R; ++r) v[r] = ok ? __ldcs(gin + (o + r * st)) : make_float2(0.f, 0.f);
    } else {
      const float2* p = gin + (c * a.N + j);
#pragma unroll
      for (int r = 0; r < R; ++r) v[r] = ok ? __ldcs(p + r * NB) : make_float2(0.f, 0.f);
    }
    if (a.conj_in) {
#pragma unroll
      for (int r = 0; r < R; ++r) v[r].y = -v[r].y;
    }
  }

  template <int R>
  __device__ __forceinline__ void load_tile(float2* v, int c, int j, int NB) const {
    if constexpr (PAD) {
#pragma unroll
      for (int r = 0; r < R; ++r) v[r] = sm[at(c, j + r * NB)];
    } else {
      const float2* p = sm + at(c, j);
      const int st = STR ? NB * a.pitch : NB;
#pragma unroll
      for (int r = 0; r < R; ++r) v[r] = p[r * st];
    }
  }

  template <int R>
  __device__ __forceinline__ void store_tile(const float2* v, int c, int m0, int Ns) const {
    if constexpr (PAD) {
#pragma unroll
      for (int q = 0; q < R; ++q) sm[at(c, m0 + q * Ns)] = v[q];
    } else {
      float2* p = sm + at(c, m0);
      const int st = STR ? Ns * a.pitch : Ns;
#pragma unroll
      for (int q = 0; q < R; ++q) p[q * st] = v[q];
    }
  }

  // outputs k0 + q Ns of column c
  template <int R>
  __device__ __forceinline__ void store_global(float2* v, int c, int k0, int Ns) const {
    if (c >= valid) return;
    if constexpr (STR) {
      if (a.ft) {   // four-step twiddle W_Nt^{col k}: one table row per output index k
        const float2* f = a.ft + (size_t)(unsigned)k0 * a.ft_cols + (col0 + c);
        const size_t fs = (size_t)(unsigned)Ns * a.ft_cols;
#pragma unroll
        for (int q = 0; q < R; ++q) v[q] = cmul(v[q], __ldg(f + q * fs));
      } else if (a.ft_lo) {   // the same from two table levels
        const unsigned col = col0 + (unsigned)c;
        const unsigned mask = (1u << a.ft_s) - 1u;
        unsigned e = col * (unsigned)k0;
        const unsigned es = col * (unsigned)Ns;
#pragma unroll
        for (int q = 0; q < R; ++q) {
          v[q] = cmul(v[q], cmul(__ldg(a.ft_lo + (e & mask)), __ldg(a.ft_hi + (e >> a.ft_s))));
          e += es;
        }
      }
    }
    if (a.scale_out) {
#pragma unroll
      for (int q = 0; q < R; ++q) v[q] = make_float2(v[q].x * a.sx, v[q].y * a.sy);
    }
    if constexpr (STR) {
      const unsigned o = (unsigned)c * a.out_cs + (unsigned)k0 * a.out_ns, st = (unsigned)Ns * a.out_ns;
#pragma unroll
      for (int q = 0; q < R; ++q) __stcs(gout + (o + q * st), v[q]);
    } else {
      float2* p = gout + (c * a.N + k0);
#pragma unroll
      for (int q = 0; q < R; ++q) __stcs(p + q * Ns, v[q]);
    }
  }

  template <int R>
  __device__ __forceinline__ void first() const {
    const int NB = (int)a.nb[0], total = a.C * NB;
    for (int b = threadIdx.x; b < total; b += blockDim.x) {
      int c, j;
      split(b, 0, c, j);
      float2 v[R];
      load_global<R>(v, c, j, NB);
      ct_dft<R>(v);
      store_tile<R>(v, c, j * R, 1);
    }
  }

  // in place: every butterfly's inputs are read before any output is written
  template <int R, int K>
  __device__ __forceinline__ void middle(int s) const {
    const int NB = (int)a.nb[s], Ns = (int)a.ns[s], total = a.C * NB;
    float2 v[K][R];
#pragma unroll
    for (int i = 0; i < K; ++i) {
      const int b = threadIdx.x + i * blockDim.x;
      if (b < total) {
        int c, j;
        split(b, s, c, j);
        load_tile<R>(v[i], c, j, NB);
      } else {   // (defined on every path, so that nothing lives across the pass loop)
#pragma unroll
        for (int r = 0; r < R; ++r) v[i][r] = make_float2(0.f, 0.f);
      }
    }
    __syncthreads();
#pragma unroll
    for (int i = 0; i < K; ++i) {
      const int b = threadIdx.x + i * blockDim.x;
      if (b < total) {
        int c, j;
        split(b, s, c, j);
        const int jq = (int)fdiv((unsigned)j, a.ns_m[s]);
        const int k = j - jq * Ns;
        mixr_twiddles<R>(v[i], a.tw + a.tw_off[s], Ns, k);
        ct_dft<R>(v[i]);
        store_tile<R>(v[i], c, jq * Ns * R + k, Ns);
      }
    }
  }

  template <int R>
  __device__ __forceinline__ void last(int s) const {
    const int NB = (int)a.nb[s], total = a.C * NB;   // Ns == NB
    for (int b = threadIdx.x; b < total; b += blockDim.x) {
      int c, j;
      split(b, s, c, j);
      float2 v[R];
      load_tile<R>(v, c, j, NB);
      mixr_twiddles<R>(v, a.tw + a.tw_off[s], NB, j);
      ct_dft<R>(v);
      store_global<R>(v, c, j, NB);
    }
  }

  // N is a single radix
  template <int R>
  __device__ __forceinline__ void only() const {
    for (int b = threadIdx.x; b < a.C; b += blockDim.x) {
      float2 v[R];
      load_global<R>(v, b, 0, 1);
      ct_dft<R>(v);
      store_global<R>(v, b, 0, 1);
    }
  }
};

#define GBFFT_MIXR_SWITCH(r, CALL) \
  switch (r) {                     \
    case 2: CALL(2); break;        \
    case 3: CALL(3); break;        \
    case 4: CALL(4); break;        \
    case 5: CALL(5); break;        \
    case 7: CALL(7); break;        \
    case 8: CALL(8); break;        \
    case 9: CALL(9); break;        \
    case 10: CALL(10); break;      \
    case 12: CALL(12); break;      \
    case 14: CALL(14); break;      \
    case 15: CALL(15); break;      \
    case 16: CALL(16); break;      \
    case 20: CALL(20); break;      \
    case 21: CALL(21); break;      \
    case 24: CALL(24); break;      \
    default: CALL(25); break;      \
  }

template <bool STR, bool PAD, int KP>
__device__ __forceinline__ void mixr_tile(const MixrArgs& a, float2* sm) {
  const long long t = a.tile0 + blockIdx.x;
  const float2* gin;
  float2* gout;
  unsigned col0;
  int valid;
  if constexpr (STR) {
    const long long bt = t / a.tiles_per_batch;
    const long long c0 = (t - bt * a.tiles_per_batch) << a.csh;
    col0 = (unsigned)c0;
    valid = (int)(a.ncols - c0 < a.C ? a.ncols - c0 : a.C);
    gin = a.in + bt * a.in_bs + c0 * a.in_cs;
    gout = a.out + bt * a.out_bs + c0 * a.out_cs;
  } else {
    const long long c0 = t * a.C;
    col0 = 0;
    valid = (int)(a.ncols - c0 < a.C ? a.ncols - c0 : a.C);
    gin = a.in + c0 * a.N;
    gout = a.out + c0 * a.N;
  }
  const MixrTile<STR, PAD> T{a, sm, gin, gout, col0, valid};
  const int last = a.nrad - 1;
  if (last == 0) {
#define CALL(R) T.template only<R>()
    GBFFT_MIXR_SWITCH(a.rad[0], CALL)
#undef CALL
    return;
  }
#define CALL(R) T.template first<R>()
  GBFFT_MIXR_SWITCH(a.rad[0], CALL)
#undef CALL
  __syncthreads();
  for (int s = 1; s < last; ++s) {
#define CALL(R) T.template middle<R, MixrK<R, KP>::value>(s)
    GBFFT_MIXR_SWITCH(a.rad[s], CALL)
#undef CALL
    __syncthreads();
  }
#define CALL(R) T.template last<R>(last)
  GBFFT_MIXR_SWITCH(a.rad[last], CALL)
#undef CALL
}

// Two shapes of CTA.  Up to 384 threads of 80 registers, so that two CTAs of
// 384, three of 256 or six of 128 share an SM; middle passes hold up to 25
// points a thread.  Up to 512 threads of 128 registers for tiles of more than
// 9600 points (one CTA per SM); middle passes hold up to 32 points.
template <bool STR, bool PAD>
__global__ void __launch_bounds__(384, 2) mixr_kernel(const MixrArgs a) {
  extern __shared__ __align__(16) unsigned char mixr_smem[];
  mixr_tile<STR, PAD, 25>(a, (float2*)mixr_smem);
}
template <bool STR, bool PAD>
__global__ void __launch_bounds__(512, 1) mixr_big_kernel(const MixrArgs a) {
  extern __shared__ __align__(16) unsigned char mixr_smem[];
  mixr_tile<STR, PAD, 32>(a, (float2*)mixr_smem);
}

}  // namespace gbfft
