// mixed_ct.cu -- mixed-radix transforms (FP32) with everything fixed at
// compile time -- length, radices, every divisor -- for the common lengths
// where that still measures faster than the run-time schedules of mixr.cuh
// (per 2^25 points on GB300, this kernel against that one: 2000 109 against
// 112 us, 4000 113 against 125, 10000 172 against 185, 12000 168 against 177;
// the run-time kernel is faster at 1000, 1200, 1500, 2400, 3000, 5000, 6000
// and 8000).
//
// Three passes of composite register radices, two exchanges through two
// shared-memory buffers.
//
// Passes follow the Stockham recurrence of mixr.cuh (natural order in and
// out): butterfly j of a pass with radix R and Ns = the product of the
// earlier radices reads a[j + r N/R], multiplies by W_{Ns R}^{r (j mod Ns)}
// (powers of one W_N table entry), runs the R-point DFT and writes
// b[(j div Ns) Ns R + (j mod Ns) + q Ns].
#include <cuda_runtime.h>

#include "gbfft_internal.h"
#include "mixed_ct.cuh"

namespace gbfft {

// One pass over the tile's C transforms: radix R, Ns = NS.
template <int N, int R, int NS, bool PAD, bool FIRST, bool LAST>
__device__ __forceinline__ void ct_pass(const MixedArgs& a, const float2* src, float2* dst, long long col0) {
  constexpr int NB = N / R;
  constexpr int STRIDE = N / (NS * R);
  static_assert(N % (NS * R) == 0, "schedule");
  const float2* tw = (const float2*)a.tw;
  const int total = a.C * NB;
  for (int b = threadIdx.x; b < total; b += blockDim.x) {
    const int c = b / NB, j = b - c * NB;
    const bool ok = col0 + c < a.batch;
    float2 v[R];
    const int n0 = c * N + j;
#pragma unroll
    for (int r = 0; r < R; ++r) {
      if constexpr (FIRST)
        v[r] = ok ? __ldcs(src + n0 + r * NB) : make_float2(0.f, 0.f);
      else
        v[r] = src[msidx<PAD>(n0 + r * NB)];
    }
    if (FIRST && a.conj_in) {
#pragma unroll
      for (int r = 0; r < R; ++r) v[r].y = -v[r].y;
    }
    const int jq = j / NS, k = j - jq * NS;
    if constexpr (NS > 1) ct_twiddles<R>(v, tw, k * STRIDE);
    ct_dft<R>(v);
    const int m0 = c * N + jq * NS * R + k;
    if constexpr (LAST) {
      if (!ok) continue;
#pragma unroll
      for (int q = 0; q < R; ++q) {
        float2 y = v[q];
        if (a.scale_out) y = make_float2(y.x * a.fsx, y.y * a.fsy);
        __stcs(dst + m0 + q * NS, y);
      }
    } else {
#pragma unroll
      for (int q = 0; q < R; ++q) dst[msidx<PAD>(m0 + q * NS)] = v[q];
    }
  }
}

// The tile of C transforms: three passes R0, R1, R2 (in == out is safe: the
// first pass reads the whole tile into shared memory before the last writes).
template <int N, int R0, int R1, int R2, bool PAD, int THREADS>
__global__ void __launch_bounds__(THREADS, THREADS <= 256 ? 2 : 1) mixed_ct_kernel(const MixedArgs a) {
  static_assert(R0 * R1 * R2 == N, "schedule");
  extern __shared__ __align__(16) unsigned char ct_smem[];
  float2* const buf0 = (float2*)ct_smem;
  float2* const buf1 = buf0 + msidx<PAD>(a.C * N - 1) + 1;
  const long long col0 = (long long)blockIdx.x * a.C;
  const float2* in = (const float2*)a.in + col0 * N;
  float2* out = (float2*)a.out + col0 * N;
  ct_pass<N, R0, 1, PAD, true, false>(a, in, buf0, col0);
  __syncthreads();
  ct_pass<N, R1, R0, PAD, false, false>(a, buf0, buf1, col0);
  __syncthreads();
  ct_pass<N, R2, R0 * R1, PAD, false, true>(a, buf1, out, col0);
}

// Compiled schedules, each the fastest of the orders and factorisations
// measured on GB300 for its length, the transforms per CTA and the threads per
// CTA (512 where one CTA fills an SM's shared memory, 256 below, where two or
// three CTAs share an SM).  The padded layout where the first pass writes at
// an even stride.
#define GBFFT_CT(N, R0, R1, R2, C, T) \
  {N, R0, R1, R2, C, T, (R0 % 2 == 0), (const void*)&mixed_ct_kernel<N, R0, R1, R2, (R0 % 2 == 0), T>}

const MixedCtInfo* mixed_ct_lookup(long long N) {
  static const MixedCtInfo tab[] = {
      GBFFT_CT(2000, 25, 16, 5, 2, 256),
      GBFFT_CT(4000, 25, 16, 10, 1, 256),
      GBFFT_CT(10000, 25, 16, 25, 1, 512),
      GBFFT_CT(12000, 25, 24, 20, 1, 512),
  };
  for (const MixedCtInfo& t : tab)
    if (t.N == N) return &t;
  return nullptr;
}

}  // namespace gbfft
