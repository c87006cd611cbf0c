// mixed.cu -- transforms of one on-chip pass whose length is a product
// N = 2^a 3^b 5^c 7^d: plans of FP32 lengths that are not powers of two
// (N <= 14336; kernels in mixr.cuh and mixed_ct.cu), and the FP64 (complex128)
// kernel for every such N <= 7168, powers of two included.
//
// Eq. 1 holds for any N; the paper's Cooley-Tukey split (Sec. 2.1) works for
// any factorisation N = R_1 R_2 ... R_s.  The FP64 kernel runs the same Stockham
// autosort recurrence as the power-of-two tiles (natural order in and out),
// with the radix of every pass chosen at run time from {16, 8, 4, 2, 3, 5, 7}:
//   pass with radix R, Ns = product of the earlier radices, butterfly j:
//     v[r] = a[j + r N/R] * W_{Ns R}^{r (j mod Ns)},   r = 0..R-1
//     V    = R-point DFT of v
//     b[(j div Ns) Ns R + (j mod Ns) + q Ns] = V[q].
// The first pass reads global memory, the last writes it; the passes in
// between go through two shared-memory buffers in turn.  Twiddles come from
// one table W_N^m, m < N (FP64 sincospi), since
// W_{Ns R}^{r k} = W_N^{r k N / (Ns R)}.
#include <cuda_runtime.h>

#include <algorithm>

#include "gbfft_internal.h"
#include "mixed_common.cuh"

namespace gbfft {

// One pass s over the tile: C transforms of length N at src (global when
// FIRST, else shared memory), written to dst (global when LAST).
template <int R, bool PAD>
__device__ __forceinline__ void mixed_pass(const MixedArgs& a, int s, const double2* src, double2* dst, bool first,
                                           bool last, long long col0) {
  using T = double2;
  const T* tw = (const T*)a.tw;
  const int N = a.N;
  const unsigned NB = a.nb[s], nbm = a.nb_m[s], Ns = a.ns[s], nsm = a.ns_m[s];
  const int total = a.C * (int)NB;
  const int stride = (int)a.tws[s];
  for (int b = threadIdx.x; b < total; b += blockDim.x) {
    const int c = (int)fdiv((unsigned)b, nbm), j = b - c * (int)NB;
    const bool ok = col0 + c < a.batch;
    T v[R];
    const int n0 = c * N + j;   // tile index of input r = 0
#pragma unroll
    for (int r = 0; r < R; ++r) {
      if (first)
        v[r] = ok ? __ldcs(src + n0 + r * NB) : Cx<T>::make(0, 0);
      else
        v[r] = src[msidx<PAD>(n0 + r * (int)NB)];
    }
    if (first && a.conj_in) {
#pragma unroll
      for (int r = 0; r < R; ++r) v[r].y = -v[r].y;
    }
    const int jq = (int)fdiv((unsigned)j, nsm);
    const int k = j - jq * (int)Ns;
    if (Ns > 1) mixed_twiddles<R>(v, tw, k * stride);
    dft_any<R>(v);
    const int m0 = c * N + jq * (int)Ns * R + k;   // tile index of output q = 0
    if (last) {
      if (!ok) continue;
#pragma unroll
      for (int q = 0; q < R; ++q) {
        T y = v[q];
        if (a.scale_out) y = Cx<T>::make(y.x * a.sx, y.y * a.sy);
        __stcs(dst + m0 + q * (int)Ns, y);
      }
    } else {
#pragma unroll
      for (int q = 0; q < R; ++q) dst[msidx<PAD>(m0 + q * (int)Ns)] = v[q];
    }
  }
}

template <bool PAD>
__device__ __forceinline__ void mixed_tile(const MixedArgs& a, double2* smem) {
  using T = double2;
  const long long tile = blockIdx.x;
  const long long col0 = tile * a.C;
  const long long off = col0 * a.N;
  const T* in = (const T*)a.in + off;
  T* out = (T*)a.out + off;
  T* const buf1 = smem + msidx<PAD>(a.C * a.N - 1) + 1;
  for (int s = 0; s < a.nrad; ++s) {
    const bool first = s == 0, last = s == a.nrad - 1;
    const T* src = first ? in : ((s & 1) ? smem : buf1);
    T* dst = last ? out : ((s & 1) ? buf1 : smem);
    switch (a.rad[s]) {
      case 2: mixed_pass<2, PAD>(a, s, src, dst, first, last, col0); break;
      case 3: mixed_pass<3, PAD>(a, s, src, dst, first, last, col0); break;
      case 4: mixed_pass<4, PAD>(a, s, src, dst, first, last, col0); break;
      case 5: mixed_pass<5, PAD>(a, s, src, dst, first, last, col0); break;
      case 7: mixed_pass<7, PAD>(a, s, src, dst, first, last, col0); break;
      case 8: mixed_pass<8, PAD>(a, s, src, dst, first, last, col0); break;
      default: mixed_pass<16, PAD>(a, s, src, dst, first, last, col0); break;
    }
    __syncthreads();
  }
}

template <bool PAD>
__global__ void __launch_bounds__(512, 1) mixed_kernel64(const MixedArgs a) {
  extern __shared__ __align__(16) unsigned char mixed_smem[];
  mixed_tile<PAD>(a, (double2*)mixed_smem);
}

static const void* mixed_fn(bool pad) {
  return pad ? (const void*)mixed_kernel64<true> : (const void*)mixed_kernel64<false>;
}

// Radix schedule: radix-16 passes for 2^a and one 8/4/2 pass for the rest of
// 2^a first, then the 3s, 5s and 7s.  The first pass (Ns = 1) needs no
// twiddles, so it gets the largest radix.  (A bank model prefers the
// power-of-two radices last -- their first-pass writes at stride 8 or 16
// conflict -- but measured on GB300 that order is 10-25 % slower: the
// twiddle loads and products of a radix-16 pass cost more than the
// conflicts.)  Returns the number of passes, 0 if N has another prime factor
// or needs more than kMixedMaxPasses passes.
int mixed_radices(long long N, int* rad) {
  int n = 0;
  long long m = N;
  int a = 0;
  while (m % 2 == 0) {
    m /= 2;
    ++a;
  }
  while (a >= 4 && n < kMixedMaxPasses) {
    rad[n++] = 16;
    a -= 4;
  }
  if (a > 0 && n < kMixedMaxPasses) rad[n++] = 1 << a;
  const int odd[3] = {3, 5, 7};
  for (int i = 0; i < 3; ++i)
    while (m % odd[i] == 0 && n < kMixedMaxPasses) {
      m /= odd[i];
      rad[n++] = odd[i];
    }
  return (m == 1) ? n : 0;
}

// The pass schedule of length N into a: radices, N/R and Ns per pass with
// their reciprocals, and the twiddle strides into the W_N table.  Returns
// false when N is not 7-smooth or needs too many passes.
bool mixed_schedule(MixedArgs& a, long long N) {
  a.nrad = mixed_radices(N, a.rad);
  if (a.nrad == 0 || N > kMixedMaxN) return false;
  a.N = (int)N;
  unsigned ns = 1;
  for (int s = 0; s < a.nrad; ++s) {
    const unsigned nb = (unsigned)(N / a.rad[s]);
    a.nb[s] = nb;
    a.nb_m[s] = nb == 1 ? 0u : (unsigned)((0x100000000ULL + nb - 1) / nb);
    a.ns[s] = ns;
    a.ns_m[s] = ns == 1 ? 0u : (unsigned)((0x100000000ULL + ns - 1) / ns);
    ns *= (unsigned)a.rad[s];
    a.tws[s] = (unsigned)(N / ns);
  }
  return true;
}

// FP32: the tile kernel of mixr.cuh.
static int mixr_plan_one_pass(fft_plan* p) {
  MixrLaunch& L = p->mr[0];
  int rc = mixr_init(L, p->n, p->batch, 1, nullptr);
  if (rc) return rc;
  const size_t tw_bytes = (mixr_table_entries(L.a) * 8 + 255) & ~(size_t)255;
  if (cudaMalloc(&p->d_tables, tw_bytes + 256) != cudaSuccess) return FFT_ERR_ALLOC;
  p->d_status = (int*)((char*)p->d_tables + tw_bytes);
  if (cudaMemset(p->d_status, 0, sizeof(int)) != cudaSuccess) return FFT_ERR_CUDA;
  rc = mixr_fill_tables(L, (float2*)p->d_tables, 0);
  if (rc) return rc;
  if (cudaStreamSynchronize(0) != cudaSuccess) return FFT_ERR_CUDA;
  p->launches = 1;
  return FFT_OK;
}

int mixed_plan_init(fft_plan* p) {
  MixedArgs& a = p->mixed;
  const long long N = p->n;
  const bool fp64 = p->prec == FFT_PREC_FP64;
  p->mixed_ct = fp64 ? nullptr : mixed_ct_lookup(N);
  if (!fp64 && !p->mixed_ct) return mixr_plan_one_pass(p);
  const size_t esz = fp64 ? 16 : 8;
  constexpr long long tile = 2048;   // points per CTA when several FP64 transforms share one
  if (!mixed_schedule(a, N) || N > (fp64 ? kMixedMaxN64 : kMixedMaxN)) return FFT_ERR_UNSUPPORTED;
  a.C = p->mixed_ct ? p->mixed_ct->C : N <= tile ? (int)(tile / N) : 1;
  if (a.C > p->batch) a.C = (int)p->batch;
  a.batch = p->batch;
  p->mixed_threads = p->mixed_ct ? p->mixed_ct->threads : a.C * N <= tile ? 256 : 512;
  // padding pays when a radix-8 or -16 pass leads (its writes are strided by
  // the radix) and the padded buffers fit; pure odd-radix lengths keep the
  // unpadded layout
  const size_t pts = (size_t)a.C * (size_t)N;
  const size_t padded = pts + ((pts - 1) >> 4) + 1;
  p->mixed_pad = p->mixed_ct ? p->mixed_ct->pad : (a.rad[0] >= 8 && 2 * padded * esz <= 227 * 1024);
  p->mixed_smem = (int)(2 * (p->mixed_pad ? padded : pts) * esz);
  if (p->mixed_smem > 227 * 1024) return FFT_ERR_UNSUPPORTED;
  const void* fn = p->mixed_ct ? p->mixed_ct->fn : mixed_fn(p->mixed_pad);
  // the limit is a property of the kernel, which plans of other lengths share:
  // always the largest, or a later plan would lower it under an earlier one
  if (p->mixed_smem > 48 * 1024 &&
      cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024) != cudaSuccess)
    return FFT_ERR_UNSUPPORTED;
  const size_t tw_bytes = ((size_t)N * esz + 255) & ~(size_t)255;
  if (cudaMalloc(&p->d_tables, tw_bytes + 256) != cudaSuccess) return FFT_ERR_ALLOC;
  a.tw = p->d_tables;
  p->d_status = (int*)((char*)p->d_tables + tw_bytes);
  const cudaError_t e = fp64 ? launch_gen_twiddles_n64((double2*)p->d_tables, N, N, 0)
                             : launch_gen_twiddles_n((float2*)p->d_tables, N, N, 0);
  if (cudaMemset(p->d_status, 0, sizeof(int)) != cudaSuccess || e != cudaSuccess ||
      cudaStreamSynchronize(0) != cudaSuccess)
    return FFT_ERR_CUDA;
  p->launches = 1;
  return FFT_OK;
}

int mixed_exec(fft_plan* p, const void* in, void* out, int conj, double sx, double sy, int scale_out,
               cudaStream_t s) {
  // in == out is safe: a tile's first pass reads all of it (into shared
  // memory, or into one thread's registers when N is a single radix) before
  // its last pass writes
  if (p->prec == FFT_PREC_FP32 && !p->mixed_ct)
    return mixr_launch(p->mr[0], (const float2*)in, (float2*)out, conj, (float)sx, (float)sy, scale_out, s);
  MixedArgs a = p->mixed;
  a.in = in;
  a.out = out;
  a.conj_in = conj;
  a.scale_out = scale_out;
  a.sx = sx;
  a.sy = sy;
  a.fsx = (float)sx;
  a.fsy = (float)sy;
  const long long tiles = (p->batch + a.C - 1) / a.C;
  if (tiles > 0x7fffffffLL) return FFT_ERR_UNSUPPORTED;
  void* args[] = {(void*)&a};
  const void* fn = p->mixed_ct ? p->mixed_ct->fn : mixed_fn(p->mixed_pad);
  return cudaLaunchKernel(fn, dim3((unsigned)tiles), dim3(p->mixed_threads), args, (size_t)p->mixed_smem, s) ==
                 cudaSuccess
             ? FFT_OK
             : FFT_ERR_CUDA;
}

}  // namespace gbfft
