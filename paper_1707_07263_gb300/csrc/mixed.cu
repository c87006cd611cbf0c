// mixed.cu -- plans of one on-chip pass per transform for lengths that are a
// product N = 2^a 3^b 5^c 7^d: FP32 lengths that are not powers of two
// (N <= 14336; kernels in mixr.cuh and mixed_ct.cu), and every FP64
// (complex128) length N <= 7168, powers of two included (fx64.cuh).
//
// Eq. 1 holds for any N; the paper's Cooley-Tukey split (Sec. 2.1) works for
// any factorisation N = R_1 R_2 ... R_s.
#include <cuda_runtime.h>

#include <algorithm>

#include "gbfft_internal.h"

namespace gbfft {

// The compiled schedules' tile: transforms per CTA, buffers, W_N table.
static int mixed_ct_plan(fft_plan* p) {
  MixedArgs& a = p->mixed;
  const MixedCtInfo* k = p->mixed_ct;
  a.N = (int)p->n;
  a.C = (int)std::min<long long>(k->C, p->batch);
  a.batch = p->batch;
  const size_t pts = (size_t)a.C * (size_t)p->n;
  p->mixed_smem = (int)(2 * (k->pad ? pts + ((pts - 1) >> 4) + 1 : pts) * 8);
  if (p->mixed_smem > 48 * 1024 &&
      cudaFuncSetAttribute(k->fn, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024) != cudaSuccess)
    return FFT_ERR_CUDA;
  return FFT_OK;
}

int mixed_plan_init(fft_plan* p) {
  const bool fp64 = p->prec == FFT_PREC_FP64;
  const long long N = p->n;
  if (N > (fp64 ? kMixedMaxN64 : kMixedMaxN)) return FFT_ERR_UNSUPPORTED;
  p->mixed_ct = fp64 ? nullptr : mixed_ct_lookup(N);
  int rc;
  size_t tw_bytes;
  if (p->mixed_ct) {
    rc = mixed_ct_plan(p);
    tw_bytes = (size_t)N * 8;
  } else if (fp64) {
    rc = fx_init(p->fx[0], N, p->batch, 1, nullptr);
    tw_bytes = fx_table_entries(p->fx[0].a) * 16;
  } else {
    rc = mixr_init(p->mr[0], N, p->batch, 1, nullptr);
    tw_bytes = mixr_table_entries(p->mr[0].a) * 8;
  }
  if (rc) return rc;
  tw_bytes = (tw_bytes + 255) & ~(size_t)255;
  if (cudaMalloc(&p->d_tables, tw_bytes + 256) != cudaSuccess) return FFT_ERR_ALLOC;
  p->d_status = (int*)((char*)p->d_tables + tw_bytes);
  if (cudaMemset(p->d_status, 0, sizeof(int)) != cudaSuccess) return FFT_ERR_CUDA;
  if (p->mixed_ct) {
    p->mixed.tw = p->d_tables;
    rc = launch_gen_twiddles_step(p->d_tables, false, N, N, 1, 0) == cudaSuccess ? FFT_OK : FFT_ERR_CUDA;
  } else {
    rc = fp64 ? fx_fill_tables(p->fx[0], (int4*)p->d_tables, 0) : mixr_fill_tables(p->mr[0], (float2*)p->d_tables, 0);
  }
  if (rc) return rc;
  if (cudaStreamSynchronize(0) != cudaSuccess) return FFT_ERR_CUDA;
  p->launches = 1;
  return FFT_OK;
}

int mixed_exec(fft_plan* p, const void* in, void* out, int conj, double sx, double sy, int scale_out,
               cudaStream_t s) {
  // in == out is safe: a tile's first pass reads all of it (into shared
  // memory, or into one thread's registers when N is a single radix) before
  // its last pass writes
  if (p->prec == FFT_PREC_FP64) return fx_launch(p->fx[0], (const double2*)in, (double2*)out, conj, sy < 0, sx, s);
  if (!p->mixed_ct)
    return mixr_launch(p->mr[0], (const float2*)in, (float2*)out, conj, (float)sx, (float)sy, scale_out, s);
  MixedArgs a = p->mixed;
  a.in = in;
  a.out = out;
  a.conj_in = conj;
  a.scale_out = scale_out;
  a.fsx = (float)sx;
  a.fsy = (float)sy;
  const long long tiles = (p->batch + a.C - 1) / a.C;
  if (tiles > 0x7fffffffLL) return FFT_ERR_UNSUPPORTED;
  void* args[] = {(void*)&a};
  return cudaLaunchKernel(p->mixed_ct->fn, dim3((unsigned)tiles), dim3(p->mixed_ct->threads), args,
                          (size_t)p->mixed_smem, s) == cudaSuccess
             ? FFT_OK
             : FFT_ERR_CUDA;
}

}  // namespace gbfft
