// mixed4.cu -- plans of two mixed-radix passes (kernels: FP32 mixr.cuh, FP64
// fx64.cuh):
//  * 1-D lengths beyond one on-chip pass: FP64 (complex128) N > 7168 and FP32
//    7-smooth N > 14336 that are not powers of two.  Sec. 2.3.2's partition:
//    N = N1 N2, n = n1 N2 + n2, k = k1 + N1 k2,
//      column pass  Y[k1][n2] = W_N^{n2 k1} sum_{n1} x[n1 N2 + n2] W_N1^{n1 k1}
//      row pass     X[k1 + N1 k2] = sum_{n2} Y[k1][n2] W_N2^{n2 k2},
//    through a workspace of N complex values per transform (Y stored as
//    ws[k1 N2 + n2]).  Both lengths are one on-chip mixed-radix sub-transform.
//  * 2-D transforms in FP64, and in FP32 when a side is not a power of two:
//    the transforms of every row, then of every column (Sec. 2.3.2), in place
//    in the output.
#include <cuda_runtime.h>

#include <cstring>

#include "gbfft_internal.h"

namespace gbfft {

static size_t al256(size_t b) { return (b + 255) & ~(size_t)255; }

// Table bytes of the two passes, and their contents.
static void pass_tables(fft_plan* p, size_t& ba, size_t& bb) {
  const bool fp64 = p->prec == FFT_PREC_FP64;
  ba = al256(fp64 ? fx_table_entries(p->fx[0].a) * 16 : mixr_table_entries(p->mr[0].a) * 8);
  bb = al256(fp64 ? fx_table_entries(p->fx[1].a) * 16 : mixr_table_entries(p->mr[1].a) * 8);
}
static int fill_pass_tables(fft_plan* p, char* a, char* b) {
  if (p->prec == FFT_PREC_FP64) {
    const int rc = fx_fill_tables(p->fx[0], (int4*)a, 0);
    return rc ? rc : fx_fill_tables(p->fx[1], (int4*)b, 0);
  }
  const int rc = mixr_fill_tables(p->mr[0], (float2*)a, 0);
  return rc ? rc : mixr_fill_tables(p->mr[1], (float2*)b, 0);
}

// N = N1 N2 with the split of the least modelled cost.
int mixed4_plan_1d(fft_plan* p) {
  const bool fp64 = p->prec == FFT_PREC_FP64;
  const size_t esz = fp64 ? 16 : 8;
  const long long N = p->n;
  const long long n1 = mixr::choose_split(fp64 ? mixr::family_fx() : mixr::family_f32(), N, p->batch,
                                          fp64 ? kMixedMaxN64 : kMixedMaxN);
  if (n1 == 0) return FFT_ERR_UNSUPPORTED;
  const long long n2 = N / n1;
  // column pass: adjacent n2, the length-N1 transform over n1, times W_N^{n2 k1};
  // row pass: adjacent k1, the length-N2 transform over n2, to X[k1 + N1 k2]
  const MixrLayout la = {N, 1, n2, N, 1, n2}, lb = {N, n2, 1, N, 1, n1};
  int rc = fp64 ? fx_init(p->fx[0], n1, n2, p->batch, &la) : mixr_init(p->mr[0], n1, n2, p->batch, &la);
  if (!rc) rc = fp64 ? fx_init(p->fx[1], n2, n1, p->batch, &lb) : mixr_init(p->mr[1], n2, n1, p->batch, &lb);
  if (rc) return rc;
  p->kind = KIND_MIXED_PASSES;
  p->m4_n1 = n1;
  p->m4_n2 = n2;
  // the dense twiddle table of the column pass's outputs while it stays small
  // beside L2 (8 MB FP32, 4 MB FP64), else two levels
  const bool dense = N <= (fp64 ? 1LL << 18 : 1LL << 20);
  int s = 0;
  if (!dense) {
    int bits = 0;
    while ((1LL << bits) < N) ++bits;
    s = (bits + 1) / 2;
  }
  const long long nlo = dense ? N : 1LL << s, nhi = dense ? 0 : ((N - 1) >> s) + 1;
  size_t ba, bb;
  pass_tables(p, ba, bb);
  const size_t olo = ba + bb, ohi = olo + al256(nlo * esz), ost = ohi + al256(nhi * esz);
  if (cudaMalloc(&p->d_tables, ost + 256) != cudaSuccess) return FFT_ERR_ALLOC;
  char* base = (char*)p->d_tables;
  p->d_status = (int*)(base + ost);
  if (cudaMemset(p->d_status, 0, sizeof(int)) != cudaSuccess) return FFT_ERR_CUDA;
  rc = fill_pass_tables(p, base, base + ba);
  if (rc) return rc;
  cudaError_t e;
  if (fp64) {
    FxArgs& a = p->fx[0].a;
    (dense ? a.ft : a.ft_lo) = (const int4*)(base + olo);
    a.ft_hi = (const int4*)(base + ohi);
    a.ft_cols = (unsigned)n2;
    a.ft_s = s;
    e = dense ? launch_gen_fx_four_step((int4*)(base + olo), N, (int)n1, (int)n2, 0)
              : launch_gen_fx_power((int4*)(base + olo), N, nlo, 1, 0);
    if (e == cudaSuccess && !dense) e = launch_gen_fx_power((int4*)(base + ohi), N, nhi, nlo, 0);
  } else {
    MixrArgs& a = p->mr[0].a;
    (dense ? a.ft : a.ft_lo) = (const float2*)(base + olo);
    a.ft_hi = (const float2*)(base + ohi);
    a.ft_cols = (unsigned)n2;
    a.ft_s = s;
    e = dense ? launch_gen_four_step((float2*)(base + olo), N, (int)n1, (int)n2, 0)
              : launch_gen_twiddles_step(base + olo, false, N, nlo, 1, 0);
    if (e == cudaSuccess && !dense) e = launch_gen_twiddles_step(base + ohi, false, N, nhi, nlo, 0);
  }
  if (e != cudaSuccess || cudaStreamSynchronize(0) != cudaSuccess) return FFT_ERR_CUDA;
  p->ws_bytes = (size_t)N * (size_t)p->batch * esz;
  p->launches = 2;
  return FFT_OK;
}

// ny-by-nx images: contiguous rows (input -> output), then columns in place in
// the output.
int mixed4_plan_2d(fft_plan* p) {
  const bool fp64 = p->prec == FFT_PREC_FP64;
  const long long ny = p->ny, nx = p->nx, img = ny * nx;
  const MixrLayout lc = {img, 1, nx, img, 1, nx};
  int rc = fp64 ? fx_init(p->fx[0], nx, ny * p->batch, 1, nullptr) : mixr_init(p->mr[0], nx, ny * p->batch, 1, nullptr);
  if (!rc) rc = fp64 ? fx_init(p->fx[1], ny, nx, p->batch, &lc) : mixr_init(p->mr[1], ny, nx, p->batch, &lc);
  if (rc) return rc;
  p->kind = KIND_MIXED_PASSES;
  p->m4_n1 = ny;
  p->m4_n2 = nx;
  size_t ba, bb;
  pass_tables(p, ba, bb);
  if (cudaMalloc(&p->d_tables, ba + bb + 256) != cudaSuccess) return FFT_ERR_ALLOC;
  char* base = (char*)p->d_tables;
  p->d_status = (int*)(base + ba + bb);
  if (cudaMemset(p->d_status, 0, sizeof(int)) != cudaSuccess) return FFT_ERR_CUDA;
  rc = fill_pass_tables(p, base, base + ba);
  if (rc) return rc;
  if (cudaStreamSynchronize(0) != cudaSuccess) return FFT_ERR_CUDA;
  p->ws_bytes = 0;
  p->launches = 2;
  return FFT_OK;
}

int mixed4_exec(fft_plan* p, const void* in, void* out, int conj, double sx, double sy, int scale_out,
                cudaStream_t s) {
  const bool two_d = p->ws_bytes == 0;
  if (!two_d && !p->ws) return FFT_ERR_NO_WORKSPACE;
  void* mid = two_d ? out : p->ws;
  if (p->prec == FFT_PREC_FP64) {
    const int rc = fx_launch(p->fx[0], (const double2*)in, (double2*)mid, conj, 0, 1.0, s);
    return rc ? rc : fx_launch(p->fx[1], (const double2*)mid, (double2*)out, 0, sy < 0, sx, s);
  }
  const int rc = mixr_launch(p->mr[0], (const float2*)in, (float2*)mid, conj, 1.f, 1.f, 0, s);
  return rc ? rc : mixr_launch(p->mr[1], (const float2*)mid, (float2*)out, 0, (float)sx, (float)sy, scale_out, s);
}

}  // namespace gbfft
