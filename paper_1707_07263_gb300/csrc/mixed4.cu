// mixed4.cu -- plans of two mixed-radix passes (kernels: FP32 mixr.cuh, FP64
// mixed4.cuh):
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

#include <cmath>
#include <cstring>

#include "gbfft_internal.h"

namespace gbfft {

constexpr int kMixed4Threads = 256;
constexpr size_t kMixed4SmemLimit = 227 * 1024;

static size_t m4_smem(long long L, int csh, bool pad, size_t esz) {
  const size_t rows = pad ? (size_t)(L + ((L - 1) >> 4)) : (size_t)L;
  return 2 * rows * ((size_t)1 << csh) * esz;
}

// One FP64 pass: sub-length L, ncols columns in each of `batches` batches, element
// n of column col of batch b at b*bs + col*cs + n*ns on either side.  Columns
// per CTA: as many as make a tile of about 2048 points, at most 8 and at most ncols, fewer when the buffers do not fit.
static int m4_pass_init(fft_plan* p, Mixed4Pass& P, long long L, long long ncols, long long batches,
                        long long in_bs, long long in_cs, long long in_ns, long long out_bs, long long out_cs,
                        long long out_ns, const void* tw, int in_role, int out_role) {
  constexpr size_t esz = 16;
  memset(&P, 0, sizeof(P));
  Mixed4Args& a = P.a;
  if (!mixed_schedule(a.m, L)) return FFT_ERR_UNSUPPORTED;
  a.m.tw = tw;
  constexpr long long target = 2048;
  constexpr int csh_max = 3;
  int csh = 0;
  while (csh < csh_max && (L << (csh + 1)) <= target && (2LL << csh) <= ncols) ++csh;
  while (csh > 0 && m4_smem(L, csh, true, esz) > kMixed4SmemLimit) --csh;
  const bool pad = m4_smem(L, csh, true, esz) <= kMixed4SmemLimit;
  const size_t smem = m4_smem(L, csh, pad, esz);
  if (smem > kMixed4SmemLimit) return FFT_ERR_UNSUPPORTED;
  P.fn = mixed4_kernel_fn64(csh, pad);
  if (!P.fn) return FFT_ERR_UNSUPPORTED;
  // (the kernel's limit, which other plans share: always the largest)
  if (smem > 48 * 1024 &&
      cudaFuncSetAttribute(P.fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kMixed4SmemLimit) != cudaSuccess)
    return FFT_ERR_CUDA;
  const int C = 1 << csh;
  a.m.C = C;
  a.m.batch = batches;
  a.in_bs = in_bs;
  a.in_cs = in_cs;
  a.in_ns = in_ns;
  a.out_bs = out_bs;
  a.out_cs = out_cs;
  a.out_ns = out_ns;
  a.ncols = ncols;
  a.tiles_per_batch = (ncols + C - 1) / C;
  a.ntiles = a.tiles_per_batch * batches;
  int per_sm = 0, sms = 0, dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
      cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, P.fn, kMixed4Threads, smem) != cudaSuccess ||
      per_sm < 1)
    return FFT_ERR_CUDA;
  const long long resident = (long long)per_sm * sms;
  P.grid = a.ntiles < resident ? a.ntiles : resident;
  P.threads = kMixed4Threads;
  P.smem = (int)smem;
  P.in_role = in_role;
  P.out_role = out_role;
  return FFT_OK;
}

static size_t al256(size_t b) { return (b + 255) & ~(size_t)255; }

// The twiddle tables of an FP64 plan in one allocation: W_La^m (m < La), W_Lb^m
// (m < Lb; shared when La == Lb), and for a four-step plan the two levels
// of W_N^e, e < N: lo[i] = W_N^i (i < 2^s), hi[j] = W_N^{j 2^s}; then the
// status word.  Entries are FP64 sincospi values.
struct M4Tables {
  const void *wa, *wb, *lo, *hi;
  int s;
};
static int m4_tables(fft_plan* p, long long La, long long Lb, long long Nft, M4Tables* t) {
  constexpr size_t esz = 16;
  int s = 0;
  long long nlo = 0, nhi = 0;
  if (Nft > 0) {
    int bits = 0;
    while ((1LL << bits) < Nft) ++bits;
    s = (bits + 1) / 2;
    nlo = 1LL << s;
    nhi = ((Nft - 1) >> s) + 1;
  }
  const size_t oa = 0, ob = al256(La * esz);
  const size_t olo = ob + (Lb == La ? 0 : al256(Lb * esz));
  const size_t ohi = olo + al256(nlo * esz);
  const size_t ost = ohi + al256(nhi * esz);
  if (cudaMalloc(&p->d_tables, ost + 256) != cudaSuccess) return FFT_ERR_ALLOC;
  char* base = (char*)p->d_tables;
  t->wa = base + oa;
  t->wb = Lb == La ? t->wa : (const void*)(base + ob);
  t->lo = Nft > 0 ? base + olo : nullptr;
  t->hi = Nft > 0 ? base + ohi : nullptr;
  t->s = s;
  p->d_status = (int*)(base + ost);
  cudaError_t e = launch_gen_twiddles_step(base + oa, true, La, La, 1, 0);
  if (e == cudaSuccess && Lb != La) e = launch_gen_twiddles_step(base + ob, true, Lb, Lb, 1, 0);
  if (e == cudaSuccess && Nft > 0) e = launch_gen_twiddles_step(base + olo, true, Nft, nlo, 1, 0);
  if (e == cudaSuccess && Nft > 0) e = launch_gen_twiddles_step(base + ohi, true, Nft, nhi, nlo, 0);
  if (e != cudaSuccess || cudaMemset(p->d_status, 0, sizeof(int)) != cudaSuccess ||
      cudaStreamSynchronize(0) != cudaSuccess)
    return FFT_ERR_CUDA;
  return FFT_OK;
}

// FP32: N = N1 N2 with the split of the least modelled cost, both passes on
// the tile kernel of mixr.cuh.
static int mixr_plan_1d(fft_plan* p) {
  const long long N = p->n;
  long long b1 = 0;
  float best = 0;
  // factors within 8 : 1 of each other unless there are none
  for (int wide = 0; wide < 2 && b1 == 0; ++wide) {
    for (long long d = 2; d * d <= N; ++d) {
      if (N % d || N / d > kMixedMaxN || (!wide && N / d > 8 * d)) continue;
      for (const long long n1 : {d, N / d}) {
        const float ca = mixr_strided_cost(n1, N / n1, p->batch, false);
        const float cb = mixr_strided_cost(N / n1, n1, p->batch, true);
        if (ca < 0 || cb < 0) continue;
        if (b1 == 0 || ca + cb < best) {
          b1 = n1;
          best = ca + cb;
        }
      }
    }
  }
  if (b1 == 0) return FFT_ERR_UNSUPPORTED;
  const long long n2 = N / b1;
  const MixrLayout la = {N, 1, n2, N, 1, n2}, lb = {N, n2, 1, N, 1, b1};
  int rc = mixr_init(p->mr[0], b1, n2, p->batch, &la);
  if (!rc) rc = mixr_init(p->mr[1], n2, b1, p->batch, &lb);
  if (rc) return rc;
  p->kind = KIND_MIXED_PASSES;
  p->m4_n1 = b1;
  p->m4_n2 = N / b1;
  // the dense twiddle table of the column pass's outputs while it stays small
  // beside L2, else two levels
  const bool dense = N <= (1LL << 20);
  int s = 0;
  if (!dense) {
    int bits = 0;
    while ((1LL << bits) < N) ++bits;
    s = (bits + 1) / 2;
  }
  const long long nlo = dense ? N : 1LL << s, nhi = dense ? 0 : ((N - 1) >> s) + 1;
  const size_t ob = al256(mixr_table_entries(p->mr[0].a) * 8);
  const size_t olo = ob + al256(mixr_table_entries(p->mr[1].a) * 8);
  const size_t ohi = olo + al256(nlo * 8), ost = ohi + al256(nhi * 8);
  if (cudaMalloc(&p->d_tables, ost + 256) != cudaSuccess) return FFT_ERR_ALLOC;
  char* base = (char*)p->d_tables;
  p->d_status = (int*)(base + ost);
  if (cudaMemset(p->d_status, 0, sizeof(int)) != cudaSuccess) return FFT_ERR_CUDA;
  rc = mixr_fill_tables(p->mr[0], (float2*)base, 0);
  if (!rc) rc = mixr_fill_tables(p->mr[1], (float2*)(base + ob), 0);
  if (rc) return rc;
  MixrArgs& a = p->mr[0].a;
  cudaError_t e;
  if (dense) {
    a.ft = (const float2*)(base + olo);
    a.ft_cols = (unsigned)p->m4_n2;
    e = launch_gen_four_step((float2*)(base + olo), N, (int)b1, (int)p->m4_n2, 0);
  } else {
    a.ft_lo = (const float2*)(base + olo);
    a.ft_hi = (const float2*)(base + ohi);
    a.ft_s = s;
    e = launch_gen_twiddles_step(base + olo, false, N, nlo, 1, 0);
    if (e == cudaSuccess) e = launch_gen_twiddles_step(base + ohi, false, N, nhi, nlo, 0);
  }
  if (e != cudaSuccess || cudaStreamSynchronize(0) != cudaSuccess) return FFT_ERR_CUDA;
  p->ws_bytes = (size_t)N * (size_t)p->batch * 8;
  p->launches = 2;
  return FFT_OK;
}

// FP32 images: contiguous rows, then columns in place in the output.
static int mixr_plan_2d(fft_plan* p) {
  const long long ny = p->ny, nx = p->nx, img = ny * nx;
  const MixrLayout lc = {img, 1, nx, img, 1, nx};
  int rc = mixr_init(p->mr[0], nx, ny * p->batch, 1, nullptr);
  if (!rc) rc = mixr_init(p->mr[1], ny, nx, p->batch, &lc);
  if (rc) return rc;
  p->kind = KIND_MIXED_PASSES;
  p->m4_n1 = ny;
  p->m4_n2 = nx;
  const size_t ob = al256(mixr_table_entries(p->mr[0].a) * 8), ost = ob + al256(mixr_table_entries(p->mr[1].a) * 8);
  if (cudaMalloc(&p->d_tables, ost + 256) != cudaSuccess) return FFT_ERR_ALLOC;
  char* base = (char*)p->d_tables;
  p->d_status = (int*)(base + ost);
  if (cudaMemset(p->d_status, 0, sizeof(int)) != cudaSuccess) return FFT_ERR_CUDA;
  rc = mixr_fill_tables(p->mr[0], (float2*)base, 0);
  if (!rc) rc = mixr_fill_tables(p->mr[1], (float2*)(base + ob), 0);
  if (rc) return rc;
  if (cudaStreamSynchronize(0) != cudaSuccess) return FFT_ERR_CUDA;
  p->ws_bytes = 0;
  p->launches = 2;
  return FFT_OK;
}

// FP64: N = N1 N2 with N1 the largest divisor of N at most sqrt(N) whose
// cofactor is one on-chip sub-transform.
int mixed4_plan_1d(fft_plan* p) {
  if (p->prec == FFT_PREC_FP32) return mixr_plan_1d(p);
  const long long N = p->n;
  long long n1 = 0;
  long long d = (long long)std::sqrt((double)N) + 1;
  while (d * d > N) --d;
  for (; d >= 2 && n1 == 0; --d)
    if (N % d == 0 && N / d <= kMixedMaxN64) n1 = d;
  if (n1 == 0) return FFT_ERR_UNSUPPORTED;
  const long long n2 = N / n1;
  M4Tables t;
  int rc = m4_tables(p, n1, n2, N, &t);
  if (rc) return rc;
  p->kind = KIND_MIXED_PASSES;
  p->m4_n1 = n1;
  p->m4_n2 = n2;
  p->m4n = 2;
  // column pass: C adjacent n2, the length-N1 transform over n1, times W_N^{n2 k1}
  rc = m4_pass_init(p, p->m4[0], n1, n2, p->batch, N, 1, n2, N, 1, n2, t.wa, 0, 2);
  if (rc) return rc;
  p->m4[0].a.ft_lo = t.lo;
  p->m4[0].a.ft_hi = t.hi;
  p->m4[0].a.ft_s = t.s;
  // row pass: C adjacent k1, the length-N2 transform over n2, to X[k1 + N1 k2]
  rc = m4_pass_init(p, p->m4[1], n2, n1, p->batch, N, n2, 1, N, 1, n1, t.wb, 2, 1);
  if (rc) return rc;
  p->ws_bytes = (size_t)N * (size_t)p->batch * 16;
  p->launches = 2;
  return FFT_OK;
}

// ny-by-nx images: row transforms (input -> output), then column transforms in
// place in the output.
int mixed4_plan_2d(fft_plan* p) {
  if (p->prec == FFT_PREC_FP32) return mixr_plan_2d(p);
  const long long ny = p->ny, nx = p->nx, img = ny * nx;
  M4Tables t;
  int rc = m4_tables(p, nx, ny, 0, &t);
  if (rc) return rc;
  p->kind = KIND_MIXED_PASSES;
  p->m4_n1 = ny;
  p->m4_n2 = nx;
  p->m4n = 2;
  rc = m4_pass_init(p, p->m4[0], nx, ny, p->batch, img, nx, 1, img, nx, 1, t.wa, 0, 1);
  if (rc) return rc;
  rc = m4_pass_init(p, p->m4[1], ny, nx, p->batch, img, 1, nx, img, 1, nx, t.wb, 1, 1);
  if (rc) return rc;
  p->ws_bytes = 0;
  p->launches = 2;
  return FFT_OK;
}

int mixed4_exec(fft_plan* p, const void* in, void* out, int conj, double sx, double sy, int scale_out,
                cudaStream_t s) {
  if (p->prec == FFT_PREC_FP32) {
    const bool two_d = p->ws_bytes == 0;
    if (!two_d && !p->ws) return FFT_ERR_NO_WORKSPACE;
    float2* mid = two_d ? (float2*)out : (float2*)p->ws;
    const int rc = mixr_launch(p->mr[0], (const float2*)in, mid, conj, 1.f, 1.f, 0, s);
    if (rc) return rc;
    return mixr_launch(p->mr[1], mid, (float2*)out, 0, (float)sx, (float)sy, scale_out, s);
  }
  void* bufs[3] = {(void*)in, out, p->ws};
  for (int i = 0; i < p->m4n; ++i)
    if ((p->m4[i].in_role == 2 || p->m4[i].out_role == 2) && !p->ws) return FFT_ERR_NO_WORKSPACE;
  for (int i = 0; i < p->m4n; ++i) {
    const Mixed4Pass& P = p->m4[i];
    Mixed4Args a = P.a;
    a.m.in = bufs[P.in_role];
    a.m.out = bufs[P.out_role];
    a.m.conj_in = i == 0 ? conj : 0;
    a.m.scale_out = i == p->m4n - 1 ? scale_out : 0;
    a.m.sx = sx;
    a.m.sy = sy;
    a.m.fsx = (float)sx;
    a.m.fsy = (float)sy;
    if (P.grid < 1 || P.grid > 0x7fffffffLL) return FFT_ERR_UNSUPPORTED;
    void* args[] = {(void*)&a};
    if (cudaLaunchKernel(P.fn, dim3((unsigned)P.grid), dim3(P.threads), args, (size_t)P.smem, s) != cudaSuccess)
      return FFT_ERR_CUDA;
  }
  return FFT_OK;
}

}  // namespace gbfft
