// fx64.cu -- plans and launches of the FP64 tile kernel (fx64.cuh); the choice
// of schedule, columns and threads is in mixr_plan.h.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstring>

#include "gbfft_internal.h"
#include "mixr_plan.h"

namespace gbfft {

using namespace mixr;

// contiguous transforms (0_) or strided columns (1_), any pad (_0) or evenly spaced (_1);
// only: N is a single radix
const void* fx_fn_0_0(bool only);
const void* fx_fn_0_1(bool only);
const void* fx_fn_1_0(bool only);
const void* fx_fn_1_1(bool only);

static unsigned recip(unsigned d) { return d == 1 ? 0u : (unsigned)((0x100000000ULL + d - 1) / d); }

// Entries of the plan's tables: the twiddles of every pass after the first,
// then W_N^m for FP64 arithmetic.
size_t fx_table_entries(const FxArgs& a) {
  size_t n = (size_t)a.N;
  for (int s = 1; s < a.nrad; ++s) n += (size_t)(a.rad[s] - 1) * a.ns[s];
  return n;
}

int fx_fill_tables(FxLaunch& L, int4* tab, cudaStream_t s) {
  FxArgs& a = L.a;
  a.tw = tab;
  for (int i = 1; i < a.nrad; ++i)
    if (launch_gen_fx_twiddles(tab + a.tw_off[i], a.rad[i], (int)a.ns[i], s) != cudaSuccess) return FFT_ERR_CUDA;
  a.wn = (const double2*)(tab + fx_table_entries(a) - a.N);
  return launch_gen_twiddles_step((void*)a.wn, true, a.N, a.N, 1, s) == cudaSuccess ? FFT_OK : FFT_ERR_CUDA;
}

// Fills L for `batches` batches of ncols sub-transforms of length N
// (contiguous when lay is NULL: then batches must be 1).
int fx_init(FxLaunch& L, long long N, long long ncols, long long batches, const MixrLayout* lay) {
  memset(&L, 0, sizeof(L));
  const Family& f = family_fx();
  const bool strided = lay != nullptr, in_rows = lay && lay->in_ns == 1 && lay->in_cs != 1;
  Choice best;
  const int rc = choose(f, best, N, ncols, ncols * batches, strided, in_rows);
  if (rc) return rc;
  FxArgs& a = L.a;
  a.N = (int)N;
  a.C = best.C;
  a.nrad = best.q.n;
  unsigned ns = 1, off = 0;
  for (int s = 0; s < a.nrad; ++s) {
    const int r = best.q.rad[s];
    a.rad[s] = r;
    a.head[s] = fx_headroom(r);
    a.nb[s] = (unsigned)(N / r);
    a.nb_m[s] = recip(a.nb[s]);
    a.ns[s] = ns;
    a.ns_m[s] = recip(ns);
    a.tw_off[s] = off;
    if (s > 0) off += (unsigned)(r - 1) * ns;
    ns *= (unsigned)r;
  }
  a.ncols = ncols;
  const bool pad = needs_pad(f, a.rad[0], strided, in_rows, a.C);
  a.pad_sh = pad ? 4 : 31;
  if (lay) {
    while ((1 << a.csh) < a.C) ++a.csh;
    a.in_rows = in_rows;
    a.pitch = in_rows ? a.C + 1 : a.C;
    a.in_bs = lay->in_bs;
    a.out_bs = lay->out_bs;
    a.in_cs = (unsigned)lay->in_cs;
    a.in_ns = (unsigned)lay->in_ns;
    a.out_cs = (unsigned)lay->out_cs;
    a.out_ns = (unsigned)lay->out_ns;
    a.tiles_per_batch = (ncols + a.C - 1) / a.C;
    L.ntiles = a.tiles_per_batch * batches;
  } else {
    L.ntiles = (ncols + a.C - 1) / a.C;
  }
  if (a.nrad > 1) {
    a.slot_off = (int)tile_bytes(f, N, a.C, strided, in_rows, pad);
    L.smem = a.slot_off + f.slot_bytes * a.nrad * a.C;
  }
  // whether a pad entry every 16 leaves every butterfly's elements evenly
  // spaced: steps that are multiples of 16, or all R within one block of 16
  bool lin = true;
  const int unit = lay ? a.pitch : 1;
  for (int s = 0; s < a.nrad; ++s) {
    const int nb = (int)a.nb[s], n1 = (int)a.ns[s], r = a.rad[s];
    if (pad && s > 0) lin = lin && nb % 16 == 0;
    if (pad && s + 1 < a.nrad) lin = lin && (n1 % 16 == 0 || 16 % (n1 * r) == 0);
    a.ld_st[s] = (nb + (pad ? nb >> 4 : 0)) * unit;
    a.st_st[s] = (n1 + (pad ? n1 >> 4 : 0)) * unit;
  }
  L.threads = best.T;
  const bool only = a.nrad == 1;
  L.fn = lay ? (lin ? fx_fn_1_1(only) : fx_fn_1_0(only)) : (lin ? fx_fn_0_1(only) : fx_fn_0_0(only));
  if (L.smem > 48 * 1024 &&
      cudaFuncSetAttribute(L.fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmemLimit) != cudaSuccess)
    return FFT_ERR_CUDA;
  return FFT_OK;
}

int fx_launch(const FxLaunch& L, const double2* in, double2* out, int conj_in, int conj_out, double scale,
              cudaStream_t s) {
  FxArgs a = L.a;
  a.in = in;
  a.out = out;
  a.conj_in = conj_in;
  a.conj_out = conj_out;
  a.scale = scale;
  int e = 0;
  const double m = std::frexp(scale, &e);   // scale = m 2^e, m in [0.5, 1)
  if (m == 0.5) {
    a.scale_ex = e - 1;
  } else {
    a.scale_q = q62_split(4 * ((long long)std::ldexp(m, 62) - (1LL << 62)));   // x m = x + x (m - 1)
    a.scale_ex = e;
  }
  for (long long t = 0; t < L.ntiles; t += 1LL << 30) {   // (grids hold at most 2^31 - 1 CTAs)
    a.tile0 = t;
    const unsigned grid = (unsigned)std::min(L.ntiles - t, 1LL << 30);
    void* args[] = {(void*)&a};
    if (cudaLaunchKernel(L.fn, dim3(grid), dim3(L.threads), args, (size_t)L.smem, s) != cudaSuccess)
      return FFT_ERR_CUDA;
  }
  return FFT_OK;
}

}  // namespace gbfft
