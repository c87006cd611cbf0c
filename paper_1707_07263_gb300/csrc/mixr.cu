// mixr.cu -- plans and launches of the FP32 mixed-radix tile kernel (mixr.cuh);
// the choice of schedule, columns and threads is in mixr_plan.h.
#include <cuda_runtime.h>

#include <algorithm>
#include <cstring>

#include "gbfft_internal.h"
#include "mixr_plan.h"

namespace gbfft {

using namespace mixr;

const void* mixr_fn_contig_0(bool big);
const void* mixr_fn_contig_1(bool big);
const void* mixr_fn_strided_0(bool big);
const void* mixr_fn_strided_1(bool big);

namespace {

const void* mixr_fn(bool strided, bool pad, bool big) {
  if (strided) return pad ? mixr_fn_strided_1(big) : mixr_fn_strided_0(big);
  return pad ? mixr_fn_contig_1(big) : mixr_fn_contig_0(big);
}

unsigned recip(unsigned d) { return d == 1 ? 0u : (unsigned)((0x100000000ULL + d - 1) / d); }

}  // namespace

// Entries of the twiddle tables of every pass after the first (16-byte aligned).
size_t mixr_table_entries(const MixrArgs& a) {
  size_t n = 0;
  for (int s = 1; s < a.nrad; ++s) n = ((n + 1) & ~(size_t)1) + (size_t)(a.rad[s] - 1) * a.ns[s];
  return n;
}

int mixr_fill_tables(MixrLaunch& L, float2* tab, cudaStream_t s) {
  L.a.tw = tab;
  for (int i = 1; i < L.a.nrad; ++i)
    if (launch_gen_mixr_twiddles(tab + L.a.tw_off[i], L.a.rad[i], (int)L.a.ns[i], s) != cudaSuccess)
      return FFT_ERR_CUDA;
  return FFT_OK;
}

// Fills L for `batches` batches of ncols sub-transforms of length N
// (contiguous when lay is NULL: then batches must be 1).
int mixr_init(MixrLaunch& L, long long N, long long ncols, long long batches, const MixrLayout* lay) {
  memset(&L, 0, sizeof(L));
  const bool strided = lay != nullptr, in_rows = lay && lay->in_ns == 1 && lay->in_cs != 1;
  Choice best;
  const Family& f = family_f32();
  const int rc = choose(f, best, N, ncols, ncols * batches, strided, in_rows);
  if (rc) return rc;
  const int* rad = best.q.rad;
  MixrArgs& a = L.a;
  a.N = (int)N;
  a.C = best.C;
  a.nrad = best.q.n;
  unsigned ns = 1, off = 0;
  for (int s = 0; s < a.nrad; ++s) {
    a.rad[s] = rad[s];
    a.nb[s] = (unsigned)(N / rad[s]);
    a.nb_m[s] = recip(a.nb[s]);
    a.ns[s] = ns;
    a.ns_m[s] = recip(ns);
    off = (off + 1) & ~1u;   // 16-byte pairs
    a.tw_off[s] = off;
    if (s > 0) off += (unsigned)(rad[s] - 1) * ns;
    ns *= (unsigned)rad[s];
  }
  a.ncols = ncols;
  const bool pad = needs_pad(f, rad[0], strided, in_rows, best.C);
  if (lay) {
    while ((1 << a.csh) < best.C) ++a.csh;
    a.in_rows = in_rows;
    a.pitch = in_rows ? best.C + 1 : best.C;
    a.in_bs = lay->in_bs;
    a.out_bs = lay->out_bs;
    a.in_cs = (unsigned)lay->in_cs;
    a.in_ns = (unsigned)lay->in_ns;
    a.out_cs = (unsigned)lay->out_cs;
    a.out_ns = (unsigned)lay->out_ns;
    a.tiles_per_batch = (ncols + best.C - 1) / best.C;
    L.ntiles = a.tiles_per_batch * batches;
  } else {
    L.ntiles = (ncols + best.C - 1) / best.C;
  }
  L.smem = a.nrad > 1 ? (int)tile_bytes(f, N, best.C, strided, in_rows, pad) : 0;
  L.threads = best.T;
  L.fn = mixr_fn(lay != nullptr, pad, best.big);
  if (L.smem > 48 * 1024 &&
      cudaFuncSetAttribute(L.fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmemLimit) != cudaSuccess)
    return FFT_ERR_CUDA;
  return FFT_OK;
}

int mixr_launch(const MixrLaunch& L, const float2* in, float2* out, int conj, float sx, float sy, int scale_out,
                cudaStream_t s) {
  MixrArgs a = L.a;
  a.in = in;
  a.out = out;
  a.conj_in = conj;
  a.scale_out = scale_out;
  a.sx = sx;
  a.sy = sy;
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
