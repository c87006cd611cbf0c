// gbfft_internal.h -- plan representation shared by the host-side planner and
// the kernel launchers.  Not part of the public ABI.
#pragma once
#include <cuda_runtime.h>
#include <stddef.h>
#include <stdint.h>

#include <mutex>

#include "../../include/gbfft.h"
#include "fx64_math.h"
#include "mixr_plan.h"
#include "tile_fft.cuh"

namespace gbfft {

struct TileKernelInfo;
struct ManyPlan;
struct FusedPlan;

// One launch of a multi-pass plan.  Buffers are named by role so a plan can
// run on any (in, out) pair: 0 = the caller's input, 1 = the caller's output,
// 2 = the workspace.  conj-in is applied by the first pass, the output
// scale / conj by the last.
struct PassDesc {
  const TileKernelInfo* k;
  TileArgs a;
  int in_role, out_role;
  long long ntiles;
  const TileKernelInfo* kcol;  // tensor-TMA variant of a column pass (or NULL)
  int col_grid;                // its resident-CTA grid
  const TileKernelInfo* kst;   // row pass with a tensor-TMA output store (or NULL)
  const TileKernelInfo* kpfs;  // contiguous one-pass rows: the persistent staged kernel (or NULL)
  long long pf_grid;           // its resident-CTA grid
};
constexpr int kMaxPasses = 4;

enum PlanKind {
  KIND_SINGLE = 0,
  KIND_FOURSTEP = 1,
  KIND_2D = 2,
  KIND_MANY = 3,
  KIND_REAL = 4,
  KIND_MIXED = 5,
  KIND_MIXED_PASSES = 6   // strided mixed-radix passes: four-step 1-D or 2-D (mixed4.cu)
};

// Lengths N = 2^a 3^b 5^c 7^d (mixed.cu, mixed4.cu): the largest of one on-chip pass.
constexpr long long kMixedMaxN = 14336;
constexpr long long kMixedMaxN64 = 7168;
// One launch of a compiled schedule (mixed_ct.cu).
struct MixedArgs {
  const void* in;
  void* out;
  const void* tw;     // W_N^m, m < N
  int N, C;           // length; transforms per CTA
  long long batch;
  int conj_in, scale_out;
  float fsx, fsy;     // output scale
};
// One launch of the FP32 mixed-radix tile kernel (mixr.cuh).
struct MixrArgs {
  const float2* in;
  float2* out;
  const float2* tw;            // twiddles of every pass, pass s at tw_off[s] (mixr_twiddles)
  int N, C;                    // length; columns per CTA
  int csh, pitch, in_rows;     // strided tiles: C == 2^csh, tile row pitch, input columns are contiguous rows
  int nrad;
  int rad[mixr::kMaxPasses];
  unsigned nb[mixr::kMaxPasses], nb_m[mixr::kMaxPasses];   // N/R and its reciprocal (fdiv)
  unsigned ns[mixr::kMaxPasses], ns_m[mixr::kMaxPasses];   // Ns and its reciprocal
  unsigned tw_off[mixr::kMaxPasses];
  long long ncols;             // columns (strided: per batch)
  long long tile0;             // first tile of the launch
  // strided tiles: element (column c, row n) of batch b at b*bs + c*cs + n*ns
  long long tiles_per_batch, in_bs, out_bs;
  unsigned in_cs, in_ns, out_cs, out_ns;
  // four-step twiddle W_Nt^{col k} of output k: dense table ft[k * ft_cols + col], or two
  // levels ft_lo[e & (2^ft_s - 1)] * ft_hi[e >> ft_s], e = col k < Nt < 2^32, or none
  const float2* ft;
  unsigned ft_cols;
  const float2* ft_lo;
  const float2* ft_hi;
  int ft_s;
  int conj_in, scale_out;
  float sx, sy;
};
struct MixrLaunch {
  MixrArgs a;
  const void* fn;
  int threads, smem;
  long long ntiles;
};
// Strided layout of a pass: batches of ncols columns.
struct MixrLayout {
  long long in_bs, in_cs, in_ns, out_bs, out_cs, out_ns;
};
size_t mixr_table_entries(const MixrArgs& a);
int mixr_init(MixrLaunch& L, long long N, long long ncols, long long batches, const MixrLayout* lay);
int mixr_fill_tables(MixrLaunch& L, float2* tab, cudaStream_t s);
int mixr_launch(const MixrLaunch& L, const float2* in, float2* out, int conj, float sx, float sy, int scale_out,
                cudaStream_t s);
cudaError_t launch_gen_mixr_twiddles(float2* tab, int R, int Ns, cudaStream_t s);
cudaError_t launch_gen_four_step(float2* tab, long long N, int n1, int n2, cudaStream_t s);

// One launch of the FP64 tile kernel (fx64.cuh), laid out as MixrArgs.
struct FxArgs {
  const double2* in;
  double2* out;
  const int4* tw;              // Q62 twiddles of every pass, pass s at tw_off[s]: (r - 1) Ns + k
  const double2* wn;           // W_N^m, m < N (transforms in FP64 arithmetic)
  int N, C;
  int csh, pitch, in_rows;
  int pad_sh, slot_off;        // one pad entry every 2^pad_sh; byte offset of the exponent slots
  int nrad;
  int rad[mixr::kMaxPasses], head[mixr::kMaxPasses];   // radix and its headroom bits
  unsigned nb[mixr::kMaxPasses], nb_m[mixr::kMaxPasses];
  unsigned ns[mixr::kMaxPasses], ns_m[mixr::kMaxPasses];
  int ld_st[mixr::kMaxPasses], st_st[mixr::kMaxPasses];   // tile strides of a butterfly's inputs and outputs
  unsigned tw_off[mixr::kMaxPasses];
  long long ncols;
  long long tile0;
  long long tiles_per_batch, in_bs, out_bs;
  unsigned in_cs, in_ns, out_cs, out_ns;
  const int4* ft;              // four-step twiddles, dense or in two levels
  unsigned ft_cols;
  const int4* ft_lo;
  const int4* ft_hi;
  int ft_s;
  int conj_in, conj_out;
  // output scale: times 2^scale_ex, and scale_q (times 1/4) unless it is a power of two
  int scale_ex;
  Q62 scale_q;
  double scale;                // the same in FP64
};
struct FxLaunch {
  FxArgs a;
  const void* fn;
  int threads, smem;
  long long ntiles;
};
size_t fx_table_entries(const FxArgs& a);
int fx_init(FxLaunch& L, long long N, long long ncols, long long batches, const MixrLayout* lay);
int fx_fill_tables(FxLaunch& L, int4* tab, cudaStream_t s);
int fx_launch(const FxLaunch& L, const double2* in, double2* out, int conj_in, int conj_out, double scale,
              cudaStream_t s);
cudaError_t launch_gen_fx_twiddles(int4* tab, int R, int Ns, cudaStream_t s);
cudaError_t launch_gen_fx_power(int4* tab, long long N, long long count, long long step, cudaStream_t s);
cudaError_t launch_gen_fx_four_step(int4* tab, long long N, int n1, int n2, cudaStream_t s);

// Mixed-radix lengths with a compile-time three-pass schedule (mixed_ct.cu).
struct MixedCtInfo {
  long long N;
  int r0, r1, r2;
  int C;           // transforms per CTA
  int threads;     // threads per CTA
  bool pad;        // padded shared-memory index (msidx)
  const void* fn;  // kernel void(MixedArgs)
};
const MixedCtInfo* mixed_ct_lookup(long long N);

int mixed_plan_init(fft_plan* p);
int mixed4_plan_1d(fft_plan* p);
int mixed4_plan_2d(fft_plan* p);
int mixed4_exec(fft_plan* p, const void* in, void* out, int conj, double sx, double sy, int scale_out,
                cudaStream_t s);
cudaError_t launch_gen_twiddles_step(void* tab, bool fp64, long long N, long long count, long long step,
                                     cudaStream_t s);
int mixed_exec(fft_plan* p, const void* in, void* out, int conj, double sx, double sy, int scale_out,
               cudaStream_t s);
cudaError_t launch_gen_twiddles_n64(double2* tab, long long N, long long count, cudaStream_t s);

cudaError_t launch_gen_stage_twiddles(float2* tab, int lg, cudaStream_t s, bool rev = false, int lgm = 4);
cudaError_t launch_gen_stage_table(float2* tab, int lg, cudaStream_t s);
cudaError_t launch_gen_power_twiddles(float2* tab, int lgN, long long count, long long step, cudaStream_t s);
// Real-to-complex transforms of N = 2M reals, M a two-pass four-step length
// with rows of 2^6..2^12 points: the even/odd split folded into the row pass
// (real_fold.cu).
struct TileKernelInfo;
const TileKernelInfo* r2c_fold_kernel_info(int lg2);
// complex to real: the split folded into the inner column pass (columns of
// 2^lg1 points, C per CTA), or NULL
const TileKernelInfo* c2r_fold_kernel_info(int lg1, int C);
int r2c_fold_launch(const TileKernelInfo* k, const TileArgs& a, long long M, int N1, long long batch,
                    const float2* r_lo, const float2* r_hi, int r_s, int scale, float s_int, float s_end,
                    cudaStream_t s);
cudaError_t launch_r2c_split(const float2* z, float2* x, long long M, long long batch, const float2* lo,
                             const float2* hi, int s, float s_int, float s_end, cudaStream_t st);
cudaError_t launch_c2r_split(const float2* x, float2* z, long long M, long long batch, const float2* lo,
                             const float2* hi, int s, float end_mul, cudaStream_t st);
cudaError_t launch_r2c_split64(const double2* z, double2* x, long long M, long long batch, const double2* lo,
                               const double2* hi, int s, double s_int, double s_end, cudaStream_t st);
cudaError_t launch_c2r_split64(const double2* x, double2* z, long long M, long long batch, const double2* lo,
                               const double2* hi, int s, double end_mul, cudaStream_t st);

// What orders the executions of a plan that share its workspace and counters:
// the lock keeps one execution's launches together, the event marks the end of
// the last one, which an execution on another stream waits for on the device.
struct PlanOrder {
  std::mutex mu;
  cudaEvent_t done = nullptr;
  cudaStream_t last = nullptr;
  bool ran = false;
};

}  // namespace gbfft

struct fft_plan {
  int kind;
  int64_t n;       // transform length (1-D), ny*nx (2-D), total points (many)
  int64_t batch;   // transforms (1-D), images (2-D), count (many)
  int64_t ny, nx;  // 2-D sides
  int dir, prec;
  int device;

  // single pass: lg; four-step: lg1 = log2 N1 (column length), lg2 = log2 N2
  // (row length); 2-D: lg1 = log2 ny, lg2 = log2 nx.
  int lg, lg1, lg2;
  int c1, c2;  // transforms per CTA of the first / second pass
  const gbfft::TileKernelInfo* k1;
  const gbfft::TileKernelInfo* k2;
  const gbfft::TileKernelInfo* ktma;  // persistent TMA-staged single-pass kernel (or NULL)
  const gbfft::TileKernelInfo* kdif2; // two-CTA radix-2 split kernel (or NULL)
  const gbfft::TileKernelInfo* kpf;   // persistent L2-prefetching single-pass kernel (or NULL)
  const gbfft::TileKernelInfo* kpfs;  // its variant staging the next transform by a bulk copy (or NULL;
                                      // kpf is then the fallback for inputs not 16-byte aligned)
  long long pf_grid;                  // its resident-CTA grid
  const gbfft::TileKernelInfo* kradix;  // single pass with radix-8 / radix-4 passes (config radix), or NULL
  void* d_radtw;                        // its stage table (schedule of largest radix 2^radix_lgm)
  int radix_lgm;
  const gbfft::TileKernelInfo* krc;   // fused range-compression kernel of the length (or NULL)
  void* d_rctw;                       // its remainder-last stage table (NULL: the length's own table)
  long long rc_grid;                  // its grid when persistent (0: one tile per CTA)

  // real-data plans (KIND_REAL, n = N reals, M = N/2): fused kernels for
  // M <= 2^14, else the complex length-M plan `inner` plus the split kernels
  // through `zbuf` (batch*M complex values after the inner workspace)
  const gbfft::TileKernelInfo* kr2c;
  const gbfft::TileKernelInfo* kc2r;
  const gbfft::TileKernelInfo* krfold;   // real-to-complex: split folded into the inner row pass (or NULL)
  const gbfft::TileKernelInfo* kcfold;   // complex-to-real: split folded into the inner column pass (or NULL)
  fft_plan* inner;
  void* d_rtw;        // W_N^k, k < M, two-level: r_lo[k & (2^r_s - 1)] * r_hi[k >> r_s]
  const float2* r_lo;
  const float2* r_hi;
  int r_s;
  float2* zbuf;

  // mixed-radix plans (KIND_MIXED)
  gbfft::MixedArgs mixed;
  int mixed_smem;
  const gbfft::MixedCtInfo* mixed_ct;   // compile-time schedule for this length (FP32), or NULL
  gbfft::MixrLaunch mr[2];   // FP32 mixed radix: one tile pass, or the two passes of a split
  gbfft::FxLaunch fx[2];     // FP64: the same
  long long m4_n1, m4_n2;   // four-step: column length N1, row length N2 (N = N1 N2); 2-D: ny, nx
  const float2* pre_tw;               // its W_N^n table, n < N/2
  long long tma_grid;                 // its resident-CTA grid

  // all twiddle tables live in one device allocation
  void* d_tables;
  const float2* tw1;  // stage table for the first pass length
  const float2* tw2;  // stage table for the second pass length
  const float2* ft_lo;
  const float2* ft_hi;
  int ft_s;

  // tensor-core radix-16 path (prec != FFT_PREC_FP32)
  void* d_tc;   // full twiddle tables of the tensor-core passes
  const gbfft::TileKernelInfo* ktc1;
  const gbfft::TileKernelInfo* ktc2;
  const float2* tctw1;
  const float2* tctw2;

  size_t ws_bytes;
  void* ws;
  int ws_owned;
  gbfft::PlanOrder* order;   // plans whose executions write a workspace or counters (NULL for others)

  int* d_status;  // device status word (bounded waits)

  gbfft::ManyPlan* many;
  gbfft::FusedPlan* fused;  // both passes in one persistent launch (fused.cu)
  int launches;

  // multi-pass plans (four-step with two or three passes, 2-D)
  gbfft::PassDesc pass[gbfft::kMaxPasses];
  int npass;
  int lg3;            // three-pass split: log2 N3
  const float2* tw3;  // stage table of the third length
  const float2* ft2_lo;  // two-level table of the second four-step level
  const float2* ft2_hi;
  int ft2_s;
};
