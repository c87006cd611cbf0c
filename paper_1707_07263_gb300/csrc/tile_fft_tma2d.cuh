// tile_fft_tma2d.cuh -- persistent column-pass kernel staged by tensor TMA.
//
// The column passes of the multi-pass plans (four-step pass 1, the first two
// passes of the three-pass split, the 2-D column passes) read C adjacent
// columns of L rows that lie far apart in memory.  Here each CTA loops over
// tiles; one thread issues cp.async.bulk.tensor for the C x L box of the next
// tile (a 4-D tensor map: columns, rows, inner batch, outer batch) into a
// staging buffer while the CTA computes the current one, completion on an
// mbarrier with a bounded wait.  The first pass reads the staged box [n][c]
// from shared memory; the remaining passes, the four-step twiddle and the
// stores are those of tile_fft.cuh.
#pragma once
#include <cuda.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "tile_fft_tma.cuh"

namespace gbfft {

template <int LG, int C>
struct ColTmaCfg {
  using Tile = TileCfg<LG, C, true, true>;
  static constexpr int L = Tile::L;
  static constexpr int T = Tile::T;
  static constexpr int S_ELEMS = C * L;  // staged box
  static constexpr int SMEM_BYTES = S_ELEMS * 8 + Tile::SMEM_BYTES;
  static constexpr int MIN_BLOCKS = T <= 256 ? 3 : 1;
};

__device__ __forceinline__ void tma_load_4d(void* dst, const CUtensorMap* map, int x, int y, int z, int w,
                                            uint32_t bytes, uint64_t* mbar) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(mbar)), "r"(bytes)
               : "memory");
  asm volatile(
      "cp.async.bulk.tensor.4d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4, "
      "%5}], [%6];" ::"r"(smem_u32(dst)),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(z), "r"(w), "r"(smem_u32(mbar))
      : "memory");
}

template <int LG, int C>
__global__ void __launch_bounds__(ColTmaCfg<LG, C>::T, ColTmaCfg<LG, C>::MIN_BLOCKS)
    col_tma_kernel(const __grid_constant__ CUtensorMap tmap, const TileArgs a, long long ntiles, int* status) {
  using Cfg = ColTmaCfg<LG, C>;
  using Tile = typename Cfg::Tile;
  static_assert(Tile::NST >= 2, "the staged pass is followed by at least one more");
  extern __shared__ __align__(128) unsigned char smraw[];
  __shared__ __align__(8) uint64_t mbar;
  float2* S = (float2*)smraw;
  float2* X = S + Cfg::S_ELEMS;
  float2* epi = X + Tile::SM_TILE;
  const int tid = threadIdx.x;

  auto split = [&](long long t, long long& b2, long long& b, long long& g) {
    b = t / a.tiles_per_batch;
    g = t - b * a.tiles_per_batch;
    b2 = 0;
    if (a.nb1) {
      b2 = b / a.nb1;
      b -= b2 * a.nb1;
    }
  };
  auto issue = [&](long long t) {
    long long b2, b, g;
    split(t, b2, b, g);
    tma_load_4d(S, &tmap, (int)(g * C), 0, (int)b, (int)b2, (uint32_t)(Cfg::S_ELEMS * 8), &mbar);
  };

  if (tid == 0) {
    mbar_init(&mbar, 1);
    fence_mbar_init();
  }
  __syncthreads();
  long long tile = blockIdx.x;
  if (tid == 0 && tile < ntiles) issue(tile);
  uint32_t parity = 0;
  for (; tile < ntiles; tile += gridDim.x) {
    long long b2, b, g;
    split(tile, b2, b, g);
    const long long col0 = g * C;
    float2* gout = a.out + b2 * a.out_b2stride + b * a.out_bstride + g * a.out_gstride;
    __syncthreads();  // the previous tile's last pass has finished reading X and epi
    if (a.ft_lgN) tile_step_table<LG, C, 4>(a, col0, b, epi);
    if (!mbar_wait(&mbar, parity)) {
      if (tid == 0) atomicExch(status, FFT_ERR_TIMEOUT);
      mbar_wait(&mbar, parity);  // second bounded wait for the copy in flight
      return;
    }
    parity ^= 1u;
    float2 v[Tile::P];
    // pass 0 from the staged box; its closing barrier frees the staging buffer
    tile_pass<LG, C, true, true, 0, false, 2>(v, X, a, S, gout, col0, b, epi);
    if (tid == 0 && tile + gridDim.x < ntiles) {
      fence_proxy_async();
      issue(tile + gridDim.x);
    }
    tile_stage<LG, C, true, true, 1, false, 0>(v, X, a, S, gout, col0, b, epi);
  }
}

// The same for long columns, whose box and exchange tile do not both fit: the
// box of the next tile is copied into the exchange buffer itself once the last
// pass of this one has read it, while that pass computes and stores (as
// tile_fft_pfs_kernel does for rows).  A box holds 256 rows at most, so the
// copy is L / 256 of them on one barrier.  The column pass without it waits for
// its loads (ncu at 2^20: long_scoreboard the top stall, 16 warps an SM, DRAM
// 49 %).  Measured per 2^26 points, 2^10-point columns 8 a tile: 2^20 416 ->
// 367 us, 2^21 446 -> 401, 2^22 (as 2^10 x 2^12) 527 -> 474, 1024 x 4096 images
// 400 -> 356, 1024 x 256 380 -> 342.
template <int LG, int C, int LGM>
struct ColStageCfg {
  using Tile = TileCfg<LG, C, true, true, 0, LGM>;
  static constexpr int T = Tile::T;
  static constexpr int SMEM_BYTES = Tile::SMEM_BYTES + 16;   // and the barrier
  static constexpr int MIN_BLOCKS = cmax(1, 512 / T);
};

struct ColStageHook {
  static constexpr bool on = true;
  const CUtensorMap* map;
  float2* sm;
  uint64_t* mbar;
  int x, z, w, rows, cols;   // first column (negative: no next tile), batches, tile shape
  __device__ __forceinline__ void operator()() const {
    if (threadIdx.x != 0 || x < 0) return;
    fence_proxy_async();   // the generic-proxy reads of the buffer before the async-proxy writes
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(mbar)),
                 "r"((uint32_t)(rows * cols * 8))
                 : "memory");
#pragma unroll 1
    for (int y = 0; y < rows; y += 256)
      asm volatile(
          "cp.async.bulk.tensor.4d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4, "
          "%5}], [%6];" ::"r"(smem_u32(sm + y * cols)),
          "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(z), "r"(w), "r"(smem_u32(mbar))
          : "memory");
  }
};

template <int LG, int C, int LGM>
__global__ void __launch_bounds__(ColStageCfg<LG, C, LGM>::T, ColStageCfg<LG, C, LGM>::MIN_BLOCKS)
    col_stage_kernel(const __grid_constant__ CUtensorMap tmap, const TileArgs a, long long ntiles, int* status) {
  using Cfg = ColStageCfg<LG, C, LGM>;
  using Tile = typename Cfg::Tile;
  static_assert(Tile::NST >= 2 && Tile::SM_TILE >= C * Tile::L && LG >= 8, "the box must fit the exchange tile");
  extern __shared__ __align__(128) unsigned char smraw[];
  float2* const X = (float2*)smraw;
  float2* const epi = X + Tile::SM_TILE;
  uint64_t* const mbar = (uint64_t*)(smraw + Tile::SMEM_BYTES);
  const int tid = threadIdx.x;
  auto split = [&](long long t, long long& b2, long long& b, long long& g) {
    b = t / a.tiles_per_batch;
    g = t - b * a.tiles_per_batch;
    b2 = 0;
    if (a.nb1) {
      b2 = b / a.nb1;
      b -= b2 * a.nb1;
    }
  };
  auto copy_of = [&](long long t) {
    ColStageHook h{&tmap, X, mbar, -1, 0, 0, Tile::L, C};
    if (t < ntiles) {
      long long b2, b, g;
      split(t, b2, b, g);
      h.x = (int)(g * C);
      h.z = (int)b;
      h.w = (int)b2;
    }
    return h;
  };
  if (tid == 0) {
    mbar_init(mbar, 1);
    fence_mbar_init();
  }
  __syncthreads();
  copy_of(blockIdx.x)();
  uint32_t parity = 0;
  float2 v[Tile::P];
  for (long long tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
    long long b2, b, g;
    split(tile, b2, b, g);
    const long long col0 = g * C;
    float2* gout = a.out + b2 * a.out_b2stride + b * a.out_bstride + g * a.out_gstride;
    if (a.ft_lgN) {
      __syncthreads();   // the previous tile's last pass has finished reading epi
      tile_step_table<LG, C, LGM>(a, col0, b, epi);
    }
    if (!mbar_wait(mbar, parity)) {
      if (tid == 0) atomicExch(status, FFT_ERR_TIMEOUT);
      mbar_wait(mbar, parity);   // second bounded wait for the copy in flight
      return;
    }
    parity ^= 1u;
    const ColStageHook next = copy_of(tile + gridDim.x);
    tile_stage<LG, C, true, true, 0, false, 9, 0, false, LGM, ColStageHook>(v, X, a, X, gout, col0, b, epi, next);
  }
}

}  // namespace gbfft
