// tile_inst_real.cu -- compiled fused real-to-complex and complex-to-real
// kernels, one per half length L = 2^1..2^14 (N = 2L reals) with
// jj_cols(lg) rows per CTA.
#include "real_pair.cuh"
#include "tile_registry.h"

namespace gbfft {

#define GBFFT_REAL(KERNEL, LG)                                                          \
  {(const void*)&KERNEL<LG, jj_cols(LG)>, TileCfg<LG, jj_cols(LG), false, false>::T,    \
   jj_cols(LG) * TileCfg<LG, jj_cols(LG), false, false>::LP * 8, LG, jj_cols(LG), MAP_JJ, 0}
#define GBFFT_PAIR(KERNEL, LG)                                               \
  {(const void*)&KERNEL<LG, jj_cols(LG)>, PairCfg<LG, jj_cols(LG)>::T,       \
   PairCfg<LG, jj_cols(LG)>::SMEM_BYTES, LG, jj_cols(LG), MAP_JJ, 0}

// Both halves of a split pair in one thread (real_pair.cuh) where a row is long
// enough for its runs of L/32 (r2c) or L/2R (c2r) values to coalesce.  Measured
// per 2^26 reals on GB300, the exchanged split -> this (a copy takes 79 us):
//   reals  2^6       2^7       2^8       2^9      2^10     2^12      2^13     2^14      2^15
//   r2c                               87 -> 90  102 -> 86 100 -> 88 101 -> 89 126 -> 110 161 -> 142
//   c2r 141 -> 124 108 -> 99 105 -> 85 107 -> 82 117 -> 83 110 -> 94 119 -> 91 144 -> 112 171 -> 149
const TileKernelInfo* tile_kernel_r2c(int lg) {
  static const TileKernelInfo tab[] = {
      GBFFT_REAL(tile_r2c_kernel, 1),  GBFFT_REAL(tile_r2c_kernel, 2),  GBFFT_REAL(tile_r2c_kernel, 3),
      GBFFT_REAL(tile_r2c_kernel, 4),  GBFFT_REAL(tile_r2c_kernel, 5),  GBFFT_REAL(tile_r2c_kernel, 6),
      GBFFT_REAL(tile_r2c_kernel, 7),  GBFFT_REAL(tile_r2c_kernel, 8),  GBFFT_PAIR(pair_r2c_kernel, 9),
      GBFFT_PAIR(pair_r2c_kernel, 10), GBFFT_PAIR(pair_r2c_kernel, 11), GBFFT_PAIR(pair_r2c_kernel, 12),
      GBFFT_PAIR(pair_r2c_kernel, 13), GBFFT_PAIR(pair_r2c_kernel, 14),
  };
  if (lg < 1 || lg > 14) return nullptr;
  return &tab[lg - 1];
}

const TileKernelInfo* tile_kernel_c2r(int lg) {
  static const TileKernelInfo tab[] = {
      GBFFT_REAL(tile_c2r_kernel, 1),  GBFFT_REAL(tile_c2r_kernel, 2),  GBFFT_REAL(tile_c2r_kernel, 3),
      GBFFT_REAL(tile_c2r_kernel, 4),  GBFFT_PAIR(pair_c2r_kernel, 5),  GBFFT_PAIR(pair_c2r_kernel, 6),
      GBFFT_PAIR(pair_c2r_kernel, 7),  GBFFT_PAIR(pair_c2r_kernel, 8),  GBFFT_PAIR(pair_c2r_kernel, 9),
      GBFFT_PAIR(pair_c2r_kernel, 10), GBFFT_PAIR(pair_c2r_kernel, 11), GBFFT_PAIR(pair_c2r_kernel, 12),
      GBFFT_PAIR(pair_c2r_kernel, 13), GBFFT_PAIR(pair_c2r_kernel, 14),
  };
  if (lg < 1 || lg > 14) return nullptr;
  return &tab[lg - 1];
}

}  // namespace gbfft
