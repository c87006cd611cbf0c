// fft_radix32.cuh -- the register-resident 32-point DFT of the single-pass
// kernels with 32 points a thread: 4 x 8, the inner twiddles W_32^{n2 k1} as
// compile-time constants.
#pragma once
#include "mixed_ct.cuh"

namespace gbfft {

template <>
__device__ __forceinline__ void dft_fwd<32>(float2* v) {
  ct_dft_split<4, 8>(v);
}

}  // namespace gbfft
