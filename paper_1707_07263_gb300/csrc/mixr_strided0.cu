// mixr_strided0.cu -- instances of the FP32 mixed-radix tile kernel: strided columns, unpadded tiles.
#include "mixr.cuh"
namespace gbfft {
const void* mixr_fn_strided_0(bool big) {
  return big ? (const void*)mixr_big_kernel<true, 0> : (const void*)mixr_kernel<true, 0>;
}
}  // namespace gbfft
