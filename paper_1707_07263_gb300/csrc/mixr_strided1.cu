// mixr_strided1.cu -- instances of the FP32 mixed-radix tile kernel: strided columns, padded tiles (even first radix).
#include "mixr.cuh"
namespace gbfft {
const void* mixr_fn_strided_1(bool big) {
  return big ? (const void*)mixr_big_kernel<true, 1> : (const void*)mixr_kernel<true, 1>;
}
}  // namespace gbfft
