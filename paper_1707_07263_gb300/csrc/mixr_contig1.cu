// mixr_contig1.cu -- instances of the FP32 mixed-radix tile kernel: contiguous transforms, padded tiles (even first radix).
#include "mixr.cuh"
namespace gbfft {
const void* mixr_fn_contig_1(bool big) {
  return big ? (const void*)mixr_big_kernel<false, 1> : (const void*)mixr_kernel<false, 1>;
}
}  // namespace gbfft
