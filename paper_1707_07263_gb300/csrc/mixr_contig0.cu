// mixr_contig0.cu -- instances of the FP32 mixed-radix tile kernel: contiguous transforms, unpadded tiles.
#include "mixr.cuh"
namespace gbfft {
const void* mixr_fn_contig_0(bool big) {
  return big ? (const void*)mixr_big_kernel<false, 0> : (const void*)mixr_kernel<false, 0>;
}
}  // namespace gbfft
