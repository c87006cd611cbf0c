// fx64_01.cu -- instance of the FP64 tile kernel: contiguous transforms, evenly spaced tile.
#include "fx64.cuh"

namespace gbfft {
const void* fx_fn_0_1(bool only) {
  return only ? (const void*)fx_only_kernel<false, true> : (const void*)fx_kernel<false, true>;
}
}  // namespace gbfft
