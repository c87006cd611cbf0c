// fx64_00.cu -- instance of the FP64 tile kernel: contiguous transforms, any pad.
#include "fx64.cuh"

namespace gbfft {
const void* fx_fn_0_0(bool only) {
  return only ? (const void*)fx_only_kernel<false, false> : (const void*)fx_kernel<false, false>;
}
}  // namespace gbfft
