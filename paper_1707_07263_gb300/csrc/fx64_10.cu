// fx64_10.cu -- instance of the FP64 tile kernel: strided columns, any pad.
#include "fx64.cuh"

namespace gbfft {
const void* fx_fn_1_0(bool only) {
  return only ? (const void*)fx_only_kernel<true, false> : (const void*)fx_kernel<true, false>;
}
}  // namespace gbfft
