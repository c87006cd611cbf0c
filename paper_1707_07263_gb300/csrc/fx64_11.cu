// fx64_11.cu -- instance of the FP64 tile kernel: strided columns, evenly spaced tile.
#include "fx64.cuh"

namespace gbfft {
const void* fx_fn_1_1(bool only) {
  return only ? (const void*)fx_only_kernel<true, true> : (const void*)fx_kernel<true, true>;
}
}  // namespace gbfft
