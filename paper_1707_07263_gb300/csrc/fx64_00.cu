// fx64_00.cu -- instance of the FP64 tile kernel: contiguous transforms, any pad.
#include "fx64.cuh"

namespace gbfft {
const void* fx_fn_0_0() { return (const void*)fx_kernel<false, false>; }
}  // namespace gbfft
