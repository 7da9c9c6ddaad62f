// FP64 axis transforms, a quarter of the compiled edges (fft_axis64.cuh).
#include "fft_axis64_impl.cuh"

namespace pwh {
PWH_AXIS_UNIT(c, PWH_AXIS_SIZES_C)
}  // namespace pwh
