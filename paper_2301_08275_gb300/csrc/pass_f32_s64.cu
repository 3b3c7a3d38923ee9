// pass_f32_s64.cu - complex64 strided (y, z) sweeps of 64 and 128 points.
#include "pass_kernels.cuh"

namespace gpe {

GPE_PASS_TU(float, 64, false, 0)
GPE_PASS_TU(float, 64, false, 1)
GPE_PASS_TU(float, 128, false, 0)
GPE_PASS_TU(float, 128, false, 1)

}  // namespace gpe
