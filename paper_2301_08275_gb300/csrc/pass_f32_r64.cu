// pass_f32_r64.cu - complex64 row (x) sweeps of 64 and 128 points.
#include "pass_kernels.cuh"

namespace gpe {

GPE_PASS_TU(float, 64, true, 0)
GPE_PASS_TU(float, 64, true, 1)
GPE_PASS_TU(float, 128, true, 0)
GPE_PASS_TU(float, 128, true, 1)

}  // namespace gpe
