// pass_f32_r256.cu - complex64 row (x) sweeps of 256 points.
#include "pass_kernels.cuh"

namespace gpe {

GPE_PASS_TU(float, 256, true, 0)
GPE_PASS_TU(float, 256, true, 1)

}  // namespace gpe
