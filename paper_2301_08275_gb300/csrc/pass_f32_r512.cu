// pass_f32_r512.cu - complex64 row (x) sweeps of 512 points.
#include "pass_kernels.cuh"

namespace gpe {

GPE_PASS_TU(float, 512, true, 0)
GPE_PASS_TU(float, 512, true, 1)

}  // namespace gpe
