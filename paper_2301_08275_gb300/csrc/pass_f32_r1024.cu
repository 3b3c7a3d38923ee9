// pass_f32_r1024.cu - complex64 row (x) sweeps of 1024 points.
#include "pass_kernels.cuh"

namespace gpe {

GPE_PASS_TU(float, 1024, true, 0)
GPE_PASS_TU(float, 1024, true, 1)

}  // namespace gpe
