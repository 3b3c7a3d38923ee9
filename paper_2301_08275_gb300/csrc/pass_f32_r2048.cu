// pass_f32_r2048.cu - complex64 row (x) sweeps of 2048 and 4096 points.
#include "pass_kernels.cuh"

namespace gpe {

GPE_PASS_TU(float, 2048, true, 0)
GPE_PASS_TU(float, 2048, true, 1)
GPE_PASS_TU(float, 4096, true, 0)
GPE_PASS_TU(float, 4096, true, 1)

}  // namespace gpe
