// pass_f64_s128.cu - complex128 strided (y, z) sweeps of 128 points.
#include "pass_kernels.cuh"

namespace gpe {

GPE_PASS_TU(double, 128, false, 0)
GPE_PASS_TU(double, 128, false, 1)

}  // namespace gpe
