// pass_f64_s64.cu - complex128 strided (y, z) sweeps of 64 points.
#include "pass_kernels.cuh"

namespace gpe {

GPE_PASS_TU(double, 64, false, 0)
GPE_PASS_TU(double, 64, false, 1)

}  // namespace gpe
