// pass_f64_s1024.cu - complex128 strided (y, z) sweeps of 1024 points.
#include "pass_kernels.cuh"

namespace gpe {

GPE_PASS_TU(double, 1024, false, 0)
GPE_PASS_TU(double, 1024, false, 1)

}  // namespace gpe
