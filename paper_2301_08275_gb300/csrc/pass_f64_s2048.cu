// pass_f64_s2048.cu - complex128 strided (y, z) sweeps of 2048 and 4096 points.
#include "pass_kernels.cuh"

namespace gpe {

GPE_PASS_TU(double, 2048, false, 0)
GPE_PASS_TU(double, 2048, false, 1)
GPE_PASS_TU(double, 4096, false, 0)
GPE_PASS_TU(double, 4096, false, 1)

}  // namespace gpe
