// pass_f64_s256.cu - complex128 strided (y, z) sweeps of 256 points.
#include "pass_kernels.cuh"

namespace gpe {

GPE_PASS_TU(double, 256, false, 0)
GPE_PASS_TU(double, 256, false, 1)

}  // namespace gpe
