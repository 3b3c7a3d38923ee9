// pass_f64_s512.cu - complex128 strided (y, z) sweeps of 512 points.
#include "pass_kernels.cuh"

namespace gpe {

GPE_PASS_TU(double, 512, false, 0)
GPE_PASS_TU(double, 512, false, 1)

}  // namespace gpe
