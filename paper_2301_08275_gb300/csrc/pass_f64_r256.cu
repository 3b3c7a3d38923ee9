// pass_f64_r256.cu - complex128 row (x) sweeps of 256 points.
#include "pass_kernels.cuh"

namespace gpe {

GPE_PASS_TU(double, 256, true, 0)
GPE_PASS_TU(double, 256, true, 1)

}  // namespace gpe
