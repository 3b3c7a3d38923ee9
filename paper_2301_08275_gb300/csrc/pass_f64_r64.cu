// pass_f64_r64.cu - complex128 row (x) sweeps of 64 points.
#include "pass_kernels.cuh"

namespace gpe {

GPE_PASS_TU(double, 64, true, 0)
GPE_PASS_TU(double, 64, true, 1)

}  // namespace gpe
