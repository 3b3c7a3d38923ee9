// pass_f64_r128.cu - complex128 row (x) sweeps of 128 points.
#include "pass_kernels.cuh"

namespace gpe {

GPE_PASS_TU(double, 128, true, 0)
GPE_PASS_TU(double, 128, true, 1)

}  // namespace gpe
