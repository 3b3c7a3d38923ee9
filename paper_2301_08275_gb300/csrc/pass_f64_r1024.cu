// pass_f64_r1024.cu - complex128 row (x) sweeps of 1024 points.
#include "pass_kernels.cuh"

namespace gpe {

GPE_PASS_TU(double, 1024, true, 0)
GPE_PASS_TU(double, 1024, true, 1)

}  // namespace gpe
