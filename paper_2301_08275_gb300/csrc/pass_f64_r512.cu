// pass_f64_r512.cu - complex128 row (x) sweeps of 512 points.
#include "pass_kernels.cuh"

namespace gpe {

GPE_PASS_TU(double, 512, true, 0)
GPE_PASS_TU(double, 512, true, 1)

}  // namespace gpe
