// pass_f32_s1024_0.cu - complex64 strided (y, z) sweeps of 1024 points.
#include "pass_kernels.cuh"

namespace gpe {

GPE_PASS_TU(float, 1024, false, 0)

}  // namespace gpe
