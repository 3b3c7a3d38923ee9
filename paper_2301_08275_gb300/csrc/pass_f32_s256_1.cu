// pass_f32_s256_1.cu - complex64 strided (y, z) sweeps of 256 points.
#include "pass_kernels.cuh"

namespace gpe {

GPE_PASS_TU(float, 256, false, 1)

}  // namespace gpe
