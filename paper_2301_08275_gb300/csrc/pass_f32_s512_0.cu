// pass_f32_s512_0.cu - complex64 strided (y, z) sweeps of 512 points.
#include "pass_kernels.cuh"

namespace gpe {

GPE_PASS_TU(float, 512, false, 0)

}  // namespace gpe
