// line1d_f32.cu - the on-chip 1D kernels, complex64.
#include "pass_kernels.cuh"

namespace gpe {

cudaError_t launch_line1d_f32(const Line1DArgs &a, cudaStream_t st) { return launch_line1d_r<float>(a, st); }

}  // namespace gpe
