// line1d_f64.cu - the on-chip 1D kernels, complex128.
#include "pass_kernels.cuh"

namespace gpe {

cudaError_t launch_line1d_f64(const Line1DArgs &a, cudaStream_t st) { return launch_line1d_r<double>(a, st); }

}  // namespace gpe
