// pass_f64.cu - complex128 sweeps of lines of less than 64 points and the dispatcher of
// all complex128 sweeps.
#include "pass_kernels.cuh"

namespace gpe {

cudaError_t launch_pass_f64(bool rows, int var, const PassArgs &a, cudaStream_t st, const CUtensorMap *tmap)
{
    if (rows) return var ? launch_pass_r<double, true, 1>(a, st, nullptr) : launch_pass_r<double, true, 0>(a, st, nullptr);
    return var ? launch_pass_r<double, false, 1>(a, st, tmap) : launch_pass_r<double, false, 0>(a, st, tmap);
}
int lines_per_tile_f64(bool rows, int n, int var) { return lines_per_tile_r<double>(rows, n, var); }

}  // namespace gpe
