// pass_f32.cu - complex64 sweeps of lines of less than 64 points and the dispatcher of
// all complex64 sweeps.
#include "pass_kernels.cuh"

namespace gpe {

cudaError_t launch_pass_f32(bool rows, int var, const PassArgs &a, cudaStream_t st, const CUtensorMap *tmap)
{
    if (rows) return var ? launch_pass_r<float, true, 1>(a, st, nullptr) : launch_pass_r<float, true, 0>(a, st, nullptr);
    return var ? launch_pass_r<float, false, 1>(a, st, tmap) : launch_pass_r<float, false, 0>(a, st, tmap);
}
int lines_per_tile_f32(bool rows, int n, int var) { return lines_per_tile_r<float>(rows, n, var); }

}  // namespace gpe
