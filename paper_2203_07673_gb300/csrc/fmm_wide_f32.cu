// Warp-per-long-row passes, float32 dense operands.
#include "fmm_wide.cuh"

namespace fmm {
cudaError_t launch_wide_f32(int mode, const PassArgs &a, int n_wide, bool ring, cudaStream_t st)
{
    return launch_wide_typed<float>(mode, a, n_wide, ring, st);
}
}  // namespace fmm
