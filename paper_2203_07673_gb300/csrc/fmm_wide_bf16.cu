// Warp-per-long-row passes, bfloat16 dense operands.
#include "fmm_wide.cuh"

namespace fmm {
cudaError_t launch_wide_bf16(int mode, const PassArgs &a, int n_wide, bool ring, cudaStream_t st)
{
    return launch_wide_typed<bf16_t>(mode, a, n_wide, ring, st);
}
}  // namespace fmm
