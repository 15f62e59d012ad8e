// Flexible-width row passes, float32 dense operands.
#include "fmm_flex.cuh"

namespace fmm {
cudaError_t launch_flex_f32(int mode, const PassArgs &a, int vb, int ng, cudaStream_t st)
{
    return launch_flex_typed<float>(mode, a, vb, ng, st);
}
}  // namespace fmm
