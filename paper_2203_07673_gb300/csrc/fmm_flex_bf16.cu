// Flexible-width row passes, bfloat16 dense operands.
#include "fmm_flex.cuh"

namespace fmm {
cudaError_t launch_flex_bf16(int mode, const PassArgs &a, int vb, int ng, cudaStream_t st)
{
    return launch_flex_typed<bf16_t>(mode, a, vb, ng, st);
}
}  // namespace fmm
