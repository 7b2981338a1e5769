// Fused sparse pass, closed-form weights.
#include "sparse_step.cuh"

namespace vsa {

cudaError_t launch_step(const StepParams& p, int threads, cudaStream_t stream)
{
    return launch_step_family<kHeadDim, false>(p, threads, stream);
}

}  // namespace vsa
