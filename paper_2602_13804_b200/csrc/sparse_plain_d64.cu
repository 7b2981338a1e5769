// Fused sparse pass, closed-form weights, head dimension 64.
#include "sparse_step.cuh"

namespace vsa {

cudaError_t launch_step_d64(const StepParams& p, int threads, cudaStream_t stream)
{
    return launch_step_family<64, false>(p, threads, stream);
}

}  // namespace vsa
