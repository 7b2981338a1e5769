// Fused sparse pass, closed-form weights, fp8 (e4m3) cache, head dimension 128.
#include "sparse_step.cuh"

namespace vsa {

cudaError_t launch_step_fp8(const StepParams& p, int threads, cudaStream_t stream)
{
    return launch_step_family<kHeadDim, true>(p, threads, stream);
}

}  // namespace vsa
