// Fused sparse pass with an iterative solve on the candidate set: entropic mirror descent (kind 1) and
// Frank-Wolfe (kind 2), 256 threads.
#include "sparse_step.cuh"

namespace vsa {

cudaError_t launch_step_solve(const StepParams& p, int kind, cudaStream_t stream)
{
    const bool fused = p.page_scores != nullptr;
    if (p.bounds) return cudaErrorInvalidValue;
    if (p.summaries) {
        if (p.scan_mma)
            return kind == 2 ? launch_step_variant<256, 4, kHeadDim, false, 2>(p, stream) : launch_step_variant<256, 4, kHeadDim, false, 1>(p, stream);
        return kind == 2 ? launch_step_variant<256, 2, kHeadDim, false, 2>(p, stream) : launch_step_variant<256, 2, kHeadDim, false, 1>(p, stream);
    }
    if (kind == 2)
        return fused ? launch_step_variant<256, 1, kHeadDim, false, 2>(p, stream)
                     : launch_step_variant<256, 0, kHeadDim, false, 2>(p, stream);
    return fused ? launch_step_variant<256, 1, kHeadDim, false, 1>(p, stream)
                 : launch_step_variant<256, 0, kHeadDim, false, 1>(p, stream);
}

}  // namespace vsa
