// Fused sparse pass with the routing certificate: every page score of the unit in registers.
#include "sparse_kernel.cuh"

namespace vsa {

namespace {

// page-score registers per thread from the block-table width
template <int THREADS>
cudaError_t launch_cert_threads(const SparseArgs& a)
{
    if (a.g.max_pages <= 8 * THREADS) return launch_tok<THREADS, 8, true>(a);
    if (a.g.max_pages <= 16 * THREADS) return launch_tok<THREADS, 16, true>(a);
    if (a.g.max_pages <= 32 * THREADS) return launch_tok<THREADS, 32, true>(a);
    return cudaErrorInvalidValue;   // (refused by the entry point before any launch)
}

}  // namespace

cudaError_t launch_sparse_cert(const SparseArgs& a, int threads)
{
    if (threads == 128) return launch_cert_threads<128>(a);
    return threads == 512 ? launch_cert_threads<512>(a) : launch_cert_threads<256>(a);
}

}  // namespace vsa
