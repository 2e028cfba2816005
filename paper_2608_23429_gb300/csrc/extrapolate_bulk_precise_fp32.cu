// Bulk-copy pipeline kernels with fp32 predictions or hidden states, fp32 sources.
#include "extrapolate_bulk_precise.cuh"

namespace cbk {

cudaError_t prepare_extrapolate_bulk_precise_fp32(int K, bool gated, size_t smem) {
    return prepare_type<false, false>(K, gated, smem);
}

cudaError_t launch_extrapolate_bulk_precise_fp32(const ExtrapArgs& a, int K, bool grouped, bool gated, int grid,
                                                 size_t smem, cudaStream_t s) {
    return launch_type<false, false>(a, K, grouped, gated, grid, smem, s);
}

}  // namespace cbk
