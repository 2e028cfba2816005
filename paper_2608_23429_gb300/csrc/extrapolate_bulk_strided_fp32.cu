// Bulk-copy pipeline kernels for items off the 16-byte grid on their way out, fp32 sources.
#include "extrapolate_bulk_precise.cuh"

namespace cbk {

cudaError_t prepare_extrapolate_bulk_strided_fp32(int K, bool gated, size_t smem) {
    return prepare_type<false, true>(K, gated, smem);
}

cudaError_t launch_extrapolate_bulk_strided_fp32(const ExtrapArgs& a, int K, bool grouped, bool gated, int grid,
                                                 size_t smem, cudaStream_t s) {
    return launch_type<false, true>(a, K, grouped, gated, grid, smem, s);
}

}  // namespace cbk
