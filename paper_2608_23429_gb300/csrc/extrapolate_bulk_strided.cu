// Bulk-copy pipeline kernels for items off the 16-byte grid on their way out, bf16 sources.
#include "extrapolate_bulk_precise.cuh"

namespace cbk {

cudaError_t prepare_extrapolate_bulk_strided_fp32(int K, bool gated, size_t smem);
cudaError_t launch_extrapolate_bulk_strided_fp32(const ExtrapArgs& a, int K, bool grouped, bool gated, int grid,
                                                 size_t smem, cudaStream_t s);

cudaError_t prepare_extrapolate_bulk_strided(int K, bool cache_bf16, bool gated, size_t smem) {
    return cache_bf16 ? prepare_type<true, true>(K, gated, smem) : prepare_extrapolate_bulk_strided_fp32(K, gated, smem);
}

cudaError_t launch_extrapolate_bulk_strided(const ExtrapArgs& a, int K, bool cache_bf16, bool grouped, bool gated,
                                            int grid, size_t smem, cudaStream_t s) {
    return cache_bf16 ? launch_type<true, true>(a, K, grouped, gated, grid, smem, s)
                      : launch_extrapolate_bulk_strided_fp32(a, K, grouped, gated, grid, smem, s);
}

}  // namespace cbk
