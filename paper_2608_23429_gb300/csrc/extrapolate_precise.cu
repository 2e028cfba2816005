// Instantiations of the direct-load kernel (direct_kernel.cuh) with fp32
// predictions or hidden states, gated or not.
#include "direct_kernel.cuh"

namespace cbk {
namespace {

template <int K, bool CB16>
cudaError_t launch_k(const ExtrapArgs& a, bool gated, int grid, cudaStream_t s) {
    if (gated)
        extrapolate_kernel<K, CB16, true, true><<<grid, kThreads, 0, s>>>(a);
    else
        extrapolate_kernel<K, CB16, false, true><<<grid, kThreads, 0, s>>>(a);
    return cudaGetLastError();
}

template <bool CB16>
cudaError_t dispatch(const ExtrapArgs& a, int K, bool gated, int grid, cudaStream_t s) {
    switch (K) {
    case 1: return launch_k<1, CB16>(a, gated, grid, s);
    case 2: return launch_k<2, CB16>(a, gated, grid, s);
    case 3: return launch_k<3, CB16>(a, gated, grid, s);
    case 4: return launch_k<4, CB16>(a, gated, grid, s);
    case 5: return launch_k<5, CB16>(a, gated, grid, s);
    case 6: return launch_k<6, CB16>(a, gated, grid, s);
    case 7: return launch_k<7, CB16>(a, gated, grid, s);
    case 8: return launch_k<8, CB16>(a, gated, grid, s);
    default: return cudaErrorInvalidValue;
    }
}

}  // namespace

cudaError_t launch_extrapolate_precise(const ExtrapArgs& a, int K, bool cache_bf16, bool gated, int grid,
                                       cudaStream_t s) {
    return cache_bf16 ? dispatch<true>(a, K, gated, grid, s) : dispatch<false>(a, K, gated, grid, s);
}

}  // namespace cbk
