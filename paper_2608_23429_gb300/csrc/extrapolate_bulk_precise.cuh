// Launchers of the bulk-copy pipeline kernel (bulk_kernel.cuh) for launches with
// fp32 predictions or hidden states, and (STRIDED) for items off the 16-byte
// grid on their way out. One translation
// unit per source type keeps the build parallel.
#pragma once

#include "bulk_kernel.cuh"

namespace cbk {
namespace {

template <int K, bool CB16, bool GROUPED, bool GATED, bool STRIDED>
cudaError_t launch_one(const ExtrapArgs& a, int grid, size_t smem, cudaStream_t s) {
    return launch_overlapped(extrapolate_bulk_kernel<K, CB16, GROUPED, GATED, false, true, STRIDED>, grid,
                             Shape<CB16, K, GROUPED, GATED, true, STRIDED>::threads, smem, s, a);
}

template <int K, bool CB16, bool STRIDED>
cudaError_t launch_k(const ExtrapArgs& a, bool grouped, bool gated, int grid, size_t smem, cudaStream_t s) {
    if (gated) return launch_one<K, CB16, true, true, STRIDED>(a, grid, smem, s);
    return grouped ? launch_one<K, CB16, true, false, STRIDED>(a, grid, smem, s)
                   : launch_one<K, CB16, false, false, STRIDED>(a, grid, smem, s);
}

template <int K, bool CB16, bool STRIDED>
cudaError_t prepare_k(bool gated, size_t smem) {
    constexpr auto attr = cudaFuncAttributeMaxDynamicSharedMemorySize;
    if (gated) return cudaFuncSetAttribute(extrapolate_bulk_kernel<K, CB16, true, true, false, true, STRIDED>, attr, (int)smem);
    const cudaError_t e =
        cudaFuncSetAttribute(extrapolate_bulk_kernel<K, CB16, true, false, false, true, STRIDED>, attr, (int)smem);
    if (e != cudaSuccess) return e;
    return cudaFuncSetAttribute(extrapolate_bulk_kernel<K, CB16, false, false, false, true, STRIDED>, attr, (int)smem);
}

template <bool CB16, bool STRIDED>
cudaError_t prepare_type(int K, bool gated, size_t smem) {
    switch (K) {
    case 1: return prepare_k<1, CB16, STRIDED>(gated, smem);
    case 2: return prepare_k<2, CB16, STRIDED>(gated, smem);
    case 3: return prepare_k<3, CB16, STRIDED>(gated, smem);
    case 4: return prepare_k<4, CB16, STRIDED>(gated, smem);
    case 5: return prepare_k<5, CB16, STRIDED>(gated, smem);
    case 6: return prepare_k<6, CB16, STRIDED>(gated, smem);
    case 7: return prepare_k<7, CB16, STRIDED>(gated, smem);
    case 8: return prepare_k<8, CB16, STRIDED>(gated, smem);
    default: return cudaErrorInvalidValue;
    }
}

template <bool CB16, bool STRIDED>
cudaError_t launch_type(const ExtrapArgs& a, int K, bool grouped, bool gated, int grid, size_t smem, cudaStream_t s) {
    switch (K) {
    case 1: return launch_k<1, CB16, STRIDED>(a, grouped, gated, grid, smem, s);
    case 2: return launch_k<2, CB16, STRIDED>(a, grouped, gated, grid, smem, s);
    case 3: return launch_k<3, CB16, STRIDED>(a, grouped, gated, grid, smem, s);
    case 4: return launch_k<4, CB16, STRIDED>(a, grouped, gated, grid, smem, s);
    case 5: return launch_k<5, CB16, STRIDED>(a, grouped, gated, grid, smem, s);
    case 6: return launch_k<6, CB16, STRIDED>(a, grouped, gated, grid, smem, s);
    case 7: return launch_k<7, CB16, STRIDED>(a, grouped, gated, grid, smem, s);
    case 8: return launch_k<8, CB16, STRIDED>(a, grouped, gated, grid, smem, s);
    default: return cudaErrorInvalidValue;
    }
}

}  // namespace
}  // namespace cbk
