// The library's host side (plan.cpp) over stand-ins for the CUDA runtime and the
// kernel launchers, for the CPU tests of its dispatch and of its error paths
// (test_dispatch_cpu.py). Nothing here runs a kernel: a launcher notes what it
// was given. Device properties are a GB300's.
#include <cuda_runtime.h>

#include <cstdio>
#include <cstring>
#include <string>

#include "../paper_2608_23429_gb300/csrc/cb_device.h"

namespace {
std::string g_log;           // one line per call noted
std::string g_fail;          // the next call of this name fails
cudaError_t g_last = cudaSuccess;
bool g_pinned = false;       // what host pointers count as
bool g_capturing = false;
int g_word = 0;              // the no-alloc status word

cudaError_t call(const char* name, const std::string& note = "") {
    const bool bad = g_fail == name;
    g_log += std::string(name) + (bad ? " FAILED" : "") + " " + note + "\n";
    if (!bad) return cudaSuccess;
    g_fail.clear();
    return g_last = cudaErrorMemoryAllocation;
}

std::string note(const cbk::ExtrapArgs& a, int K, bool src_bf16, int grid, size_t smem) {
    char b[256];
    std::snprintf(b, sizeof b, "K=%d src_bf16=%d grid=%d smem=%zu stages=%d x=%u gates=%u overlap=%d precise=%d items=%d",
                  K, src_bf16, grid, smem, a.stages, a.stage_x_bytes, a.stage_gate_bytes, a.overlap, a.precise, a.n_items);
    return b;
}

void kernel(cbk::PushArgs) {}
}  // namespace

extern "C" {
const char* stub_log() { return g_log.c_str(); }
void stub_reset() {
    g_log.clear();
    g_fail.clear();
    g_last = cudaSuccess;
    g_pinned = g_capturing = false;
}
void stub_fail(const char* name) { g_fail = name; }
void stub_host_memory(int pinned) { g_pinned = pinned != 0; }
void stub_capturing(int on) { g_capturing = on != 0; }
int stub_last_error() { return g_last; }

cudaError_t cudaGetDevice(int* d) { return *d = 0, cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr a, int) {
    *v = a == cudaDevAttrMultiProcessorCount                    ? 152
         : a == cudaDevAttrMaxSharedMemoryPerBlockOptin         ? 232448
         : a == cudaDevAttrMaxSharedMemoryPerMultiprocessor     ? 233472
         : a == cudaDevAttrL2CacheSize                          ? 135266304
                                                                : 0;
    return cudaSuccess;
}
const char* cudaGetErrorName(cudaError_t) { return "stub"; }
const char* cudaGetErrorString(cudaError_t) { return "stub"; }
cudaError_t cudaGetLastError() {
    const cudaError_t e = g_last;
    g_last = cudaSuccess;
    return e;
}
cudaError_t cudaMemsetAsync(void*, int, size_t, cudaStream_t) { return call("memset"); }
cudaError_t cudaMemcpyAsync(void* dst, const void*, size_t n, cudaMemcpyKind, cudaStream_t) {
    std::memset(dst, 0, n);
    return call("memcpy");
}
cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamIsCapturing(cudaStream_t, cudaStreamCaptureStatus* s) {
    *s = g_capturing ? cudaStreamCaptureStatusActive : cudaStreamCaptureStatusNone;
    return cudaSuccess;
}
cudaError_t cudaPointerGetAttributes(cudaPointerAttributes* at, const void* p) {
    at->type = g_pinned ? cudaMemoryTypeHost : cudaMemoryTypeUnregistered;
    at->devicePointer = g_pinned ? const_cast<void*>(p) : nullptr;
    return cudaSuccess;
}
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t*, const void*, void**) { return call("launch"); }
}

namespace cbk {
cudaError_t launch_extrapolate(const ExtrapArgs& a, int K, bool bf, int grid, cudaStream_t) {
    return call("direct", note(a, K, bf, grid, 0));
}
cudaError_t launch_extrapolate_gated(const ExtrapArgs& a, int K, bool bf, int grid, cudaStream_t) {
    return call("direct_gated", note(a, K, bf, grid, 0));
}
cudaError_t launch_extrapolate_precise(const ExtrapArgs& a, int K, bool bf, bool, int grid, cudaStream_t) {
    return call("direct_precise", note(a, K, bf, grid, 0));
}
cudaError_t extrapolate_blocks_per_sm(int, bool, int* n) { return *n = 2, cudaSuccess; }
size_t bulk_smem_bytes(size_t stage_bytes, int stages) { return 256 + (size_t)stages * stage_bytes; }
cudaError_t prepare_extrapolate_bulk(int, bool, size_t) { return cudaSuccess; }
cudaError_t launch_extrapolate_bulk(const ExtrapArgs& a, int K, bool bf, bool, int grid, size_t smem, cudaStream_t) {
    return call("bulk", note(a, K, bf, grid, smem));
}
cudaError_t prepare_extrapolate_bulk_precise(int, bool, bool, size_t) { return cudaSuccess; }
cudaError_t launch_extrapolate_bulk_precise(const ExtrapArgs& a, int K, bool bf, bool, bool, int grid, size_t smem,
                                            cudaStream_t) {
    return call("bulk_precise", note(a, K, bf, grid, smem));
}
cudaError_t prepare_extrapolate_bulk_strided(int, bool, bool, size_t) { return cudaSuccess; }
cudaError_t launch_extrapolate_bulk_strided(const ExtrapArgs& a, int K, bool bf, bool, bool, int grid, size_t smem,
                                            cudaStream_t) {
    return call("bulk_strided", note(a, K, bf, grid, smem));
}
cudaError_t prepare_extrapolate_bulk_gated(int, bool, size_t) { return cudaSuccess; }
cudaError_t launch_extrapolate_bulk_gated(const ExtrapArgs& a, int K, bool bf, int grid, size_t smem, cudaStream_t) {
    return call("bulk_gated", note(a, K, bf, grid, smem));
}
cudaError_t launch_epilogue(const ExtrapArgs& a, int grid, cudaStream_t) { return call("epilogue", note(a, 1, true, grid, 0)); }
cudaError_t epilogue_blocks_per_sm(int* n) { return *n = 3, cudaSuccess; }
cudaError_t launch_push(const PushArgs& a, bool, bool, int grid, size_t smem, cudaStream_t s) {
    return launch_overlapped(kernel, grid, kThreads, smem, s, a);
}
cudaError_t push_blocks_per_sm(bool, bool, size_t, int* n) { return *n = 4, cudaSuccess; }
cudaError_t noalloc_status_word(int, int** word) { return *word = &g_word, cudaSuccess; }
cudaError_t take_status(int*, int* status, cudaStream_t) {
    const cudaError_t e = call("take_status");
    if (e == cudaSuccess) *status = 0;
    return e;
}
}  // namespace cbk
