// Internal: kernel argument blocks and launchers shared by the host plan
// (plan.cpp) and the kernels (extrapolate*.cu, epilogue.cu, push.cu), and the
// library's own status block (static_status.cu). Not part of the ABI.
#pragma once

#include <cuda_runtime.h>

#include <cstdint>

namespace cbk {

constexpr int kThreads = 256;     // threads per CTA
constexpr int kVecElems = 8;      // elements per vector (16 B of bf16, 32 B of fp32)
constexpr int kMaxItems = 256;    // work items (tensors, or residual groups) per launch
constexpr int kMaxMembers = 256;  // branch tensors per launch

// Launches a kernel that, with a.overlap, may start while the stream's previous
// one is still ending (programmatic dependent launch): its blocks are placed as
// that one's leave, and wait, before they touch global memory (after_previous),
// until it has ended and its writes are visible. GB300: one step of 2 x [1, 256,
// 1152] 5.0 -> 4.4 us, of the tiny fp32 workload 6.2 -> 5.0 us, a DDIM-50 run of
// one DiT-XL/2 256^2 image 1170 -> 1126 us. Grids that leave SMs free on purpose
// do not overlap: the next grid's blocks would fill just those, out of balance
// (FLUX.1-dev, 3/4 of the SMs: 1792 -> 1836 us).
template <typename Args>
cudaError_t launch_overlapped(void (*kernel)(Args), int grid, int threads, size_t smem, cudaStream_t s, const Args& a) {
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = a.overlap;
    cudaLaunchConfig_t c{};
    c.gridDim = dim3((unsigned)grid);
    c.blockDim = dim3((unsigned)threads);
    c.dynamicSmemBytes = smem;
    c.stream = s;
    c.attrs = &at;
    c.numAttrs = 1;
    void* args[] = {const_cast<void*>(static_cast<const void*>(&a))};
    const cudaError_t e = cudaLaunchKernelExC(&c, reinterpret_cast<const void*>(kernel), args);
    if (e != cudaSuccess) (void)cudaGetLastError();  // returned here, so not left for a check of the caller's own launches
    return e;
}

#ifdef __CUDACC__
// At the head of every kernel launched by launch_overlapped: lets the next one
// be placed, and waits for the previous one's end.
__device__ __forceinline__ void after_previous() {
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    asm volatile("griddepcontrol.wait;" ::: "memory");
}
#endif

// Vectors each thread handles per tile: two 16-B vectors for a bf16 cache,
// one 32-B vector for an fp32 cache (both give 2*K 16-B loads in flight).
__host__ __device__ constexpr int vectors_per_thread(bool cache_bf16) { return cache_bf16 ? 2 : 1; }
__host__ __device__ constexpr long long tile_elems(bool cache_bf16) {
    return (long long)kThreads * vectors_per_thread(cache_bf16) * kVecElems;
}

// One skipped-step launch. Items are the units of work: a single branch
// tensor, or (with hidden states) all branch tensors of one residual group.
// Every item is cut into tiles of tile_elems() elements; tiles are numbered
// consecutively across items and dealt to a persistent grid.
struct ExtrapArgs {
    // byte address of the history: entry j of member m starts at
    // hist_base + slot_off[j] + m_off[m] (the ring arena and offsets inside it;
    // for a full step's epilogue, base 0 and m_off the new features' addresses)
    unsigned long long hist_base;
    long long slot_off[8];       // byte offset of history entry j (0 = oldest)
    float w_hi[8];               // fp32(w_j)
    float w_lo[8];               // fp32(w_j - w_hi[j])
    unsigned w_anchor[8];        // 2 |w_j|, rounded up: fp32, or bf16 twice for bf16 sources (see sum_vec)
    float w_guard[8];            // (K+2) u (1.01) 2^9 |w_hi[j]|: the fast path's scaled error bound
    int n_items;
    int tiles_total;
    int out_bf16;    // predictions are bf16 (else fp32)
    int resid_bf16;  // hidden states are bf16 (else fp32)
    int precise;     // 1: compensated arithmetic for every element
    int copy_out;    // full-step epilogue: outputs receive the (K = 1) sources converted, not a prediction
    int stages;                  // bulk variant: shared-memory pipeline depth
    unsigned stage_x_bytes;      // bulk variant: bytes of a tile's hidden state staged behind the K chunks (0: not staged)
    unsigned stage_gate_bytes;   // bulk variant: bytes per stage for gate rows (0: gates read from global)
    unsigned long long wait_ns;  // bulk variant: limit of every barrier wait
    int* status;                 // bulk variant: device status word (codes OR-ed in)
    int overlap;                 // host only: see launch_overlapped
    int withhold_first;          // bulk variant, tests only: announce but never issue the first copies
    int keep_tiles;              // bulk variant: whole tiles whose history L2 is to keep for the next step
    // bulk variant: tile_begin and tiles_total count whole tiles only (none of
    // items with vec_ok = 0); the ragged last tiles are numbered after them
    int n_ragged;
    int any_scalar;              // bulk variant: some item has vec_ok = 0
    short ragged[kMaxItems];     // items with a ragged last tile
    int tile_begin[kMaxItems + 1];
    long long numel[kMaxItems];
    void* resid[kMaxItems];           // hidden state of the item, or null
    unsigned char nb[kMaxItems];      // member tensors of the item
    unsigned char vec_ok[kMaxItems];  // every pointer of the item is 16-B aligned
    short first[kMaxItems];           // first member index
    long long m_off[kMaxMembers];     // byte offset of the member tensor inside one slot
    void* m_out[kMaxMembers];         // prediction output of the member, or null
    // gated hidden-state update (x <- x + sum_b g_b * P_b); read by gated kernels only
    int gate_bf16;                      // gates are bf16 (else fp32)
    const void* m_gate[kMaxMembers];    // gate [batch, hidden] of the member, or null (gate 1)
    unsigned i_hidden[kMaxItems];       // hidden size of the item's tensors
    unsigned i_row[kMaxItems];          // tokens * hidden of the item's tensors
    unsigned long long i_hidden_magic[kMaxItems];  // ceil(2^64 / i_hidden) (0: i_hidden = 1)
    unsigned long long i_row_magic[kMaxItems];     // ceil(2^64 / i_row) (0: i_row = 1)
};

// One full-step launch: copy/convert every tensor into one ring slot.
struct PushArgs {
    int overlap;          // host only: see launch_overlapped
    unsigned char* slot;  // base of the destination slot
    int n_items;
    int tiles_total;
    int tile_begin[kMaxItems + 1];
    long long numel[kMaxItems];
    long long off[kMaxItems];  // byte offset of the tensor inside the slot
    const void* src[kMaxItems];
    unsigned char vec_ok[kMaxItems];
};

constexpr long long push_tile_elems = (long long)kThreads * 2 * kVecElems;


cudaError_t launch_extrapolate(const ExtrapArgs& a, int K, bool cache_bf16, int grid, cudaStream_t s);
// gated variant of the direct kernel (extrapolate_gated.cu)
cudaError_t launch_extrapolate_gated(const ExtrapArgs& a, int K, bool cache_bf16, int grid, cudaStream_t s);
// with fp32 predictions or hidden states, gated or not (extrapolate_precise.cu)
cudaError_t launch_extrapolate_precise(const ExtrapArgs& a, int K, bool cache_bf16, bool gated, int grid,
                                       cudaStream_t s);
cudaError_t extrapolate_blocks_per_sm(int K, bool cache_bf16, int* blocks);

// Bulk-copy pipeline variant (extrapolate_bulk.cu). Its barrier block holds
// the full and empty barriers of at most kMaxStages stages.
constexpr int kMaxStages = 16;
// Shape of the bulk kernel: CTAs per SM, consumer warps of a CTA, elements of
// a tile.
//
// `precise` launches (fp32 predictions or hidden states) are bound by the
// latency of their arithmetic: as many warps as hold one vector per thread
// without spilling in the loop, 20 of 96 registers for bf16 sources, 12 of 168
// for fp32 ones (with the producer a multiple of the four schedulers). GB300,
// DiT-XL/2 512^2, K = 4, fp32 hidden states, with and without gates: 7 warps
// 1048 us, 11 871 / 666 us, 15 607 / 509 us, 19 577 / 458 us, 23 (spilling)
// 746 / 512 us, at a time when the consumers branched once per pair (19 warps take
// 528 / 443 us now); 11 against 15 warps for fp32 sources, K = 8: 379 / 454 us.
//
// Others: two CTAs of 8 consumer warps, else one (16 for bf16 tiles): two
// for K = 1, for bf16 prediction-only launches (not `grouped`) with
// K <= 2 and for ungated bf16 grouped launches with K = 2..3, where two
// vectors per thread still fit the register budget. Ungated bf16 grouped
// launches with K = 1 (the full-step epilogue from bf16 features) stream
// faster as one CTA of 16 warps (GB300: FLUX 88.3 -> 94.1 %, DiT-256
// 81.2 -> 90.1 % of the copy peak, PixArt unchanged); gated ones do not
// (DiT-256 88.0 -> 63.9 %) and keep two.
struct BulkShape {
    int ctas_per_sm;
    int consumer_warps;
    int tile;
};
// Compensated launches whose gate rows are staged with their member: where the
// loads' latency counts more than the rows' room and traffic (GB300, 28 groups of
// two, [8, 256, 1152], gates from global memory -> staged: fp32 sources, K = 1, 2, 4,
// 8 247 -> 207, 288 -> 247, 382 -> 381, 670 -> 670 us; bf16 sources, K = 1..4, bf16 gates
// 204 -> 186, 228 -> 219, 251 -> 244, 280 -> 272 us, fp32 gates 185 -> 186, 217 -> 219,
// 240 -> 245, 272 -> 276 us).
__host__ __device__ constexpr bool staged_gates(int K, bool src_bf16) { return !src_bf16 || K <= 2; }
__host__ __device__ constexpr BulkShape bulk_shape(int K, bool src_bf16, bool grouped, bool gated, bool precise,
                                                   bool strided) {
    // fp32 sources with gates and K <= 2: 15 warps (K = 1: 374 -> 343 us); so for
    // the strided kernels with hidden states, which hold more (8 x 3 x [3, 333,
    // 577], gates: 63.7 -> 59.8 us, K = 8 75 -> 70 us, [8, 333, 577] the same)
    if (precise) {
        const int warps = src_bf16 ? (strided && grouped ? 15 : 19) : gated && K <= 2 ? 15 : 11;
        return BulkShape{1, warps, warps * 32 * kVecElems};
    }
    const bool two = (K == 1 && !(src_bf16 && grouped && !gated)) || (src_bf16 && !grouped && K <= 2) ||
                     (src_bf16 && grouped && !gated && K >= 2 && K <= 3);
    return BulkShape{two ? 2 : 1, (src_bf16 && !two) ? 16 : 8, (int)tile_elems(src_bf16)};
}
size_t bulk_smem_bytes(size_t stage_bytes, int stages);
cudaError_t prepare_extrapolate_bulk(int K, bool cache_bf16, size_t smem);
// grouped: some item updates a hidden state or has several members (the
// kernel's hidden-state bookkeeping); it also selects the CTA shape.
cudaError_t launch_extrapolate_bulk(const ExtrapArgs& a, int K, bool cache_bf16, bool grouped, int grid, size_t smem,
                                    cudaStream_t s);
// with fp32 predictions or hidden states, gated or not (extrapolate_bulk_precise*.cu)
cudaError_t prepare_extrapolate_bulk_precise(int K, bool cache_bf16, bool gated, size_t smem);
cudaError_t launch_extrapolate_bulk_precise(const ExtrapArgs& a, int K, bool cache_bf16, bool grouped, bool gated,
                                            int grid, size_t smem, cudaStream_t s);
// for items whose outputs, hidden states or gates are off the 16-byte grid (extrapolate_bulk_strided*.cu)
cudaError_t prepare_extrapolate_bulk_strided(int K, bool cache_bf16, bool gated, size_t smem);
cudaError_t launch_extrapolate_bulk_strided(const ExtrapArgs& a, int K, bool cache_bf16, bool grouped, bool gated,
                                            int grid, size_t smem, cudaStream_t s);
// gated variant of the bulk kernel (extrapolate_bulk_gated.cu)
cudaError_t prepare_extrapolate_bulk_gated(int K, bool cache_bf16, size_t smem);
cudaError_t launch_extrapolate_bulk_gated(const ExtrapArgs& a, int K, bool cache_bf16, int grid, size_t smem,
                                          cudaStream_t s);

// Full-step epilogue kernel (epilogue.cu) for ungated bf16 features: a
// one-entry history of weight 1 on 2048-element tiles, one 8-element vector
// per thread and tile.
constexpr long long epilogue_tile_elems = (long long)kThreads * kVecElems;
cudaError_t launch_epilogue(const ExtrapArgs& a, int grid, cudaStream_t s);
cudaError_t epilogue_blocks_per_sm(int* blocks);

cudaError_t launch_push(const PushArgs& a, bool src_bf16, bool dst_bf16, int grid, size_t smem, cudaStream_t s);
// with `smem` bytes of dynamic shared memory, for which the kernel's limit is raised
cudaError_t push_blocks_per_sm(bool src_bf16, bool dst_bf16, size_t smem, int* blocks);

// Status word of cb_extrapolate_noalloc in the library's own device block
// (static_status.cu): its device address on `device`, which must be the
// current device. The first call per device looks the address up.
constexpr int kMaxStatusDevices = 64;
cudaError_t noalloc_status_word(int device, int** word);
// Hands the word over to *status (memory the device can write) and clears it.
cudaError_t take_status(int* word, int* status, cudaStream_t s);

}  // namespace cbk
