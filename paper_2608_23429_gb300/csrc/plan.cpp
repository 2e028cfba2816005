// Host side of libchebboost: the plan (the offline weight precomputation of
// Sec. 3.3; Alg. 1 offline stage), the history buffer's ring bookkeeping, the
// online weights (Sec. 3.2 Eq. barycentric_coeff) and the kernel launches.
// Everything here is fp64 host arithmetic that runs in microseconds per call;
// all device work is in push.cu (cache write), epilogue.cu (full-step
// epilogue) and the extrapolate*.cu instantiations of the skipped-step kernels.
#include <cuda_runtime.h>

#include <algorithm>
#include <atomic>
#include <cmath>
#include <cstdint>
#include <cstring>
#include <memory>
#include <new>
#include <string>
#include <vector>

#include "../../include/chebboost.h"
#include "cb_device.h"

namespace {

thread_local std::string g_last_error;

int cuda_fail(cudaError_t e, const char* where) {
    g_last_error = std::string(where) + ": " + cudaGetErrorName(e) + ": " + cudaGetErrorString(e);
    return CB_ERR_CUDA;
}

size_t esize(cb_dtype d) { return d == CB_BF16 ? 2 : 4; }
bool valid_dtype(cb_dtype d) { return d == CB_BF16 || d == CB_FP32; }
size_t round_up(size_t x, size_t a) { return (x + a - 1) / a * a; }

// Barycentric weights rho_j = 1 / prod_{k != j} (x_j - x_k) (App. A, Eq. general_weights).
bool rho_of(const double* x, int n, double* rho) {
    for (int j = 0; j < n; ++j) {
        double d = 1.0;
        for (int k = 0; k < n; ++k)
            if (k != j) d *= x[j] - x[k];
        if (d == 0.0 || !std::isfinite(d)) return false;
        rho[j] = 1.0 / d;
    }
    return true;
}

// Interpolation coefficients w_j = (rho_j / (x - x_j)) / sum_i rho_i / (x - x_i)
// (Sec. 3.2, Eq. barycentric_coeff). A target on a node gives the unit vector.
void coeff_of(const double* x, const double* rho, int n, double xq, double* w) {
    for (int j = 0; j < n; ++j)
        if (xq == x[j]) {
            for (int i = 0; i < n; ++i) w[i] = (i == j) ? 1.0 : 0.0;
            return;
        }
    double den = 0.0;
    for (int i = 0; i < n; ++i) {
        w[i] = rho[i] / (xq - x[i]);
        den += w[i];
    }
    for (int i = 0; i < n; ++i) w[i] /= den;
}

struct DeviceInfo {
    int device = -1;
    int sms = 0;
    int smem_optin = 0;                    // largest dynamic shared memory per CTA
    int smem_per_sm = 0;                   // shared memory of one SM
    int l2_bytes = 0;                      // L2 cache
    int occ_extrap[2][CB_MAX_K + 1] = {};  // [cache_bf16][K]
    int occ_push[2][2] = {};               // [src_bf16][dst_bf16]
    int occ_epilogue = 0;                  // epilogue kernel (bf16 features, no gates)
    int bulk_stages[2][CB_MAX_K + 1] = {};  // 1 once the kernel's shared-memory limit is raised
    int bulk_gated[2][CB_MAX_K + 1] = {};   // the same for the gated kernel
    int bulk_precise[2][2][CB_MAX_K + 1] = {};  // [gated]: the same for fp32 predictions or hidden states
    int bulk_strided[2][2][CB_MAX_K + 1] = {};  // [gated]: the same for items off the 16-byte grid
};

}  // namespace

struct cb_plan {
    int K = 0;
    cb_dtype cache_dtype = CB_BF16;
    double t_min = 0, t_max = 1;
    std::vector<cb_tensor_desc> tensors;
    std::vector<std::vector<int>> groups;  // residual group -> member tensors
    std::vector<double> node_t;            // full-step timesteps, sampling order
    std::vector<double> node_tau;
    int dir = 0;                           // +1 increasing, -1 decreasing t
    std::vector<double> rho_win;           // rho of node window i: rho_win[i*K + j]
    std::vector<long long> off;            // byte offset of tensor i inside a slot
    std::vector<long long> sh_tokens;      // [batch, tokens, hidden] of each tensor (0: unset)
    std::vector<long long> sh_hidden;
    size_t slot_bytes = 0;
    // bound history buffer
    unsigned char* cache = nullptr;
    // ring state of H
    double slot_t[CB_MAX_K] = {};
    int next = 0;   // slot written by the next push
    int count = 0;  // entries held (<= K)
    bool has_last = false;
    double last_t = 0;
    bool status_clear = false;  // the device status word was zeroed since binding
    int kernel = CB_KERNEL_AUTO;
    unsigned long long wait_ns = 1000000000ull;
    int withhold_first = 0;
    bool partial = false;  // extrapolate from fewer than K entries while H fills
    DeviceInfo dev;
    // value-initialised: no field of a launch's arguments is ever left unset
    std::unique_ptr<cbk::ExtrapArgs> eargs{new cbk::ExtrapArgs()};
    std::unique_ptr<cbk::ExtrapArgs> eargs2;  // part of a call's items (made when first needed)
    std::unique_ptr<cbk::PushArgs> pargs{new cbk::PushArgs()};

    double tau(double t) const { return 2.0 * (t - t_min) / (t_max - t_min) - 1.0; }
    int* status_word() const { return reinterpret_cast<int*>(cache + slot_bytes * (size_t)K); }
    int oldest() const { return count < K ? 0 : next; }
};

namespace {

int ensure_device(cb_plan* p) {
    int d = 0;
    cudaError_t e = cudaGetDevice(&d);
    if (e != cudaSuccess) return cuda_fail(e, "cudaGetDevice");
    if (p->dev.device != d) {
        DeviceInfo info;
        info.device = d;
        e = cudaDeviceGetAttribute(&info.sms, cudaDevAttrMultiProcessorCount, d);
        if (e != cudaSuccess) return cuda_fail(e, "cudaDeviceGetAttribute");
        e = cudaDeviceGetAttribute(&info.smem_optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, d);
        if (e != cudaSuccess) return cuda_fail(e, "cudaDeviceGetAttribute");
        e = cudaDeviceGetAttribute(&info.smem_per_sm, cudaDevAttrMaxSharedMemoryPerMultiprocessor, d);
        if (e != cudaSuccess) return cuda_fail(e, "cudaDeviceGetAttribute");
        e = cudaDeviceGetAttribute(&info.l2_bytes, cudaDevAttrL2CacheSize, d);
        if (e != cudaSuccess) return cuda_fail(e, "cudaDeviceGetAttribute");
        p->dev = info;
    }
    return CB_OK;
}

int extrap_grid(cb_plan* p, int K, bool cb16, int tiles, int* grid) {
    int& occ = p->dev.occ_extrap[cb16 ? 1 : 0][K];
    if (occ == 0) {
        cudaError_t e = cbk::extrapolate_blocks_per_sm(K, cb16, &occ);
        if (e != cudaSuccess || occ <= 0) {
            occ = 0;
            return cuda_fail(e == cudaSuccess ? cudaErrorInvalidConfiguration : e, "occupancy");
        }
    }
    long long g = (long long)p->dev.sms * occ;
    *grid = (int)(tiles < g ? tiles : g);
    return CB_OK;
}

// Largest gate staging per pipeline stage (two rows of 4096 fp32 channels).
constexpr size_t kMaxStagedGateBytes = 32768;

// Pipeline of the bulk kernel: as many stages of `stage_bytes` as fit in one
// CTA's shared memory, at most kMaxStages, and the CTAs per SM. A shape made
// for two CTAs per SM runs one, with all of the SM's shared memory, when half
// of it cannot hold `min_stages`. The kernel's dynamic shared-memory limit is
// raised to the device maximum once per instantiation.
int bulk_config(cb_plan* p, int K, bool cb16, bool gated, bool precise, bool strided, int shape_ctas,
                size_t stage_bytes, int min_stages, int* stages, size_t* smem, int* ctas_per_sm) {
    int& prepared = strided ? p->dev.bulk_strided[gated ? 1 : 0][cb16 ? 1 : 0][K]
                    : precise ? p->dev.bulk_precise[gated ? 1 : 0][cb16 ? 1 : 0][K]
                    : gated ? p->dev.bulk_gated[cb16 ? 1 : 0][K]
                            : p->dev.bulk_stages[cb16 ? 1 : 0][K];
    if (prepared == 0) {
        const size_t most = (size_t)p->dev.smem_optin;
        cudaError_t e = strided   ? cbk::prepare_extrapolate_bulk_strided(K, cb16, gated, most)
                        : precise ? cbk::prepare_extrapolate_bulk_precise(K, cb16, gated, most)
                        : gated ? cbk::prepare_extrapolate_bulk_gated(K, cb16, most)
                                : cbk::prepare_extrapolate_bulk(K, cb16, most);
        if (e != cudaSuccess) return cuda_fail(e, "cudaFuncSetAttribute");
        prepared = 1;
    }
    // with several CTAs per SM each gets its share of the SM's shared memory
    // (less the 1 KB the hardware reserves per CTA)
    for (int per_sm = shape_ctas; per_sm >= 1; --per_sm) {
        size_t cap = (size_t)p->dev.smem_optin;
        if (per_sm > 1) cap = std::min(cap, (size_t)p->dev.smem_per_sm / per_sm - 1024);
        int s = cbk::kMaxStages;
        while (s > 1 && cbk::bulk_smem_bytes(stage_bytes, s) > cap) --s;
        *stages = cbk::bulk_smem_bytes(stage_bytes, s) <= cap ? s : 0;
        *smem = cbk::bulk_smem_bytes(stage_bytes, s);
        *ctas_per_sm = per_sm;
        if (*stages >= min_stages) break;
    }
    return CB_OK;
}

// The cache write's grid, and shared memory that it does not use but that keeps
// an overlapping launch's blocks from crowding on some SMs.
int push_grid(cb_plan* p, bool sb, bool db, int tiles, int* grid, size_t* smem) {
    // fewer concurrent copy streams stream faster than full occupancy (FLUX
    // cache writes: bf16 sources best at 4 CTAs per SM, fp32 sources at 3)
    const int cap = sb ? 4 : 3;
    *smem = (size_t)p->dev.smem_per_sm / (cap + 1);
    int& occ = p->dev.occ_push[sb ? 1 : 0][db ? 1 : 0];
    if (occ == 0) {
        cudaError_t e = cbk::push_blocks_per_sm(sb, db, *smem, &occ);
        if (e != cudaSuccess || occ <= 0) {
            occ = 0;
            return cuda_fail(e == cudaSuccess ? cudaErrorInvalidConfiguration : e, "occupancy");
        }
    }
    long long g = (long long)p->dev.sms * occ;
    *grid = (int)(tiles < g ? tiles : g);
    return CB_OK;
}

bool aligned(const void* ptr, size_t a) { return ((uintptr_t)ptr % a) == 0; }

// Multiplier of the kernels' division by d < 2^32: ceil(2^64 / d), 0 for d <= 1.
unsigned long long div_magic(unsigned d) { return d <= 1 ? 0ull : ~0ull / d + 1ull; }

// 2 |w| as the compensated sums take it for their anchor (sum_vec): rounded up,
// so far that K rounded additions cannot bring the sum below 2 sum_j |w_j F_j|.
// fp32 for fp32 sources; for bf16 ones bf16, twice in one word.
unsigned anchor_weight(double w, int K, bool src_bf16) {
    const float x = (float)(2.0 * w * (1.0 + K * std::ldexp(1.0, src_bf16 ? -8 : -22)));
    unsigned b;
    std::memcpy(&b, &x, sizeof b);
    if (!src_bf16) return b;
    b = (b + 0xFFFFu) >> 16;  // up to the next bf16 (infinity past the largest)
    return b << 16 | b;
}

// Logical history window: n entries, oldest first, with the slot of each.
struct Window {
    int n;
    double t[CB_MAX_K];
    double tau[CB_MAX_K];
    int slot[CB_MAX_K];
};

// rho for a window: reuse the offline table when the window is K consecutive
// nodes of the plan, otherwise compute it the same way now.
bool window_rho(const cb_plan* p, const Window& w, double* rho) {
    const int K = p->K;
    const int n = (int)p->node_t.size();
    if (w.n == K) {
        for (int i = 0; i + K <= n; ++i) {
            if (p->node_t[i] != w.t[0]) continue;
            bool match = true;
            for (int j = 1; j < K && match; ++j) match = p->node_t[i + j] == w.t[j];
            if (match) {
                std::memcpy(rho, &p->rho_win[(size_t)i * K], sizeof(double) * K);
                return true;
            }
        }
    }
    return rho_of(w.tau, w.n, rho);
}

int weights_for(const cb_plan* p, const Window& w, double t_target, double* out) {
    if (!std::isfinite(t_target)) return CB_ERR_ARG;
    double rho[CB_MAX_K];
    if (!window_rho(p, w, rho)) return CB_ERR_NODES_DEGENERATE;
    for (int j = 0; j < w.n; ++j)
        if (t_target == w.t[j]) {  // the target is a cached node: return it exactly
            for (int i = 0; i < w.n; ++i) out[i] = (i == j) ? 1.0 : 0.0;
            return CB_OK;
        }
    coeff_of(w.tau, rho, w.n, p->tau(t_target), out);
    return CB_OK;
}

// Entries a skipped step may use: all K once H is full; with partial history
// enabled, whatever H holds (at least one); otherwise none.
int live_entries(const cb_plan* p) {
    if (p->count == p->K) return p->K;
    if (p->partial && p->count >= 1) return p->count;
    return 0;
}

Window live_window(const cb_plan* p, int n) {
    Window w{};
    w.n = n;
    const int o = p->oldest();
    for (int j = 0; j < n; ++j) {
        w.slot[j] = (o + j) % p->K;
        w.t[j] = p->slot_t[w.slot[j]];
        w.tau[j] = p->tau(w.t[j]);
    }
    return w;
}

// Gates (one per tensor, [batch, hidden] of gate_dtype, null = 1) apply to the
// hidden-state update of a grouped tensor: its shape must be set, its group's
// tensors must share it, and indexing stays in 32 bits.
int check_gates(const cb_plan* p, const void* const* gates, cb_dtype gate_dtype) {
    if (!gates) return CB_OK;
    if (!valid_dtype(gate_dtype)) return CB_ERR_ARG;
    const int n = (int)p->tensors.size();
    for (int i = 0; i < n; ++i) {
        if (!gates[i]) continue;
        if (p->sh_hidden[i] <= 0) return CB_ERR_ARG;  // cb_plan_set_shapes first
        if (!aligned(gates[i], esize(gate_dtype))) return CB_ERR_ALIGN;
        if (p->tensors[i].numel > 0xFFFFFFFFLL) return CB_ERR_LIMIT;
    }
    return CB_OK;
}

// The device status word is zeroed once after binding, on the stream of the
// first launch, after that launch's arguments have all been validated.
int clear_status_once(cb_plan* p, void* stream) {
    if (p->status_clear) return CB_OK;
    cudaError_t e = cudaMemsetAsync(p->status_word(), 0, sizeof(int), (cudaStream_t)stream);
    if (e != cudaSuccess) return cuda_fail(e, "cudaMemsetAsync");
    p->status_clear = true;
    return CB_OK;
}

// A history buffer given with the call instead of the bound arena, and the
// status word of device `device` its launches record into (cb_extrapolate_noalloc;
// null: none). `launched` is set once a launch is under way.
struct CallerHistory {
    const unsigned char* hist;
    int* status;
    int device;
    bool launched;
};

// Devices whose no-alloc status word may hold a code that nobody was told: a
// call failed between its launch and the handover that clears the word.
std::atomic<bool> g_unclaimed[cbk::kMaxStatusDevices];

// What the launches of one call share.
struct Launch {
    cb_plan* p;
    int K;
    bool cb16;         // source type: bf16 (else fp32)
    bool full_step;    // the sources are a full step's new features
    size_t res;        // bytes of a hidden-state element
    cb_dtype gate_dtype;
    void* stream;
    CallerHistory* ch;
};

int clear_status(Launch& L) {
    CallerHistory* ch = L.ch;
    if (!ch) return clear_status_once(L.p, L.stream);
    // Its word is zero, but for what a failed call left there. A clearing that is
    // captured runs later: the word stays unclaimed until one has been enqueued.
    if (ch->status && !ch->launched && g_unclaimed[ch->device]) {
        const cudaStream_t s = (cudaStream_t)L.stream;
        cudaStreamCaptureStatus capture = cudaStreamCaptureStatusNone;
        cudaError_t e = cudaStreamIsCapturing(s, &capture);
        if (e == cudaSuccess) e = cudaMemsetAsync(ch->status, 0, sizeof(int), s);
        if (e != cudaSuccess) return cuda_fail(e, "status word");
        if (capture == cudaStreamCaptureStatusNone) g_unclaimed[ch->device] = false;
    }
    ch->launched = true;
    return CB_OK;
}

// Cut the items into tiles of te elements, numbered across items. `split` (the
// bulk kernel's numbering): whole tiles first, then the ragged last ones;
// items with vec_ok = 0 have none, unless the launch is `strided`.
int cut_tiles(cbk::ExtrapArgs& A, long long te, bool split, bool strided = false) {
    long long tiles = 0;
    A.n_ragged = A.any_scalar = 0;
    for (int i = 0; i < A.n_items; ++i) {
        A.tile_begin[i] = (int)tiles;
        if (split && !strided && !A.vec_ok[i]) {
            A.any_scalar = 1;
            continue;
        }
        if (split && A.numel[i] % te != 0) A.ragged[A.n_ragged++] = (short)i;
        tiles += split ? A.numel[i] / te : (A.numel[i] + te - 1) / te;
        if (tiles + A.n_ragged > 0x7FFFFFFFLL) return CB_ERR_LIMIT;
    }
    A.tile_begin[A.n_items] = A.tiles_total = (int)tiles;
    return CB_OK;
}

bool any_gate(const cbk::ExtrapArgs& A) {
    for (int i = 0; i < A.n_items; ++i)
        for (int m = 0; m < A.nb[i]; ++m)
            if (A.m_gate[A.first[i] + m]) return true;
    return false;
}

// The items of A whose flag is `want`, with their members, as B.
void take_items(const cbk::ExtrapArgs& A, const bool* flag, bool want, cbk::ExtrapArgs& B) {
    B = A;
    B.n_items = 0;
    int members = 0;
    for (int i = 0; i < A.n_items; ++i) {
        if (flag[i] != want) continue;
        const int k = B.n_items++;
        B.numel[k] = A.numel[i];
        B.resid[k] = A.resid[i];
        B.nb[k] = A.nb[i];
        B.vec_ok[k] = A.vec_ok[i];
        B.first[k] = (short)members;
        B.i_hidden[k] = A.i_hidden[i];
        B.i_row[k] = A.i_row[i];
        B.i_hidden_magic[k] = A.i_hidden_magic[i];
        B.i_row_magic[k] = A.i_row_magic[i];
        for (int m = 0; m < A.nb[i]; ++m, ++members) {
            B.m_off[members] = A.m_off[A.first[i] + m];
            B.m_out[members] = A.m_out[A.first[i] + m];
            B.m_gate[members] = A.m_gate[A.first[i] + m];
        }
    }
}

int launch_direct(Launch& L, cbk::ExtrapArgs& A) {
    int grid = 0;
    int r = cut_tiles(A, cbk::tile_elems(L.cb16), false);
    if (r == CB_OK) r = extrap_grid(L.p, L.K, L.cb16, A.tiles_total, &grid);
    if (r == CB_OK) r = clear_status(L);
    if (r != CB_OK) return r;
    const cudaStream_t s = (cudaStream_t)L.stream;
    const bool gated = any_gate(A);
    cudaError_t e = A.precise ? cbk::launch_extrapolate_precise(A, L.K, L.cb16, gated, grid, s)
                    : gated   ? cbk::launch_extrapolate_gated(A, L.K, L.cb16, grid, s)
                              : cbk::launch_extrapolate(A, L.K, L.cb16, grid, s);
    return e == cudaSuccess ? CB_OK : cuda_fail(e, "extrapolate launch");
}

int launch_epilogue(Launch& L, cbk::ExtrapArgs& A) {
    int& occ = L.p->dev.occ_epilogue;
    if (occ == 0) {
        cudaError_t e = cbk::epilogue_blocks_per_sm(&occ);
        if (e != cudaSuccess || occ <= 0) {
            occ = 0;
            return cuda_fail(e == cudaSuccess ? cudaErrorInvalidConfiguration : e, "occupancy");
        }
    }
    int r = cut_tiles(A, cbk::epilogue_tile_elems, false);
    if (r == CB_OK) r = clear_status(L);
    if (r != CB_OK) return r;
    const int grid = (int)std::min<long long>(A.tiles_total, (long long)L.p->dev.sms * occ);
    A.overlap = 1;
    cudaError_t e = cbk::launch_epilogue(A, grid, (cudaStream_t)L.stream);
    return e == cudaSuccess ? CB_OK : cuda_fail(e, "epilogue launch");
}

// The bulk-copy pipeline. `strided`: every item is off the 16-byte grid on its
// way out (see the kernel's STRIDED).
int launch_bulk(Launch& L, cbk::ExtrapArgs& A, bool strided) {
    cb_plan* p = L.p;
    const int K = L.K, items = A.n_items;
    const bool cb16 = L.cb16, gated = any_gate(A), precise = A.precise != 0 || strided;
    // the grouped kernel (hidden-state bookkeeping) for gates, hidden states or multi-member items
    int max_nb = 1;
    bool grouped = gated, any_resid = false;
    for (int i = 0; i < items; ++i) {
        max_nb = std::max(max_nb, (int)A.nb[i]);
        any_resid = any_resid || A.resid[i] != nullptr;
        grouped = grouped || A.resid[i] != nullptr || A.nb[i] > 1;
    }
    const cbk::BulkShape shape = cbk::bulk_shape(K, cb16, grouped, gated, precise, strided);
    int rc = cut_tiles(A, shape.tile, true, strided);
    if (rc != CB_OK) return rc;
    // Hidden states travel through shared memory with the first member of their
    // group (not those off the 16-byte grid). Launches that recompute guarded
    // elements hold a whole group and need one stage ahead of it; compensated
    // ones hold nothing.
    A.stage_x_bytes = any_resid && !strided ? (unsigned)(shape.tile * L.res) : 0u;
    A.stage_gate_bytes = 0;
    const bool hold = grouped && !precise;
    const int min_stages = hold ? max_nb + 1 : 2;
    // Gate rows travel with their member when every gated tile touches at
    // most two batches (a batch holds a tile or more) and two rows are small.
    if (gated && !strided && (!precise || cbk::staged_gates(K, cb16))) {
        const size_t gs = esize(L.gate_dtype);
        size_t need = 0;
        bool fits = true;
        for (int i = 0; i < items; ++i) {
            bool gated_item = false;
            for (int m = 0; m < A.nb[i]; ++m) gated_item = gated_item || A.m_gate[A.first[i] + m];
            if (!gated_item || !A.vec_ok[i]) continue;
            fits = fits && (long long)A.i_row[i] >= shape.tile;
            need = std::max(need, 2 * (size_t)A.i_hidden[i] * gs);
        }
        if (fits && need <= kMaxStagedGateBytes) A.stage_gate_bytes = (unsigned)((need + 127) / 128 * 128);
    }
    size_t smem = 0, stage_bytes = 0;
    int per_sm = 1;
    auto fit = [&] {
        stage_bytes = (size_t)K * shape.tile * esize(cb16 ? CB_BF16 : CB_FP32) + A.stage_x_bytes + A.stage_gate_bytes;
        return bulk_config(p, K, cb16, gated, precise, strided, shape.ctas_per_sm, stage_bytes, min_stages, &A.stages,
                           &smem, &per_sm);
    };
    rc = fit();
    // Gate rows too wide to lie beside the stages stay in global memory, rather than
    // that another kernel runs (GB300, [1, 4096, 3072], fp32 gates, direct kernel ->
    // here: fp32 sources, K = 8, groups of one 418 -> 288 us, of two 691 -> 512 us;
    // bf16 groups of two, K = 6 573 -> 520 us).
    if (rc == CB_OK && A.stages < min_stages && A.stage_gate_bytes) {
        A.stage_gate_bytes = 0;
        rc = fit();
    }
    if (rc != CB_OK) return rc;
    if (A.stages < min_stages) {  // too deep for shared memory
        // A group too large to hold: the compensated kernels hold none (GB300, hidden
        // states in bf16, 10 groups of 4 x [8, 256, 1152], K = 5..8: 162, 185, 219, 228 us
        // against 175, 208, 247, 288 for the direct-load kernel, with gates K = 7 and 8
        // 242 and 264 against 275 and 316; fp32 sources, 5 groups of 4 x [4, 256, 1152],
        // K = 6 and 8: 85 and 108 against 94 and 135). bf16 sources with gates and
        // K <= 6 are faster there (28 groups of 4 x [8, 256, 1152], K = 5 and 6: 484 and
        // 571 against 553 and 608 us).
        if (!hold || (cb16 && K <= 6 && gated)) return launch_direct(L, A);
        A.precise = 1;
        return launch_bulk(L, A, false);
    }
    const int stages_all = A.stages;
    const size_t smem_all = smem;
    // Bytes in flight. HBM serves a mix of reads and writes best when no more is
    // asked of it than covers its latency; beyond that reads and writes turn
    // the bus around more often. GB300, DiT-XL/2 256^2 shapes, every SM, KB in
    // flight per SM (all that fits -> here): predictions with K = 1 100.0 ->
    // 83.8 us (48), K = 2 136 -> 120 (64), K = 3 169 -> 151 (120), K = 4 206 ->
    // 188 (128); full-step epilogue from fp32 features 176 -> 159 (100). The
    // more is read per byte written, the flatter the optimum and the higher.
    // Launches that hold a group's stages keep two groups' worth; those with
    // K >= 2 are bound by their consumers and any depth serves them.
    if (!hold || K == 1) {
        double rd = 0, wr = 0, units = 0;
        for (int i = 0; i < items; ++i) {
            const double e = (double)A.numel[i], x = A.resid[i] ? (double)L.res : 0.0;
            rd += e * (A.nb[i] * K * (cb16 ? 2.0 : 4.0) + x);
            units += e * A.nb[i];
            wr += e * x;
            for (int m = 0; m < A.nb[i]; ++m)
                if (A.m_out[A.first[i] + m]) wr += e * (A.out_bf16 ? 2.0 : 4.0);
        }
        const double ratio = rd / wr, kb = hold ? 76 : ratio < 1.25 ? 48 : ratio < 2.5 ? 76 : 120;
        const double unit = rd / units * shape.tile;
        const int most = (int)(kb * 1024.0 / unit / per_sm + 0.5);
        const int least = std::max(hold ? 2 * max_nb : 2, per_sm == 1 ? 3 : 2);
        A.stages = std::min(A.stages, std::max(most, least));
        smem = cbk::bulk_smem_bytes(stage_bytes, A.stages);
    }
    // Persistent grid: every SM, except that bf16 prediction-only launches with
    // K = 5 and 6, whose stages are too large to be limited in number, limit the
    // SMs instead (FLUX.1-dev, K = 5: 3/4 of the SMs with all stages 1794 us,
    // all of them with three stages 1800 us, with all stages 1898 us; K = 8:
    // 344 and 340 us).
    double frac = 1.0;
    if (cb16 && !grouped && !precise && (K == 5 || K == 6) && A.tiles_total >= 8LL * p->dev.sms) {
        frac = 0.75;
        A.stages = stages_all;
        smem = smem_all;
    }
    // L2 residency. Consecutive skipped steps read the same history and write
    // the same buffers. A history somewhat larger than L2 would be gone by the
    // time the next step comes to it and take the step's writes along, so its
    // tiles are copied in for eviction first, but for as many as fit, with the
    // writes, in two fifths of L2 (GB300: 52 MB; each die caches for itself).
    // One DiT-XL/2 256^2 image: skipped step 27.6 -> 22.2 us (hidden states 34.2
    // -> 26.9 us), its DDIM-50 run 1119 -> 955 us; two images, hidden states alone
    // 51.9 -> 42.7 us, four 97.5 -> 92.3 us. Where the writes alone take more than
    // half of L2 the hint loses (three images 75.3 -> 77.2 us, eight 186 -> 194
    // us): those launches leave it out.
    A.keep_tiles = 0x7FFFFFFF;
    if (!L.full_step) {
        double rd = 0, wr = 0;
        for (int i = 0; i < items; ++i) {
            const double e = (double)A.numel[i];
            rd += e * A.nb[i] * K * (cb16 ? 2.0 : 4.0);
            if (A.resid[i]) wr += e * (double)L.res;
            for (int m = 0; m < A.nb[i]; ++m)
                if (A.m_out[A.first[i] + m]) wr += e * (A.out_bf16 ? 2.0 : 4.0);
        }
        const double l2 = p->dev.l2_bytes, room = 0.4 * l2;
        if (rd + wr > room && wr <= 0.55 * l2) A.keep_tiles = (int)(std::max(0.0, room - wr) / rd * A.tiles_total);
    }
    // The gated one-entry epilogue of bf16 groups of two holds more in flight than
    // the mix wants: a twentieth of the SMs less pays where a launch is long and its
    // gate rows narrow (GB300, tiles per SM 53, 71, 106, 189, 212: 66.1 -> 65.8, 85.9 ->
    // 84.4, 126.0 -> 124.9, 218.6 -> 215.6, 246 -> 243 us). Short launches lose their
    // overlap by it (0.5, 4, 8, 40 tiles per SM 4.8 -> 6.2, 7.2 -> 8.2, 13.2 -> 14.4, 51.1
    // -> 51.3 us), rows of 3072 channels 0.5 to 3 % (146 -> 150, 641 -> 646 us), groups of
    // one and three and fp32 gates 1 to 4 %.
    if (L.full_step && cb16 && gated && hold && max_nb == 2 && L.gate_dtype == CB_BF16 &&
        A.stage_gate_bytes <= 8192 && A.tiles_total >= 48LL * p->dev.sms)
        frac = 0.95;
    const long long ctas = std::max(1LL, (long long)((double)p->dev.sms * per_sm * frac));
    // An overlapping launch's blocks go wherever they fit: ask for so much shared
    // memory that no SM takes more than its share of them.
    A.overlap = frac == 1.0 ? 1 : 0;
    smem = std::max(smem, (size_t)p->dev.smem_per_sm / (per_sm + 1));
    const int grid = A.any_scalar ? (int)ctas : (int)std::min<long long>((long long)A.tiles_total + A.n_ragged, ctas);
    rc = clear_status(L);
    if (rc != CB_OK) return rc;
    const cudaStream_t s = (cudaStream_t)L.stream;
    cudaError_t e = strided   ? cbk::launch_extrapolate_bulk_strided(A, K, cb16, grouped, gated, grid, smem, s)
                    : precise ? cbk::launch_extrapolate_bulk_precise(A, K, cb16, grouped, gated, grid, smem, s)
                    : gated   ? cbk::launch_extrapolate_bulk_gated(A, K, cb16, grid, smem, s)
                              : cbk::launch_extrapolate_bulk(A, K, cb16, grouped, grid, smem, s);
    return e == cudaSuccess ? CB_OK : cuda_fail(e, "extrapolate launch");
}

// One skipped-step launch over the window `win` with the fp64 weights w[0..n).
// With `feats` it is instead a full step's epilogue: a one-entry history (the
// new features, weight 1) whose members are written, converted, into the ring
// slot `next` while the hidden states receive x + sum_b g_b f_b. With `ch` the
// window's slots are read from ch->hist and events recorded in ch->status.
int run_launch(cb_plan* p, const Window& win, const double* w, void* const* outs, cb_dtype out_dtype,
               void* const* resid, cb_dtype resid_dtype, void* stream, const void* const* gates = nullptr,
               cb_dtype gate_dtype = CB_BF16, const void* const* feats = nullptr, cb_dtype feat_dtype = CB_BF16,
               CallerHistory* ch = nullptr) {
    if (!ch && !p->cache) return CB_ERR_UNBOUND;
    const int K = win.n;
    if (K < 1 || (!feats && !ch && p->count < K)) return CB_ERR_HISTORY_NOT_FULL;
    if (!valid_dtype(out_dtype) || !valid_dtype(resid_dtype)) return CB_ERR_ARG;
    const int n = (int)p->tensors.size();
    const int ng = (int)p->groups.size();
    const size_t oes = esize(out_dtype), res = esize(resid_dtype);
    if (outs)
        for (int i = 0; i < n; ++i)
            if (outs[i] && !aligned(outs[i], oes)) return CB_ERR_ALIGN;
    if (resid)
        for (int g = 0; g < ng; ++g)
            if (resid[g] && !aligned(resid[g], res)) return CB_ERR_ALIGN;

    for (int j = 0; j < K; ++j)
        if (!std::isfinite(w[j])) return CB_ERR_ARG;
    int rc = check_gates(p, gates, gate_dtype);
    if (rc != CB_OK) return rc;

    cbk::ExtrapArgs& A = *p->eargs;
    // the kernels' source type: the cache's, or the new features'
    const bool cb16 = (feats ? feat_dtype : p->cache_dtype) == CB_BF16;
    // A full step's epilogue runs its own kernel (unless CB_OPT_KERNEL names
    // one) when its threads keep enough loads in flight: ungated bf16 features
    // and bf16 hidden states with every tensor in a residual group of three or
    // more branches.
    // Otherwise the bulk pipeline streams faster (see epilogue.cu).
    bool epilogue = feats && p->kernel == CB_KERNEL_AUTO && feat_dtype == CB_BF16 && resid &&
                    resid_dtype == CB_BF16;
    for (int i = 0; epilogue && i < n; ++i) {
        const int g = p->tensors[i].group;
        epilogue = g >= 0 && resid[g] && p->groups[g].size() >= 3 && !(gates && gates[i]);
    }
    unsigned char* slot = p->cache + (size_t)p->next * p->slot_bytes;
    A.hist_base = feats ? 0ull : (unsigned long long)(uintptr_t)(ch ? ch->hist : p->cache);
    A.copy_out = feats ? 1 : 0;
    for (int j = 0; j < CB_MAX_K; ++j) {
        const bool on = j < K;
        A.slot_off[j] = on && !feats ? (long long)win.slot[j] * (long long)p->slot_bytes : 0;
        const float hi = on ? (float)w[j] : 0.0f;
        A.w_hi[j] = hi;
        A.w_lo[j] = on ? (float)(w[j] - (double)hi) : 0.0f;
        // the fast path's bound, scaled: (K+2) u (1.01) 2^9 |w_hi[j]|, u = 2^-24
        A.w_guard[j] = (float)(std::fabs((double)hi) * (K + 2) * 1.01 * std::ldexp(1.0, -15));
        A.w_anchor[j] = anchor_weight(std::fabs((double)hi), K, cb16);
    }
    A.out_bf16 = out_dtype == CB_BF16;
    A.resid_bf16 = resid_dtype == CB_BF16;

    int items = 0, members = 0;
    bool any_out = false, any_resid = false;
    // items that can be copied in but not stored (or gated) by whole vectors
    bool strided[cbk::kMaxItems];
    A.gate_bf16 = gate_dtype == CB_BF16;
    auto add_item = [&](const int* mem, int nm, void* res_ptr) {
        const long long numel = p->tensors[mem[0]].numel;
        bool vec = !res_ptr || aligned(res_ptr, 16), src = true;
        A.first[items] = (short)members;
        A.i_hidden[items] = (unsigned)p->sh_hidden[mem[0]];
        A.i_row[items] = (unsigned)(p->sh_tokens[mem[0]] * p->sh_hidden[mem[0]]);
        A.i_hidden_magic[items] = div_magic(A.i_hidden[items]);
        A.i_row_magic[items] = div_magic(A.i_row[items]);
        for (int m = 0; m < nm; ++m) {
            const int i = mem[m];
            void* o = feats ? slot + p->off[i] : outs ? outs[i] : nullptr;
            const void* g = (res_ptr && gates) ? gates[i] : nullptr;
            A.m_off[members] = feats ? (long long)(uintptr_t)feats[i] : p->off[i];
            if (feats) src = src && aligned(feats[i], 16);
            A.m_out[members] = o;
            A.m_gate[members] = g;
            if (g) {  // vectors of 8 stay inside one gate row
                vec = vec && aligned(g, 16) && p->sh_hidden[i] % 8 == 0;
            }
            if (o) {
                any_out = true;
                vec = vec && aligned(o, 16);
            }
            ++members;
        }
        vec = vec && src;
        if (res_ptr) any_resid = true;
        A.nb[items] = (unsigned char)nm;
        A.resid[items] = res_ptr;
        A.vec_ok[items] = vec ? 1 : 0;
        strided[items] = !vec && src;
        A.numel[items] = numel;
        ++items;
    };
    std::vector<char> in_group(n, 0);
    if (resid)
        for (int g = 0; g < ng; ++g)
            if (resid[g] && !p->groups[g].empty()) {
                add_item(p->groups[g].data(), (int)p->groups[g].size(), resid[g]);
                for (int i : p->groups[g]) in_group[i] = 1;
            }
    for (int i = 0; i < n; ++i)
        if (!in_group[i] && (feats || (outs && outs[i]))) add_item(&i, 1, nullptr);
    A.n_items = items;
    // a full step's slot write is a conversion, not arithmetic
    A.precise = (any_out && !feats && out_dtype == CB_FP32) || (any_resid && resid_dtype == CB_FP32);
    if (items == 0) return CB_OK;  // nothing requested

    A.wait_ns = p->wait_ns;
    A.status = ch ? ch->status : p->status_word();
    A.withhold_first = p->withhold_first;
    A.stages = 0;
    A.stage_x_bytes = 0;
    A.stage_gate_bytes = 0;
    A.n_ragged = A.any_scalar = 0;

    rc = ensure_device(p);
    if (rc != CB_OK) return rc;
    Launch L{p, K, cb16, feats != nullptr, res, gate_dtype, stream, ch};
    if (p->kernel == CB_KERNEL_DIRECT) return launch_direct(L, A);
    auto aligned_items = [&](cbk::ExtrapArgs& B) { return epilogue ? launch_epilogue(L, B) : launch_bulk(L, B, false); };
    int n_strided = 0;
    for (int i = 0; i < items; ++i) n_strided += strided[i] ? 1 : 0;
    if (n_strided == 0) return aligned_items(A);
    if (n_strided == items) return launch_bulk(L, A, true);
    // some of each: a launch for either
    if (!p->eargs2) p->eargs2.reset(new (std::nothrow) cbk::ExtrapArgs());
    if (!p->eargs2) return CB_ERR_LIMIT;
    cbk::ExtrapArgs& B = *p->eargs2;
    take_items(A, strided, true, B);
    rc = launch_bulk(L, B, true);
    if (rc != CB_OK) return rc;
    take_items(A, strided, false, B);
    return aligned_items(B);
}

}  // namespace

extern "C" {

int cb_schedule_full(int T, int r, int s0, int s1, int K, uint8_t* is_full, int* n_full) {
    if (T <= 0 || r <= 0 || s0 < 0 || s1 < 0 || K < 0 || !is_full) return CB_ERR_ARG;
    int held = 0, nf = 0;
    for (int s = 0; s < T; ++s) {
        const bool in_range = s >= s0 && s <= T - 1 - s1;
        bool full = !in_range || (s - s0) % r == 0;
        if (held < K) full = true;  // not enough history to extrapolate yet
        is_full[s] = full ? 1 : 0;
        if (full) {
            ++nf;
            if (held < K) ++held;
        }
    }
    if (n_full) *n_full = nf;
    return CB_OK;
}

int cb_plan_create(const double* node_t, int n_nodes, int K, const cb_tensor_desc* tensors, int n_tensors,
                   cb_dtype cache_dtype, double t_min, double t_max, cb_plan** out) {
    if (!out) return CB_ERR_ARG;
    *out = nullptr;
    if (K < 1 || K > CB_MAX_K) return K < 1 ? CB_ERR_ARG : CB_ERR_LIMIT;
    if (!node_t || n_nodes < K || !tensors || n_tensors < 1) return CB_ERR_ARG;
    if (n_tensors > CB_MAX_TENSORS) return CB_ERR_LIMIT;
    if (!valid_dtype(cache_dtype)) return CB_ERR_ARG;
    if (!(std::isfinite(t_min) && std::isfinite(t_max) && t_min < t_max)) return CB_ERR_ARG;
    for (int i = 0; i < n_nodes; ++i)
        if (!std::isfinite(node_t[i])) return CB_ERR_ARG;
    int dir = 0;
    if (n_nodes >= 2) {
        for (int i = 1; i < n_nodes; ++i) {
            const double d = node_t[i] - node_t[i - 1];
            if (d == 0.0) return CB_ERR_NODES_DEGENERATE;
            const int s = d > 0 ? 1 : -1;
            if (dir == 0) dir = s;
            if (s != dir) return CB_ERR_ARG;  // nodes must be strictly monotone
        }
    }
    try {
        std::unique_ptr<cb_plan> p(new cb_plan);
        p->K = K;
        p->cache_dtype = cache_dtype;
        p->t_min = t_min;
        p->t_max = t_max;
        p->dir = dir;
        p->tensors.assign(tensors, tensors + n_tensors);
        int ng = 0;
        for (const auto& d : p->tensors) {
            if (d.numel <= 0 || d.reserved != 0 || d.group < -1) return CB_ERR_ARG;
            if (d.numel > CB_MAX_NUMEL) return CB_ERR_LIMIT;
            if (d.group + 1 > ng) ng = d.group + 1;
        }
        static_assert(cbk::kMaxItems == CB_MAX_TENSORS, "one work item per tensor or group");
        if (ng > cbk::kMaxItems) return CB_ERR_LIMIT;
        p->groups.assign(ng, {});
        for (int i = 0; i < n_tensors; ++i) {
            const auto& d = p->tensors[i];
            if (d.group < 0) continue;
            auto& g = p->groups[d.group];
            if (!g.empty() && p->tensors[g[0]].numel != d.numel) return CB_ERR_ARG;
            g.push_back(i);
            if ((int)g.size() > CB_MAX_BRANCHES) return CB_ERR_LIMIT;
        }
        p->node_t.assign(node_t, node_t + n_nodes);
        p->node_tau.resize(n_nodes);
        for (int i = 0; i < n_nodes; ++i) p->node_tau[i] = p->tau(node_t[i]);
        // offline stage: rho for every window of K consecutive nodes
        p->rho_win.resize((size_t)(n_nodes - K + 1) * K);
        for (int i = 0; i + K <= n_nodes; ++i)
            if (!rho_of(&p->node_tau[i], K, &p->rho_win[(size_t)i * K])) return CB_ERR_NODES_DEGENERATE;
        // slot layout: tensors back to back, each at a CB_CACHE_ALIGN boundary
        size_t o = 0;
        p->off.resize(n_tensors);
        for (int i = 0; i < n_tensors; ++i) {
            p->off[i] = (long long)o;
            o = round_up(o + (size_t)p->tensors[i].numel * esize(cache_dtype), CB_CACHE_ALIGN);
        }
        p->slot_bytes = o;
        p->sh_tokens.assign(n_tensors, 0);
        p->sh_hidden.assign(n_tensors, 0);
        *out = p.release();
        return CB_OK;
    } catch (const std::bad_alloc&) {
        return CB_ERR_LIMIT;
    }
}

size_t cb_plan_cache_bytes(const cb_plan* p) {
    return p ? p->slot_bytes * (size_t)p->K + CB_STATUS_BYTES : 0;
}

int cb_plan_bind_cache(cb_plan* p, void* dev_ptr, size_t bytes) {
    if (!p || !dev_ptr || bytes < cb_plan_cache_bytes(p)) return CB_ERR_ARG;
    if (!aligned(dev_ptr, CB_CACHE_ALIGN)) return CB_ERR_ALIGN;
    p->cache = static_cast<unsigned char*>(dev_ptr);
    p->next = p->count = 0;
    p->has_last = false;
    p->status_clear = false;  // zeroed on the stream of the first launch
    return CB_OK;
}

int cb_cache_push(cb_plan* p, const void* const* feats, cb_dtype feat_dtype, double t, void* stream) {
    if (!p || !feats || !valid_dtype(feat_dtype) || !std::isfinite(t)) return CB_ERR_ARG;
    if (!p->cache) return CB_ERR_UNBOUND;
    const int n = (int)p->tensors.size();
    const size_t fes = esize(feat_dtype);
    for (int i = 0; i < n; ++i) {
        if (!feats[i]) return CB_ERR_ARG;
        if (!aligned(feats[i], fes)) return CB_ERR_ALIGN;
    }
    if (p->has_last) {
        const double d = t - p->last_t;
        if (d == 0.0 || (p->dir != 0 && (d > 0 ? 1 : -1) != p->dir)) return CB_ERR_ORDER;
    }
    for (int j = 0; j < p->count; ++j)
        if (p->slot_t[(p->oldest() + j) % p->K] == t) return CB_ERR_NODES_DEGENERATE;

    cbk::PushArgs& A = *p->pargs;
    const bool sb = feat_dtype == CB_BF16, db = p->cache_dtype == CB_BF16;
    A.slot = p->cache + (size_t)p->next * p->slot_bytes;
    long long tiles = 0;
    for (int i = 0; i < n; ++i) {
        A.tile_begin[i] = (int)tiles;
        A.numel[i] = p->tensors[i].numel;
        A.off[i] = p->off[i];
        A.src[i] = feats[i];
        A.vec_ok[i] = aligned(feats[i], 16) ? 1 : 0;
        tiles += (p->tensors[i].numel + cbk::push_tile_elems - 1) / cbk::push_tile_elems;
    }
    if (tiles > 0x7FFFFFFFLL) return CB_ERR_LIMIT;
    A.tile_begin[n] = (int)tiles;
    A.n_items = n;
    A.tiles_total = (int)tiles;
    A.overlap = 1;
    int rc = ensure_device(p);
    if (rc != CB_OK) return rc;
    int grid = 0;
    size_t smem = 0;
    rc = push_grid(p, sb, db, (int)tiles, &grid, &smem);
    if (rc != CB_OK) return rc;
    rc = clear_status_once(p, stream);
    if (rc != CB_OK) return rc;
    cudaError_t e = cbk::launch_push(A, sb, db, grid, smem, (cudaStream_t)stream);
    if (e != cudaSuccess) return cuda_fail(e, "push launch");
    // the pair (t, f_t) is now in H; the oldest entry was overwritten when full
    p->slot_t[p->next] = t;
    p->next = (p->next + 1) % p->K;
    if (p->count < p->K) ++p->count;
    p->has_last = true;
    p->last_t = t;
    return CB_OK;
}

int cb_extrapolate(cb_plan* p, double t_target, void* const* outs, cb_dtype out_dtype, void* const* resid,
                   cb_dtype resid_dtype, void* stream) {
    if (!p) return CB_ERR_ARG;
    const int n = live_entries(p);
    if (n == 0) return p->cache ? CB_ERR_HISTORY_NOT_FULL : CB_ERR_UNBOUND;
    const Window win = live_window(p, n);
    double w[CB_MAX_K];
    const int rc = weights_for(p, win, t_target, w);
    if (rc != CB_OK) return rc;
    return run_launch(p, win, w, outs, out_dtype, resid, resid_dtype, stream);
}

int cb_extrapolate_ring(cb_plan* p, const double* slot_t, int head, double t_target, void* const* outs,
                        cb_dtype out_dtype, void* const* resid, cb_dtype resid_dtype, void* stream) {
    if (!p || !slot_t || head < 0 || head >= (p ? p->K : 1)) return CB_ERR_ARG;
    if (p->count < p->K) return p->cache ? CB_ERR_HISTORY_NOT_FULL : CB_ERR_UNBOUND;
    Window win{};
    win.n = p->K;
    for (int j = 0; j < p->K; ++j) {
        win.slot[j] = (head + j) % p->K;
        win.t[j] = slot_t[win.slot[j]];
        if (!std::isfinite(win.t[j])) return CB_ERR_ARG;
        win.tau[j] = p->tau(win.t[j]);
        for (int i = 0; i < j; ++i)
            if (win.t[i] == win.t[j]) return CB_ERR_NODES_DEGENERATE;
    }
    double w[CB_MAX_K];
    const int rc = weights_for(p, win, t_target, w);
    if (rc != CB_OK) return rc;
    return run_launch(p, win, w, outs, out_dtype, resid, resid_dtype, stream);
}

int cb_extrapolate_noalloc(cb_plan* p, const void* hist, size_t hist_bytes, const double* slot_t, int head,
                           double t_target, void* const* outs, cb_dtype out_dtype, void* const* resid,
                           cb_dtype resid_dtype, int* status, void* stream) {
    if (!p || !hist || !slot_t || head < 0 || head >= p->K) return CB_ERR_ARG;
    if (!aligned(hist, CB_CACHE_ALIGN)) return CB_ERR_ALIGN;
    if (hist_bytes < p->slot_bytes * (size_t)p->K) return CB_ERR_ARG;  // the K slots, no status block
    Window win{};
    win.n = p->K;
    for (int j = 0; j < p->K; ++j) {
        win.slot[j] = (head + j) % p->K;
        win.t[j] = slot_t[win.slot[j]];
        if (!std::isfinite(win.t[j])) return CB_ERR_ARG;
        win.tau[j] = p->tau(win.t[j]);
        for (int i = 0; i < j; ++i)
            if (win.t[i] == win.t[j]) return CB_ERR_NODES_DEGENERATE;
    }
    double w[CB_MAX_K];
    int rc = weights_for(p, win, t_target, w);
    if (rc != CB_OK) return rc;
    // the library's status word on the current device (looked up on the first call there)
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return cuda_fail(e, "cudaGetDevice");
    if (dev >= cbk::kMaxStatusDevices) return CB_ERR_LIMIT;
    int* word = nullptr;
    e = cbk::noalloc_status_word(dev, &word);
    if (e != cudaSuccess) return cuda_fail(e, "cudaGetSymbolAddress");
    // Only launches whose status is asked for record into the word, and handing
    // it over clears it, so that it needs no clearing before a launch (unless a
    // call failed in between: clear_status).
    CallerHistory ch{static_cast<const unsigned char*>(hist), status ? word : nullptr, dev, false};
    rc = run_launch(p, win, w, outs, out_dtype, resid, resid_dtype, stream, nullptr, CB_BF16, nullptr, CB_BF16, &ch);
    if (rc != CB_OK && status && ch.launched) g_unclaimed[dev] = true;
    if (rc != CB_OK || !status) return rc;
    if (!ch.launched) {  // nothing was requested, so nothing ran
        *status = 0;
        return CB_OK;
    }
    cudaPointerAttributes at{};
    const bool pinned = cudaPointerGetAttributes(&at, status) == cudaSuccess && at.type == cudaMemoryTypeHost &&
                        at.devicePointer != nullptr;
    if (pinned && aligned(at.devicePointer, sizeof(int))) {  // a kernel's store wants the alignment, a copy does not
        e = cbk::take_status(word, static_cast<int*>(at.devicePointer), (cudaStream_t)stream);
    } else {
        (void)cudaGetLastError();  // a pointer the runtime does not know is ordinary memory
        e = cudaMemcpyAsync(status, word, sizeof(int), cudaMemcpyDeviceToHost, (cudaStream_t)stream);
        if (e == cudaSuccess) e = cudaMemsetAsync(word, 0, sizeof(int), (cudaStream_t)stream);
    }
    if (e != cudaSuccess) {
        g_unclaimed[dev] = true;
        return cuda_fail(e, "status read-back");
    }
    return CB_OK;
}

int cb_extrapolate_weights(cb_plan* p, const double* w_logical, void* const* outs, cb_dtype out_dtype,
                           void* const* resid, cb_dtype resid_dtype, void* stream) {
    if (!p || !w_logical) return CB_ERR_ARG;
    const int n = live_entries(p);
    if (n == 0) return p->cache ? CB_ERR_HISTORY_NOT_FULL : CB_ERR_UNBOUND;
    return run_launch(p, live_window(p, n), w_logical, outs, out_dtype, resid, resid_dtype, stream);
}

int cb_plan_set_shapes(cb_plan* p, const int64_t* bth) {
    if (!p || !bth) return CB_ERR_ARG;
    const int n = (int)p->tensors.size();
    for (int i = 0; i < n; ++i) {
        const int64_t b = bth[3 * i], t = bth[3 * i + 1], h = bth[3 * i + 2];
        const int64_t numel = p->tensors[i].numel;
        // b * t * h == numel, tested by division so that no product overflows
        if (b <= 0 || t <= 0 || h <= 0 || h > numel || t > numel / h) return CB_ERR_ARG;
        if (numel % (t * h) != 0 || numel / (t * h) != b) return CB_ERR_ARG;
        if (t * h > 0xFFFFFFFFLL) return CB_ERR_LIMIT;
    }
    for (const auto& g : p->groups)  // members of a group share one hidden state, hence one shape
        for (int i : g)
            if (bth[3 * i + 1] != bth[3 * g[0] + 1] || bth[3 * i + 2] != bth[3 * g[0] + 2]) return CB_ERR_ARG;
    for (int i = 0; i < n; ++i) {
        p->sh_tokens[i] = bth[3 * i + 1];
        p->sh_hidden[i] = bth[3 * i + 2];
    }
    return CB_OK;
}

int cb_extrapolate_gated(cb_plan* p, double t_target, void* const* outs, cb_dtype out_dtype, void* const* resid,
                         cb_dtype resid_dtype, const void* const* gates, cb_dtype gate_dtype, void* stream) {
    if (!p) return CB_ERR_ARG;
    const int n = live_entries(p);
    if (n == 0) return p->cache ? CB_ERR_HISTORY_NOT_FULL : CB_ERR_UNBOUND;
    const Window win = live_window(p, n);
    double w[CB_MAX_K];
    const int rc = weights_for(p, win, t_target, w);
    if (rc != CB_OK) return rc;
    return run_launch(p, win, w, outs, out_dtype, resid, resid_dtype, stream, gates, gate_dtype);
}

int cb_cache_push_residual(cb_plan* p, const void* const* feats, cb_dtype feat_dtype, double t, void* const* resid,
                           cb_dtype resid_dtype, const void* const* gates, cb_dtype gate_dtype, void* stream) {
    if (!p || !feats || !valid_dtype(feat_dtype) || !valid_dtype(resid_dtype) || !std::isfinite(t))
        return CB_ERR_ARG;
    if (!p->cache) return CB_ERR_UNBOUND;
    const int n = (int)p->tensors.size();
    const int ng = (int)p->groups.size();
    const size_t fes = esize(feat_dtype), res = esize(resid_dtype);
    for (int i = 0; i < n; ++i) {
        if (!feats[i]) return CB_ERR_ARG;
        if (!aligned(feats[i], fes)) return CB_ERR_ALIGN;
    }
    if (resid)
        for (int g = 0; g < ng; ++g)
            if (resid[g] && !aligned(resid[g], res)) return CB_ERR_ALIGN;
    int rc = check_gates(p, gates, gate_dtype);
    if (rc != CB_OK) return rc;
    if (p->has_last) {
        const double d = t - p->last_t;
        if (d == 0.0 || (p->dir != 0 && (d > 0 ? 1 : -1) != p->dir)) return CB_ERR_ORDER;
    }
    for (int j = 0; j < p->count; ++j)
        if (p->slot_t[(p->oldest() + j) % p->K] == t) return CB_ERR_NODES_DEGENERATE;

    // one-entry history of weight 1: the new features themselves
    Window one{};
    one.n = 1;
    const double w1[1] = {1.0};
    rc = run_launch(p, one, w1, nullptr, p->cache_dtype, resid, resid_dtype, stream, gates, gate_dtype, feats,
                    feat_dtype);
    if (rc != CB_OK) return rc;
    p->slot_t[p->next] = t;
    p->next = (p->next + 1) % p->K;
    if (p->count < p->K) ++p->count;
    p->has_last = true;
    p->last_t = t;
    return CB_OK;
}

int cb_weights(const cb_plan* p, double t_target, double* w_logical) {
    if (!p || !w_logical) return CB_ERR_ARG;
    const int n = live_entries(p);
    if (n == 0) return CB_ERR_HISTORY_NOT_FULL;
    return weights_for(p, live_window(p, n), t_target, w_logical);
}

int cb_taylor_weights(const double* node_t, int n, double t_target, double* w) {
    if (!node_t || !w || n < 1 || n > CB_MAX_K || !std::isfinite(t_target)) return CB_ERR_ARG;
    for (int i = 0; i < n; ++i)
        if (!std::isfinite(node_t[i])) return CB_ERR_ARG;
    double h = 1.0;
    if (n >= 2) {
        h = node_t[n - 1] - node_t[n - 2];
        if (h == 0.0) return CB_ERR_NODES_DEGENERATE;
        for (int i = 1; i < n; ++i)  // equispaced nodes only
            if (std::fabs((node_t[i] - node_t[i - 1]) - h) > 1e-9 * std::fabs(h)) return CB_ERR_ARG;
    }
    const double theta = n >= 2 ? (t_target - node_t[n - 1]) / h : 0.0;
    // f(t) ~ sum_i theta^i / i! nabla^i f_n, nabla^i f_n = sum_k (-1)^k C(i, k) f_{n-k}
    for (int j = 0; j < n; ++j) w[j] = 0.0;
    double pow_fact = 1.0;  // theta^i / i!
    for (int i = 0; i < n; ++i) {
        if (i > 0) pow_fact *= theta / i;
        double binom = 1.0;  // C(i, k)
        for (int k = 0; k <= i; ++k) {
            if (k > 0) binom = binom * (i - k + 1) / k;
            w[n - 1 - k] += pow_fact * ((k & 1) ? -binom : binom);
        }
    }
    return CB_OK;
}

int cb_plan_export_weights(const cb_plan* p, const double* targets, int n_targets, double* table) {
    if (!p || (n_targets > 0 && (!targets || !table)) || n_targets < 0) return CB_ERR_ARG;
    const int K = p->K, n = (int)p->node_t.size();
    for (int m = 0; m < n_targets; ++m) {
        const double t = targets[m];
        if (!std::isfinite(t)) return CB_ERR_ARG;
        // the K most recent nodes that precede t in sampling order
        int last = -1;
        for (int i = 0; i < n; ++i) {
            const double d = t - p->node_t[i];
            const bool before = p->dir >= 0 ? d > 0 : d < 0;
            if (before) last = i;
        }
        if (last + 1 < K) return CB_ERR_HISTORY_NOT_FULL;
        Window w{};
        w.n = K;
        for (int j = 0; j < K; ++j) {
            w.t[j] = p->node_t[last - K + 1 + j];
            w.tau[j] = p->node_tau[last - K + 1 + j];
        }
        const int rc = weights_for(p, w, t, &table[(size_t)m * K]);
        if (rc != CB_OK) return rc;
    }
    return CB_OK;
}

int cb_plan_history(const cb_plan* p, double* slot_t, int* head, int* count) {
    if (!p) return CB_ERR_ARG;
    if (slot_t)
        for (int j = 0; j < p->K; ++j) slot_t[j] = p->slot_t[j];
    if (head) *head = p->oldest();
    if (count) *count = p->count;
    return CB_OK;
}

int cb_plan_reset(cb_plan* p) {
    if (!p) return CB_ERR_ARG;
    p->next = p->count = 0;
    p->has_last = false;
    return CB_OK;
}

int cb_plan_set_option(cb_plan* p, int option, int64_t value) {
    if (!p) return CB_ERR_ARG;
    switch (option) {
    case CB_OPT_KERNEL:
        if (value != CB_KERNEL_AUTO && value != CB_KERNEL_DIRECT && value != CB_KERNEL_BULK) return CB_ERR_ARG;
        p->kernel = (int)value;
        return CB_OK;
    case CB_OPT_WAIT_NS:
        if (value < 0 || value > 60000000000LL) return CB_ERR_ARG;
        p->wait_ns = (unsigned long long)value;
        return CB_OK;
    case CB_OPT_PARTIAL_HISTORY:
        if (value != 0 && value != 1) return CB_ERR_ARG;
        p->partial = value != 0;
        return CB_OK;
    case CB_OPT_TEST_WITHHOLD:
        if (value != 0 && value != 1) return CB_ERR_ARG;
        p->withhold_first = (int)value;
        return CB_OK;
    default: return CB_ERR_ARG;
    }
}

int cb_plan_device_status(cb_plan* p, int* status, void* stream) {
    if (!p || !status) return CB_ERR_ARG;
    if (!p->cache) return CB_ERR_UNBOUND;
    if (!p->status_clear) {  // nothing has run since binding
        *status = 0;
        return CB_OK;
    }
    cudaStream_t s = (cudaStream_t)stream;
    int v = 0;
    cudaError_t e = cudaMemcpyAsync(&v, p->status_word(), sizeof(int), cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaMemsetAsync(p->status_word(), 0, sizeof(int), s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    if (e != cudaSuccess) return cuda_fail(e, "device status");
    *status = v;
    return CB_OK;
}

int cb_plan_num_groups(const cb_plan* p) { return p ? (int)p->groups.size() : 0; }

void cb_plan_destroy(cb_plan* p) { delete p; }

const char* cb_status_string(int s) {
    switch (s) {
    case CB_OK: return "ok";
    case CB_ERR_ARG: return "invalid argument";
    case CB_ERR_ALIGN: return "misaligned pointer";
    case CB_ERR_NODES_DEGENERATE: return "duplicate node times (omega'(tau_j) = 0)";
    case CB_ERR_HISTORY_NOT_FULL: return "history buffer holds fewer than K entries";
    case CB_ERR_ORDER: return "pushed time does not continue the sampling direction";
    case CB_ERR_UNBOUND: return "no cache arena bound to the plan";
    case CB_ERR_CUDA: return "CUDA error";
    case CB_ERR_LIMIT: return "size limit exceeded";
    default: return "unknown status";
    }
}

const char* cb_last_error_message(void) { return g_last_error.c_str(); }

}  // extern "C"
