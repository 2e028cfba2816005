// Skipped-step kernel, bulk-copy pipeline variant (Sec. 3.3, Eq. for f_t; Alg. 1,
// extrapolation branch). It gives the direct kernel's bits, for finite values, in
// the whole tiles of items on the 16-byte grid, where the launch holds its groups
// or has fp32 results. The compensated sums take the place of the direct kernel's
// guarded ones in ragged last tiles and in bf16 groups too large to hold, and of
// its element-wise Dot2 for items off the grid.
//
// One or two CTAs per SM (see Shape). A producer lane moves, for every work unit
// (one tile of one branch tensor), the K history chunks of the tile (8 KB each,
// less or more in the compensated kernels) from HBM into a ring of shared-memory
// stages with cp.async.bulk (the Blackwell bulk-copy engine), each stage guarded
// by a "full" mbarrier (transaction bytes) and an "empty" mbarrier (one arrival
// per consumer warp). Consumer warps read their 8-element vectors of the K
// chunks from shared memory, compute, and store from registers, so that what is
// in flight does not depend on the consumers' registers, which bound the
// direct-load variant. How much is in flight the host decides (launch_bulk).
//
// Whole tiles come first, in a loop that tests no lengths; the ragged last tiles
// follow in a loop of their own (ragged_tiles), and items whose sources are off
// the 16-byte grid last, without the pipeline (scalar_items).
//
// Many consumer warps per scheduler hide the consumers' fixed latencies (see
// Shape for the thread map). Every consumer fences its reads of a stage
// against the async proxy before the stage goes back to the producer
// (release_stage). Two kinds of launch (GROUPED):
//   * predictions only: each stage is released as soon as it is read into
//     registers, and guarded elements are recomputed from those registers;
//   * with hidden states: stages are released after the member's arithmetic,
//     guarded elements are recomputed from shared memory (so the history
//     values die early). The producer also stages each tile's hidden state
//     (behind the chunks of the group's first member) and the consumers
//     hold the group's member stages until the hidden state is written (the
//     host guarantees more stages than members, so holding cannot starve the
//     producer). With gates, each member's stage also carries the gate rows
//     of the batches its tile touches, so that no consumer waits on a global
//     load.
// Launches with fp32 predictions or hidden states (PRECISE) and items off the
// 16-byte grid on their way out (STRIDED) have kernels of their own: see
// precise_tile.
// The same kernel runs a full step's epilogue (cb_cache_push_residual) as a
// one-entry history of weight 1 whose member addresses are the new features;
// with copy_out the outputs (the ring slot) receive the features converted.
//
// Every wait is bounded (%globaltimer). A consumer wait that runs out in any
// lane records a code in the plan's device status word and the whole warp
// returns (a warp vote, so no lane leaves a warp that goes on to a
// __syncwarp); a producer wait that runs out stops the producer, which then
// waits, with its own limit (at least 10 ms), for the copies it has issued
// before it exits. A test option makes the producer announce the first unit's
// bytes without issuing its copies, so that the consumers' wait runs out with
// no fault and nothing in flight.
#pragma once

#include "cb_async.cuh"
#include "cb_math.cuh"

namespace cbk {
namespace {

// Thread map (bulk_shape). With one CTA per SM, one 8-element vector per consumer
// thread and tile: 16 consumer warps for bf16 tiles (512 vectors; 17 warps cap
// registers at 96), 8 for fp32 tiles (256 vectors). Launches that carry few
// bytes per unit (most K = 1 launches, and bf16 launches with small K) pay the
// consumers' fixed cost per unit more often; they run two CTAs of 8
// consumer warps per SM (two independent pipelines), bf16 threads taking two
// vectors per tile. An earlier map of 8 consumer warps with two vectors each
// on one CTA left the launches with hidden states issue-bound.
template <bool CB16, int K, bool GROUPED, bool GATED, bool PRECISE, bool STRIDED = false>
struct Shape {
    static constexpr BulkShape b = bulk_shape(K, CB16, GROUPED, GATED, PRECISE, STRIDED);
    static constexpr int ctas_per_sm = b.ctas_per_sm;
    static constexpr int consumer_warps = b.consumer_warps;
    static constexpr int consumers = consumer_warps * 32;
    static constexpr int threads = consumers + 32;  // plus the producer warp
    static constexpr int tile = b.tile;             // elements of one unit
    static constexpr int chunk = tile * (CB16 ? 2 : 4);  // bytes of one history entry's share of a tile
    static constexpr int vecs = tile / kVecElems / consumers;  // vectors per consumer thread per tile
    static_assert(vecs * kVecElems * consumers == tile, "a tile's vectors spread evenly over the consumers");
};
constexpr int kBarrierBytes = 256;  // full[S] and empty[S] barriers, S <= kMaxStages
static_assert(2 * 8 * kMaxStages <= kBarrierBytes, "barrier block holds every stage's barriers");
// A consumer warp hands one stage back to the producer: every lane fences its
// shared-memory reads of the stage against the async proxy, then lane 0
// arrives on the stage's empty barrier. The refill that follows is an
// async-proxy write to the same bytes, and the mbarrier release/acquire pair
// alone does not order it after generic-proxy reads: without the fence, a
// refill landed on the start of a stage before some of a warp's loads were
// performed (half a warp's first vector took the next unit's bytes, about one
// launch in 200 on full-size PixArt shapes; none in 3000 with the fence).
__device__ __forceinline__ void release_stage(uint32_t empty_bar, int lane) {
    fence_generic_to_async();
    __syncwarp();
    if (lane == 0) mbar_arrive(empty_bar);
}

// Bytes of a ragged tile of n elements that are copied: whole 16-byte pieces.
// The history's tensors are padded to CB_CACHE_ALIGN, so the last piece may
// reach past the tensor; a full step's new features are not, and what is left
// of them (less than 16 bytes) is read from global memory.
template <int ES>
__device__ __forceinline__ uint32_t ragged_bytes(const ExtrapArgs& A, long long n) {
    const uint32_t b = (uint32_t)n * ES;
    return A.copy_out ? b & ~15u : (b + 15u) & ~15u;
}

// The producer lane: every unit's history chunks, and what travels with them,
// from global into shared memory, in the consumers' order.
template <typename Sh, int K, bool CB16, bool GROUPED, bool GATED>
__device__ __forceinline__ void produce(const ExtrapArgs& A, uint32_t full0, uint32_t empty0, uint32_t buf0,
                                        uint32_t stage_bytes) {
    constexpr long long TE = Sh::tile;
    constexpr int ES = CB16 ? 2 : 4;
    const int S = A.stages;
    unsigned u = 0;               // units issued
    uint32_t ps = 0, wraps = 0;   // stage of the next unit; times the ring has wrapped
    // one tile of item `it`: a unit per member; false when a wait ran out
    const uint64_t normal = policy_normal(), passing = policy_first();
    auto issue = [&](int it, long long e0, bool whole, uint32_t bytes, uint64_t policy) {
        const int first = A.first[it];
        const int nb = GROUPED ? A.nb[it] : 1;
        const unsigned char* resid = GROUPED ? reinterpret_cast<const unsigned char*>(A.resid[it]) : nullptr;
        // gate rows b0..b1 of the batches this tile touches (b1 <= b0 + 1:
        // the host stages gates only when a batch holds a tile or more)
        uint32_t gbytes = 0;
        size_t gsrc = 0;
        if (GATED && A.stage_gate_bytes && resid && whole && A.i_row[it] != 0) {
            const long long row = A.i_row[it];
            const long long b0 = e0 / row, b1 = (e0 + TE - 1) / row;
            const size_t gs = A.gate_bf16 ? 2 : 4;
            gsrc = (size_t)b0 * A.i_hidden[it] * gs;
            gbytes = (uint32_t)((b1 - b0 + 1) * A.i_hidden[it] * gs);
        }
        for (int m = 0; m < nb; ++m) {
            const uint32_t stage = ps;
            if (wraps > 0 && !mbar_wait(empty0 + 8u * stage, (wraps - 1) & 1u, A.wait_ns)) {
                record(A.status, 2);
                return false;
            }
            ++u;
            if (++ps == (uint32_t)S) {
                ps = 0;
                ++wraps;
            }
            // a whole tile's hidden state travels with its first member
            const uint32_t xbytes = GROUPED && resid && whole && m == 0 ? A.stage_x_bytes : 0u;
            const uint32_t gb = (GATED && A.m_gate[first + m]) ? gbytes : 0u;
            mbar_expect_tx(full0 + 8u * stage, (uint32_t)K * bytes + xbytes + gb);
            if (A.withhold_first && u == 1) continue;
            const uint32_t dst = buf0 + stage * stage_bytes;
            if (bytes) {
#pragma unroll
                for (int j = 0; j < K; ++j)
                    bulk_g2s(dst + j * (uint32_t)Sh::chunk, hist_ptr(A, j, A.m_off[first + m]) + e0 * ES, bytes,
                             full0 + 8u * stage, policy);
            }
            if (xbytes)
                bulk_g2s(dst + K * (uint32_t)Sh::chunk, resid + e0 * (A.resid_bf16 ? 2 : 4), xbytes,
                         full0 + 8u * stage, normal);
            if (gb)
                bulk_g2s(dst + K * (uint32_t)Sh::chunk + A.stage_x_bytes,
                         reinterpret_cast<const unsigned char*>(A.m_gate[first + m]) + gsrc, gb, full0 + 8u * stage,
                         normal);
        }
        return true;
    };
    int it = 0, tile = blockIdx.x;
    bool ok = true;
    for (; ok && tile < A.tiles_total; tile += gridDim.x) {
        while (tile >= A.tile_begin[it + 1]) ++it;
        ok = issue(it, (long long)(tile - A.tile_begin[it]) * TE, true, (uint32_t)Sh::chunk,
                   tile < A.keep_tiles ? normal : passing);
    }
#pragma unroll 1
    for (; ok && tile < A.tiles_total + A.n_ragged; tile += gridDim.x) {
        it = A.ragged[tile - A.tiles_total];
        const long long e0 = (long long)(A.tile_begin[it + 1] - A.tile_begin[it]) * TE;
        ok = issue(it, e0, false, ragged_bytes<ES>(A, A.numel[it] - e0), normal);
    }
    // never leave while copies into this CTA's shared memory are in flight:
    // wait for every unit still in the ring; after one wait runs out (a unit
    // whose copies were never issued) the others get the short limit
    unsigned long long drain_ns = A.wait_ns > kMinDrainNs ? A.wait_ns : kMinDrainNs;
    bool drained = true;
    for (unsigned q = u > (unsigned)S ? u - S : 0; q < u; ++q)
        if (!mbar_wait(full0 + 8u * (q % S), (q / S) & 1u, drain_ns)) {
            drained = false;
            drain_ns = kMinDrainNs;
        }
    if (!drained) record(A.status, 4);
}

// Elements i, i + 1 of a ragged tile (n elements, of which the first `staged`
// lie in the chunk at p) as words of a vector. A tensor of odd length ends inside
// a pair: its second half is then whatever the slot's padding holds (no_padding).
// TAIL: some elements may not be staged (a full step's new features).
template <bool CB16, bool TAIL>
__device__ __forceinline__ uint2 ragged_pair(const unsigned char* p, int i, int n, int staged,
                                             const unsigned char* global) {
    uint2 w = make_uint2(0u, 0u);
    if (i >= n) return w;
    if (!TAIL || i + 1 < staged) {
        if constexpr (CB16)
            w.x = *reinterpret_cast<const uint32_t*>(p + 2 * i);
        else
            w = *reinterpret_cast<const uint2*>(p + 4 * i);
    } else if constexpr (CB16) {
        const uint16_t* q = reinterpret_cast<const uint16_t*>(global) + i;
        w.x = q[0] | (i + 1 < n ? (uint32_t)q[1] << 16 : 0u);
    } else {
        const uint32_t* q = reinterpret_cast<const uint32_t*>(global) + i;
        w = make_uint2(q[0], i + 1 < n ? q[1] : 0u);
    }
    return w;
}

// Clears the second half of the pair that ends a tensor of odd length n, in the
// history values of the vector whose pair q begins at at(q): the padding is
// nobody's value, and a NaN there would decide how the thread's other elements
// are summed. Once per vector, behind a branch that tiles of even length skip:
// tested with each pair's load it cost the fp32 kernels 14 to 40 registers.
template <int K, bool CB16, typename At>
__device__ __forceinline__ void no_padding(uint4 (&raw)[K][CB16 ? 1 : 2], int n, At at) {
    if ((n & 1) == 0) return;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        if (at(q) + 1 != n) continue;
#pragma unroll
        for (int j = 0; j < K; ++j) {
            if constexpr (CB16)
                (q == 0 ? raw[j][0].x : q == 1 ? raw[j][0].y : q == 2 ? raw[j][0].z : raw[j][0].w) &= 0xFFFFu;
            else
                ((q & 1) ? raw[j][q >> 1].w : raw[j][q >> 1].y) = 0u;
        }
    }
}

// Four pairs of elements p[at(q, 0)], p[at(q, 1)]; 0 where in(q, e) is false.
template <typename At, typename In>
__device__ __forceinline__ void read_pairs(const void* p, bool bf16, float (&x)[8], At at, In in) {
    if (bf16) {
#pragma unroll
        for (int i = 0; i < 8; ++i)
            x[i] = in(i >> 1, i & 1)
                       ? __uint_as_float((uint32_t)reinterpret_cast<const uint16_t*>(p)[at(i >> 1, i & 1)] << 16)
                       : 0.0f;
    } else {
#pragma unroll
        for (int i = 0; i < 8; ++i)
            x[i] = in(i >> 1, i & 1) ? reinterpret_cast<const float*>(p)[at(i >> 1, i & 1)] : 0.0f;
    }
}

// The consumers of launches with fp32 predictions or hidden states: every
// element takes the compensated sum (sum_vec), so nothing is recomputed and
// each stage goes back to the producer as soon as its values, and the hidden
// state behind the first member's, are in registers. Predictions alone stream
// at the copy rate (DiT-XL/2 512^2, K = 8, bf16 history, fp32 predictions: 1180 us
// with Dot2 in the common kernel, 740 us here, 7.1 TB/s); with gated fp32 hidden
// states the consumers' latency bounds them (K = 4: 897 -> 528 us, 6.0 TB/s at 57 %
// of the issue slots).
//
// A thread holds vecs vectors of eight elements. In a whole tile they are
// contiguous; in the ragged last tile of a tensor they are four pairs each,
// adjacent threads on adjacent pairs, so that any length is covered from
// shared memory with the same arithmetic (and bits).
//
// precise_tile: one tile of one item. RAGGED: pairs as above; FULL: of a whole
// tile, else of any length n. False when a wait ran out.
struct Cursor {
    uint32_t stage = 0, phase = 0;  // of the next unit to consume
};
template <typename Sh, int K, bool CB16, bool GROUPED, bool GATED, bool RAGGED, bool FULL = !RAGGED>
__device__ __forceinline__ bool precise_tile(const ExtrapArgs& A, int it, long long e0, int n, Cursor& cur,
                                             uint32_t full0, uint32_t empty0, const unsigned char* stages,
                                             uint32_t stage_bytes, int lane) {
    constexpr int ES = CB16 ? 2 : 4;
    constexpr int NCT = Sh::consumers;
    constexpr int U = Sh::vecs;
    const int c = threadIdx.x;
    const int nb = GROUPED ? A.nb[it] : 1;
    const int first = A.first[it];
    void* resid = GROUPED ? A.resid[it] : nullptr;
    // Gates come with the stage (staged_gates), else from global memory, asked
    // for before the wait, and wait in registers through the sums; with bf16
    // sources and K >= 5 the sums need those, and the gates are read after them
    // (DiT-XL/2 512^2, fp32 gates, before -> after the sums: K = 4 528 -> 536 us, K = 5
    // 615 -> 600, K = 6 663 -> 646, K = 7 727 -> 711, K = 8 812 -> 780).
    constexpr bool LATE_GATES = GATED && !RAGGED && CB16 && K >= 5;
    constexpr bool STAGED_GATES = GATED && !RAGGED && staged_gates(K, CB16);
    const int held = RAGGED && !FULL ? (int)ragged_bytes<ES>(A, n) / ES : Sh::tile;  // elements in the chunks
    auto in = [&](int i) { return FULL || i < n; };
    // first element of vector v of this thread, and of pair q of its vector v
    auto at = [&](int v) { return (v * NCT + c) * kVecElems; };
    auto pair_at = [&](int v, int q) { return 2 * (c + NCT * (4 * v + q)); };
    auto put = [&](void* p, bool bf16, int v, const uint32_t (&o)[8]) {
        if constexpr (!RAGGED) {
            store_o8(p, bf16, e0 + at(v), o);
        } else {
            unsigned char* base = reinterpret_cast<unsigned char*>(p) + e0 * (bf16 ? 2 : 4);
#pragma unroll
            for (int q = 0; q < 4; ++q)
                store_o2(base, bf16, pair_at(v, q), FULL ? 2 : n - pair_at(v, q), bf16 ? o[q] : o[2 * q], o[2 * q + 1]);
        }
    };
    const bool gated = GATED && resid != nullptr && A.i_row[it] != 0;  // items without a shape carry no gate
    unsigned gi[U];
    if constexpr (GATED && !RAGGED) {
        long long ev[U];
#pragma unroll
        for (int v = 0; v < U; ++v) ev[v] = e0 + at(v);
        if (gated) gate_offsets<U>(A, it, e0, ev, gi, STAGED_GATES && A.stage_gate_bytes != 0);
    }
    // ragged: of the pairs' first elements, and whether the second one lies in
    // the next token of the same batch, hidden channels back
    const unsigned hidden = GATED && RAGGED ? A.i_hidden[it] : 0u;
    unsigned gq[U][4], back = 0u;
    if constexpr (GATED && RAGGED) {
        if (gated)
#pragma unroll
            for (int v = 0; v < U; ++v)
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    bool b;
                    gate_offset_pair(A, it, e0 + (in(pair_at(v, q)) ? pair_at(v, q) : 0), gq[v][q], b);
                    back |= b ? 1u << (4 * v + q) : 0u;
                }
    }
    Acc<U> acc;
    Finite fin;
    if (GROUPED && RAGGED && resid != nullptr)  // not staged: asked for before the wait for the stage
        resid_begin<U>(acc, [&](int v, float (&x)[8]) {
            read_pairs(
                reinterpret_cast<const unsigned char*>(resid) + e0 * (A.resid_bf16 ? 2 : 4), A.resid_bf16, x,
                [&](int q, int e) { return pair_at(v, q) + e; }, [&](int q, int e) { return in(pair_at(v, q) + e); });
        });
#pragma unroll 1
    for (int m = 0; m < nb; ++m) {
        float g[U][8];
        if constexpr (GATED) {
            const void* gp = gated ? A.m_gate[first + m] : nullptr;
#pragma unroll
            for (int v = 0; v < U; ++v) {
                if (LATE_GATES || STAGED_GATES) continue;
                if (!RAGGED && gp != nullptr) {
                    load_x8(gp, A.gate_bf16, (long long)gi[v], g[v]);
                    continue;
                }
#pragma unroll
                for (int e = 0; e < 8; ++e) g[v][e] = 1.0f;
                if (RAGGED && gp != nullptr)
                    read_pairs(
                        gp, A.gate_bf16, g[v],
                        [&](int q, int e) { return gq[v][q] + e - (e && (back >> (4 * v + q) & 1u) ? hidden : 0u); },
                        [&](int q, int e) { return in(pair_at(v, q) + e); });
            }
        }
        const uint32_t stage = cur.stage;
        if (!__all_sync(~0u, mbar_wait(full0 + 8u * stage, cur.phase, A.wait_ns))) {
            if (lane == 0) record(A.status, 1);
            return false;
        }
        if (++cur.stage == (uint32_t)A.stages) {
            cur.stage = 0;
            cur.phase ^= 1u;
        }
        const unsigned char* base = stages + stage * stage_bytes;
        RawVecs<K, CB16, U> raw;
#pragma unroll
        for (int v = 0; v < U; ++v)
#pragma unroll
            for (int j = 0; j < K; ++j) {
                const unsigned char* chunk = base + j * Sh::chunk;
                if constexpr (!RAGGED) {
                    const unsigned char* p = chunk + at(v) * ES;
                    raw[v][j][0] = *reinterpret_cast<const uint4*>(p);
                    if constexpr (!CB16) raw[v][j][CB16 ? 0 : 1] = *reinterpret_cast<const uint4*>(p + 16);
                } else {
                    const unsigned char* src = hist_ptr(A, j, A.m_off[first + m]) + e0 * ES;
                    uint2 w[4];
#pragma unroll
                    for (int q = 0; q < 4; ++q) w[q] = ragged_pair<CB16, K == 1 && !FULL>(chunk, pair_at(v, q), FULL ? Sh::tile : n, held, src);
                    if constexpr (CB16) {
                        raw[v][j][0] = make_uint4(w[0].x, w[1].x, w[2].x, w[3].x);
                    } else {
                        raw[v][j][0] = make_uint4(w[0].x, w[0].y, w[1].x, w[1].y);
                        raw[v][j][CB16 ? 0 : 1] = make_uint4(w[2].x, w[2].y, w[3].x, w[3].y);
                    }
                }
            }
        if constexpr (RAGGED && !FULL)
#pragma unroll
            for (int v = 0; v < U; ++v) no_padding<K, CB16>(raw[v], n, [&](int q) { return pair_at(v, q); });
        if constexpr (STAGED_GATES) {  // rows that came with the stage, or from global memory
            const void* gp = gated ? A.m_gate[first + m] : nullptr;
            if (gp != nullptr && A.stage_gate_bytes) gp = base + K * Sh::chunk + A.stage_x_bytes;
#pragma unroll
            for (int v = 0; v < U; ++v) {
                if (gp != nullptr)
                    load_x8(gp, A.gate_bf16, (long long)gi[v], g[v]);
                else
#pragma unroll
                    for (int e = 0; e < 8; ++e) g[v][e] = 1.0f;
            }
        }
        if (GROUPED && !RAGGED && m == 0 && resid != nullptr)
            resid_begin<U>(acc, [&](int v, float (&x)[8]) { load_x8(base + K * Sh::chunk, A.resid_bf16, at(v), x); });
        release_stage(empty0 + 8u * stage, lane);
        void* out = A.m_out[first + m];
        bool want = out != nullptr;
        if constexpr (K == 1) {
            if (want && A.copy_out) {  // a full step: the slot receives the features converted
#pragma unroll
                for (int v = 0; v < U; ++v) {
                    uint32_t o[8];
                    copy_o8<CB16>(A.out_bf16, raw[v][0], o);
                    put(out, A.out_bf16, v, o);
                }
                want = false;
            }
        }
        member_precise<K, CB16, U, GATED>(
            A, want, raw, resid != nullptr, acc, fin,
            [&](int v, float (&gv)[8]) {
                if constexpr (GATED) {
                    const void* gp = LATE_GATES && gated ? A.m_gate[first + m] : nullptr;
                    if (gp != nullptr)
                        load_x8(gp, A.gate_bf16, (long long)gi[v], gv);
                    else
#pragma unroll
                        for (int e = 0; e < 8; ++e) gv[e] = LATE_GATES ? 1.0f : g[v][e];
                }
            },
            [&](int v, bool bf16, const uint32_t (&o)[8]) { put(out, bf16, v, o); });
    }
    if (resid != nullptr ? !resid_precise<K, U>(A, acc, fin,
                                                [&](int v, bool bf16, const uint32_t (&o)[8]) { put(resid, bf16, v, o); })
                         : !fin.all()) {
#pragma unroll 1
        for (int v = 0; v < U; ++v)
#pragma unroll 1
            for (int e = 0; e < kVecElems; ++e) {
                const int i = RAGGED ? pair_at(v, e >> 1) + (e & 1) : at(v) + e;
                if (in(i)) scalar_element<CB16>(A, K, it, e0 + i);
            }
    }
    return true;
}

// The ragged last tiles, after every whole tile of the launch: a loop of its
// own, so that their loads and stores cost the loop over whole tiles neither
// registers nor instruction cache (inside it they cost 5 to 15 %).
template <typename Sh, int K, bool CB16, bool GROUPED, bool GATED>
__device__ __forceinline__ bool ragged_tiles(const ExtrapArgs& A, int tile, Cursor& cur, uint32_t full0,
                                             uint32_t empty0, const unsigned char* stages, uint32_t stage_bytes,
                                             int lane) {
#pragma unroll 1
    for (; tile < A.tiles_total + A.n_ragged; tile += gridDim.x) {
        const int it = A.ragged[tile - A.tiles_total];
        const long long e0 = (long long)(A.tile_begin[it + 1] - A.tile_begin[it]) * Sh::tile;
        if (!precise_tile<Sh, K, CB16, GROUPED, GATED, true>(A, it, e0, (int)(A.numel[it] - e0), cur, full0, empty0,
                                                             stages, stage_bytes, lane))
            return false;
    }
    return true;
}

// Items whose sources are off the 16-byte grid (a full step's new features
// only): element by element from global memory, without the pipeline.
template <typename Sh, int K, bool CB16>
__device__ __forceinline__ void scalar_items(const ExtrapArgs& A) {
    if (!A.any_scalar) return;
#pragma unroll 1
    for (int it = 0; it < A.n_items; ++it) {
        if (A.vec_ok[it]) continue;
        const long long numel = A.numel[it], step = (long long)gridDim.x * Sh::consumers;
#pragma unroll 1
        for (long long e = (long long)blockIdx.x * Sh::consumers + threadIdx.x; e < numel; e += step)
            scalar_element<CB16>(A, K, it, e);
    }
}

// The consumers of every other launch, over the whole tiles (see the head of
// this file).
template <int K, bool CB16, bool GROUPED, bool GATED, bool ONE>
__device__ __forceinline__ bool fast_tiles(const ExtrapArgs& A, int& tile, Cursor& cur, uint32_t full0,
                                           uint32_t empty0, const unsigned char* stages, uint32_t stage_bytes,
                                           uint32_t gates_at, int lane) {
    using Sh = Shape<CB16, K, GROUPED, GATED, false>;
    constexpr int NCT = Sh::consumers;
    constexpr long long TE = Sh::tile;
    constexpr int ES = CB16 ? 2 : 4;
    constexpr int U = Sh::vecs;
    // the stage stays held through the member's arithmetic (see below)
    constexpr bool LATE = GROUPED || (CB16 && K >= 7);
    const int c = threadIdx.x;
    const int S = A.stages;
    auto chunk = [&](uint32_t stage, int j) { return stages + stage * stage_bytes + (size_t)j * Sh::chunk; };
    auto gate_stage = [&](uint32_t stage) -> const void* { return stages + stage * stage_bytes + gates_at; };
    int it = 0;
    for (; tile < A.tiles_total; tile += gridDim.x) {
        while (tile >= A.tile_begin[it + 1]) ++it;
        const long long e0 = (long long)(tile - A.tile_begin[it]) * TE;
        const int nb = GROUPED ? A.nb[it] : 1;
        const int first = A.first[it];
        void* resid = GROUPED ? A.resid[it] : nullptr;
        // with a hidden state, every member's stage stays held until the hidden
        // state is written, so that its guarded elements can be recomputed
        const bool hold = GROUPED && resid != nullptr;
        // stage of member m of this tile (nb < S: one wrap at most)
        const uint32_t s0 = cur.stage;
        auto stage_of = [&](int m) { return s0 + m < (uint32_t)S ? s0 + m : s0 + m - (uint32_t)S; };
        long long ev[U];
#pragma unroll
        for (int v = 0; v < U; ++v) ev[v] = e0 + ((long long)v * NCT + c) * kVecElems;
        // gate offsets of this thread's vectors, relative to the gate rows the
        // producer staged (or absolute, when gates stay in global memory)
        unsigned gi[U];
        if constexpr (GATED) {
            if (hold && A.i_row[it] != 0)  // items without a shape carry no gate
                gate_offsets<U>(A, it, e0, ev, gi, A.stage_gate_bytes != 0);
        }
        Acc<U> acc;
        acc.zero();
        for (int m = 0; m < nb; ++m) {
            const uint32_t stage = cur.stage;
            // the give-up is warp-uniform: no lane leaves while its warp-mates
            // go on to a __syncwarp
            if (!__all_sync(~0u, mbar_wait(full0 + 8u * stage, cur.phase, A.wait_ns))) {
                if (lane == 0) record(A.status, 1);
                return false;
            }
            if (++cur.stage == (uint32_t)S) {
                cur.stage = 0;
                cur.phase ^= 1u;
            }
            RawVecs<K, CB16, U> raw;
#pragma unroll
            for (int v = 0; v < U; ++v)
#pragma unroll
                for (int j = 0; j < K; ++j) {
                    const unsigned char* p = chunk(stage, j) + (size_t)(ev[v] - e0) * ES;
                    raw[v][j][0] = *reinterpret_cast<const uint4*>(p);
                    if constexpr (!CB16) raw[v][j][CB16 ? 0 : 1] = *reinterpret_cast<const uint4*>(p + 16);
                }
            // gates of this member (staged rows or global memory), read as
            // each vector is accumulated
            const void* gp = GATED ? A.m_gate[first + m] : nullptr;
            if (GATED && gp && A.stage_gate_bytes) gp = gate_stage(stage);
            auto gate = [&](int v, float (&gv)[8]) {
                if (gp)
                    load_x8(gp, A.gate_bf16, (long long)gi[v], gv);
                else
#pragma unroll
                    for (int e = 0; e < 8; ++e) gv[e] = 1.0f;
            };
            // prediction-only launches release the stage as soon as it is read
            // and recompute guarded elements from registers; grouped launches
            // and bf16 ones with K >= 7 keep the stage until the member is done
            // and recompute from shared memory, which frees the history values'
            // registers early (bf16 K >= 7 would otherwise spill under the cap)
            if (!LATE) release_stage(empty0 + 8u * stage, lane);
            void* out = member_out<K, CB16, U>(A, first + m, ev, raw);
            if constexpr (ONE) {
                if (resid != nullptr) member_one<K, CB16, U, GATED>(raw, acc, gate);
            } else if constexpr (LATE) {
                auto exact = [&](int v, int e, float& hi, float& lo) {
                    const size_t off = (size_t)(ev[v] - e0 + e) * ES;
                    float p = 0.0f, cc = 0.0f;
#pragma unroll
                    for (int j = 0; j < K; ++j) {
                        const unsigned char* src = chunk(stage, j) + off;
                        const float f = CB16 ? __uint_as_float((uint32_t)(*reinterpret_cast<const uint16_t*>(src)) << 16)
                                             : *reinterpret_cast<const float*>(src);
                        dot2_step(A.w_hi[j], A.w_lo[j], f, p, cc);
                    }
                    two_sum(p, cc, hi, lo);
                };
                member_fast<K, CB16, U, false, GATED>(A, A.m_off[first + m], out, ev, raw, resid != nullptr,
                                                      acc, gate, exact);
            } else {
                member_fast<K, CB16, U, true, GATED>(A, A.m_off[first + m], out, ev, raw, resid != nullptr,
                                                     acc, gate);
            }
            if (LATE && !hold) release_stage(empty0 + 8u * stage, lane);
        }
        if (GROUPED && hold) {
            // the bf16 hidden state, behind the first member's chunks
            auto xload = [&](int v, float (&x)[8]) {
                unpack_bf16x8(*reinterpret_cast<const uint4*>(chunk(s0, K) + (size_t)(ev[v] - e0) * 2), x);
            };
            // Dot2 of x + sum_b P_b for one element, from the held stages
            auto exact = [&](int v, int e, float xe, float& hi, float& lo) {
                const size_t off = (size_t)(ev[v] - e0 + e) * ES;
                float tp = xe, tc = 0.0f;
                for (int m = 0; m < nb; ++m) {
                    const uint32_t st = stage_of(m);
                    float p = 0.0f, cc = 0.0f, h, l, qq;
#pragma unroll
                    for (int j = 0; j < K; ++j) {
                        const unsigned char* src = chunk(st, j) + off;
                        const float f = CB16 ? __uint_as_float((uint32_t)(*reinterpret_cast<const uint16_t*>(src)) << 16)
                                             : *reinterpret_cast<const float*>(src);
                        dot2_step(A.w_hi[j], A.w_lo[j], f, p, cc);
                    }
                    two_sum(p, cc, h, l);
                    // a member without a gate adds like an ungated one (as exact_resid)
                    const void* gm = GATED ? A.m_gate[first + m] : nullptr;
                    if (gm) {
                        const float gv = load_elem(A.stage_gate_bytes ? gate_stage(st) : gm, A.gate_bf16, gi[v] + e);
                        add_gated_pair(gv, h, l, tp, tc);
                    } else {
                        two_sum(tp, h, tp, qq);
                        tc = __fadd_rn(tc, __fadd_rn(qq, l));
                    }
                }
                two_sum(tp, tc, hi, lo);
            };
            resid_fast<K, U>(A, it, ev, acc, resid, xload, exact, ONE ? A.w_guard[0] : 1.0f);
            fence_generic_to_async();
            __syncwarp();
            if (lane == 0)
                for (int m = 0; m < nb; ++m) mbar_arrive(empty0 + 8u * stage_of(m));
        }
    }
    return true;
}

// GROUPED: some item updates a hidden state or has several members (stage
// holding, hidden-state staging); prediction-only launches compile without
// that bookkeeping. GATED (with GROUPED): the hidden state receives g_b * P_b,
// with a per-(batch, channel) gate per member.
// ONE: the full-step epilogue (copy_out with bf16 hidden states or none): a
// one-entry history of weight 1, whose member step needs no weighted sum
// (member_one); PRECISE: fp32 predictions or hidden states; STRIDED: items whose
// outputs, hidden state or gates are off the 16-byte grid (or whose gate rows
// hold no whole vectors), every tile by pairs of elements. Compiled apart so
// that each kernel carries only its own path.
template <int K, bool CB16, bool GROUPED, bool GATED, bool ONE = false, bool PRECISE = false, bool STRIDED = false>
__global__ void __launch_bounds__(Shape<CB16, K, GROUPED, GATED, PRECISE, STRIDED>::threads,
                                  Shape<CB16, K, GROUPED, GATED, PRECISE, STRIDED>::ctas_per_sm)
    extrapolate_bulk_kernel(const __grid_constant__ ExtrapArgs A) {
    static_assert(!ONE || (K == 1 && !PRECISE), "the epilogue is a one-entry history");
    static_assert(!STRIDED || PRECISE, "strided tiles are compensated");
    extern __shared__ __align__(128) unsigned char smem[];
    using Sh = Shape<CB16, K, GROUPED, GATED, PRECISE, STRIDED>;
    constexpr int NCW = Sh::consumer_warps;
    constexpr long long TE = Sh::tile;
    const int S = A.stages;
    const uint32_t full0 = smem_addr(smem);
    const uint32_t empty0 = full0 + 8u * (uint32_t)S;
    const uint32_t buf0 = smem_addr(smem + kBarrierBytes);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

    if (threadIdx.x == 0) {
        for (int s = 0; s < S; ++s) {
            mbar_init(full0 + 8u * s, 1);
            mbar_init(empty0 + 8u * s, NCW);
        }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncthreads();
    after_previous();

    // offset of the gate rows in a stage (a grouped launch has hidden states)
    const uint32_t gates_at =
        (uint32_t)K * Sh::chunk + (!GROUPED ? 0u : PRECISE ? A.stage_x_bytes : (uint32_t)Sh::tile * 2u);
    const uint32_t stage_bytes = gates_at + (GATED ? A.stage_gate_bytes : 0u);
    if (warp == NCW) {
        if (lane == 0) produce<Sh, K, CB16, GROUPED, GATED>(A, full0, empty0, buf0, stage_bytes);
        return;
    }
    const unsigned char* stages = smem + kBarrierBytes;
    Cursor cur;
    int tile = blockIdx.x;
    if constexpr (PRECISE) {
        int it = 0;
        for (; tile < A.tiles_total; tile += gridDim.x) {
            while (tile >= A.tile_begin[it + 1]) ++it;
            const long long e0 = (long long)(tile - A.tile_begin[it]) * TE;
            if (!precise_tile<Sh, K, CB16, GROUPED, GATED, STRIDED, true>(A, it, e0, (int)TE, cur, full0, empty0, stages,
                                                                          stage_bytes, lane))
                return;
        }
    } else if (!fast_tiles<K, CB16, GROUPED, GATED, ONE>(A, tile, cur, full0, empty0, stages, stage_bytes, gates_at,
                                                         lane)) {
        return;
    }
    if (!ragged_tiles<Sh, K, CB16, GROUPED, GATED>(A, tile, cur, full0, empty0, stages, stage_bytes, lane)) return;
    if constexpr (!STRIDED) scalar_items<Sh, K, CB16>(A);
}

}  // namespace
}  // namespace cbk
