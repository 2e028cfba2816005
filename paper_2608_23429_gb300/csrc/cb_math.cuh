// Internal: the per-element arithmetic of the skipped-step kernels, shared by
// the direct-load kernel (direct_kernel.cuh) and the bulk-copy pipeline kernel
// (bulk_kernel.cuh). Where both take the same of its two ways to sum, they
// produce identical bits: see the head of bulk_kernel.cuh for where they do not.
//
// Fast path. s = sum_j w_hi[j] F_j by fp32 FMA and, alongside,
// a = sum_j |w_hi[j]| |F_j|. With u = 2^-24 the FMA chain plus the dropped low
// half of each weight give |s - P| <= (K+1) u a (1 + O(Ku)). Whenever
// (K+2) u a (1.01) <= 2^-9 |s| that error is below the smallest bf16 spacing
// next to s, so bf16(s) lies within one bf16 ulp of bf16(P). The kernels
// accumulate the bound already scaled, a' = sum_j w_guard[j] |F_j| with
// w_guard[j] = (K+2) u (1.01) 2^9 |w_hi[j]| (host-computed), so the test is
// a' <= |s|; the 1 % margin covers the extra fp32 roundings of a'.
// Elements failing the test (strong cancellation, ~1e-4..3e-3 of them) are
// recomputed from the values already loaded with Dot2 (Ogita, Rump &
// Oishi, "Accurate Sum and Dot Product", SIAM J. Sci. Comput. 26(6), 2005:
// TwoProduct by FMA plus TwoSum) with the weights as fp32 pairs hi + lo, and
// the unevaluated result pair is rounded once. fp32 results always take a
// compensated sum (sum_vec below): Dot2 for K <= 2, an anchored sum from
// K = 3 on, both on pairs of elements with packed fp32 operations.
#pragma once

#include <cuda_bf16.h>

#include <type_traits>

#include "cb_device.h"

namespace cbk {
namespace {

constexpr float kU = 0x1.0p-24f;

// Plain 16-byte global load of history values (direct-load kernel). The
// streaming form (ld.global.nc with L1::no_allocate) measured slower on GB300:
// the FLUX skipped step took 2159 us with it and 1940 us without.
__device__ __forceinline__ uint4 ld_v4(const unsigned char* p) {
    uint4 v;
    asm("ld.global.v4.u32 {%0,%1,%2,%3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p));
    return v;
}

__device__ __forceinline__ void unpack_bf16x8(const uint4& v, float (&f)[8]) {
    const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        f[2 * i] = __uint_as_float(w[i] << 16);
        f[2 * i + 1] = __uint_as_float(w[i] & 0xFFFF0000u);
    }
}

__device__ __forceinline__ void unpack_f32x8(const uint4& a, const uint4& b, float (&f)[8]) {
    f[0] = __uint_as_float(a.x); f[1] = __uint_as_float(a.y);
    f[2] = __uint_as_float(a.z); f[3] = __uint_as_float(a.w);
    f[4] = __uint_as_float(b.x); f[5] = __uint_as_float(b.y);
    f[6] = __uint_as_float(b.z); f[7] = __uint_as_float(b.w);
}

template <bool CB16>
__device__ __forceinline__ void unpack(const uint4 (&r)[CB16 ? 1 : 2], float (&f)[8]) {
    if constexpr (CB16)
        unpack_bf16x8(r[0], f);
    else
        unpack_f32x8(r[0], r[CB16 ? 0 : 1], f);
}

// Elements 2q and 2q + 1 of a vector.
template <bool CB16>
__device__ __forceinline__ float2 vec_pair(const uint4 (&r)[CB16 ? 1 : 2], int q) {
    if constexpr (CB16) {
        const uint32_t w = q == 0 ? r[0].x : q == 1 ? r[0].y : q == 2 ? r[0].z : r[0].w;
        return make_float2(__uint_as_float(w << 16), __uint_as_float(w & 0xFFFF0000u));
    } else {
        const uint4 v = r[(q >> 1) & (CB16 ? 0 : 1)];
        return (q & 1) ? make_float2(__uint_as_float(v.z), __uint_as_float(v.w))
                       : make_float2(__uint_as_float(v.x), __uint_as_float(v.y));
    }
}

__device__ __forceinline__ uint32_t pack_bf16x2(float lo, float hi) {
    __nv_bfloat162 h = __floats2bfloat162_rn(lo, hi);  // RNE; .x is the low half
    return *reinterpret_cast<uint32_t*>(&h);
}

__device__ __forceinline__ uint16_t bf16_bits(float x) { return __bfloat16_as_ushort(__float2bfloat16_rn(x)); }

// ---- error-free transformations (explicitly rounded operations, never contracted)
__device__ __forceinline__ void two_sum(float a, float b, float& s, float& e) {
    s = __fadd_rn(a, b);
    const float bb = __fsub_rn(s, a);
    e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
}

// One Dot2 term: (p, c) += (w_hi + w_lo) * f, p the running sum, c its error.
__device__ __forceinline__ void dot2_step(float w_hi, float w_lo, float f, float& p, float& c) {
    const float h = __fmul_rn(w_hi, f);
    const float r = __fmaf_rn(w_hi, f, -h);  // exact: w_hi*f - h
    float q;
    two_sum(p, h, p, q);
    c = __fadd_rn(c, __fadd_rn(q, r));
    c = __fmaf_rn(w_lo, f, c);
}

// ---- the same on pairs of elements (packed operations: half the issue slots
// at the same rate per lane, 115 lane operations per clock and SM measured)
__device__ __forceinline__ float2 pair_of(float x) { return make_float2(x, x); }
__device__ __forceinline__ float2 add2(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 sub2(float2 a, float2 b) { return __ffma2_rn(b, pair_of(-1.0f), a); }  // a - b, rounded once
__device__ __forceinline__ float2 mul2(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
// x y + z in bf16, both halves of a word
__device__ __forceinline__ uint32_t fma_bf16x2(uint32_t x, uint32_t y, uint32_t z) {
    uint32_t r;
    asm("fma.rn.bf16x2 %0, %1, %2, %3;" : "=r"(r) : "r"(x), "r"(y), "r"(z));
    return r;
}
__device__ __forceinline__ void two_sum2(float2 a, float2 b, float2& s, float2& e) {
    s = add2(a, b);
    const float2 bb = sub2(s, a);
    e = add2(sub2(a, sub2(s, bb)), sub2(b, bb));
}

// bf16 of the exact value hi + lo, where hi = fl(hi + lo) (so |lo| <= ulp(hi)/2).
// Only when hi sits exactly on a bf16 rounding midpoint can lo change the
// outcome; then the sign of lo decides, otherwise hi rounds like hi + lo.
__device__ __forceinline__ uint16_t bf16_of_pair(float hi, float lo) {
    const uint32_t b = __float_as_uint(hi);
    if ((b & 0xFFFFu) == 0x8000u && lo != 0.0f && (b & 0x7F800000u) != 0x7F800000u) {
        const bool away = (lo > 0.0f) == (hi > 0.0f);
        return (uint16_t)((b >> 16) + (away ? 1u : 0u));
    }
    return bf16_bits(hi);
}

// hi + lo (hi = fl(hi + lo), finite) rounded to odd: of the two fp32 values about
// it the one with an odd last bit, unless it is exact. Rounding that to nearest
// bf16 gives what rounding hi + lo gives (Boldo & Melquiond, "Emulation of a
// FMA and correctly rounded sums: proved algorithms using rounding to odd",
// IEEE Trans. Comput. 57(4), 2008).
__device__ __forceinline__ float odd_of_pair(float hi, float lo) {
    const uint32_t b = __float_as_uint(hi);
    const bool inexact = lo != 0.0f && (b & 1u) == 0u && (b & 0x7F800000u) != 0x7F800000u;
    const uint32_t step = 1u | (uint32_t)((int)(b ^ __float_as_uint(lo)) >> 31);  // away from zero 1, towards it -1
    return __uint_as_float(inexact ? b + step : b);
}

// Start of history entry j of the member at byte offset moff.
__device__ __forceinline__ const unsigned char* hist_ptr(const ExtrapArgs& A, int j, long long moff) {
    return reinterpret_cast<const unsigned char*>(A.hist_base + (unsigned long long)A.slot_off[j] +
                                                  (unsigned long long)moff);
}

template <bool CB16>
__device__ __forceinline__ float load_cache_elem(const unsigned char* base, long long e) {
    if constexpr (CB16) {
        const uint16_t h = reinterpret_cast<const uint16_t*>(base)[e];
        return __uint_as_float((uint32_t)h << 16);
    } else {
        return reinterpret_cast<const float*>(base)[e];
    }
}

__device__ __forceinline__ float load_elem(const void* p, bool bf16, long long e) {
    if (bf16) return __uint_as_float((uint32_t)(reinterpret_cast<const uint16_t*>(p)[e]) << 16);
    return reinterpret_cast<const float*>(p)[e];
}

__device__ __forceinline__ void store_pair(void* p, bool bf16, long long e, float hi, float lo) {
    if (bf16)
        reinterpret_cast<uint16_t*>(p)[e] = bf16_of_pair(hi, lo);
    else
        reinterpret_cast<float*>(p)[e] = hi;
}

// Full-step epilogue: element e of a source converted to the output type (bit
// copy for equal types, exact widening, round-to-nearest-even narrowing).
template <bool CB16>
__device__ __forceinline__ void copy_elem(void* out, bool out_bf16, const unsigned char* src, long long e) {
    if constexpr (CB16) {
        const uint16_t h = reinterpret_cast<const uint16_t*>(src)[e];
        if (out_bf16)
            reinterpret_cast<uint16_t*>(out)[e] = h;
        else
            reinterpret_cast<uint32_t*>(out)[e] = (uint32_t)h << 16;
    } else {
        const float f = reinterpret_cast<const float*>(src)[e];
        if (out_bf16)
            reinterpret_cast<uint16_t*>(out)[e] = bf16_bits(f);
        else
            reinterpret_cast<float*>(out)[e] = f;
    }
}

// Gate of member mi (item it) at element e: g[b * hidden + h] for element
// e = (b * tokens + token) * hidden + h; 1 when the member has no gate.
__device__ __forceinline__ float gate_at(const ExtrapArgs& A, int mi, int it, long long e) {
    const void* g = A.m_gate[mi];
    if (!g) return 1.0f;
    const unsigned long long row = A.i_row[it], H = A.i_hidden[it], ue = (unsigned long long)e;
    return load_elem(g, A.gate_bf16, (long long)(ue / row * H + ue % H));
}

// Exact product g * (h + l) added to the unevaluated sum tp + tc.
__device__ __forceinline__ void add_gated_pair(float g, float h, float l, float& tp, float& tc) {
    const float gh = __fmul_rn(g, h);
    const float gr = __fmaf_rn(g, h, -gh);  // exact: g*h - gh
    float q;
    two_sum(tp, gh, tp, q);
    tc = __fadd_rn(tc, __fadd_rn(q, gr));
    tc = __fmaf_rn(g, l, tc);
}

// Compensated value of member tensor (byte offset moff) at element e.
template <bool CB16>
__device__ __noinline__ void exact_member(const ExtrapArgs& A, int K, long long moff, long long e, float& hi,
                                          float& lo) {
    float p = 0.0f, c = 0.0f;
    for (int j = 0; j < K; ++j) {
        const float f = load_cache_elem<CB16>(hist_ptr(A, j, moff), e);
        dot2_step(A.w_hi[j], A.w_lo[j], f, p, c);
    }
    two_sum(p, c, hi, lo);
}

// Compensated hidden-state update of item `it` at element e: x + sum_b P_b.
template <bool CB16>
__device__ __noinline__ void exact_resid(const ExtrapArgs& A, int K, int it, long long e, float x, float& hi,
                                         float& lo) {
    float tp = x, tc = 0.0f;
    const int first = A.first[it];
    for (int m = 0; m < A.nb[it]; ++m) {
        float h, l, q;
        exact_member<CB16>(A, K, A.m_off[first + m], e, h, l);
        if (A.m_gate[first + m]) {
            add_gated_pair(gate_at(A, first + m, it, e), h, l, tp, tc);
        } else {
            two_sum(tp, h, tp, q);
            tc = __fadd_rn(tc, __fadd_rn(q, l));
        }
    }
    two_sum(tp, tc, hi, lo);
}

// One element of item `it` through the compensated path, the hidden state and
// every member (misaligned items and ragged tails).
template <bool CB16>
__device__ __noinline__ void scalar_element(const ExtrapArgs& A, int K, int it, long long e) {
    const int first = A.first[it];
    void* resid = A.resid[it];
    float tp = resid ? load_elem(resid, A.resid_bf16, e) : 0.0f, tc = 0.0f;
    for (int m = 0; m < A.nb[it]; ++m) {
        float hi, lo, q;
        exact_member<CB16>(A, K, A.m_off[first + m], e, hi, lo);
        void* out = A.m_out[first + m];
        if (out && A.copy_out)
            copy_elem<CB16>(out, A.out_bf16, hist_ptr(A, 0, A.m_off[first + m]), e);
        else if (out)
            store_pair(out, A.out_bf16, e, hi, lo);
        if (A.m_gate[first + m]) {
            add_gated_pair(gate_at(A, first + m, it, e), hi, lo, tp, tc);
        } else {
            two_sum(tp, hi, tp, q);
            tc = __fadd_rn(tc, __fadd_rn(q, lo));
        }
    }
    if (resid) {
        float hi, lo;
        two_sum(tp, tc, hi, lo);
        store_pair(resid, A.resid_bf16, e, hi, lo);
    }
}

__device__ __forceinline__ void load_x8(const void* p, bool bf16, long long e, float (&x)[8]) {
    if (bf16) {
        const uint4 v = *reinterpret_cast<const uint4*>(reinterpret_cast<const uint16_t*>(p) + e);
        unpack_bf16x8(v, x);
    } else {
        const uint4* q = reinterpret_cast<const uint4*>(reinterpret_cast<const float*>(p) + e);
        unpack_f32x8(q[0], q[1], x);
    }
}

__device__ __forceinline__ void store_bf16x8(void* p, long long e, const uint32_t (&pk)[4]) {
    *reinterpret_cast<uint4*>(reinterpret_cast<uint16_t*>(p) + e) = make_uint4(pk[0], pk[1], pk[2], pk[3]);
}

__device__ __forceinline__ void store_f32x8(void* p, long long e, const float (&v)[8]) {
    uint4* q = reinterpret_cast<uint4*>(reinterpret_cast<float*>(p) + e);
    q[0] = make_uint4(__float_as_uint(v[0]), __float_as_uint(v[1]), __float_as_uint(v[2]), __float_as_uint(v[3]));
    q[1] = make_uint4(__float_as_uint(v[4]), __float_as_uint(v[5]), __float_as_uint(v[6]), __float_as_uint(v[7]));
}

// Running sums of one item across its members (the fused hidden-state update):
// fast path x = sum_b s_b, y = sum_b a_b; compensated path x + y is the
// unevaluated sum (running value and its error), begun from the hidden state.
template <int UV>
struct Acc {
    float x[UV][8];
    float y[UV][8];
    __device__ __forceinline__ void zero() {
#pragma unroll
        for (int u = 0; u < UV; ++u)
#pragma unroll
            for (int e = 0; e < 8; ++e) x[u][e] = y[u][e] = 0.0f;
    }
};

template <int K, bool CB16, int UV>
using RawVecs = uint4[UV][K][CB16 ? 1 : 2];

// Elements 2q, 2q + 1 (the pairs hi + lo, one rounding) into the eight output
// elements of a vector: fp32 in o[0..7], or bf16 in o[0..3].
__device__ __forceinline__ void put_pair(uint32_t (&o)[8], bool bf16, int q, float2 hi, float2 lo) {
    if (bf16) {
        o[q] = pack_bf16x2(odd_of_pair(hi.x, lo.x), odd_of_pair(hi.y, lo.y));
    } else {
        o[2 * q] = __float_as_uint(hi.x);
        o[2 * q + 1] = __float_as_uint(hi.y);
    }
}

// One pair of output elements e, e + 1 (words w0, w1 as put_pair leaves them);
// n of the two exist. Adjacent threads hold adjacent pairs.
__device__ __forceinline__ void store_o2(void* p, bool bf16, long long e, int n, uint32_t w0, uint32_t w1) {
    if (n <= 0) return;
    if (bf16) {
        uint16_t* q = reinterpret_cast<uint16_t*>(p) + e;
        if (n > 1 && (reinterpret_cast<uintptr_t>(q) & 3) == 0) {
            *reinterpret_cast<uint32_t*>(q) = w0;
        } else {
            q[0] = (uint16_t)w0;
            if (n > 1) q[1] = (uint16_t)(w0 >> 16);
        }
    } else {
        uint32_t* q = reinterpret_cast<uint32_t*>(p) + e;
        if (n > 1 && (reinterpret_cast<uintptr_t>(q) & 7) == 0) {
            *reinterpret_cast<uint2*>(q) = make_uint2(w0, w1);
        } else {
            q[0] = w0;
            if (n > 1) q[1] = w1;
        }
    }
}

__device__ __forceinline__ void store_o8(void* p, bool bf16, long long e, const uint32_t (&o)[8]) {
    if (bf16) {
        *reinterpret_cast<uint4*>(reinterpret_cast<uint16_t*>(p) + e) = make_uint4(o[0], o[1], o[2], o[3]);
    } else {
        uint4* q = reinterpret_cast<uint4*>(reinterpret_cast<float*>(p) + e);
        q[0] = make_uint4(o[0], o[1], o[2], o[3]);
        q[1] = make_uint4(o[4], o[5], o[6], o[7]);
    }
}

// Full-step epilogue: the 8 source values of a vector in the output type (see
// copy_elem): fp32 in o[0..7], or bf16 in o[0..3].
template <bool CB16>
__device__ __forceinline__ void copy_o8(bool out_bf16, const uint4 (&r)[CB16 ? 1 : 2], uint32_t (&o)[8]) {
    const uint4 a = r[0], b = r[CB16 ? 0 : 1];
    const uint32_t w[8] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w};
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        if constexpr (CB16) {
            if (out_bf16) {
                o[i] = w[i];
            } else {
                o[2 * i] = w[i] << 16;
                o[2 * i + 1] = w[i] & 0xFFFF0000u;
            }
        } else {
            if (out_bf16) {
                o[i] = pack_bf16x2(__uint_as_float(w[2 * i]), __uint_as_float(w[2 * i + 1]));
            } else {
                o[2 * i] = w[2 * i];
                o[2 * i + 1] = w[2 * i + 1];
            }
        }
    }
}

// ... written to out at element e.
template <bool CB16>
__device__ __forceinline__ void copy_vec(void* out, bool out_bf16, long long e, const uint4 (&r)[CB16 ? 1 : 2]) {
    uint32_t o[8];
    if (out_bf16) {  // two branches with their stores: one store behind a choice of words costs the epilogue 15 %
        copy_o8<CB16>(true, r, o);
        store_o8(out, true, e, o);
    } else {
        copy_o8<CB16>(false, r, o);
        store_o8(out, false, e, o);
    }
}

// Output pointer handed to member_fast / member_precise for member mi: in the
// full-step epilogue the sources are written out converted here and no
// prediction is stored (null); otherwise the member's prediction output.
template <int K, bool CB16, int UV>
__device__ __forceinline__ void* member_out(const ExtrapArgs& A, int mi, const long long (&ev)[UV],
                                            const RawVecs<K, CB16, UV>& raw) {
    void* out = A.m_out[mi];
    if (!A.copy_out) return out;
    if (out)
#pragma unroll
        for (int u = 0; u < UV; ++u) copy_vec<CB16>(out, A.out_bf16, ev[u], raw[u][0]);
    return nullptr;
}

// Gate source of an ungated accumulation (never called).
struct NoGate {
    __device__ void operator()(int, float (&)[8]) const {}
};

// Placeholder for "no recompute functor" (never called).
struct NoExact {
    __device__ void operator()(int, int, float&, float&) const {}
};

// Dot2 value of element e of vector u from its K history values as loaded
// (registers or shared memory); used where the fast path's guard fails.
template <int K, bool CB16, int UV>
__device__ __forceinline__ void exact_from_raw(const ExtrapArgs& A, const RawVecs<K, CB16, UV>& raw, int u, int e,
                                               float& hi, float& lo) {
    float p = 0.0f, c = 0.0f;
#pragma unroll
    for (int j = 0; j < K; ++j) {
        float f[8];
        unpack<CB16>(raw[u][j], f);
        float fe = f[0];
#pragma unroll
        for (int i = 1; i < 8; ++i) fe = (e == i) ? f[i] : fe;
        dot2_step(A.w_hi[j], A.w_lo[j], fe, p, c);
    }
    two_sum(p, c, hi, lo);
}

// Fast-path guard: with |s - P| <= (K+1) u a (1 + O(Ku)), the test
// (K+2) u a (1.01) <= 2^-9 |s| keeps the interval between s and P shorter than
// the smallest bf16 spacing next to s (2^-8 |s| in s's binade, 2^-9 |s| below
// it), so it holds at most one rounding midpoint and bf16(s) is within one ulp
// of bf16(P). With the scaled bound a' (see above) the test is a' <= |s|.
__device__ __forceinline__ bool guard_ok(float a_scaled, float s) { return a_scaled <= fabsf(s); }

// s0, s1 += w * (f0, f1): one paired fp32 FMA, each lane rounded like fmaf.
__device__ __forceinline__ void fma_pair(float w, float f0, float f1, float& s0, float& s1) {
    const float2 r = __ffma2_rn(make_float2(w, w), make_float2(f0, f1), make_float2(s0, s1));
    s0 = r.x;
    s1 = r.y;
}

// Fast path for one member over UV aligned 8-element vectors already loaded
// into registers: bf16 prediction (if out) and accumulation into acc. The
// rare guarded elements are recomputed by exact(u, e, hi, lo) when given
// (e.g. from shared memory), else from the loaded values (FROM_RAW: no memory
// latency, but the values stay live and cost registers) or re-read from
// global memory (member byte offset moff).
// GATED: gate(u, g) supplies the 8 gate values of vector u when it is
// accumulated (late, so that they are not live beside the history values).
template <int K, bool CB16, int UV, bool FROM_RAW, bool GATED = false, typename Gate = NoGate,
          typename Exact = NoExact>
__device__ __forceinline__ void member_fast(const ExtrapArgs& A, long long moff, void* out,
                                            const long long (&ev)[UV], const RawVecs<K, CB16, UV>& raw,
                                            bool accumulate, Acc<UV>& acc, Gate gate = {}, Exact exact = {}) {
#pragma unroll
    for (int u = 0; u < UV; ++u) {
        float s[8], a[8];
#pragma unroll
        for (int e = 0; e < 8; ++e) s[e] = a[e] = 0.0f;
#pragma unroll
        for (int j = 0; j < K; ++j) {
            float f[8];
            unpack<CB16>(raw[u][j], f);
#pragma unroll
            for (int e = 0; e < 8; e += 2) fma_pair(A.w_hi[j], f[e], f[e + 1], s[e], s[e + 1]);
#pragma unroll
            for (int e = 0; e < 8; ++e) a[e] = fmaf(A.w_guard[j], fabsf(f[e]), a[e]);
        }
        if (out) {
            uint32_t pk[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) pk[i] = pack_bf16x2(s[2 * i], s[2 * i + 1]);
            unsigned bad = 0;
#pragma unroll
            for (int e = 0; e < 8; ++e) bad |= guard_ok(a[e], s[e]) ? 0u : (1u << e);
            store_bf16x8(out, ev[u], pk);
            // rare: the failing elements get their Dot2 value, stored by this
            // thread over the fast-path bf16 it has just written (the vector is
            // dead by then, so the loop keeps nothing of the fast path live)
            while (bad) {
                const int e = __ffs(bad) - 1;
                bad &= bad - 1;
                float hi, lo;
                if constexpr (!std::is_same_v<Exact, NoExact>)
                    exact(u, e, hi, lo);
                else if constexpr (FROM_RAW)
                    exact_from_raw<K, CB16, UV>(A, raw, u, e, hi, lo);
                else
                    exact_member<CB16>(A, K, moff, ev[u] + e, hi, lo);
                reinterpret_cast<uint16_t*>(out)[ev[u] + e] = bf16_of_pair(hi, lo);
            }
        }
        if (accumulate) {
            float g[8];
            if constexpr (GATED) gate(u, g);
#pragma unroll
            for (int e = 0; e < 8; ++e) {
                if constexpr (GATED) {  // x + g * s: one rounding, bound |g| a'
                    acc.x[u][e] = fmaf(g[e], s[e], acc.x[u][e]);
                    acc.y[u][e] = fmaf(fabsf(g[e]), a[e], acc.y[u][e]);
                } else {
                    acc.x[u][e] += s[e];
                    acc.y[u][e] += a[e];
                }
            }
        }
    }
}

// Full-step epilogue (a one-entry history of weight 1): member features f,
// taken exactly, added into the hidden-state sums, acc.x += g f and the
// unscaled bound acc.y += |g f| (g = 1 without gates). resid_fast scales the
// bound with yscale = w_guard[0] = 3 u (1.01) 2^9, the scaled bound the general
// path would have accumulated for K = 1.
template <int K, bool CB16, int UV, bool GATED = false, typename Gate = NoGate>
__device__ __forceinline__ void member_one(const RawVecs<K, CB16, UV>& raw, Acc<UV>& acc, Gate gate = {}) {
    static_assert(K == 1, "a one-entry history");
#pragma unroll
    for (int u = 0; u < UV; ++u) {
        float g[8];
        if constexpr (GATED) gate(u, g);  // first: each feature is then unpacked as it is used
        const uint32_t w[8] = {raw[u][0][0].x, raw[u][0][0].y, raw[u][0][0].z, raw[u][0][0].w,
                               raw[u][0][CB16 ? 0 : 1].x, raw[u][0][CB16 ? 0 : 1].y, raw[u][0][CB16 ? 0 : 1].z,
                               raw[u][0][CB16 ? 0 : 1].w};
#pragma unroll
        for (int e = 0; e < 8; ++e) {
            const float f = CB16 ? __uint_as_float((e & 1) ? (w[e >> 1] & 0xFFFF0000u) : (w[e >> 1] << 16))
                                 : __uint_as_float(w[e]);
            if constexpr (GATED) {
                acc.x[u][e] = fmaf(g[e], f, acc.x[u][e]);
                acc.y[u][e] = fmaf(fabsf(g[e]), fabsf(f), acc.y[u][e]);
            } else {
                acc.x[u][e] += f;
                acc.y[u][e] += fabsf(f);
            }
        }
    }
}

// Fast path: hidden state <- bf16(x + sum_b s_b), guarded like the members.
// xload(u, x) supplies the 8 hidden-state values of vector u (global or shared
// memory); exact(u, e, x_e, hi, lo) recomputes one guarded element with Dot2.
// yscale: factor that turns acc.y into the scaled bound (1 when the members
// accumulated scaled bounds; w_guard[0] after member_one's unscaled sums).
template <int K, int UV, typename XLoad, typename Exact>
__device__ __forceinline__ void resid_fast(const ExtrapArgs& A, int it, const long long (&ev)[UV],
                                           const Acc<UV>& acc, void* resid, XLoad xload, Exact exact,
                                           float yscale = 1.0f) {
    // the test g_res (sum_b a_b + |x|) <= 2^-9 |t|, g_res = (K + nb + 3) u 1.01,
    // on the scaled bounds acc.y = (K+2) u 1.01 2^9 sum_b a_b:
    // q acc.y + r |x| <= |t| with q = (K + nb + 3) / (K + 2), r = g_res 2^9
    const float kn = (float)(K + A.nb[it] + 3);
    const float q = kn * (1.0f / (float)(K + 2)) * 1.0000005f * yscale;  // rounded up past fp32 error
    const float r = kn * (kU * 1.01f * 512.0f);
#pragma unroll
    for (int u = 0; u < UV; ++u) {
        float x[8], t[8];
        uint32_t pk[4];
        xload(u, x);
#pragma unroll
        for (int e = 0; e < 8; ++e) t[e] = acc.x[u][e] + x[e];
#pragma unroll
        for (int i = 0; i < 4; ++i) pk[i] = pack_bf16x2(t[2 * i], t[2 * i + 1]);
        float b[8];
        bool pass = true;
#pragma unroll
        for (int e = 0; e < 8; ++e) {
            b[e] = fmaf(r, fabsf(x[e]), q * acc.y[u][e]);
            pass = pass && guard_ok(b[e], t[e]);
        }
        unsigned bad = 0;
        if (!pass)
#pragma unroll
            for (int e = 0; e < 8; ++e) bad |= guard_ok(b[e], t[e]) ? 0u : (1u << e);
        store_bf16x8(resid, ev[u], pk);
        // rare: Dot2 values stored over the fast-path bf16 just written
        while (bad) {
            const int e = __ffs(bad) - 1;
            bad &= bad - 1;
            float xe = x[0];
#pragma unroll
            for (int i = 1; i < 8; ++i) xe = (e == i) ? x[i] : xe;
            float hi, lo;
            exact(u, e, xe, hi, lo);
            reinterpret_cast<uint16_t*>(resid)[ev[u] + e] = bf16_of_pair(hi, lo);
        }
    }
}

// Unevaluated compensated sums s[q] + c[q] = sum_j w_j F_j of the elements
// 2q, 2q + 1 of one vector.
//
// K <= 2: Dot2 (its first TwoSum adds to zero and is left out). K >= 3: an
// anchored sum. With M >= 2 T, T = sum_j |w_hi[j] F_j|, every S_j =
// fl(w_hi[j] F_j + S_{j-1}), S_{-1} = M, is at least T, so d_j = S_j - S_{j-1},
// at most T, is exact, as is S_{K-1} - M; what the rounding left out, w_hi[j] F_j -
// d_j, is one FMA, a second one adds the weight's low half to it, and c collects
// the sum (the error-free extraction by a large constant of Rump, Ogita & Oishi,
// "Accurate floating-point summation", SIAM J. Sci. Comput. 31(1), 2008, with the
// product folded into the FMA).
//
// Error. With u = 2^-24, S_j <= (3 + small) T, so what is left out is at most
// 3.3 u T each, and the roundings of its FMA, of the second one and of the K - 1
// additions give |s + c - P| <= u^2 T (3.3 (K (K + 1) / 2 - 1) + 6.5 K): 2^-42 T
// for K = 4, 2^-40.6 T for K = 8. Seen, over 2.9e7 sums against quad precision
// (K = 3..8, bf16 and fp32 features, entries of one size and 2^30 apart, weights
// of zero, cancelling terms): at most 2^-43.1 T, Dot2 2^-44.0 T; the fp32 results'
// 2-norm error equals Dot2's to seven digits. An anchor from sum |w_j| times
// max |F_j| is cheaper by an operation per term and no bound in T: a large
// feature under a small weight takes the other terms' low bits (2^-22 T seen).
//
// Cost: seven operations per term of a pair (T is summed in bf16 for bf16 sources)
// against Dot2's eleven: with fp32 results the kernels are bound by the FMA pipe
// and the issue slots. The cheaper anchor measured DiT-XL/2 512^2, K = 8, fp32
// predictions 734 us (737 us here) and K = 4 with gated fp32 hidden states 527 us (528).
// Where M overflows (T >= 2^127) or a feature is not finite, s or c is not
// finite: the callers then take scalar_element, which has no anchor.
//
// Two pairs advance together, term by term (four at once take registers from
// the other warps; one at a time is as fast with five warps per scheduler).
template <int K, bool CB16>
__device__ __forceinline__ void sum_vec(const ExtrapArgs& A, const uint4 (&raw)[K][CB16 ? 1 : 2], float2 (&s)[4],
                                        float2 (&c)[4]) {
    if constexpr (K <= 2) {
#pragma unroll
        for (int j = 0; j < K; ++j) {
            const float2 w = pair_of(A.w_hi[j]), wl = pair_of(A.w_lo[j]);
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const float2 f = vec_pair<CB16>(raw[j], q);
                if (j == 0) {
                    s[q] = mul2(w, f);
                    c[q] = fma2(w, f, mul2(pair_of(-A.w_hi[j]), f));  // exact: w_hi*f - s
                } else {
                    const float2 h = mul2(w, f);
                    float2 e;
                    two_sum2(s[q], h, s[q], e);
                    c[q] = add2(c[q], add2(e, fma2(w, f, mul2(pair_of(-A.w_hi[j]), f))));
                }
                c[q] = fma2(wl, f, c[q]);
            }
        }
    } else {
        float2 anchor[4];
#pragma unroll
        for (int q0 = 0; q0 < 4; q0 += 2) {
#pragma unroll
            for (int q = q0; q < q0 + 2; ++q) {
                if constexpr (CB16) {
                    uint32_t x = 0u;
#pragma unroll
                    for (int j = 0; j < K; ++j) {
                        const uint4 v = raw[j][0];
                        x = fma_bf16x2(A.w_anchor[j], (q == 0 ? v.x : q == 1 ? v.y : q == 2 ? v.z : v.w) & 0x7FFF7FFFu, x);
                    }
                    anchor[q] = make_float2(__uint_as_float(x << 16), __uint_as_float(x & 0xFFFF0000u));
                } else {
                    float2 x = pair_of(0.0f);
#pragma unroll
                    for (int j = 0; j < K; ++j) {
                        const float w = __uint_as_float(A.w_anchor[j]);
                        const float2 f = vec_pair<CB16>(raw[j], q);
                        x = make_float2(fmaf(w, fabsf(f.x), x.x), fmaf(w, fabsf(f.y), x.y));
                    }
                    anchor[q] = x;
                }
                s[q] = anchor[q];
            }
#pragma unroll
            for (int j = 0; j < K; ++j) {
                const float2 w = pair_of(A.w_hi[j]), wl = pair_of(A.w_lo[j]);
#pragma unroll
                for (int q = q0; q < q0 + 2; ++q) {
                    const float2 f = vec_pair<CB16>(raw[j], q);
                    const float2 t = fma2(w, f, s[q]);
                    const float2 r = fma2(wl, f, fma2(w, f, sub2(s[q], t)));
                    c[q] = j == 0 ? r : add2(c[q], r);
                    s[q] = t;
                }
            }
#pragma unroll
            for (int q = q0; q < q0 + 2; ++q) s[q] = sub2(s[q], anchor[q]);
        }
    }
}

// Finiteness of a thread's compensated results: `zero` stays +-0 exactly as
// long as every value given to it is finite.
struct Finite {
    float2 zero = {0.0f, 0.0f};
    __device__ __forceinline__ void see(float2 v) { zero = fma2(v, pair_of(0.0f), zero); }
    __device__ __forceinline__ bool all() const { return zero.x == 0.0f && zero.y == 0.0f; }
};

// Compensated path for one member (any launch with fp32 predictions or hidden
// states): the prediction's output elements to put(u, bf16, o) when wanted (o as
// put_pair leaves it, for vector u), and accumulation into acc.
//
// The output type and what is wanted are asked once per vector, not per pair:
// branches between the pairs kept their chains from overlapping and held 10 to
// 30 registers more (gated fp32 hidden states, DiT-XL/2 512^2: K = 2 520 -> 430 us,
// K = 4 585 -> 528; the off-grid gated step of 24 x [3, 333, 577] 54 -> 48; a full
// step of DiT-XL/2 256^2 with fp32 hidden states and gates 230 -> 198). fp32
// predictions alone, which HBM bounds, are as fast either way (K = 4..8 504, 564,
// 606, 670, 735 -> 492, 570, 586, 670, 736 us).
template <int K, bool CB16, int UV, bool GATED, typename Gate, typename Put>
__device__ __forceinline__ void member_precise(const ExtrapArgs& A, bool want, const RawVecs<K, CB16, UV>& raw,
                                               bool accumulate, Acc<UV>& acc, Finite& fin, Gate gate, Put put) {
#pragma unroll
    for (int u = 0; u < UV; ++u) {
        float2 sv[4], cv[4];
        sum_vec<K, CB16>(A, raw[u], sv, cv);
        float g[8];
        if constexpr (GATED)
            if (accumulate) gate(u, g);
        if (want) {
            uint32_t o[8];
            auto pairs = [&](bool bf16) {
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    float2 hi = add2(sv[q], cv[q]), lo = hi;
                    if (bf16) two_sum2(sv[q], cv[q], hi, lo);
                    put_pair(o, bf16, q, hi, lo);
                    if (K > 2) fin.see(hi);
                }
                put(u, bf16, o);
            };
            if (A.out_bf16) {
                pairs(true);
            } else {
                pairs(false);
            }
        }
        if (accumulate) {
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const float2 s = sv[q], c = cv[q];
                float2 x = make_float2(acc.x[u][2 * q], acc.x[u][2 * q + 1]);
                float2 y = make_float2(acc.y[u][2 * q], acc.y[u][2 * q + 1]), e;
                if constexpr (GATED) {
                    const float2 gq = make_float2(g[2 * q], g[2 * q + 1]);
                    const float2 gs = mul2(gq, s);
                    const float2 gr = fma2(gq, s, make_float2(-gs.x, -gs.y));  // exact: g*s - gs
                    two_sum2(x, gs, x, e);
                    y = fma2(gq, c, add2(y, add2(e, gr)));
                } else {
                    two_sum2(x, s, x, e);
                    y = add2(y, add2(e, c));
                }
                acc.x[u][2 * q] = x.x;
                acc.x[u][2 * q + 1] = x.y;
                acc.y[u][2 * q] = y.x;
                acc.y[u][2 * q + 1] = y.y;
            }
        }
    }
}

// The compensated sums start from the hidden state (xload(u, x), as resid_fast).
template <int UV, typename XLoad>
__device__ __forceinline__ void resid_begin(Acc<UV>& acc, XLoad xload) {
#pragma unroll
    for (int u = 0; u < UV; ++u) {
        xload(u, acc.x[u]);
#pragma unroll
        for (int e = 0; e < 8; ++e) acc.y[u][e] = 0.0f;
    }
}

// Rounds the compensated hidden state to put(u, bf16, o), unless a result was not
// finite (then nothing is stored and the caller recomputes the elements).
template <int K, int UV, typename Put>
__device__ __forceinline__ bool resid_precise(const ExtrapArgs& A, const Acc<UV>& acc, Finite& fin, Put put) {
    float2 hi[UV][4], lo[UV][4];
#pragma unroll
    for (int u = 0; u < UV; ++u) {
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const float2 x = make_float2(acc.x[u][2 * q], acc.x[u][2 * q + 1]);
            const float2 y = make_float2(acc.y[u][2 * q], acc.y[u][2 * q + 1]);
            two_sum2(x, y, hi[u][q], lo[u][q]);
            if (K > 2) fin.see(hi[u][q]);
        }
    }
    if (K > 2 && !fin.all()) return false;
    auto store = [&](bool bf16) {
#pragma unroll
        for (int u = 0; u < UV; ++u) {
            uint32_t o[8];
#pragma unroll
            for (int q = 0; q < 4; ++q) put_pair(o, bf16, q, hi[u][q], lo[u][q]);
            put(u, bf16, o);
        }
    };
    if (A.resid_bf16)
        store(true);
    else
        store(false);
    return true;
}

// n / d for n, d < 2^32 from M = ceil(2^64 / d) (M = 0 encodes d = 1):
// n M / 2^64 = n / d + n delta / (d 2^64) with 0 <= delta < d, and the excess
// n delta / (d 2^64) < 2^-32 < 1 / d cannot carry frac(n / d) <= (d - 1) / d
// past the next integer (division by invariant integers, after Granlund &
// Montgomery, PLDI 1994).
__device__ __forceinline__ unsigned div_magic(unsigned n, unsigned long long M) {
    return M ? (unsigned)__umul64hi((unsigned long long)n, M) : n;
}

// Gate offsets b * hidden + h of UV vectors of a tile starting at element e0
// (32-bit arithmetic: gated tensors have fewer than 2^32 elements); with
// `relative`, b counts from the tile's first batch (the staged gate rows).
// Rows of tokens * hidden are multiples of hidden, so h = e mod hidden.
template <int UV>
__device__ __forceinline__ void gate_offsets(const ExtrapArgs& A, int it, long long e0,
                                             const long long (&ev)[UV], unsigned (&gi)[UV], bool relative = false) {
    const unsigned row = A.i_row[it], H = A.i_hidden[it], ue0 = (unsigned)e0;
    if (row == 0 || H == 0) {  // no shape: no gate
#pragma unroll
        for (int u = 0; u < UV; ++u) gi[u] = 0;
        return;
    }
    // what the tile's first element fixes is the same for every thread; a
    // thread's own channel is (h0 + d) mod H for its offset d in the tile. With
    // m = ceil(2^32 / H), x < 2^32 / H has x / H = x m / 2^32 exactly (as in
    // div_magic), and wider rows than that hold a tile, so that x < 2 H.
    const unsigned q0 = div_magic(ue0, A.i_row_magic[it]), r0 = ue0 - q0 * row;
    const unsigned h0 = r0 - div_magic(r0, A.i_hidden_magic[it]) * H;
    const unsigned m32 = (unsigned)((A.i_hidden_magic[it] + 0xFFFFFFFFull) >> 32);
#pragma unroll
    for (int u = 0; u < UV; ++u) {
        const unsigned d = (unsigned)(ev[u] - e0), x = h0 + d;
        unsigned h;
        if (H > 16384u)
            h = x >= H ? x - H : x;
        else
            h = m32 ? x - __umulhi(x, m32) * H : 0u;
        unsigned r = r0 + d, b = relative ? 0u : q0;
        while (r >= row) {  // a tile spans few rows
            r -= row;
            ++b;
        }
        gi[u] = b * H + h;
    }
}

// Gate offset g0 of element e (32-bit, as above), of an item with a shape; that
// of e + 1 is g0 + 1, less the hidden size where it begins the batch's next
// token (`back`).
__device__ __forceinline__ void gate_offset_pair(const ExtrapArgs& A, int it, long long e, unsigned& g0, bool& back) {
    const unsigned row = A.i_row[it], H = A.i_hidden[it], ue = (unsigned)e;
    const unsigned b = div_magic(ue, A.i_row_magic[it]), r = ue - b * row;
    const unsigned h = r - div_magic(r, A.i_hidden_magic[it]) * H;
    g0 = b * H + h;
    back = h + 1 == H && r + 1 < row;
}

// The 8 gate values of member mi for each of UV vectors (1 without a gate).
template <int UV>
__device__ __forceinline__ void load_gates(const ExtrapArgs& A, int mi, const unsigned (&gi)[UV], float (&g)[UV][8]) {
    const void* gp = A.m_gate[mi];
#pragma unroll
    for (int u = 0; u < UV; ++u) {
        if (gp)
            load_x8(gp, A.gate_bf16, (long long)gi[u], g[u]);
        else
#pragma unroll
            for (int e = 0; e < 8; ++e) g[u][e] = 1.0f;
    }
}

}  // namespace
}  // namespace cbk
