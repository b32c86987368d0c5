// forces.cuh -- the ForceAtlas2 arithmetic of one body or node (Section 3.1;
// the force model of Jacomy et al. 2014), shared by the kernels that run over
// the whole GPU (fa2.cu) and the ones that keep a small graph in shared memory
// (small.cuh): both give the same bits.
#pragma once

#include "bgv_internal.cuh"

namespace bgv {
namespace {

typedef unsigned __int128 u128;

__device__ __forceinline__ unsigned long long spread_bits(uint32_t v) {
    unsigned long long x = v;
    x = (x | (x << 16)) & 0x0000FFFF0000FFFFull;
    x = (x | (x << 8)) & 0x00FF00FF00FF00FFull;
    x = (x | (x << 4)) & 0x0F0F0F0F0F0F0F0Full;
    x = (x | (x << 2)) & 0x3333333333333333ull;
    x = (x | (x << 1)) & 0x5555555555555555ull;
    return x;
}

// ----------------------------------------------------------------- frame
// Frame of a bounding box: origin, side = max extent * (1 + 2^-20).
__device__ __forceinline__ float4 frame_of(float lx, float ly, float hx, float hy) {
    const float ex = __fsub_rn(hx, lx), ey = __fsub_rn(hy, ly);
    const float ext = ex > ey ? ex : ey;
    float side = __fmul_rn(ext, 1.00000095367431640625f);  // 1 + 2^-20
    if (!(ext > 0.0f)) side = 1.0f;
    return make_float4(lx, ly, side, 0.0f);
}

__device__ __forceinline__ float4 box_empty() { return make_float4(INFINITY, INFINITY, -INFINITY, -INFINITY); }
__device__ __forceinline__ void box_add(float4 &b, float2 p) {
    b.x = fminf(b.x, p.x); b.y = fminf(b.y, p.y);
    b.z = fmaxf(b.z, p.x); b.w = fmaxf(b.w, p.y);
}
__device__ __forceinline__ void box_merge(float4 &b, const float4 &o) {
    b.x = fminf(b.x, o.x); b.y = fminf(b.y, o.y);
    b.z = fmaxf(b.z, o.z); b.w = fmaxf(b.w, o.w);
}
__device__ __forceinline__ void box_warp(float4 &b) {
#pragma unroll
    for (int d = 16; d > 0; d >>= 1)
        box_merge(b, make_float4(__shfl_xor_sync(0xFFFFFFFFu, b.x, d), __shfl_xor_sync(0xFFFFFFFFu, b.y, d),
                                 __shfl_xor_sync(0xFFFFFFFFu, b.z, d), __shfl_xor_sync(0xFFFFFFFFu, b.w, d)));
}
// -------------------------------------------------------------- repulsion
// One body's Barnes-Hut walk without a stack over a pre-order array.  At
// element `cur` (a cell or a body) it accepts the element -- sums its monopole
// and moves to skip[cur], past its subtree -- or enters it (cur + 1).  A body is
// always accepted except the walker's own (its side^2 is -1); a cell holding the
// body is always entered; any other cell is accepted by the FP32 opening test
// of the definition.
template <class Skip>
__device__ __forceinline__ float2 bh_walk(const float4 *geo, const Skip *skip, float4 bi,
                                          float kmi, float theta2, uint32_t self, uint32_t cur, uint32_t end,
                                          unsigned &inter) {
    float fx = 0.0f, fy = 0.0f;
    while (cur < end) {
        const float4 e = geo[cur];
        const uint32_t sk = uint32_t(skip[cur]);
        const float dx = __fsub_rn(bi.x, e.x), dy = __fsub_rn(bi.y, e.y);
        const float d2 = __fadd_rn(__fmul_rn(dx, dx), __fmul_rn(dy, dy));
        // accepted: not an element holding the body (cur <= self < sk) and
        // the opening test passes; no branch, so lanes stay converged
        const bool accept = self - cur >= sk - cur && e.w < __fmul_rn(theta2, d2);
        const float f = accept && d2 > 0.0f ? __fdividef(kmi * e.z, d2) : 0.0f;
        fx += f * dx;
        fy += f * dy;
        inter += accept ? 1u : 0u;
        cur = accept ? sk : cur + 1;
    }
    return make_float2(fx, fy);
}

// ------------------------------------------------------------ attraction
// Rows of more than att_short and up to this many entries are summed by one
// warp, longer ones by a block.
constexpr int kAttMedium = 4096;
__device__ __forceinline__ bool valid_row(int32_t j, int64_t K) {
    return static_cast<uint64_t>(int64_t(j)) < static_cast<uint64_t>(K);  // an invalid entry adds nothing
}

// --------------------------------------------- node forces, swing, speed
// Global swing and traction (the sums that set the adaptive speed):
// S = sum m_i swing_i and T = sum m_i traction_i over FP32 per-node products,
// which are non-negative.  They are summed EXACTLY: each product f * 2^q
// (f its 24-bit significand) is added as a fixed-point integer into a
// 128-bit accumulator V whose unit 2^q0 sits kXHead binary places below the
// largest term seen so far (q0 moves up, with V shifted down, when a larger
// term arrives).  A term below the unit loses only its bits under 2^q0, less
// than 2^-95 of the largest term, so the accumulated value equals the exact
// sum to about 2^-64 relative even over 2^31 terms; integer addition does not
// depend on the order of the merges.  The total is rounded once to FP64, so S
// and T are the correctly rounded sums of the products (Kahan or Neumaier
// compensation in FP64 would leave about two units in the last place, and
// FP64 arithmetic runs at a small fraction of the integer rate on this GPU).
constexpr int kXHead = 72;          // each term < 2^(24 + 72): 2^31 terms fit in 127 bits
constexpr int kXNoAnchor = -100000; // anchor of an empty accumulator
struct XSum {
    u128 V;
    int q0;
    int bad;  // 1: an infinite term, 2: a NaN term
};
__device__ __forceinline__ XSum xsum_zero() { return XSum{0, kXNoAnchor, 0}; }

__device__ __forceinline__ void xsum_add(XSum &a, float x) {
    const uint32_t b = __float_as_uint(x) & 0x7FFFFFFFu;  // terms are >= 0 (a -0 adds nothing)
    const int e = int(b >> 23);
    if (e == 255) {
        a.bad |= (b & 0x7FFFFFu) ? 2 : 1;
        return;
    }
    const uint32_t f = e ? ((b & 0x7FFFFFu) | 0x800000u) : b;
    const int q = (e ? e : 1) - 150;  // x = f * 2^q
    if (f == 0u) return;
    if (q - kXHead > a.q0) {  // a new largest term: move the anchor up
        const int d = q - kXHead - a.q0;
        a.V = d >= 128 ? u128(0) : (a.V >> d);
        a.q0 = q - kXHead;
    }
    const int sh = q - a.q0;  // <= kXHead
    if (sh >= 0)
        a.V += u128(f) << sh;
    else if (sh > -24)
        a.V += u128(f >> -sh);
}

__device__ __forceinline__ XSum xsum_merge(XSum a, XSum b) {
    if (b.q0 > a.q0) {
        const XSum t = a;
        a = b;
        b = t;
    }
    const int d = a.q0 - b.q0;
    if (d < 128) a.V += b.V >> d;
    a.bad |= b.bad;
    return a;
}

__device__ __forceinline__ XSum xsum_shfl_down(const XSum &a, int d) {
    XSum r;
    r.V = (u128(__shfl_down_sync(0xFFFFFFFFu, static_cast<unsigned long long>(a.V >> 64), d)) << 64) |
          __shfl_down_sync(0xFFFFFFFFu, static_cast<unsigned long long>(a.V), d);
    r.q0 = __shfl_down_sync(0xFFFFFFFFu, a.q0, d);
    r.bad = __shfl_down_sync(0xFFFFFFFFu, a.bad, d);
    return r;
}

// The accumulated value rounded once to FP64 (round to nearest even): the top
// 64 bits of V, with a sticky bit for the rest, converted, then scaled.
__device__ __forceinline__ double xsum_value(const XSum &a) {
    if (a.bad) return (a.bad & 2) ? __longlong_as_double(0x7FF8000000000000ll) : __longlong_as_double(0x7FF0000000000000ll);
    const unsigned long long hi = static_cast<unsigned long long>(a.V >> 64);
    if (!hi) return ldexp(__ull2double_rn(static_cast<unsigned long long>(a.V)), a.q0);
    const int sh = 64 - __clzll(static_cast<long long>(hi));  // bits of V above its top 64
    unsigned long long t = static_cast<unsigned long long>(a.V >> sh);
    if (a.V & ((u128(1) << sh) - 1)) t |= 1ull;  // sticky: far below the rounding position
    return ldexp(__ull2double_rn(t), a.q0 + sh);
}

// Stored form of one accumulator (per-block partials).
struct XPart {
    unsigned long long lo, hi;
    int q0, bad;
};
__device__ __forceinline__ XPart xsum_pack(const XSum &a) {
    return XPart{static_cast<unsigned long long>(a.V), static_cast<unsigned long long>(a.V >> 64), a.q0, a.bad};
}
__device__ __forceinline__ XSum xsum_unpack(const XPart *p) {  // from L2: written by other blocks
    const unsigned long long lo = __ldcg(&p->lo), hi = __ldcg(&p->hi);
    return XSum{(u128(hi) << 64) | lo, __ldcg(&p->q0), __ldcg(&p->bad)};
}

// Merge of one (S, T) pair per lane; lane 0 receives the result.
__device__ __forceinline__ void xsum_warp(XSum &S, XSum &T) {
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) {
        const XSum oS = xsum_shfl_down(S, d), oT = xsum_shfl_down(T, d);
        S = xsum_merge(S, oS);
        T = xsum_merge(T, oT);
    }
}

// The sum of one value below 2^104 per lane, in every lane: 26 bits per reduction.
__device__ __forceinline__ u128 warp_sum_u104(u128 v) {
    u128 sum = 0;
#pragma unroll
    for (int k = 0; k < 4; ++k)
        sum += u128(__reduce_add_sync(0xFFFFFFFFu, uint32_t(v >> (26 * k)) & 0x3FFFFFFu)) << (26 * k);
    return sum;
}
// The sum of one term per lane, in every lane: at the scale of the largest term
// they are integers below 2^96, so the whole warp takes six reductions.
__device__ __forceinline__ XSum xsum_warp_terms(float x) {
    const uint32_t b = __float_as_uint(x) & 0x7FFFFFFFu;
    const int e = int(b >> 23);
    const int bad = int(__reduce_or_sync(0xFFFFFFFFu, e == 255 ? (b & 0x7FFFFFu ? 2u : 1u) : 0u));
    const uint32_t f = e == 255 ? 0u : e ? ((b & 0x7FFFFFu) | 0x800000u) : b;
    const int q = (e ? e : 1) - 150;
    const int top = __reduce_max_sync(0xFFFFFFFFu, f ? q : -1000);
    if (top == -1000) return XSum{0, kXNoAnchor, bad};
    const int q0 = top - kXHead, sh = q - q0;
    return XSum{warp_sum_u104(sh >= 0 ? u128(f) << (f ? sh : 0) : sh > -24 ? u128(f >> -sh) : u128(0)), q0, bad};
}
// The merge of two accumulators of at most 2^6 terms per lane, in every lane.
__device__ __forceinline__ XSum xsum_warp_merge(const XSum &a, const XSum &b) {
    const int q0 = __reduce_max_sync(0xFFFFFFFFu, a.q0 > b.q0 ? a.q0 : b.q0);
    const int bad = int(__reduce_or_sync(0xFFFFFFFFu, uint32_t(a.bad | b.bad)));
    const u128 va = q0 - a.q0 < 128 ? a.V >> (q0 - a.q0) : u128(0), vb = q0 - b.q0 < 128 ? b.V >> (q0 - b.q0) : u128(0);
    return XSum{warp_sum_u104(va + vb), q0, bad};
}

// Block-wide merge of one (S, T) pair per thread; thread 0 receives the result.
template <int kBlock>
__device__ __forceinline__ void xsum_block(XSum &S, XSum &T) {
    constexpr int kWarps = kBlock / 32;
    __shared__ XPart part[2][kWarps];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    xsum_warp(S, T);
    if (lane == 0) {
        part[0][warp] = xsum_pack(S);
        part[1][warp] = xsum_pack(T);
    }
    __syncthreads();
    if (warp == 0) {
        auto get = [&](int k) {
            const XPart &x = part[k][lane];
            return lane < kWarps ? XSum{(u128(x.hi) << 64) | x.lo, x.q0, x.bad} : xsum_zero();
        };
        S = get(0);
        T = get(1);
#pragma unroll
        for (int d = kWarps / 2; d > 0; d >>= 1) {
            const XSum oS = xsum_shfl_down(S, d), oT = xsum_shfl_down(T, d);
            S = xsum_merge(S, oS);
            T = xsum_merge(T, oT);
        }
    }
    __syncthreads();
}

__device__ __forceinline__ double speed_update(double sp, double Ssum, double Tsum, float tau) {
    if (Ssum > 0.0) {
        const double target = double(tau) * Tsum / Ssum;
        const double rise = target - sp, cap = 0.5 * sp;
        sp += rise < cap ? rise : cap;
    }
    return sp;
}

// Per-node swing and traction products, FP32 with every rounding explicit
// (no contraction), so they can be recomputed bit for bit from F, Fprev and
// the mass: m |F - Fprev| and (m / 2) |F + Fprev|.
__device__ __forceinline__ float2 swing_traction(float m, float fx, float fy, float px, float py) {
    const float sx = __fsub_rn(fx, px), sy = __fsub_rn(fy, py), tx = __fadd_rn(fx, px), ty = __fadd_rn(fy, py);
    const float sw = sqrtf(__fadd_rn(__fmul_rn(sx, sx), __fmul_rn(sy, sy)));
    const float tr = sqrtf(__fadd_rn(__fmul_rn(tx, tx), __fmul_rn(ty, ty)));
    return make_float2(__fmul_rn(m, sw), __fmul_rn(__fmul_rn(0.5f, m), tr));
}

// x^2 + y^2 with its one fused step named, so that every kernel rounds alike.
__device__ __forceinline__ float norm2(float x, float y) { return __fmaf_rn(x, x, __fmul_rn(y, y)); }

__device__ __forceinline__ float2 force_sum(float2 fa, float m, float2 pi, float2 fr, float kg, int strong) {
    float gx, gy;
    if (strong) {
        gx = -kg * m * pi.x;
        gy = -kg * m * pi.y;
    } else {
        const float rr = sqrtf(norm2(pi.x, pi.y));
        gx = rr > 0.0f ? -kg * m * pi.x / rr : 0.0f;
        gy = rr > 0.0f ? -kg * m * pi.y / rr : 0.0f;
    }
    return make_float2(fr.x + fa.x + gx, fr.y + fa.y + gy);
}

// Total force on node i: repulsion fr, attraction full[i] (none if null),
// gravity.
__device__ __forceinline__ float2 node_force(int64_t i, const float2 *__restrict__ full, float m, float2 pi, float2 fr,
                                             float kg, int strong) {
    return force_sum(full ? full[i] : make_float2(0.0f, 0.0f), m, pi, fr, kg, strong);
}

__device__ __forceinline__ float2 displaced(float2 p, float2 f, float2 fp, float sp, float ks, float ksmax) {
    const float sx = f.x - fp.x, sy = f.y - fp.y;
    const float swing = sqrtf(norm2(sx, sy));
    float s = ks * sp / __fmaf_rn(sp, sqrtf(swing), 1.0f);
    const float fn = sqrtf(norm2(f.x, f.y));
    if (fn > 0.0f && s * fn > ksmax) s = ksmax / fn;
    p.x = __fmaf_rn(s, f.x, p.x);
    p.y = __fmaf_rn(s, f.y, p.y);
    return p;
}

}  // namespace
}  // namespace bgv
