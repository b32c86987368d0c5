// tree.cuh -- the Barnes-Hut quadtree over the Morton-sorted bodies, laid out
// in depth-first pre-order for the traversal (three kernels, no tree search).
//
// A cell of the quadtree (with chains of single-child cells collapsed into the
// deepest) is a maximal interval of sorted bodies whose neighbouring keys agree
// down to at least some level, with equality somewhere.  With D[i] = the level
// down to which the keys of bodies i - 1 and i agree, stored plus one (0: another
// graph, or past either end), the boundary j inside it with D[j] = v is the first
// of its smallest ones: the nearest boundary before j with D <= v has D < v and
// starts the cell, and the nearest after j with D < v ends it.  So every
// boundary asks for itself, with two short searches, whether it stands for a
// cell and for which; a tile of bodies finds nearly all of its cells in shared
// memory (a bit row per level, LevelBits).  (Walking all the cells
// that start at a body instead left most lanes waiting for the one with the
// longest chain: 207 us for k_tile at 3.2 M bodies.)
//   k_tile       gathers the bodies of a tile in Morton order, their levels D
//                and moment prefixes; finds the tile's cells, their centres from
//                exact integer moments, and what the others need: for every
//                level the first boundary below it, and the cells still open at
//                the tile's end (at most one per level); moment totals before
//                the tile by a decoupled look-back
//   k_tile_cross closes the open cells, a warp per tile: the first later tile
//                with a boundary below the level, by the tiles' minima; the last
//                block sums the cells of the tiles before each
//   k_tile_emit  pre-order positions of the tile's bodies and cells
// A radix-tree form with one thread per binary node took 335 us at 3.2 M bodies
// (gather and moment scan 110, candidates 21, range searches 143, scan 19, layout
// 42).  500 steps at 1 M bodies and 16 M CSR entries: 224.6 ms with it, 211.2 with
// the tiles.
// k_tile is bound by instruction issue.  Searching the bytes of D, four per
// comparison and 64 per skip, it took 34 warp instructions a body with 18 lanes
// active, as a warp waits for its longest search; with the bit rows (about one
// ballot and one store per level and 32 bodies, then two words per search) 500
// steps of 1 M bodies fell from 188.7 to 177.5 ms and 300 steps of 160 graphs
// (6.0 M bodies) from 484.4 to 456.6 ms.  Before that, moments of light bodies in 32 and 64 bits,
// with the centre's division by an estimate: 190.0 -> 188.7 and 488.5 -> 484.4 ms.
#pragma once

#include <type_traits>

#include "bgv_internal.cuh"

namespace bgv {
namespace {

typedef unsigned __int128 u128;

// Exact power-of-two scale 2^-level for 0 <= level <= 126.
__device__ __forceinline__ float pow2_neg(int level) { return __int_as_float((127 - level) << 23); }

// Fixed-point position of a body in its graph's frame: U = floor(2^32 (p -
// origin) / side) per axis, FP32 with round-to-nearest steps.
__device__ __forceinline__ uint2 fixed_point(float2 p, float4 fr) {
    const float ux = __fdiv_rn(__fsub_rn(p.x, fr.x), fr.z);
    const float uy = __fdiv_rn(__fsub_rn(p.y, fr.y), fr.z);
    return make_uint2(__float2uint_rz(__fmul_rn(ux, 4294967296.0f)), __float2uint_rz(__fmul_rn(uy, 4294967296.0f)));
}

// Exact moments (m, m Ux, m Uy) in 64/128-bit integers, so sums do not depend
// on their order.
struct Mom {
    unsigned long long M;
    u128 X, Y;
};
__device__ __forceinline__ Mom mom_zero() { return Mom{0ull, 0, 0}; }
__device__ __forceinline__ Mom mom_add(Mom a, const Mom &b) {
    a.M += b.M;
    a.X += b.X;
    a.Y += b.Y;
    return a;
}
__device__ __forceinline__ Mom mom_sub(Mom a, const Mom &b) {
    a.M -= b.M;
    a.X -= b.X;
    a.Y -= b.Y;
    return a;
}
__device__ __forceinline__ Mom mom_body(uint32_t m, uint32_t ux, uint32_t uy) {
    return Mom{m, static_cast<unsigned long long>(m) * ux, static_cast<unsigned long long>(m) * uy};
}
__device__ __forceinline__ Mom mom_shfl_up(const Mom &a, int d) {
    Mom r;
    r.M = __shfl_up_sync(0xFFFFFFFFu, a.M, d);
    const unsigned long long xl = __shfl_up_sync(0xFFFFFFFFu, static_cast<unsigned long long>(a.X), d);
    const unsigned long long xh = __shfl_up_sync(0xFFFFFFFFu, static_cast<unsigned long long>(a.X >> 64), d);
    const unsigned long long yl = __shfl_up_sync(0xFFFFFFFFu, static_cast<unsigned long long>(a.Y), d);
    const unsigned long long yh = __shfl_up_sync(0xFFFFFFFFu, static_cast<unsigned long long>(a.Y >> 64), d);
    r.X = (u128(xh) << 64) | xl;
    r.Y = (u128(yh) << 64) | yl;
    return r;
}

// One moment record in 32 bytes (one sector): M in 64 bits, the coordinate
// sums in 96 (their totals stay below 2^95).
struct __align__(32) MomP {
    uint4 a, b;
};
__device__ __forceinline__ void momp_store(MomP *p, const Mom &v) {
    p->a = make_uint4(uint32_t(v.M), uint32_t(v.M >> 32), uint32_t(v.X), uint32_t(v.X >> 32));
    p->b = make_uint4(uint32_t(v.Y), uint32_t(v.Y >> 32), uint32_t(v.X >> 64), uint32_t(v.Y >> 64));
}
__device__ __forceinline__ Mom momp_load(const MomP *p) {
    const uint4 a = p->a, b = p->b;
    const unsigned long long xl = (static_cast<unsigned long long>(a.w) << 32) | a.z;
    const unsigned long long yl = (static_cast<unsigned long long>(b.y) << 32) | b.x;
    return Mom{(static_cast<unsigned long long>(a.y) << 32) | a.x, (u128(b.z) << 64) | xl, (u128(b.w) << 64) | yl};
}
__device__ __forceinline__ Mom momp_load_cg(const MomP *p) {  // from L2: written by other blocks of this kernel
    MomP q;
    q.a = __ldcg(&p->a);
    q.b = __ldcg(&p->b);
    return momp_load(&q);
}

constexpr int kTileThreads = 256;
constexpr int kTileItems = 4;
constexpr int kTile = kTileThreads * kTileItems;  // bodies per tile
constexpr int kTileLevels = 26;                   // values of D: 0 .. max_depth + 1
constexpr int kTileGroup = 64;                    // tiles per group minimum
enum : uint32_t { kMomAgg = 1u, kMomIncl = 2u };  // look-back flags (0: nothing published)
constexpr int kMomLBItems = 4;                           // predecessors per thread and round
constexpr int kMomLookBack = kTileThreads * kMomLBItems;  // predecessors per round

inline int64_t tile_count(int64_t K) { return (K + kTile - 1) / kTile; }
inline int64_t tile_groups(int64_t K) { return (tile_count(K) + kTileGroup - 1) / kTileGroup; }

// What the tiles leave for each other (device arrays).
struct TileArrays {
    uint32_t *flags;     // [tiles] look-back flags, [tiles] tile counter, [tiles + 1] ticket, then per group of tiles
                         // 31 - its smallest D; all zero before k_tile
    MomP *agg, *incl;    // [tiles] moment totals: of the tile, of all up to it
    uint8_t *tmin;       // [tiles, padded to 16] smallest D of the tile's boundaries
    uint32_t *first;     // [tiles][levels] first boundary with D < v: place (11 bits) | its D << 11 | cells that
                         // start before it in the tile << 16; place 0: none
    MomP *first_mom;     // [tiles][levels] moments of the tile's bodies before that boundary
    uint32_t *open_n;    // [tiles] cells open at the tile's end
    uint32_t *open;      // [tiles][levels] first body (10 bits) | level << 10 | the first body's D << 15
    MomP *open_mom;      // [tiles][levels] moments of the tile's bodies before the first body
    uint32_t *open_cells;  // [tiles][levels] cells closed from that entry
    uint32_t *cells;     // [tiles] cells inside the tile
    uint32_t *base;      // [tiles + 1] cells that start before the tile
    uint8_t *starts;     // [K] cells inside the tile that start at the body
    float4 *cell;        // [K] per tile: centre, mass, side^2 of its cells
    uint32_t *meta;      // [K] per tile: first body (10 bits) | last << 10 | outer cells from it inside the tile << 20
    uint32_t *cross_mask;  // [tiles] levels of the cells that leave the tile
    float4 *cross;       // [tiles][levels] their centre, mass, side^2
    uint2 *cross_meta;   // [tiles][levels] first body | inner ones of these cells from it << 10, last body (of all)
};
inline int64_t tile_flag_words(int64_t K) { return tile_count(K) + 2 + tile_groups(K); }
inline void carve_tiles(Carver &c, int64_t K, TileArrays &t) {
    const size_t n = size_t(tile_count(K)), k = size_t(K);
    t.flags = c.take<uint32_t>(size_t(tile_flag_words(K)));
    t.agg = c.take<MomP>(n);
    t.incl = c.take<MomP>(n);
    t.tmin = c.take<uint8_t>((n + 15) / 16 * 16);
    t.first = c.take<uint32_t>(n * kTileLevels);
    t.first_mom = c.take<MomP>(n * kTileLevels);
    t.open_n = c.take<uint32_t>(n);
    t.open = c.take<uint32_t>(n * kTileLevels);
    t.open_mom = c.take<MomP>(n * kTileLevels);
    t.open_cells = c.take<uint32_t>(n * kTileLevels);
    t.cells = c.take<uint32_t>(n);
    t.base = c.take<uint32_t>(n + 1);
    t.starts = c.take<uint8_t>((k + 3) / 4 * 4);
    t.cell = c.take<float4>(k);
    t.meta = c.take<uint32_t>(k);
    t.cross_mask = c.take<uint32_t>(n);
    t.cross = c.take<float4>(n * kTileLevels);
    t.cross_meta = c.take<uint2>(n * kTileLevels);
}

// floor(X / M) when it is below 2^32: an FP32 estimate (relative error below
// 2^-21, so off by at most 2^11), corrected by its exact remainder, and once more
// by one.
__device__ __forceinline__ uint32_t mean_u32(unsigned long long X, uint32_t M) {
    const float r = __frcp_rn(__uint2float_rn(M));
    uint32_t q = __float2uint_rz(__fmul_rn(__ull2float_rn(X), r));  // saturates
    long long R = static_cast<long long>(X - static_cast<unsigned long long>(q) * M);
    const int dq = __float2int_rd(__fmul_rn(__ll2float_rn(R), r));
    q += uint32_t(dq);
    R -= static_cast<long long>(dq) * static_cast<long long>(static_cast<unsigned long long>(M));
    if (R < 0) --q;
    if (R >= static_cast<long long>(static_cast<unsigned long long>(M))) ++q;
    return q;
}

// The same for moments of any width (X < 2^32 M, M < 2^63): the remainder of the
// estimate is at most 2^12 M, and that of its correction a few M.  (A 128-bit
// division is a loop of hundreds of instructions; the cells across tiles are few,
// and wait for it.)
__device__ __forceinline__ float u128_to_float(u128 x) {
    return __fmaf_rn(__ull2float_rn(static_cast<unsigned long long>(x >> 64)), 18446744073709551616.0f,
                     __ull2float_rn(static_cast<unsigned long long>(x)));
}
__device__ __forceinline__ uint32_t mean_wide(u128 X, unsigned long long M) {
    const float r = __frcp_rn(__ull2float_rn(M));
    uint32_t q = __float2uint_rz(__fmul_rn(u128_to_float(X), r));  // saturates
    __int128 R = static_cast<__int128>(X - u128(q) * M);
    const bool over = R < 0;
    const uint32_t dq = __float2uint_rz(__fmul_rn(u128_to_float(over ? u128(0) - u128(R) : u128(R)), r));
    const __int128 by = static_cast<__int128>(u128(dq) * M);
    q = over ? q - dq : q + dq;
    R = over ? R + by : R - by;
    while (R < 0) {
        --q;
        R += M;
    }
    while (R >= static_cast<__int128>(u128(M))) {
        ++q;
        R -= M;
    }
    return q;
}

// The element of one cell: FP32 centre from the exact moments, mass, and the
// squared side of the opening test (+inf for a leaf that is never accepted).
// v, pv: its level and its parent's, plus one; n bodies.
// qx, qy: the centre in fixed point; Mf: the mass.
__device__ __forceinline__ float4 cell_element(uint32_t qx, uint32_t qy, float Mf, int v, int pv, int64_t n, int L,
                                               int leaf_cap, float4 fr) {
    const int lev = v - 1, par_lev = pv - 1;
    const bool leaf = n <= leaf_cap || lev >= L;
    // A leaf made by the depth limit (coincident keys, more than leaf_cap
    // bodies) hides a chain of non-leaf cells with the same bodies between its
    // parent's level and L; the deepest of them, at level L - 1, takes the
    // opening test for the whole chain.
    const bool testable = leaf && n > leaf_cap && par_lev + 1 <= L - 1;
    const float two_m32 = 2.3283064365386963e-10f;  // 2^-32
    const float cx = __fadd_rn(fr.x, __fmul_rn(fr.z, __fmul_rn(__uint2float_rn(qx), two_m32)));
    const float cy = __fadd_rn(fr.y, __fmul_rn(fr.z, __fmul_rn(__uint2float_rn(qy), two_m32)));
    const float sl = __fmul_rn(fr.z, pow2_neg(testable ? L - 1 : lev));
    const float side2 = (leaf && !testable) ? INFINITY : __fmul_rn(sl, sl);
    return make_float4(cx, cy, Mf, side2);
}
__device__ __forceinline__ float4 cell_element(const Mom &mom, int v, int pv, int64_t n, int L, int leaf_cap, float4 fr) {
    uint32_t qx = 0u, qy = 0u;
    if (mom.M) {
        qx = mean_wide(mom.X, mom.M);
        qy = mean_wide(mom.Y, mom.M);
    }
    return cell_element(qx, qy, __ull2float_rn(mom.M), v, pv, n, L, leaf_cap, fr);
}

// Bodies lighter than this: the moments of kSmallMax or kTile of them fit in 32
// (mass) and 64 bits (coordinates), a third of the work of the full width.
constexpr uint32_t kLightMass = 1u << 21;
struct Mom64 {
    uint32_t M;
    unsigned long long X, Y;
};
__device__ __forceinline__ Mom64 mom64_add(Mom64 a, uint32_t m, uint32_t ux, uint32_t uy) {
    a.M += m;
    a.X += static_cast<unsigned long long>(m) * ux;
    a.Y += static_cast<unsigned long long>(m) * uy;
    return a;
}
// A prefix stored by momp_store whose values fit.
__device__ __forceinline__ Mom64 mom64_load(const MomP *p) {
    const uint4 a = p->a;
    const uint2 b = *reinterpret_cast<const uint2 *>(&p->b);
    return Mom64{a.x, (static_cast<unsigned long long>(a.w) << 32) | a.z, (static_cast<unsigned long long>(b.y) << 32) | b.x};
}
__device__ __forceinline__ float4 cell_element(const Mom64 &lo, const Mom64 &hi, int v, int pv, int n, int L,
                                               int leaf_cap, float4 fr) {
    const uint32_t M = hi.M - lo.M;
    return cell_element(M ? mean_u32(hi.X - lo.X, M) : 0u, M ? mean_u32(hi.Y - lo.Y, M) : 0u, __uint2float_rn(M), v, pv,
                        n, L, leaf_cap, fr);
}
// Inclusive warp scan.
__device__ __forceinline__ Mom64 mom64_warp_scan(Mom64 a) {
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const uint32_t M = __shfl_up_sync(0xFFFFFFFFu, a.M, d);
        const unsigned long long X = __shfl_up_sync(0xFFFFFFFFu, a.X, d), Y = __shfl_up_sync(0xFFFFFFFFu, a.Y, d);
        if (lane >= d) {
            a.M += M;
            a.X += X;
            a.Y += Y;
        }
    }
    return a;
}
__device__ __forceinline__ Mom mom_warp_scan(Mom a) {
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const Mom o = mom_shfl_up(a, d);
        if (lane >= d) a = mom_add(a, o);
    }
    return a;
}

// Level down to which two keys agree, plus one (the graph bits come first).
__device__ __forceinline__ uint32_t level_between(unsigned long long a, unsigned long long b, int L, int gbits) {
    if (a == b) return uint32_t(L) + 1u;
    const int delta = __clzll(static_cast<long long>(a ^ b)) - (64 - 2 * L - gbits);
    return delta < gbits ? 0u : uint32_t((delta - gbits) >> 1) + 1u;
}

// Where D <= v, a bit per place, for every level v between the least and the
// greatest of a tile: a row of kWords words per level (kept kWords + 1 apart, as
// neighbouring threads ask different rows for the same word) and a word that
// tells which of them are not zero.  The nearest place before or after another
// takes at most two words, however far it is.
template <int kWords>
struct LevelBits {
    using Some = typename std::conditional<kWords == 32, uint32_t, unsigned long long>::type;
    uint32_t row[32][kWords + 1];
    // Every thread of a warp, with the value of its place of word w; lo <= hi, at most 32 levels.
    __device__ __forceinline__ void add(uint32_t d, int w, uint32_t lo, uint32_t hi, uint32_t *some) {
        const uint32_t lane = threadIdx.x & 31;
        uint32_t keep = 0u;
        for (uint32_t v = lo; v <= hi; ++v) {
            const uint32_t x = __ballot_sync(0xFFFFFFFFu, d <= v);
            if (lane == v - lo) keep = x;
        }
        if (lane <= hi - lo) row[lane][w] = keep;
        if (keep) atomicOr(&some[lane * (kWords / 32) + (w >> 5)], 1u << (w & 31));  // 32 bits: a native operation
    }
    // Last place <= from in row r; -1 if there is none.
    __device__ __forceinline__ int last(int r, Some some, int from) const {
        int w = from >> 5;
        uint32_t x = row[r][w] & (0xFFFFFFFFu >> (31 - (from & 31)));
        if (!x) {
            const Some s = some & ((Some(1) << w) - 1);
            if (!s) return -1;
            w = kWords == 32 ? 31 - __clz(int(s)) : 63 - __clzll(static_cast<long long>(s));
            x = row[r][w];
        }
        return 32 * w + 31 - __clz(int(x));
    }
    // First place >= from (below 32 kWords) in row r; -1 if there is none.
    __device__ __forceinline__ int first(int r, Some some, int from) const {
        int w = from >> 5;
        uint32_t x = row[r][w] & (0xFFFFFFFFu << (from & 31));
        if (!x) {
            const Some s = some & (~Some(1) << w);
            if (!s) return -1;
            w = (kWords == 32 ? __ffs(int(s)) : __ffsll(static_cast<long long>(s))) - 1;
            x = row[r][w];
        }
        return 32 * w + __ffs(int(x)) - 1;
    }
};

// Gather, levels, moments and the cells inside each tile of kTile bodies.  A
// tile's blocks take tiles in order from a counter, so a tile's look-back waits
// only for tiles that already run.
__global__ void __launch_bounds__(kTileThreads, 4) k_tile(
    const unsigned long long *keys, const uint32_t *perm, int64_t K,
    const float2 *__restrict__ pos, const uint32_t *__restrict__ mass, const float4 *__restrict__ frames,
    const int32_t *__restrict__ bgraph, int L, int gbits, int leaf_cap, float4 *__restrict__ body, TileArrays T,
    uint32_t *dev_status, int spin_limit) {
    chain_wait();
    __shared__ __align__(16) uint32_t sm[kTile], sux[kTile], suy[kTile];  // masses, fixed-point coordinates
    __shared__ union {
        LevelBits<kTile / 32> bits;
        MomP Pq[kTileThreads + 1];                        // then: moments before every fourth body
    } u;
    __shared__ uint32_t some[32];                         // of the bits
    __shared__ uint32_t D4[kTile / 4 + 1];                // D of places 0 .. kTile (bytes)
    __shared__ uint32_t nst4[kTile / 4];                  // cells starting at each body (bytes)
    __shared__ uint16_t npre[kTileThreads + 1];           // cells starting before every fourth body
    __shared__ uint32_t list[kTile];                      // cells: first | last << 10 | level << 20
    __shared__ uint32_t levels[kTile];                    // levels of the cells that start at each body (bit mask)
    __shared__ uint32_t open_sh[kTileLevels + 6];
    __shared__ uint32_t wsum[kTileThreads / 32];
    __shared__ unsigned long long red_sh[kTileThreads / 32][5];
    __shared__ uint32_t cells_sh, opens_sh, min_sh, max_sh;
    __shared__ unsigned tile_sh;
    __shared__ int near_sh;
    uint8_t *D = reinterpret_cast<uint8_t *>(D4), *nst = reinterpret_cast<uint8_t *>(nst4);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int64_t tiles = (K + kTile - 1) / kTile;
    if (tid == 0) {
        tile_sh = atomicAdd(&T.flags[tiles], 1u);
        cells_sh = 0u;
        opens_sh = 0u;
        min_sh = 255u;
        max_sh = 0u;
    }
    if (tid < 32) some[tid] = 0u;
    __syncthreads();
    const int64_t tile = tile_sh;
    if (tile >= tiles) return;
    const int64_t t0 = tile * kTile;
    const int n = K - t0 < kTile ? int(K - t0) : kTile;

    // bodies and boundaries, neighbouring threads on neighbouring bodies
    uint32_t heaviest = 0u, least = 255u, greatest = 0u, ds = 0u;
    uint32_t ids[kTileItems];
#pragma unroll
    for (int r = 0; r < kTileItems; ++r) {  // every load before any store: plain loads do not pass them
        const int64_t s = t0 + r * kTileThreads + tid;
        ids[r] = s < t0 + n ? perm[s] : 0u;
    }
#pragma unroll
    for (int r = 0; r < kTileItems; ++r) {
        const int e = r * kTileThreads + tid;
        const int64_t s = t0 + e;
        uint32_t m = 0u, d = 255u;
        uint2 U = make_uint2(0u, 0u);
        if (e < n) {
            const uint32_t i = ids[r];
            const float2 p = pos[i];
            U = fixed_point(p, frames[bgraph ? bgraph[i] : 0]);
            m = mass[i];
            body[s] = make_float4(p.x, p.y, __uint2float_rn(m), __uint_as_float(i));
            d = s > 0 ? level_between(keys[s - 1], keys[s], L, gbits) : 0u;
        } else if (e == n) {
            d = s < K ? level_between(keys[s - 1], keys[s], L, gbits) : 0u;
        }
        levels[e] = 0u;
        heaviest = max(heaviest, m);
        sm[e] = m;
        sux[e] = U.x;
        suy[e] = U.y;
        D[e] = uint8_t(d);
        ds |= d << (8 * r);
        if (e > 0) least = min(least, d);
        if (d != 255u) greatest = max(greatest, d);
    }
    if (tid == 0) {  // place kTile
        uint32_t d = 255u;
        if (n == kTile) {
            d = t0 + kTile < K ? level_between(keys[t0 + kTile - 1], keys[t0 + kTile], L, gbits) : 0u;
            least = min(least, d);
            greatest = max(greatest, d);
        }
        D[kTile] = uint8_t(d);
    }
    least = __reduce_min_sync(0xFFFFFFFFu, least);
    greatest = __reduce_max_sync(0xFFFFFFFFu, greatest);
    if (lane == 0) {
        atomicMin(&min_sh, least);  // over the tile's own boundaries 1 .. n
        atomicMax(&max_sh, greatest);
    }
    const bool light = !__syncthreads_or(heaviest >= kLightMass);
    const uint32_t lo = min(min_sh, uint32_t(D[0])), top = max_sh;
#pragma unroll
    for (int r = 0; r < kTileItems; ++r) u.bits.add((ds >> (8 * r)) & 255u, r * (kTileThreads / 32) + warp, lo, top, some);
    __syncthreads();

    // the cells: boundary j stands for one if it is the first of its smallest
    auto next_below = [&](int from, uint32_t v) {  // first place >= from with D < v
        int e = -1;
        if (v > lo && from < kTile) {
            const int r = int(min(v - 1u, top) - lo);
            e = u.bits.first(r, some[r], from);
        }
        return e >= 0 ? e : D[kTile] < v ? kTile : kTile + 1;
    };
#pragma unroll
    for (int r = 0; r < kTileItems; ++r) {
        const int j = r * kTileThreads + tid + 1;
        const uint32_t v = j <= n ? D[j] : 0u;
        if (v == 0u) continue;
        const int a = u.bits.last(int(v - lo), some[v - lo], j - 1);
        if (a < 0 || D[a] == v) continue;  // the cell starts before the tile, or an earlier boundary stands for it
        const int e = next_below(j + 1, v);
        if (e > n) {  // still open at the tile's end
            open_sh[atomicAdd(&opens_sh, 1u)] = uint32_t(a) | (v << 10) | (uint32_t(D[a]) << 15);
        } else {
            list[atomicAdd(&cells_sh, 1u)] = uint32_t(a) | (uint32_t(e - 1) << 10) | (v << 20);
            atomicOr(&levels[a], 1u << v);
        }
    }
    const int first_below = warp == 0 && lane > 0 ? next_below(1, uint32_t(lane)) : kTile + 1;  // of level `lane`
    __syncthreads();  // the bits are done with: their memory takes the moments

    // moment prefixes, a thread on four consecutive bodies
    const uint4 m4 = reinterpret_cast<const uint4 *>(sm)[tid];
    const uint4 x4 = reinterpret_cast<const uint4 *>(sux)[tid], y4 = reinterpret_cast<const uint4 *>(suy)[tid];
    Mom total;
    {
        Mom acc, inc;
        if (light) {
            const Mom64 a = mom64_add(mom64_add(mom64_add(mom64_add(Mom64{0u, 0ull, 0ull}, m4.x, x4.x, y4.x), m4.y, x4.y,
                                                          y4.y), m4.z, x4.z, y4.z), m4.w, x4.w, y4.w);
            const Mom64 i = mom64_warp_scan(a);
            acc = Mom{a.M, a.X, a.Y};
            inc = Mom{i.M, i.X, i.Y};
        } else {
            acc = mom_add(mom_add(mom_body(m4.x, x4.x, y4.x), mom_body(m4.y, x4.y, y4.y)),
                          mom_add(mom_body(m4.z, x4.z, y4.z), mom_body(m4.w, x4.w, y4.w)));
            inc = mom_warp_scan(acc);
        }
        if (lane == 31) {
            red_sh[warp][0] = inc.M;
            red_sh[warp][1] = static_cast<unsigned long long>(inc.X);
            red_sh[warp][2] = static_cast<unsigned long long>(inc.X >> 64);
            red_sh[warp][3] = static_cast<unsigned long long>(inc.Y);
            red_sh[warp][4] = static_cast<unsigned long long>(inc.Y >> 64);
        }
        __syncthreads();
        Mom before = mom_zero();
        total = mom_zero();
        if (light) {
            Mom64 b{0u, 0ull, 0ull}, t = b;
            for (int w = 0; w < kTileThreads / 32; ++w) {
                if (w == warp) b = t;
                t = Mom64{t.M + uint32_t(red_sh[w][0]), t.X + red_sh[w][1], t.Y + red_sh[w][3]};
            }
            before = Mom{b.M, b.X, b.Y};
            total = Mom{t.M, t.X, t.Y};
        } else for (int w = 0; w < kTileThreads / 32; ++w) {
            const Mom t{red_sh[w][0], (u128(red_sh[w][2]) << 64) | red_sh[w][1], (u128(red_sh[w][4]) << 64) | red_sh[w][3]};
            if (w < warp) before = mom_add(before, t);
            total = mom_add(total, t);
        }
        momp_store(&u.Pq[tid], mom_sub(mom_add(before, inc), acc));
        if (tid == 0) momp_store(&u.Pq[kTileThreads], total);
    }
    if (tid == 0) {
        momp_store(tile == 0 ? &T.incl[0] : &T.agg[tile], total);
        __threadfence();
        atomicExch(&T.flags[tile], tile == 0 ? kMomIncl : kMomAgg);
    }
#pragma unroll
    for (int r = 0; r < kTileItems; ++r) nst[r * kTileThreads + tid] = uint8_t(__popc(levels[r * kTileThreads + tid]));
    __syncthreads();
    const uint32_t cells = cells_sh, opens = opens_sh;
    // cells that start before every fourth body
    {
        const uint32_t x = nst4[tid];
        const uint32_t mine = (x & 0xFFu) + ((x >> 8) & 0xFFu) + ((x >> 16) & 0xFFu) + (x >> 24);
        uint32_t inc = mine;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, inc, d);
            if (lane >= d) inc += y;
        }
        if (lane == 31) wsum[warp] = inc;
        __syncthreads();
        uint32_t before = 0u;
        for (int w = 0; w < warp; ++w) before += wsum[w];
        npre[tid] = uint16_t(before + inc - mine);
        if (tid == 0) npre[kTileThreads] = uint16_t(cells);
        if (4 * tid < n) reinterpret_cast<uint32_t *>(T.starts + t0)[tid] = x;
    }
    __syncthreads();
    // moments of the tile's bodies before place j
    auto before_place = [&](int j) {
        Mom v = momp_load(&u.Pq[j >> 2]);
        for (int q = j & ~3; q < j; ++q) v = mom_add(v, mom_body(sm[q], sux[q], suy[q]));
        return v;
    };
    if (warp == 0 && lane < kTileLevels) {  // the first boundary below each level
        const int j = first_below;
        uint32_t word = 0u;
        if (j <= n) {
            uint32_t c = npre[j >> 2];
            for (int q = j & ~3; q < j; ++q) c += nst[q];
            word = uint32_t(j) | (uint32_t(D[j]) << 11) | (c << 16);
            momp_store(&T.first_mom[tile * kTileLevels + lane], before_place(j));
        }
        T.first[tile * kTileLevels + lane] = word;
    }
    if (warp == 1 && lane < int(opens)) {
        T.open[tile * kTileLevels + lane] = open_sh[lane];
        momp_store(&T.open_mom[tile * kTileLevels + lane], before_place(int(open_sh[lane] & 1023u)));
    }
    if (tid == 64) {
        T.open_n[tile] = opens;
        T.cells[tile] = cells;
        T.tmin[tile] = uint8_t(min_sh);
        atomicMax(&T.flags[tiles + 2 + tile / kTileGroup], 31u - min_sh);
    }
    for (uint32_t q = tid; q < cells; q += kTileThreads) {
        const uint32_t c = list[q];
        const int a = int(c & 1023u), b = int((c >> 10) & 1023u), v = int(c >> 20);
        const int pv = max(int(D[a]), int(D[b + 1]));
        // positions of graph g in Morton order are its index range too
        const float4 fr = frames[bgraph ? bgraph[t0 + a] : 0];
        if (light) {
            auto before = [&](int j) {
                Mom64 x = mom64_load(&u.Pq[j >> 2]);
                for (int k = j & ~3; k < j; ++k) x = mom64_add(x, sm[k], sux[k], suy[k]);
                return x;
            };
            T.cell[t0 + q] = cell_element(before(a), before(b + 1), v, pv, b - a + 1, L, leaf_cap, fr);
        } else {
            T.cell[t0 + q] = cell_element(mom_sub(before_place(b + 1), before_place(a)), v, pv, b - a + 1, L, leaf_cap, fr);
        }
        T.meta[t0 + q] = (c & 0xFFFFFu) | (uint32_t(__popc(levels[a] & ((1u << v) - 1u))) << 20);
    }

    // Look-back by the whole block, kMomLookBack predecessors per round: the
    // nearest tile with an inclusive prefix in the window ends it; the tiles
    // after it must have published their totals (they did long ago, as a rule:
    // the cells were found in the meantime).
    if (tile == 0) return;
    Mom excl = mom_zero();
    int64_t hi = tile - 1;
    int spins = 0;
    while (hi >= 0) {
        if (tid == 0) near_sh = -1;
        __syncthreads();
        uint32_t f[kMomLBItems];
#pragma unroll
        for (int r = 0; r < kMomLBItems; ++r) {
            const int64_t idx = hi - (r * kTileThreads + tid);
            f[r] = idx >= 0 ? *reinterpret_cast<volatile uint32_t *>(&T.flags[idx]) : 0u;
            if (idx >= 0 && f[r] == kMomIncl) atomicMax(&near_sh, int(idx));
        }
        __syncthreads();
        const int64_t near = near_sh;
        const int64_t win_lo = hi - kMomLookBack + 1 > 0 ? hi - kMomLookBack + 1 : 0;
        const int64_t lo = near >= 0 ? near : win_lo;
        bool pending = false;
#pragma unroll
        for (int r = 0; r < kMomLBItems; ++r) {
            const int64_t idx = hi - (r * kTileThreads + tid);
            pending |= idx >= lo && f[r] == 0u;
        }
        if (__syncthreads_or(pending)) {
            if (++spins > spin_limit) {
                if (tid == 0) raise_status(dev_status, BGV_DEV_TIMEOUT);
                break;
            }
            __nanosleep(64);
            continue;
        }
        __threadfence();
        Mom v = mom_zero();
#pragma unroll
        for (int r = 0; r < kMomLBItems; ++r) {
            const int64_t idx = hi - (r * kTileThreads + tid);
            if (idx >= lo) v = mom_add(v, momp_load_cg(f[r] == kMomIncl ? &T.incl[idx] : &T.agg[idx]));
        }
#pragma unroll
        for (int d = 16; d > 0; d >>= 1) {
            Mom o;
            o.M = __shfl_xor_sync(0xFFFFFFFFu, v.M, d);
            const unsigned long long xl = __shfl_xor_sync(0xFFFFFFFFu, static_cast<unsigned long long>(v.X), d);
            const unsigned long long xh = __shfl_xor_sync(0xFFFFFFFFu, static_cast<unsigned long long>(v.X >> 64), d);
            const unsigned long long yl = __shfl_xor_sync(0xFFFFFFFFu, static_cast<unsigned long long>(v.Y), d);
            const unsigned long long yh = __shfl_xor_sync(0xFFFFFFFFu, static_cast<unsigned long long>(v.Y >> 64), d);
            o.X = (u128(xh) << 64) | xl;
            o.Y = (u128(yh) << 64) | yl;
            v = mom_add(v, o);
        }
        if (lane == 0) {
            red_sh[warp][0] = v.M;
            red_sh[warp][1] = static_cast<unsigned long long>(v.X);
            red_sh[warp][2] = static_cast<unsigned long long>(v.X >> 64);
            red_sh[warp][3] = static_cast<unsigned long long>(v.Y);
            red_sh[warp][4] = static_cast<unsigned long long>(v.Y >> 64);
        }
        __syncthreads();
#pragma unroll
        for (int w = 0; w < kTileThreads / 32; ++w)
            excl = mom_add(excl, Mom{red_sh[w][0], (u128(red_sh[w][2]) << 64) | red_sh[w][1],
                                     (u128(red_sh[w][4]) << 64) | red_sh[w][3]});
        if (near >= 0) break;
        hi = lo - 1;
    }
    if (tid == 0) {
        momp_store(&T.incl[tile], mom_add(excl, total));
        __threadfence();
        atomicExch(&T.flags[tile], kMomIncl);
    }
}

// First tile after t with a boundary below level v (the last tile's end is one).
__device__ __forceinline__ int64_t next_tile_below(const TileArrays &T, int64_t tiles, int64_t t, uint32_t v) {
    const uint32_t vv = v * 0x01010101u;
    int64_t at = t + 1;
    while (at < tiles) {
        if (at % kTileGroup == 0 && 31u - T.flags[tiles + 2 + at / kTileGroup] >= v) {
            at += kTileGroup;
            continue;
        }
        const int64_t base = at & ~int64_t(15);
        const uint4 q = *reinterpret_cast<const uint4 *>(T.tmin + base);  // 16 tiles; past the last: not reached
        const uint32_t x[4] = {q.x, q.y, q.z, q.w};
        int found = 16;
#pragma unroll
        for (int w = 3; w >= 0; --w) {
            uint32_t y = x[w];
            const int skip = int(at - base) - 4 * w;  // bytes of this word before `at`
            if (skip >= 4) continue;
            if (skip > 0) y |= (1u << (8 * skip)) - 1u;
            const uint32_t hit = __vcmpltu4(y, vv);
            if (hit) found = 4 * w + ((__ffs(int(hit)) - 1) >> 3);
        }
        if (found < 16) return base + found;
        at = base + 16;
    }
    return tiles - 1;
}

// The cells open at each tile's end, a lane per open first body of the tile.
// Bound by latency: a lane closes its cells one after the other, outwards (20 us at
// 1 M bodies with 128-bit divisions and every search from the tile on; a single
// step of 60,000 bodies 133.9 -> 131.7 us with neither).
__global__ void __launch_bounds__(kTileThreads) k_tile_cross(int64_t K, int L, int leaf_cap,
                                                             const float4 *__restrict__ frames,
                                                             const int32_t *__restrict__ bgraph, TileArrays T,
                                                             unsigned long long *tree_nodes) {
    chain_wait();
    const int lane = threadIdx.x & 31;
    const int64_t tiles = (K + kTile - 1) / kTile;
    const int64_t tile = (int64_t(blockIdx.x) * kTileThreads + threadIdx.x) >> 5;
    if (tile < tiles) {
        uint32_t mask = 0u, made = 0u;
        if (lane < int(T.open_n[tile])) {
            const int64_t slot = tile * kTileLevels + lane;
            const uint32_t o = T.open[slot];
            const uint32_t a = o & 1023u, dl = o >> 15;
            uint32_t v = (o >> 10) & 31u;
            Mom lo = momp_load(&T.open_mom[slot]);
            if (tile) lo = mom_add(lo, momp_load(&T.incl[tile - 1]));
            const int64_t first = tile * kTile + a;
            const float4 fr = frames[bgraph ? bgraph[first] : 0];
            int64_t te = tile;
            while (true) {  // outwards: a boundary below a lower level is no nearer
                te = next_tile_below(T, tiles, te == tile ? tile : te - 1, v);
                const uint32_t w = T.first[te * kTileLevels + v];
                const uint32_t j = w & 2047u, dj = (w >> 11) & 31u;
                Mom hi = momp_load(&T.first_mom[te * kTileLevels + v]);
                hi = mom_add(hi, momp_load(&T.incl[te - 1]));  // te > tile >= 0
                const int64_t last = te * kTile + j - 1;
                T.cross[tile * kTileLevels + v] =
                    cell_element(mom_sub(hi, lo), int(v), int(max(dl, dj)), last - first + 1, L, leaf_cap, fr);
                T.cross_meta[tile * kTileLevels + v] = make_uint2(a | (made << 10), uint32_t(last));
                mask |= 1u << v;
                ++made;
                if (dj <= dl) break;
                v = dj;
            }
            T.open_cells[slot] = made;
        }
        mask = __reduce_or_sync(0xFFFFFFFFu, mask);
        made = __reduce_add_sync(0xFFFFFFFFu, made);
        if (lane == 0) {
            T.cross_mask[tile] = mask;
            T.base[tile] = T.cells[tile] + made;
        }
    }
    // the last block turns the tiles' cell counts into prefix sums
    __shared__ uint32_t wsum[kTileThreads / 32];
    __shared__ bool last_block;
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        last_block = atomicAdd(&T.flags[tiles + 1], 1u) == gridDim.x - 1;
    }
    __syncthreads();
    if (!last_block) return;
    __threadfence();
    constexpr int kPer = 4;
    const int warp = threadIdx.x >> 5;
    uint32_t carry = 0u;
    for (int64_t b0 = 0; b0 < tiles; b0 += kTileThreads * kPer) {
        const int64_t i0 = b0 + int64_t(threadIdx.x) * kPer;
        uint32_t c[kPer], mine = 0u;
#pragma unroll
        for (int q = 0; q < kPer; ++q) {
            c[q] = i0 + q < tiles ? __ldcg(&T.base[i0 + q]) : 0u;
            mine += c[q];
        }
        uint32_t inc = mine;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, inc, d);
            if (lane >= d) inc += y;
        }
        if (lane == 31) wsum[warp] = inc;
        __syncthreads();
        uint32_t before = carry, all = 0u;
        for (int w = 0; w < kTileThreads / 32; ++w) {
            if (w < warp) before += wsum[w];
            all += wsum[w];
        }
        uint32_t run = before + inc - mine;
#pragma unroll
        for (int q = 0; q < kPer; ++q) {
            if (i0 + q < tiles) T.base[i0 + q] = run;
            run += c[q];
        }
        carry += all;
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        T.base[tiles] = carry;
        *tree_nodes = carry;
    }
}

// Pre-order layout.  With S[s] = cells whose first body precedes s:
//   body s           -> s + S[s + 1]     (every cell starting at or before s
//                                          comes first)
//   cell [a, b]      -> a + S[a] + (its ancestors that also start at a: the cells
//                                   that leave the tile, then the outer ones inside)
//   skip(cell [a,b]) -> b + 1 + S[b + 1] (the element after its subtree)
// Elements are float4 (x, y, mass, side^2), side^2 = -1 for a body.  Also leaves
// the tiles' flags and the step's interaction counter at zero, for the next
// step's k_tile and the traversal after this kernel.
__global__ void __launch_bounds__(kTileThreads) k_tile_emit(int64_t K, const float4 *__restrict__ body, TileArrays T,
                                                            uint32_t *__restrict__ S, float4 *__restrict__ geo,
                                                            int32_t *__restrict__ skip,
                                                            unsigned long long *interactions) {
    chain_wait();
    __shared__ uint32_t nst4[kTile / 4], loc4[kTile / 4];  // cells that start at each body: all, inside the tile
    __shared__ uint32_t pre[kTile + 1];  // cells starting before each body, in this tile
    __shared__ uint32_t wsum[kTileThreads / 32];
    uint8_t *nst = reinterpret_cast<uint8_t *>(nst4), *loc = reinterpret_cast<uint8_t *>(loc4);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int64_t tile = blockIdx.x, t0 = tile * kTile;
    const int n = K - t0 < kTile ? int(K - t0) : kTile;
    nst4[tid] = loc4[tid] = 4 * tid < n ? reinterpret_cast<const uint32_t *>(T.starts + t0)[tid] : 0u;
    if (tid == 0) {
        const int64_t tiles = gridDim.x;
        T.flags[tile] = 0u;
        if (tile % kTileGroup == 0) T.flags[tiles + 2 + tile / kTileGroup] = 0u;
        if (tile == 0) {
            T.flags[tiles] = T.flags[tiles + 1] = 0u;
            *interactions = 0ull;
        }
    }
    const uint32_t base = T.base[tile], cells = T.cells[tile], opens = T.open_n[tile];
    __syncthreads();
    if (tid < int(opens)) {  // one entry per first body
        const int64_t slot = tile * kTileLevels + tid;
        nst[T.open[slot] & 1023u] += uint8_t(T.open_cells[slot]);
    }
    __syncthreads();
    {
        const uint32_t x = nst4[tid];
        const uint32_t c0 = x & 0xFFu, c1 = (x >> 8) & 0xFFu, c2 = (x >> 16) & 0xFFu, c3 = x >> 24;
        const uint32_t mine = c0 + c1 + c2 + c3;
        uint32_t inc = mine;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, inc, d);
            if (lane >= d) inc += y;
        }
        if (lane == 31) wsum[warp] = inc;
        __syncthreads();
        uint32_t run = inc - mine;
        for (int w = 0; w < warp; ++w) run += wsum[w];
        pre[4 * tid] = run;
        pre[4 * tid + 1] = run + c0;
        pre[4 * tid + 2] = run + c0 + c1;
        pre[4 * tid + 3] = run + c0 + c1 + c2;
        if (tid == kTileThreads - 1) pre[kTile] = run + mine;
    }
    __syncthreads();
#pragma unroll
    for (int r = 0; r < kTileItems; ++r) {
        const int e = r * kTileThreads + tid;
        if (e >= n) continue;
        const float4 b = body[t0 + e];
        const int64_t at = t0 + e + base + pre[e + 1];
        S[t0 + e] = base + pre[e];
        geo[at] = make_float4(b.x, b.y, b.z, -1.0f);
        skip[at] = int32_t(at + 1);
    }
    if (tid == 0 && t0 + n == K) S[K] = T.base[tile + 1];
    for (uint32_t q = tid; q < cells; q += kTileThreads) {
        const uint32_t c = T.meta[t0 + q];
        const int a = int(c & 1023u), b = int((c >> 10) & 1023u);
        const int64_t at = t0 + a + base + (pre[a + 1] - loc[a]) + (c >> 20);
        geo[at] = T.cell[t0 + q];
        skip[at] = int32_t(t0 + b + 1 + base + pre[b + 1]);
    }
    const uint32_t mask = T.cross_mask[tile];
    if (tid < kTileLevels && ((mask >> tid) & 1u)) {  // cells that end in a later tile
        const int64_t slot = tile * kTileLevels + tid;
        const uint2 c = T.cross_meta[slot];
        const int a = int(c.x & 1023u), k = int(c.x >> 10);
        const int64_t at = t0 + a + base + (pre[a + 1] - loc[a] - 1u - uint32_t(k));
        // cells starting before the end's boundary: the tiles before its tile,
        // the cells inside that tile, and the open ones that start before it
        const int64_t te = int64_t(c.y) / kTile;
        const uint32_t j = c.y % kTile + 1u;
        uint32_t s = T.base[te] + (T.first[te * kTileLevels + tid] >> 16);
        const uint32_t on = T.open_n[te];
        for (uint32_t q = 0; q < on; ++q)
            if ((T.open[te * kTileLevels + q] & 1023u) < j) s += T.open_cells[te * kTileLevels + q];
        geo[at] = T.cross[slot];
        skip[at] = int32_t(int64_t(c.y) + 1 + s);
    }
}

}  // namespace
}  // namespace bgv
