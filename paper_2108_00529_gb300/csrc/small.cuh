// small.cuh -- whole ForceAtlas2 runs on graphs of up to kSmallMax bodies.
//
// With few bodies a step of the general path is a chain of a dozen kernels that
// each last a few microseconds (72 us per step at 219 bodies, 94 at 1,764; here
// 15.1 and 26).
// Here one cluster of blocks keeps a graph in shared memory and takes every
// step of the run in one launch: each block builds the whole quadtree for
// itself (sorting 2,048 bodies costs less than fetching a tree from elsewhere),
// half of its threads walk its share of the bodies in Morton order while the
// other half sums the attraction of its share of the nodes; repulsions, sums of
// swing and traction, and new positions go straight into the other blocks'
// shared memory.  Three cluster barriers per step.
// Bound by latency: at 1,764 bodies a step was 73,000 cycles, 20,500 of them the
// search for cells, 14,600 the walk, 9,300 the sort, 9,000 the exact sums and the
// speed, the rest short phases between barriers.  Cells found by LevelBits: 200
// steps 7,239 -> 5,996 us (219 bodies: 3,975 -> 3,605); the sort binned by the
// frame's own bits and sums by warp reductions of integers at one scale: 5,327
// (3,037); the bits' summary words set by 32-bit atomics, as 64-bit ones loop:
// 5,184 (3,020).  A step at 1,764 bodies is then about 52,000 cycles, the walk
// 14,400, cells 7,900, sort 6,000, no other phase more than 4,000.
// All arithmetic is that of the general path (forces.cuh, tree.cuh), and every
// sum is taken in the same order or exactly, so the results are the same bits.
#pragma once

#include <cooperative_groups.h>

#include "forces.cuh"
#include "tree.cuh"

namespace bgv {
namespace {

constexpr int kSmallMax = 2048;
constexpr int kSmallThreads = 512;
constexpr int kSmallHalf = kSmallThreads / 2;
constexpr int kSmallSums = kSmallHalf / 32;  // warps of nodes
constexpr int kSmallCluster = 8;         // blocks per cluster, at most
constexpr int kSmallIdBits = 11;         // ids < kSmallMax
constexpr int kSmallRank = 32;           // largest bin ranked by counting
// CSR entries a block keeps (weights below 2^21): what is left of its shared
// memory.  200 steps at 1,764 bodies took 9,683 us with 8,192, and 7,239 with
// 10,240, lighter moments and the sums merged by a warp.
constexpr int kSmallCache = 9664;
// CSR entries of a graph, at most.  Half of them may lie in one block's rows, and are
// read from memory in every step: 100 steps of 2,048 bodies 4.4 ms with 118,286 even
// entries (general path 7.5), 7.6 with 489,116, but 16.4 with 332,304 of which half
// lie in an eighth of the rows.
constexpr int64_t kSmallEntries = int64_t(1) << 17;
constexpr int kSmallChunk = 256;         // steps per launch, at most
static_assert(kSmallMax == 4 * kSmallThreads, "four bodies a thread");
static_assert(kSmallMax <= kSmallCluster * kSmallHalf, "a thread per node");

// Blocks per cluster for graphs of up to K bodies: a block has at least about
// 128 bodies, one warp's worth per scheduler.
inline int small_cluster(int64_t K) { return K <= 128 ? 1 : K <= 256 ? 2 : K <= 512 ? 4 : kSmallCluster; }

struct SmallArgs {
    int64_t K;              // bodies (one graph)
    const int64_t *koff;    // batched: [G + 1] first body of each graph, else null
    const int32_t *off, *adj;  // off null: no CSR entries
    const uint32_t *w, *mass;
    float2 *pos, *F, *Fprev;
    double *speed;
    WsHeader *hdr;
    float theta2, kr, kg, tau, ks, ksmax;
    int strong, L, leaf_cap, att_short, iterations;
};

struct SmallMem {
    float2 pos[kSmallMax];
    float4 body[kSmallMax];              // Morton order: x, y, mass, id
    uint32_t mass[kSmallMax];            // by id
    uint32_t sm[kSmallMax], sux[kSmallMax], suy[kSmallMax];  // Morton order: mass, fixed-point position
    union {
        LevelBits<kSmallMax / 32> bits;
        MomP Pq[kSmallThreads + 1];      // then: moments before every fourth body
        float2 fa[kSmallHalf];           // then: attraction of the block's long rows
    } w;
    unsigned long long some[32];         // of the bits
    union {
        struct {
            unsigned long long a[kSmallMax], b[kSmallMax];  // key << kSmallIdBits | id
            uint32_t bins[kSmallMax];            // then the levels of the cells that start at each body
        } sort;
        struct {
            float4 geo[2 * kSmallMax];
            uint16_t skip[2 * kSmallMax];
        } tree;
        XPart xpart[kSmallCluster * kSmallSums][2];  // after the walks: S and T of every block's node warps
    } u;
    uint32_t list[kSmallMax];            // cells: first | last << 11 | outer cells from it << 22 | level << 27
    uint32_t D4[kSmallThreads + 1];
    uint16_t S[kSmallMax + 2];           // cells that start before each body
    uint32_t cache[kSmallCache];         // neighbour << 21 | weight
    float2 frep[kSmallHalf];             // repulsion of the block's nodes (written by the walkers of all blocks)
    unsigned long long red[kSmallThreads / 32][5];
    float4 box[kSmallThreads / 32];
    uint32_t wsum[2][kSmallThreads / 32];  // of the sort, of the cells
    int2 long_span[kSmallHalf];          // the block's rows of more than att_short entries
    uint8_t long_rows[kSmallHalf];       // their nodes in the block
    uint32_t longs, next;                // how many, and the next of them to sum
    uint32_t cells, greatest;
    double speed;
};
static_assert(sizeof(SmallMem) <= 227 * 1024, "shared memory of a block");

// Exclusive block scan of one value per thread.
__device__ __forceinline__ uint32_t small_scan(uint32_t x, uint32_t *wsum) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint32_t inc = x;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, inc, d);
        if (lane >= d) inc += y;
    }
    if (lane == 31) wsum[warp] = inc;
    __syncthreads();
    return __reduce_add_sync(0xFFFFFFFFu, lane < warp ? wsum[lane] : 0u) + inc - x;
}

// The words w (four per thread; item r of thread t is body r * kSmallThreads +
// t) in ascending order into sort.a: binned by their high bits, then ranked
// inside the bins; a bitonic network when a bin is too full.
__device__ void small_sort(SmallMem &m, const unsigned long long (&w)[4], int K, int L) {
    const int tid = threadIdx.x;
    const int sh = 2 * L;  // kSmallMax bins over the keys, which fill their range (the frame is the bodies' box)
    uint32_t r4[4];
#pragma unroll
    for (int r = 0; r < 4; ++r)
        r4[r] = r * kSmallThreads + tid < K ? atomicAdd(&m.u.sort.bins[uint32_t(w[r] >> sh)], 1u) : 0u;
    __syncthreads();
    uint4 c = reinterpret_cast<uint4 *>(m.u.sort.bins)[tid];
    const uint32_t most = max(max(c.x, c.y), max(c.z, c.w));
    const uint32_t run = small_scan(c.x + c.y + c.z + c.w, m.wsum[0]);
    c = make_uint4(run, run + c.x, run + c.x + c.y, run + c.x + c.y + c.z);
    reinterpret_cast<uint4 *>(m.u.sort.bins)[tid] = c;
    if (!__syncthreads_or(most > kSmallRank)) {
#pragma unroll
        for (int r = 0; r < 4; ++r)
            if (r * kSmallThreads + tid < K) m.u.sort.b[m.u.sort.bins[uint32_t(w[r] >> sh)] + r4[r]] = w[r];
        __syncthreads();
        for (int s = tid; s < K; s += kSmallThreads) {
            const unsigned long long x = m.u.sort.b[s];
            const uint32_t bin = uint32_t(x >> sh);
            const int b0 = int(m.u.sort.bins[bin]), b1 = bin + 1 < kSmallMax ? int(m.u.sort.bins[bin + 1]) : K;
            int at = b0;
            for (int t = b0; t < b1; ++t) at += m.u.sort.b[t] < x ? 1 : 0;  // words differ by their ids
            m.u.sort.a[at] = x;
        }
        __syncthreads();
        return;
    }
    int lg = 1;
    while ((1 << lg) < K) ++lg;
#pragma unroll
    for (int r = 0; r < 4; ++r) {
        const int i = r * kSmallThreads + tid;
        if (i < K) m.u.sort.a[i] = w[r];
    }
    __syncthreads();
    // every comparator puts the smaller word first, so places past K count as
    // +infinity and stay away
    auto exchange = [&](int i, int j) {
        if (j >= K) return;
        const unsigned long long x = m.u.sort.a[i], y = m.u.sort.a[j];
        if (x > y) {
            m.u.sort.a[i] = y;
            m.u.sort.a[j] = x;
        }
    };
    for (int l = 1; l <= lg; ++l) {
        const int half = 1 << (l - 1);
        for (int q = tid; q < (1 << (lg - 1)); q += kSmallThreads) {
            const int base = (q >> (l - 1)) << l, o = q & (half - 1);
            exchange(base + o, base + 2 * half - 1 - o);
        }
        __syncthreads();
        for (int j = l - 2; j >= 0; --j) {
            for (int q = tid; q < (1 << (lg - 1)); q += kSmallThreads) {
                const int i = ((q >> j) << (j + 1)) + (q & ((1 << j) - 1));
                exchange(i, i + (1 << j));
            }
            __syncthreads();
        }
    }
}

// The quadtree of the positions in m.pos, in pre-order in m.u.tree (see
// tree.cuh; all K <= kSmallMax bodies are one tile).  Returns the cells.
__device__ uint32_t small_tree(SmallMem &m, int K, int L, int leaf_cap) {
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    uint8_t *D = reinterpret_cast<uint8_t *>(m.D4);
    uint32_t *levels = m.u.sort.bins;
    float4 box = box_empty();
    for (int i = tid; i < K; i += kSmallThreads) box_add(box, m.pos[i]);
#pragma unroll
    for (int r = 0; r < 4; ++r) m.u.sort.bins[r * kSmallThreads + tid] = 0u;
    box_warp(box);
    if (lane == 0) m.box[warp] = box;
    if (tid == 0) m.cells = m.greatest = 0u;
    if (tid < 32) m.some[tid] = 0ull;
    __syncthreads();
    box = m.box[0];
    for (int q = 1; q < kSmallThreads / 32; ++q) box_merge(box, m.box[q]);
    const float4 fr = frame_of(box.x, box.y, box.z, box.w);
    {
        unsigned long long w[4];
#pragma unroll
        for (int r = 0; r < 4; ++r) {
            const int i = r * kSmallThreads + tid;
            const uint2 U = i < K ? fixed_point(m.pos[i], fr) : make_uint2(0u, 0u);
            const unsigned long long key = (spread_bits(U.x >> (32 - L)) << 1) | spread_bits(U.y >> (32 - L));
            w[r] = (key << kSmallIdBits) | unsigned(i);
        }
        small_sort(m, w, K, L);
    }
    // Morton order: bodies and the levels between neighbours
    uint32_t heaviest = 0u, greatest = 0u, ds = 0u;
#pragma unroll
    for (int r = 0; r < 4; ++r) {
        const int s = r * kSmallThreads + tid;
        uint32_t mass = 0u, d = 255u;
        uint2 U = make_uint2(0u, 0u);
        if (s < K) {
            const unsigned long long x = m.u.sort.a[s];
            const uint32_t id = uint32_t(x) & (kSmallMax - 1);
            const float2 p = m.pos[id];
            U = fixed_point(p, fr);
            mass = m.mass[id];
            m.body[s] = make_float4(p.x, p.y, __uint2float_rn(mass), __uint_as_float(id));
            d = s ? level_between(m.u.sort.a[s - 1] >> kSmallIdBits, x >> kSmallIdBits, L, 0) : 0u;
        } else if (s == K) {
            d = 0u;
        }
        levels[s] = 0u;
        heaviest = max(heaviest, mass);
        m.sm[s] = mass;
        m.sux[s] = U.x;
        m.suy[s] = U.y;
        D[s] = uint8_t(d);
        ds |= d << (8 * r);
        if (d != 255u) greatest = max(greatest, d);
    }
    if (tid == 0) D[kSmallMax] = K == kSmallMax ? 0u : 255u;
    greatest = __reduce_max_sync(0xFFFFFFFFu, greatest);
    if (lane == 0) atomicMax(&m.greatest, greatest);
    const bool light = !__syncthreads_or(heaviest >= kLightMass);
    {
        const uint32_t hi = m.greatest;  // the least is 0, at place 0
#pragma unroll
        for (int r = 0; r < 4; ++r)
            if (r * kSmallThreads + warp * 32 <= K)  // words past the end are not asked for
                m.w.bits.add((ds >> (8 * r)) & 255u, r * (kSmallThreads / 32) + warp, 0u, hi,
                             reinterpret_cast<uint32_t *>(m.some));
    }
    __syncthreads();
#pragma unroll
    for (int r = 0; r < 4; ++r) {
        const int j = r * kSmallThreads + tid + 1;
        const uint32_t v = j < K ? D[j] : 0u;  // the end of all bodies closes every cell and stands for none
        if (v == 0u) continue;
        const int a = m.w.bits.last(int(v), m.some[v], j - 1);  // place 0 is not above any
        if (D[a] == v) continue;
        int e = m.w.bits.first(int(v) - 1, m.some[v - 1], j + 1 < kSmallMax ? j + 1 : kSmallMax - 1);
        if (e <= j) e = kSmallMax;
        m.list[atomicAdd(&m.cells, 1u)] = uint32_t(a) | (uint32_t(e - 1) << 11) | (v << 27);
        atomicOr(&levels[a], 1u << v);
    }
    __syncthreads();  // the bits are done with: their memory takes the moments
    const uint32_t cells = m.cells;
    {
        const uint4 m4 = reinterpret_cast<const uint4 *>(m.sm)[tid];
        const uint4 x4 = reinterpret_cast<const uint4 *>(m.sux)[tid], y4 = reinterpret_cast<const uint4 *>(m.suy)[tid];
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
            m.red[warp][0] = inc.M;
            m.red[warp][1] = static_cast<unsigned long long>(inc.X);
            m.red[warp][2] = static_cast<unsigned long long>(inc.X >> 64);
            m.red[warp][3] = static_cast<unsigned long long>(inc.Y);
            m.red[warp][4] = static_cast<unsigned long long>(inc.Y >> 64);
        }
        const uint4 x = reinterpret_cast<const uint4 *>(levels)[tid];
        const uint32_t c0 = __popc(x.x), c1 = __popc(x.y), c2 = __popc(x.z), c3 = __popc(x.w);
        const uint32_t run = small_scan(c0 + c1 + c2 + c3, m.wsum[1]);  // its barrier orders m.red too
        m.S[4 * tid] = uint16_t(run);
        m.S[4 * tid + 1] = uint16_t(run + c0);
        m.S[4 * tid + 2] = uint16_t(run + c0 + c1);
        m.S[4 * tid + 3] = uint16_t(run + c0 + c1 + c2);
        if (tid == kSmallThreads - 1) m.S[kSmallMax] = uint16_t(run + c0 + c1 + c2 + c3);
        Mom before = mom_zero();
        if (light) {
            Mom64 b{0u, 0ull, 0ull};
            for (int q = 0; q < warp; ++q)
                b = Mom64{b.M + uint32_t(m.red[q][0]), b.X + m.red[q][1], b.Y + m.red[q][3]};
            before = Mom{b.M, b.X, b.Y};
        } else {
            for (int q = 0; q < warp; ++q)
                before = mom_add(before, Mom{m.red[q][0], (u128(m.red[q][2]) << 64) | m.red[q][1],
                                             (u128(m.red[q][4]) << 64) | m.red[q][3]});
        }
        before = mom_add(before, inc);
        momp_store(&m.w.Pq[tid], mom_sub(before, acc));
        if (tid == kSmallThreads - 1) momp_store(&m.w.Pq[kSmallThreads], before);
    }
    for (uint32_t q = tid; q < cells; q += kSmallThreads) {
        const uint32_t c = m.list[q];
        m.list[q] = c | (uint32_t(__popc(levels[c & 2047u] & ((1u << (c >> 27)) - 1u))) << 22);
    }
    __syncthreads();
    auto before_place = [&](int j) {
        Mom v = momp_load(&m.w.Pq[j >> 2]);
        for (int q = j & ~3; q < j; ++q) v = mom_add(v, mom_body(m.sm[q], m.sux[q], m.suy[q]));
        return v;
    };
    // the sorted words are done with: their memory becomes the tree
    for (uint32_t q = tid; q < cells; q += kSmallThreads) {
        const uint32_t c = m.list[q];
        const int a = int(c & 2047u), b = int((c >> 11) & 2047u), v = int(c >> 27);
        const int at = a + m.S[a] + int((c >> 22) & 31u);
        const int pv = max(int(D[a]), int(D[b + 1]));
        if (light) {
            auto before = [&](int j) {
                Mom64 x = mom64_load(&m.w.Pq[j >> 2]);
                for (int k = j & ~3; k < j; ++k) x = mom64_add(x, m.sm[k], m.sux[k], m.suy[k]);
                return x;
            };
            m.u.tree.geo[at] = cell_element(before(a), before(b + 1), v, pv, b - a + 1, L, leaf_cap, fr);
        } else {
            m.u.tree.geo[at] = cell_element(mom_sub(before_place(b + 1), before_place(a)), v, pv, b - a + 1, L, leaf_cap, fr);
        }
        m.u.tree.skip[at] = uint16_t(b + 1 + m.S[b + 1]);
    }
    for (int s = tid; s < K; s += kSmallThreads) {
        const float4 b = m.body[s];
        const int at = s + m.S[s + 1];
        m.u.tree.geo[at] = make_float4(b.x, b.y, b.z, -1.0f);
        m.u.tree.skip[at] = uint16_t(at + 1);
    }
    __syncthreads();
    return cells;
}

// Attraction of one row [b, e) summed in the general path's order (k_att_*): a
// short row by its thread, a longer one by a warp.  entry(x, p, &wf): position and
// weight of CSR entry x (weight 0: none).
template <class Entry>
__device__ __forceinline__ float2 small_short_row(int64_t b, int64_t e, float2 p, Entry entry) {
    float ax = 0.0f, ay = 0.0f;
#pragma unroll 4
    for (int64_t x = b; x < e; ++x) {
        float wf;
        const float2 pj = entry(x, p, &wf);
        ax += wf * (pj.x - p.x);
        ay += wf * (pj.y - p.y);
    }
    return make_float2(ax, ay);
}
// kIn: entries of a lane in flight.
template <int kIn, class Entry>
__device__ __forceinline__ float2 small_warp_row(int64_t b, int64_t e, float2 p, Entry entry) {
    const int lane = threadIdx.x & 31;
    const bool block_row = e - b > kAttMedium;  // a block's 256 threads: eight warps' sums, added in order
    const int stride = block_row ? 256 : 32;
    float tx = 0.0f, ty = 0.0f;
    for (int vw = 0; vw < (block_row ? 8 : 1); ++vw) {
        float sx = 0.0f, sy = 0.0f;
        for (int64_t x0 = b + vw * 32 + lane; x0 < e; x0 += kIn * stride) {
            float wf[kIn];
            float2 pj[kIn];
#pragma unroll
            for (int k = 0; k < kIn; ++k) {
                const int64_t x = x0 + k * stride;
                wf[k] = 0.0f;
                if (x < e) pj[k] = entry(x, p, &wf[k]);
            }
#pragma unroll
            for (int k = 0; k < kIn; ++k) {
                if (x0 + k * stride >= e) break;
                sx += wf[k] * (pj[k].x - p.x);
                sy += wf[k] * (pj[k].y - p.y);
            }
        }
#pragma unroll
        for (int d = 16; d > 0; d >>= 1) {
            sx += __shfl_xor_sync(0xFFFFFFFFu, sx, d);
            sy += __shfl_xor_sync(0xFFFFFFFFu, sy, d);
        }
        tx = vw ? tx + sx : sx;
        ty = vw ? ty + sy : sy;
    }
    return make_float2(tx, ty);
}
// The block's long rows, taken one after the other by whichever warp is free;
// row(b, e, p): the sum of the row [b, e), whose node is at p.  Whole warps call it,
// the walkers when they are done, as long as more than kSmallKeep rows are left: fewer
// are summed before the last walker is done.  (A thread's own rows summed by its
// warp, one after the other, left hubs to one warp: 100 steps of 1,500 bodies and
// 226,212 entries, half of them in an eighth of the rows, 24.7 ms; so 11.6.)
constexpr uint32_t kSmallKeep = 16;
__device__ __forceinline__ bool small_rows_left(const SmallMem &m, uint32_t all) {
    const uint32_t keep = threadIdx.x >= kSmallHalf ? kSmallKeep : 0u;
    return __shfl_sync(0xFFFFFFFFu, *static_cast<const volatile uint32_t *>(&m.next), 0) + keep < all;
}
template <class Row>
__device__ __forceinline__ void small_long_rows(SmallMem &m, int lo, Row row) {
    const int lane = threadIdx.x & 31;
    const uint32_t all = m.longs;
    while (small_rows_left(m, all)) {
        const uint32_t q = __shfl_sync(0xFFFFFFFFu, lane == 0 ? atomicAdd(&m.next, 1u) : 0u, 0);
        if (q >= all) break;
        const int local = m.long_rows[q];
        const int2 span = m.long_span[q];
        const float2 f = row(span.x, span.y, m.pos[lo + local]);
        if (lane == 0) m.w.fa[local] = f;
    }
}

__global__ void __launch_bounds__(kSmallThreads, 1) k_small(const __grid_constant__ SmallArgs A) {
    namespace cg = cooperative_groups;
    extern __shared__ __align__(32) unsigned char small_raw[];
    SmallMem &m = *reinterpret_cast<SmallMem *>(small_raw);
    cg::cluster_group cluster = cg::this_cluster();
    const int C = int(cluster.num_blocks()), rank = int(cluster.block_rank());
    const int tid = threadIdx.x, lane = tid & 31;
    const int64_t g = blockIdx.x / C;
    const int64_t k0 = A.koff ? A.koff[g] : 0;
    const int K = int((A.koff ? A.koff[g + 1] : A.K) - k0);
    for (int i = tid; i < K; i += kSmallThreads) {
        m.pos[i] = A.pos[k0 + i];
        m.mass[i] = A.mass[k0 + i];
    }
    // the block's nodes (the first half's threads, one each) and bodies in
    // Morton order (the other half's)
    const int per = (K + C - 1) / C;
    const int lo = min(rank * per, K), hi = min(lo + per, K);
    const int warp = tid >> 5;
    const bool walker = tid >= kSmallHalf;
    const int mine = lo + (walker ? tid - kSmallHalf : tid);
    const bool have = mine < hi;
    const bool node = have && !walker;
    int64_t rb = 0, re = 0;
    float2 f = make_float2(0.0f, 0.0f), fp = f;
    float mass = 0.0f;
    if (node) {
        if (A.off) {
            rb = A.off[k0 + mine];
            re = A.off[k0 + mine + 1];
        }
        fp = A.Fprev[k0 + mine];
        mass = __uint2float_rn(A.mass[k0 + mine]);
    }
    // the rows of the block's nodes, kept if they fit
    const int64_t c_lo = A.off && lo < hi ? A.off[k0 + lo] : 0, c_hi = A.off && lo < hi ? A.off[k0 + hi] : 0;
    bool cached = c_hi - c_lo <= kSmallCache;
    if (cached) {
        bool wide = false;
        for (int r = lo + (tid >> 5); r < hi && A.off; r += kSmallThreads / 32) {
            const int64_t b = A.off[k0 + r], e = A.off[k0 + r + 1];
            wide |= b < e && (b < c_lo || e > c_hi);  // offsets that fall somewhere: rows past the block's range
            for (int64_t x = b + lane; x < e; x += 32) {
                const int64_t j = int64_t(A.adj[x]) - k0;
                const bool ok = j >= 0 && j < K;  // an invalid entry adds nothing
                const uint32_t w = ok ? A.w[x] : 0u;
                wide |= w >= (1u << 21);
                if (x >= c_lo && x < c_hi) m.cache[x - c_lo] = (uint32_t(ok ? j : r) << 21) | (w & 0x1FFFFFu);
            }
        }
        cached = !__syncthreads_or(wide);
    }
    auto entry_cached = [&](int64_t x, float2, float *wf) {
        const uint32_t q = m.cache[x - c_lo];
        *wf = __uint2float_rn(q & 0x1FFFFFu);
        return m.pos[q >> 21];
    };
    auto entry_global = [&](int64_t x, float2 own, float *wf) {
        const int64_t j = int64_t(__ldg(A.adj + x)) - k0;
        const bool ok = j >= 0 && j < K;
        *wf = ok ? __uint2float_rn(__ldg(A.w + x)) : 0.0f;
        return ok ? m.pos[j] : own;
    };
    auto row_cached = [&](int b, int e, float2 p) { return small_warp_row<2>(b, e, p, entry_cached); };
    auto row_global = [&](int b, int e, float2 p) { return small_warp_row<8>(b, e, p, entry_global); };
    if (tid == 0) {
        m.speed = A.speed[g];
        m.longs = m.next = 0u;
    }
    __syncthreads();
    const bool is_long = re - rb > A.att_short;
    if (is_long) {
        const uint32_t q = atomicAdd(&m.longs, 1u);
        m.long_rows[q] = uint8_t(tid);
        m.long_span[q] = make_int2(int(rb), int(re));
    }
    cluster.sync();
    unsigned long long inter_total = 0ull;
    unsigned inter = 0u;
    uint32_t cells = 0u;
    double Ssum = 0.0, Tsum = 0.0;
    for (int it = 0; it < A.iterations; ++it) {
        cells = small_tree(m, K, A.L, A.leaf_cap);
        float2 p = make_float2(0.0f, 0.0f), fa = p;
        inter = 0u;
        if (walker) {
            if (have) {
                const float4 bi = m.body[mine];
                const float2 fr = bh_walk(m.u.tree.geo, m.u.tree.skip, bi, A.kr * bi.z, A.theta2,
                                          uint32_t(mine + m.S[mine + 1]), 0u, uint32_t(K) + m.S[K], inter);
                const int id = __float_as_int(bi.w);
                const int owner = id / per;
                cluster.map_shared_rank(m.frep, owner)[id - owner * per] = fr;
            }
            inter_total += inter;
        } else if (node) {
            p = m.pos[mine];
            if (!is_long) fa = cached ? small_short_row(rb, re, p, entry_cached) : small_short_row(rb, re, p, entry_global);
        }
        if (small_rows_left(m, m.longs)) {
            if (cached) small_long_rows(m, lo, row_cached); else small_long_rows(m, lo, row_global);
        }
        cluster.sync();  // the repulsions have arrived
        float2 st = make_float2(0.0f, 0.0f);
        if (node) {
            if (is_long) fa = m.w.fa[tid];
            f = force_sum(fa, mass, p, m.frep[mine - lo], A.kg, A.strong);
            st = swing_traction(mass, f.x, f.y, fp.x, fp.y);
        }
        if (!walker) {
            const XSum S = xsum_warp_terms(st.x), T = xsum_warp_terms(st.y);
            if (lane < C) {
                XPart(*to)[2] = cluster.map_shared_rank(m.u.xpart, lane) + rank * kSmallSums + warp;
                (*to)[0] = xsum_pack(S);
                (*to)[1] = xsum_pack(T);
            }
        }
        cluster.sync();  // every block's sums, and nobody reads positions any more
        if (tid == 0) m.next = 0u;
        if (warp == 0) {
            auto part = [&](int q, int k) {
                if (q >= C * kSmallSums) return xsum_zero();
                const XPart &x = m.u.xpart[q][k];
                return XSum{(u128(x.hi) << 64) | x.lo, x.q0, x.bad};
            };
            const XSum S = xsum_warp_merge(part(lane, 0), part(lane + 32, 0));
            const XSum T = xsum_warp_merge(part(lane, 1), part(lane + 32, 1));
            Ssum = xsum_value(S);
            Tsum = xsum_value(T);
            const double sp = speed_update(m.speed, Ssum, Tsum, A.tau);
            __syncwarp();
            if (lane == 0) m.speed = sp;
        }
        __syncthreads();
        if (node) {
            p = displaced(p, f, fp, float(m.speed), A.ks, A.ksmax);
            fp = f;
            for (int q = 0; q < C; ++q) cluster.map_shared_rank(m.pos, q)[mine] = p;
        }
        cluster.sync();  // the new positions have arrived
    }
    if (node) {
        A.pos[k0 + mine] = m.pos[mine];
        A.F[k0 + mine] = f;
        A.Fprev[k0 + mine] = fp;
    }
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) {
        inter += __shfl_xor_sync(0xFFFFFFFFu, inter, d);
        inter_total += __shfl_xor_sync(0xFFFFFFFFu, inter_total, d);
    }
    if (lane == 0 && inter_total) {
        atomicAdd(&A.hdr->interactions, static_cast<unsigned long long>(inter));
        atomicAdd(&A.hdr->interactions_total, inter_total);
    }
    if (tid == 0 && rank == 0) {
        A.speed[g] = m.speed;
        atomicAdd(&A.hdr->tree_nodes, static_cast<unsigned long long>(cells));
        if (g == 0) {
            A.hdr->S = Ssum;
            A.hdr->T = Tsum;
            A.hdr->steps_total += static_cast<unsigned long long>(A.iterations);
        }
    }
}

}  // namespace
}  // namespace bgv
