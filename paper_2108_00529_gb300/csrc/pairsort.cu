// pairsort.cu -- the (row, col) pairs of all cut edges, in both directions, as
// sorted 64-bit keys row << b | col (Section 4.1: the superedges and the CSR
// the attraction reads), b = bits of the supernode ids.
//
// An LSD sort of the 68 M keys of a 34 M-edge graph moves every key six times
// through HBM and ranks it stably six times (3.3 ms on GB300, after 0.4 ms
// to write the keys).  Keys are all that is sorted, so equal keys need no order
// and no pass has to be stable: a key goes to its place with one shared-memory
// atomic per level, and two levels suffice.
//   1. k_ps_hist     counts the keys' top 15 bits (32,768 fine bins in shared
//                    memory), straight from the edge list
//   2. k_ps_plan     groups neighbouring fine bins into buckets that one block
//                    sorts in shared memory (at most kPsW keys and rows); a bin
//                    larger than that is an oversize bucket of its own
//   3. k_ps_coarse   reads the edges again and writes each key to one of 256 runs
//      k_ps_place    of neighbouring buckets, then from there to its bucket: a
//                    tile of 8,192 keys orders its keys in shared memory first, so
//                    that they leave in long pieces
//   4. k_ps_sort     one block per oversize bucket (the hubs of a skewed graph)
//                    splits it by the next 15 bits of its keys (ps_split), beside
//                    the other buckets; the pieces take a second launch
//                    One block per bucket sorts it: bins per row (and per part of a long
//                    row) by shared-memory atomics, then every key's rank inside
//                    its bin, which holds a few keys; bins that hold many keys
//                    go through a bitonic network
// A bucket of keys that only differ below the splits' 30 bits is counted out
// (k_ps_sort), and a bucket of equal keys needs no sorting.  When one fine bin
// holds more than kPsGiant keys, or too many equal top bits are left, *guard is
// set and the caller sorts the keys with the LSD sort instead; the decision
// stays on the device.
// Supergraph of 34 M R-MAT edges (68 M keys): 4.62 ms with the LSD sort, 2.36 with
// this (and one pass less over the sorted keys); whole-graph CSR of 8 M edges 1.09
// and 0.62 ms.  The 68 M keys: histogram 75 us, plan 36, moves 277 and 304, split
// 185, sort 832 (instruction issue: about 260 thread instructions a key).
#include "bgv_internal.cuh"
#include "pieces.cuh"

namespace bgv {
namespace {
constexpr int kThreads = 1024;
constexpr int kFineBits = 15;
constexpr int kFine = 1 << kFineBits;
constexpr uint32_t kPsW = 24576;       // keys plus rows (primaries) a block sorts in shared memory
constexpr uint32_t kPsT = kPsW / 2;    // small bins are grouped up to this weight (and one bin more)
constexpr uint32_t kPsGiant = 1u << 21;
constexpr int kPsMaxPrim = 2048;       // primaries of a bucket whose bins are parts of rows
constexpr int kPsRank = 32;            // bins up to this size are ranked by counting
constexpr int kPsWarpBin = 1024;       // bins up to this size are sorted by one warp
constexpr int kPsMaxSlices = 64;       // 15-bit slices of a bucket that is counted out

enum : uint32_t { kSrcSplit = 1u, kEqual = 2u };
// a bin's rows stay a fraction of kPsT, and every low part of a key fits 32 bits
static_assert((1u << (kPairSortBits - kFineBits)) < kPsT, "rows of one fine bin");

__device__ __forceinline__ int key_bits(int64_t K) {  // bits_for(K)
    return K <= 2 ? 1 : 64 - __clzll(K - 1);
}
__device__ __forceinline__ int fine_shift(int b) { return 2 * b > kFineBits ? 2 * b - kFineBits : 0; }

// Exclusive block scan of one value per thread (kThreads threads).
template <class T>
__device__ __forceinline__ T ps_scan(T x, T *total) {
    __shared__ T wsum[kThreads / 32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    T inc = x;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const T y = __shfl_up_sync(0xFFFFFFFFu, inc, d);
        if (lane >= d) inc += y;
    }
    if (lane == 31) wsum[warp] = inc;
    __syncthreads();
    if (warp == 0) {
        const T w = wsum[lane];
        T wi = w;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const T y = __shfl_up_sync(0xFFFFFFFFu, wi, d);
            if (lane >= d) wi += y;
        }
        wsum[lane] = wi;
    }
    __syncthreads();
    const T r = (warp ? wsum[warp - 1] : T(0)) + inc - x;
    *total = wsum[kThreads / 32 - 1];
    __syncthreads();
    return r;
}

// ---------------------------------------------------------- 1. histogram
__device__ __forceinline__ bool ps_pair(int32_t u, int32_t v, int32_t n, const int32_t *__restrict__ node_map,
                                        bool identity, int32_t *a, int32_t *c, uint32_t *status) {
    if (static_cast<uint32_t>(u) >= static_cast<uint32_t>(n) || static_cast<uint32_t>(v) >= static_cast<uint32_t>(n)) {
        raise_status(status, BGV_DEV_BADEDGE);
        *a = *c = 0;
        return false;
    }
    *a = identity ? u : node_map[u];
    *c = identity ? v : node_map[v];
    return *a != *c;
}

__global__ void __launch_bounds__(kThreads, 1) k_ps_hist(const int32_t *__restrict__ edges, int64_t m, int32_t n,
                                                      const int32_t *__restrict__ node_map, const int64_t *K_dev,
                                                      const uint32_t *moved, int4 *__restrict__ mapped,
                                                      uint32_t *total, uint32_t *status) {
    extern __shared__ uint32_t h[];
    for (int f = threadIdx.x; f < kFine; f += kThreads) h[f] = 0u;
    __syncthreads();
    const int b = key_bits(*K_dev), s1 = fine_shift(b);
    const bool identity = *moved == 0u;  // node_map[v] == v for every node: no gathers
    const int4 *e2 = reinterpret_cast<const int4 *>(edges);
    const int64_t full = m >> 1, pairs = (m + 1) >> 1;
    const int64_t stride = int64_t(gridDim.x) * kThreads;
    constexpr int kIn = 4;
    auto count = [&](int32_t a, int32_t c) {
        const unsigned long long ka = (static_cast<unsigned long long>(uint32_t(a)) << b) | uint32_t(c);
        const unsigned long long kc = (static_cast<unsigned long long>(uint32_t(c)) << b) | uint32_t(a);
        atomicAdd(&h[swz(uint32_t(ka >> s1))], 1u);
        atomicAdd(&h[swz(uint32_t(kc >> s1))], 1u);
    };
    for (int64_t q0 = int64_t(blockIdx.x) * kThreads + threadIdx.x; q0 < pairs; q0 += stride * kIn) {
        int4 e[kIn], t[kIn];
#pragma unroll
        for (int r = 0; r < kIn; ++r) {
            const int64_t q = q0 + r * stride;
            e[r] = q < full ? __ldcs(e2 + q) : make_int4(0, 0, 0, 0);
            if (q >= full && q < pairs) e[r] = make_int4(edges[2 * (m - 1)], edges[2 * (m - 1) + 1], 0, 0);
        }
        bool g0[kIn], g1[kIn];
#pragma unroll
        for (int r = 0; r < kIn; ++r) {
            const bool in = q0 + r * stride < pairs;
            g0[r] = in && ps_pair(e[r].x, e[r].y, n, node_map, identity, &t[r].x, &t[r].y, status);
            g1[r] = in && ps_pair(e[r].z, e[r].w, n, node_map, identity, &t[r].z, &t[r].w, status);
        }
#pragma unroll
        for (int r = 0; r < kIn; ++r) {
            const int64_t q = q0 + r * stride;
            if (q < pairs && !identity) mapped[q] = t[r];
            if (g0[r]) count(t[r].x, t[r].y);
            if (g1[r]) count(t[r].z, t[r].w);
        }
    }
    __syncthreads();
    for (int f = threadIdx.x; f < kFine; f += kThreads) {
        const uint32_t c = h[swz(f)];
        if (c) atomicAdd(&total[f], c);
    }
}

// --------------------------------------------------------------- 2. plan
// Grouping of NF neighbouring bins by their counts (any memory): bins heavier
// than kPsT stand alone, runs of others share a group as long as the group's
// first kPsT of weight lasts.  With B = weight of the small bins before f and G
// = heavy bins before f, the group of f is B / kPsT + 2 G (+ 1 if heavy), which
// never falls along f; the bins where it changes start the groups.  Calls
// head(group index, bin, keys before bin) for every group and returns the
// number of groups; keys before bin f go to prefix(f, keys).
template <class Count, class Prefix, class Head>
__device__ __forceinline__ uint32_t ps_groups(int NF, uint32_t rows_per_bin, uint32_t key0, Count count, Prefix prefix,
                                              Head head) {
    __shared__ uint32_t last_id[kThreads];
    constexpr int kPer = kFine / kThreads;
    const int f0 = threadIdx.x * kPer, f1 = min(f0 + kPer, NF);
    unsigned long long keys = 0, small = 0, heavy = 0;
    for (int f = f0; f < f1; ++f) {
        const uint32_t c = count(f);
        const unsigned long long w = static_cast<unsigned long long>(c) + rows_per_bin;
        keys += c;
        if (w > kPsT) heavy += 1; else small += w;
    }
    unsigned long long tot;
    const unsigned long long key_pre = ps_scan<unsigned long long>(keys, &tot) + key0;
    const unsigned long long small_pre = ps_scan<unsigned long long>(small, &tot);
    const unsigned long long heavy_pre = ps_scan<unsigned long long>(heavy, &tot);
    auto walk = [&](auto each) {  // each(f, id, keys before f)
        unsigned long long k = key_pre, s = small_pre, g = heavy_pre;
        for (int f = f0; f < f1; ++f) {
            const uint32_t c = count(f);
            const unsigned long long w = static_cast<unsigned long long>(c) + rows_per_bin;
            const bool hv = w > kPsT;
            each(f, uint32_t(s / kPsT + 2 * g + (hv ? 1 : 0)), uint32_t(k));
            k += c;
            if (hv) g += 1; else s += w;
        }
    };
    uint32_t id = 0xFFFFFFFFu, heads = 0;
    walk([&](int, uint32_t x, uint32_t) {
        if (id != 0xFFFFFFFFu && x != id) ++heads;
        id = x;
    });
    last_id[threadIdx.x] = id;
    __syncthreads();
    // the first bin of a thread starts a group unless the bin before it (the
    // previous thread's last) has the same id
    uint32_t before = threadIdx.x ? last_id[threadIdx.x - 1] : 0xFFFFFFFFu;
    uint32_t first = 0xFFFFFFFFu;
    walk([&](int, uint32_t x, uint32_t) { first = first == 0xFFFFFFFFu ? x : first; });
    if (first != 0xFFFFFFFFu && first != before) ++heads;
    uint32_t groups;
    uint32_t at = ps_scan<uint32_t>(heads, &groups);
    id = before;
    walk([&](int f, uint32_t x, uint32_t k) {
        if (x != id) {
            head(at, f, k);
            ++at;
        }
        id = x;
        prefix(f, k, at - 1);
    });
    __syncthreads();
    return groups;
}

__device__ __forceinline__ void ps_append(const PsBucket &e, PsControl *ctl, PsBucket *list, uint32_t cap) {
    const uint32_t at = atomicAdd(&ctl->buckets, 1u);
    if (at < cap)
        list[at] = e;
    else
        ctl->guard = 1u;  // cannot happen (the list is sized for every group); the LSD sort takes over
}
// Equal keys need no sorting, only a place: shared out in pieces.
__device__ __forceinline__ void ps_append_equal(PsBucket e, PsControl *ctl, PsBucket *list, uint32_t cap) {
    const uint32_t start = e.start, end = e.start + e.count, pieces = pieces_of(e.count, kPsW);
    e.flags |= kEqual;
    for (uint32_t p = 0; p < pieces; ++p) {
        e.start = start + p * kPsW;
        e.count = piece_size(e.start, end, kPsW);
        ps_append(e, ctl, list, cap);
    }
}

constexpr int kCoarse = 256;  // runs of buckets, at most 128 buckets each
// Groups of one run; run c holds groups [c * per, c * per + per).
__device__ __forceinline__ uint32_t groups_per_run(uint32_t groups) {
    return groups > uint32_t(kCoarse) ? (groups + kCoarse - 1) / kCoarse : 1u;
}

// One block.  ctl and list counters are zero before.  Bound by the latency of its
// passes (the bins' groups go out through shared memory: written by the threads
// that walk the bins, 32 apart, they took 20 us more).
__global__ void __launch_bounds__(kThreads, 1) k_ps_plan(const uint32_t *__restrict__ total, const int64_t *K_dev,
                                                      PsControl *ctl, uint32_t *__restrict__ bstart,
                                                      uint32_t *__restrict__ bfine, uint16_t *__restrict__ bmap,
                                                      uint32_t *__restrict__ cursor, uint32_t *__restrict__ run_cursor,
                                                      PsBucket *list, uint32_t list_cap,
                                                      PsBucket *over, uint32_t over_cap, unsigned long long *nkeys) {
    const int64_t K = *K_dev;
    const int b = key_bits(K), s1 = fine_shift(b);
    const int NF = K > 0 ? int((((static_cast<unsigned long long>(K) << b) - 1) >> s1) + 1) : 1;
    const uint32_t rows_per_bin = s1 >= b ? 1u << (s1 - b) : 0u;
    extern __shared__ uint32_t c_sh[];  // [kFine] the counts: the grouping walks them several times
    uint32_t mine = 0;
    for (int f = threadIdx.x; f < kFine; f += kThreads) {
        const uint32_t c = f < NF ? total[f] : 0u;
        c_sh[swz(f)] = c;
        mine += c;
    }
    uint32_t all;
    ps_scan<uint32_t>(mine, &all);
    const uint32_t groups = ps_groups(
        NF, rows_per_bin, 0u, [&](int f) { return c_sh[swz(f)]; },
        [&](int f, uint32_t, uint32_t g) { c_sh[swz(f)] = g; },  // its count has been read for the last time
        [&](uint32_t g, int f, uint32_t k) {
            bstart[g] = k;
            bfine[g] = uint32_t(f);
            cursor[g] = k;
        });
    if (threadIdx.x == 0) {
        ctl->groups = groups;
        *nkeys = all;
    }
    __syncthreads();
    for (int f = threadIdx.x; f < NF; f += kThreads) bmap[f] = uint16_t(c_sh[swz(f)]);
    if (threadIdx.x < kCoarse) {
        const uint32_t g = threadIdx.x * groups_per_run(groups);
        run_cursor[threadIdx.x] = g < groups ? bstart[g] : all;
    }
    for (uint32_t g = threadIdx.x; g < groups; g += kThreads) {
        const uint32_t f0 = bfine[g], f1 = g + 1 < groups ? bfine[g + 1] : uint32_t(NF);
        const uint32_t k0 = bstart[g], k1 = g + 1 < groups ? bstart[g + 1] : all;
        if (k1 == k0) continue;
        PsBucket e{k0, k1 - k0, static_cast<unsigned long long>(f0) << s1,
                   static_cast<unsigned long long>(f1 - f0) << s1, 0u, 0u};
        if (f1 - f0 == 1 && s1 == 0) {
            ps_append_equal(e, ctl, list, list_cap);
        } else if (static_cast<unsigned long long>(e.count) + (f1 - f0) * static_cast<unsigned long long>(rows_per_bin) <=
                   kPsW) {
            ps_append(e, ctl, list, list_cap);
        } else {
            // more than kPsW: a single bin, as groups of small ones stay within 2 kPsT
            if (e.count > kPsGiant) ctl->guard = 1u;
            const uint32_t at = atomicAdd(&ctl->over, 1u);
            if (at < over_cap)
                over[at] = e;
            else
                ctl->guard = 1u;
        }
    }
    __syncthreads();
    if (threadIdx.x == 0) ctl->planned = atomicAdd(&ctl->buckets, 0u);
}

// -------------------------------------------------------------- 3. moves
// A tile of kMoveKeys keys is ordered by destination in shared memory and written
// in pieces: about 32 keys to a run of buckets, then about a hundred to a bucket.
// (Written straight to thousands of buckets, a few keys each, the store requests
// -- one 8-byte piece of a sector at a time -- and the phases that one large
// block per SM cannot overlap took 1,215 us for 68 M keys; these two take 277 and 304.)
constexpr int kMoveThreads = 512;
constexpr int kMoveIn = 16;   // keys per thread
constexpr int kMoveKeys = kMoveThreads * kMoveIn;
static_assert(kFine / kCoarse <= kCoarse && kMoveKeys < 65536, "ranks in 16 bits");

struct MoveBins {
    uint32_t cnt[kCoarse + 32];   // keys per bin, then their first place in the tile; the last 32: no keys
    uint32_t delta[kCoarse];      // from a place in the tile to the place in the output
    uint32_t wsum[kMoveThreads / 32];
    uint32_t total;
};

// Counts to places, and room in the output for every bin; ends in a barrier.
__device__ void ps_move_plan(MoveBins &mb, int bins, uint32_t *cursor) {
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    const uint32_t c = t < bins ? mb.cnt[t] : 0u;
    const uint32_t room = c ? atomicAdd(&cursor[t], c) : 0u;
    uint32_t inc = c;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, inc, d);
        if (lane >= d) inc += y;
    }
    if (lane == 31) mb.wsum[warp] = inc;
    __syncthreads();
    const uint32_t start = __reduce_add_sync(0xFFFFFFFFu, lane < warp ? mb.wsum[lane] : 0u) + inc - c;
    if (t < bins) {
        mb.cnt[t] = start;
        mb.delta[t] = room - start;
    }
    if (t == kMoveThreads - 1) mb.total = start + c;
    __syncthreads();
}

// The tile's keys out of `stage`, which holds them by bin; ends in a barrier.
template <class BinOf>
__device__ void ps_move_out(const MoveBins &mb, const unsigned long long *stage, BinOf bin_of,
                            unsigned long long *__restrict__ out, int64_t cap) {
    const uint32_t total = mb.total;
#pragma unroll 4
    for (uint32_t i = threadIdx.x; i < total; i += kMoveThreads) {
        const unsigned long long key = stage[i];
        const uint32_t to = mb.delta[bin_of(key)] + i;
        if (to < cap) out[to] = key;
    }
    __syncthreads();
}

constexpr size_t kCoarseSmem = size_t(kMoveKeys) * sizeof(unsigned long long) + kFine;
constexpr size_t kPlaceSmem = size_t(kMoveKeys) * sizeof(unsigned long long);

__global__ void __launch_bounds__(kMoveThreads, 2) k_ps_coarse(const int32_t *__restrict__ edges, int64_t m, int32_t n,
                                                            const int64_t *K_dev, const uint32_t *moved,
                                                            const int4 *__restrict__ mapped,
                                                            const uint16_t *__restrict__ bmap, uint32_t *run_cursor,
                                                            const PsControl *ctl,
                                                            unsigned long long *__restrict__ out, int64_t cap) {
    if (ctl->guard) return;
    extern __shared__ __align__(16) unsigned long long stage[];  // [kMoveKeys], then the fine bins' runs (bytes)
    __shared__ MoveBins mb;
    uint8_t *run_of = reinterpret_cast<uint8_t *>(stage + kMoveKeys);
    const int64_t K = *K_dev;
    const int b = key_bits(K), s1 = fine_shift(b);
    const int NF = K > 0 ? int((((static_cast<unsigned long long>(K) << b) - 1) >> s1) + 1) : 1;
    const uint32_t per = groups_per_run(ctl->groups);
    for (int f = threadIdx.x; f < NF; f += kMoveThreads) run_of[f] = uint8_t(bmap[f] / per);
    const bool identity = *moved == 0u;
    const int4 *e2 = identity ? reinterpret_cast<const int4 *>(edges) : mapped;
    const int64_t full = identity ? m >> 1 : (m + 1) >> 1, pairs = (m + 1) >> 1;
    // a pair in one supernode, and a bad endpoint (stored as a loop, or out of range here), has no keys
    auto has_keys = [&](int32_t a, int32_t c) {
        return a != c && static_cast<uint32_t>(a) < static_cast<uint32_t>(n) &&
               static_cast<uint32_t>(c) < static_cast<uint32_t>(n);
    };
    auto key_of = [&](int32_t a, int32_t c) {
        return (static_cast<unsigned long long>(uint32_t(a)) << b) | uint32_t(c);
    };
    constexpr int kIn = kMoveIn / 4;  // two edges, four keys
    int4 e[kIn];
    auto load = [&](int64_t p0) {
#pragma unroll
        for (int r = 0; r < kIn; ++r) {
            const int64_t q = p0 + r * kMoveThreads + threadIdx.x;
            e[r] = q < full ? __ldcs(e2 + q) : make_int4(0, 0, 0, 0);
            if (q >= full && q < pairs) e[r] = make_int4(edges[2 * (m - 1)], edges[2 * (m - 1) + 1], 0, 0);
        }
    };
    constexpr int64_t kPairs = kMoveKeys / 4;  // int4 pairs per tile
    int64_t p0 = int64_t(blockIdx.x) * kPairs;
    if (p0 < pairs) load(p0);
    while (p0 < pairs) {
        if (threadIdx.x < kCoarse) mb.cnt[threadIdx.x] = 0u;
        __syncthreads();
        // every key's run (no keys: one of the last 32 counters) and its rank there
        uint32_t at[kMoveIn];
        const uint32_t none = kCoarse + (threadIdx.x & 31);
#pragma unroll
        for (int r = 0; r < kIn; ++r) {
            const bool ok0 = has_keys(e[r].x, e[r].y), ok1 = has_keys(e[r].z, e[r].w);
            at[4 * r] = ok0 ? run_of[uint32_t(key_of(e[r].x, e[r].y) >> s1)] : none;
            at[4 * r + 1] = ok0 ? run_of[uint32_t(key_of(e[r].y, e[r].x) >> s1)] : none;
            at[4 * r + 2] = ok1 ? run_of[uint32_t(key_of(e[r].z, e[r].w) >> s1)] : none;
            at[4 * r + 3] = ok1 ? run_of[uint32_t(key_of(e[r].w, e[r].z) >> s1)] : none;
        }
#pragma unroll
        for (int k = 0; k < kMoveIn; ++k) at[k] |= atomicAdd(&mb.cnt[at[k]], 1u) << 16;
        __syncthreads();
        ps_move_plan(mb, kCoarse, run_cursor);
        auto put = [&](uint32_t x, int32_t a, int32_t c) {
            const uint32_t r = x & 0xFFFFu;
            if (r < kCoarse) stage[mb.cnt[r] + (x >> 16)] = key_of(a, c);
        };
#pragma unroll
        for (int r = 0; r < kIn; ++r) {
            put(at[4 * r], e[r].x, e[r].y);
            put(at[4 * r + 1], e[r].y, e[r].x);
            put(at[4 * r + 2], e[r].z, e[r].w);
            put(at[4 * r + 3], e[r].w, e[r].z);
        }
        p0 += int64_t(gridDim.x) * kPairs;
        if (p0 < pairs) load(p0);  // in flight while this tile is written
        __syncthreads();
        ps_move_out(mb, stage, [&](unsigned long long key) { return uint32_t(run_of[uint32_t(key >> s1)]); }, out, cap);
    }
}

// run_cursor: the ends of the runs, as k_ps_coarse leaves it.
__global__ void __launch_bounds__(kMoveThreads, 2) k_ps_place(const unsigned long long *__restrict__ in,
                                                           const int64_t *K_dev, const uint16_t *__restrict__ bmap,
                                                           const uint32_t *__restrict__ bstart,
                                                           const uint32_t *__restrict__ run_cursor,
                                                           const PsControl *ctl, uint32_t *cursor,
                                                           unsigned long long *__restrict__ out, int64_t cap) {
    if (ctl->guard) return;
    extern __shared__ __align__(16) unsigned long long stage[];
    __shared__ MoveBins mb;
    __shared__ uint32_t tiles_before[kCoarse + 1], run_start[kCoarse], run_end[kCoarse];
    const int s1 = fine_shift(key_bits(*K_dev));
    const uint32_t groups = ctl->groups, per = groups_per_run(groups);
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    {  // tiles of every run
        uint32_t tiles = 0u;
        if (t < kCoarse && uint32_t(t) * per < groups) {
            run_start[t] = bstart[t * per];
            run_end[t] = run_cursor[t];
            tiles = pieces_of(run_end[t] - run_start[t], kMoveKeys);
        }
        uint32_t inc = tiles;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, inc, d);
            if (lane >= d) inc += y;
        }
        if (lane == 31) mb.wsum[warp] = inc;
        __syncthreads();
        inc += __reduce_add_sync(0xFFFFFFFFu, lane < warp ? mb.wsum[lane] : 0u);
        if (t < kCoarse) tiles_before[t + 1] = inc;
        if (t == 0) tiles_before[0] = 0u;
        __syncthreads();
    }
    const uint32_t all = tiles_before[kCoarse];
    for (uint32_t tile = blockIdx.x; tile < all; tile += gridDim.x) {
        int c = 0;  // the last run that starts at or before the tile
#pragma unroll
        for (int d = kCoarse / 2; d > 0; d >>= 1)
            if (tiles_before[c + d] <= tile) c += d;
        const uint32_t k0 = run_start[c] + (tile - tiles_before[c]) * kMoveKeys;
        const uint32_t count = min(uint32_t(kMoveKeys), run_end[c] - k0);
        const uint32_t g0 = uint32_t(c) * per;
        const int bins = int(min(per, groups - g0));
        if (t < kCoarse) mb.cnt[t] = 0u;
        unsigned long long k[kMoveIn];
#pragma unroll
        for (int r = 0; r < kMoveIn; ++r) {
            const uint32_t i = r * kMoveThreads + t;
            k[r] = i < count ? __ldcs(in + k0 + i) : 0ull;
        }
        __syncthreads();
        uint32_t at[kMoveIn];
#pragma unroll
        for (int r = 0; r < kMoveIn; ++r) {
            const bool ok = uint32_t(r * kMoveThreads + t) < count;
            at[r] = ok ? uint32_t(__ldg(bmap + uint32_t(k[r] >> s1))) - g0 : uint32_t(kCoarse + lane);
        }
#pragma unroll
        for (int r = 0; r < kMoveIn; ++r) {
            // a large bucket fills whole tiles: one add for a warp of its keys
            const uint32_t first = __shfl_sync(0xFFFFFFFFu, at[r], 0);
            uint32_t rank;
            if (__all_sync(0xFFFFFFFFu, at[r] == first)) {
                uint32_t base = 0u;
                if (lane == 0) base = atomicAdd(&mb.cnt[first], 32u);
                rank = __shfl_sync(0xFFFFFFFFu, base, 0) + lane;
            } else {
                rank = atomicAdd(&mb.cnt[at[r]], 1u);
            }
            at[r] |= rank << 16;
        }
        __syncthreads();
        ps_move_plan(mb, bins, cursor + g0);
#pragma unroll
        for (int r = 0; r < kMoveIn; ++r) {
            const uint32_t x = at[r] & 0xFFFFu;
            if (x < kCoarse) stage[mb.cnt[x] + (at[r] >> 16)] = k[r];
        }
        __syncthreads();
        ps_move_out(mb, stage, [&](unsigned long long key) { return uint32_t(__ldg(bmap + uint32_t(key >> s1))) - g0; }, out,
                    cap);
    }
}

// -------------------------------------------------------------- 4. split
// Oversize buckets (one fine bin each): counted by the next 15 bits of their
// keys, grouped as above, and moved bin by bin from `in` to the same range of
// `out`.  One block per bucket; a bucket has at most kPsGiant keys.
constexpr int kSplitGroups = 2048;  // of one bucket: at most 3 kPsGiant / kPsT + 4
// h: [kFine] counts, then cursors; after them [2 * kSplitGroups].  Every thread of
// the block calls it; ends in a barrier.
__device__ void ps_split(const PsBucket &o, int b, const unsigned long long *__restrict__ in,
                         unsigned long long *__restrict__ out, PsControl *ctl, PsBucket *list, uint32_t list_cap,
                         uint32_t *h) {
    uint32_t *gstart = h + kFine, *gfine = gstart + kSplitGroups;
    const int s1 = fine_shift(b), s2 = s1 > kFineBits ? s1 - kFineBits : 0;
    const uint32_t rows_per_bin = s2 >= b ? 1u << (s2 - b) : 0u;
    const int NF = int(o.span >> s2);  // a power of two up to kFine
    for (int f = threadIdx.x; f < kFine; f += kThreads) h[f] = 0u;
    __syncthreads();
    const unsigned long long *src = in + o.start;
    constexpr int kIn = 8;
    for (uint32_t i0 = threadIdx.x; i0 < o.count; i0 += kThreads * kIn) {
        unsigned long long k[kIn];
#pragma unroll
        for (int r = 0; r < kIn; ++r) k[r] = i0 + r * kThreads < o.count ? src[i0 + r * kThreads] : o.lo;
#pragma unroll
        for (int r = 0; r < kIn; ++r)
            if (i0 + r * kThreads < o.count) atomicAdd(&h[swz(uint32_t((k[r] - o.lo) >> s2) & (kFine - 1))], 1u);
    }
    __syncthreads();
    const uint32_t groups = ps_groups(
        NF, rows_per_bin, 0u, [&](int f) { return h[swz(f)]; }, [&](int, uint32_t, uint32_t) {},
        [&](uint32_t g, int f, uint32_t k) {
            if (g < kSplitGroups) {
                gstart[g] = k;
                gfine[g] = uint32_t(f);
            }
        });
    if (groups > kSplitGroups) {  // cannot happen, see kSplitGroups
        if (threadIdx.x == 0) ctl->guard = 1u;
        return;
    }
    for (uint32_t g = threadIdx.x; g < groups; g += kThreads) {
        const uint32_t f0 = gfine[g], f1 = g + 1 < groups ? gfine[g + 1] : uint32_t(NF);
        const uint32_t k0 = gstart[g], k1 = g + 1 < groups ? gstart[g + 1] : o.count;
        if (k1 == k0) continue;
        PsBucket e{o.start + k0, k1 - k0, o.lo + (static_cast<unsigned long long>(f0) << s2),
                   static_cast<unsigned long long>(f1 - f0) << s2, kSrcSplit, 0u};
        if (f1 - f0 == 1 && s2 == 0) continue;  // equal keys, in their place already
        if (e.count > kPsW && s2 > kFineBits && (1 << (s2 - kFineBits)) > kPsMaxSlices) ctl->guard = 1u;
        ps_append(e, ctl, list, list_cap);
    }
    __syncthreads();
    // counts -> exclusive prefix (a cursor per bin), then every key to its bin
    constexpr int kPer = kFine / kThreads;
    uint32_t sum = 0, all;
    for (int f = 0; f < kPer; ++f) sum += h[swz(threadIdx.x * kPer + f)];
    uint32_t run = ps_scan<uint32_t>(sum, &all);
    for (int f = 0; f < kPer; ++f) {
        uint32_t &x = h[swz(threadIdx.x * kPer + f)];
        const uint32_t c = x;
        x = run;
        run += c;
    }
    __syncthreads();
    unsigned long long *dst = out + o.start;
    for (uint32_t i0 = threadIdx.x; i0 < o.count; i0 += kThreads * kIn) {
        unsigned long long k[kIn];
#pragma unroll
        for (int r = 0; r < kIn; ++r) k[r] = i0 + r * kThreads < o.count ? src[i0 + r * kThreads] : o.lo;
#pragma unroll
        for (int r = 0; r < kIn; ++r)
            if (i0 + r * kThreads < o.count) {
                const uint32_t pos = atomicAdd(&h[swz(uint32_t((k[r] - o.lo) >> s2) & (kFine - 1))], 1u);
                if (pos < o.count) dst[pos] = k[r];
            }
    }
    __syncthreads();
}

// --------------------------------------------------------------- 5. sort
// Ascending bitonic network on v[0, n), over the threads t = 0 .. T-1 of one
// warp (kWarp) or the block: every comparator puts the smaller value first, so
// places past n count as +infinity and stay away.
template <bool kWarp>
__device__ void ps_bitonic(uint32_t *v, int n) {
    const int t = kWarp ? (threadIdx.x & 31) : threadIdx.x, T = kWarp ? 32 : kThreads;
    int lg = 1;  // a network over 2^lg places
    while ((1 << lg) < n) ++lg;
    const int pairs = 1 << (lg - 1);
    auto exchange = [&](int i, int j) {
        if (j >= n) return;
        const uint32_t x = v[i], y = v[j];
        if (x > y) {
            v[i] = y;
            v[j] = x;
        }
    };
    auto sync = [&]() {
        if (kWarp) __syncwarp(); else __syncthreads();
    };
    for (int l = 1; l <= lg; ++l) {
        const int half = 1 << (l - 1);
        for (int q = t; q < pairs; q += T) {
            const int base = (q >> (l - 1)) << l, off = q & (half - 1);
            exchange(base + off, base + 2 * half - 1 - off);
        }
        sync();
        for (int j = l - 2; j >= 0; --j) {
            for (int q = t; q < pairs; q += T) {
                const int i = ((q >> j) << (j + 1)) + (q & ((1 << j) - 1));
                exchange(i, i + (1 << j));
            }
            sync();
        }
    }
}

// A bucket of more than kPsW keys whose keys share all but their lowest bits:
// counted in slices of 2^15 key values and written out in order (through `tmp`,
// as the keys stay in `buf` until the last slice is counted).
__device__ void ps_count_out(const PsBucket &e, unsigned long long *buf, unsigned long long *tmp, uint32_t *h) {
    constexpr int kPer = kFine / kThreads;
    uint32_t done = 0;
    for (unsigned long long s0 = 0; s0 < e.span; s0 += kFine) {
        for (int f = threadIdx.x; f < kFine; f += kThreads) h[f] = 0u;
        __syncthreads();
        for (uint32_t i = threadIdx.x; i < e.count; i += kThreads) {
            const unsigned long long rel = buf[e.start + i] - e.lo - s0;  // wraps below the slice
            if (rel < kFine) atomicAdd(&h[uint32_t(rel)], 1u);
        }
        __syncthreads();
        uint32_t sum = 0, all;
        for (int f = 0; f < kPer; ++f) sum += h[threadIdx.x * kPer + f];
        const uint32_t pre = ps_scan<uint32_t>(sum, &all);
        uint32_t run = done + pre;
        for (int f = 0; f < kPer; ++f) {  // exclusive starts
            const uint32_t c = h[threadIdx.x * kPer + f];
            h[threadIdx.x * kPer + f] = run;
            run += c;
        }
        __syncthreads();
        // every output place finds its key: the last bin that starts at or before it
        for (uint32_t i = done + threadIdx.x; i < done + all; i += kThreads) {
            int lo = 0, hi = kFine;
            while (hi - lo > 1) {
                const int mid = (lo + hi) >> 1;
                if (h[mid] <= i) lo = mid; else hi = mid;
            }
            if (i < e.count) tmp[e.start + i] = e.lo + s0 + uint32_t(lo);
        }
        done += all;
        __syncthreads();
    }
    for (uint32_t i = threadIdx.x; i < e.count; i += kThreads) buf[e.start + i] = tmp[e.start + i];
    __syncthreads();
}

// kSplit: the splits of the oversize buckets first, then the buckets listed before
// them; else the buckets that the splits have listed.  The largest hub takes one
// block as long as hundreds of small buckets, which the other blocks sort
// meanwhile; nothing waits for anything inside a launch.  (As a kernel of its own
// the split of a 34 M-edge R-MAT graph took 185 us, nearly all of it one hub.)
template <bool kSplit>
__global__ void __launch_bounds__(kThreads, 1) k_ps_sort(unsigned long long *buf0, unsigned long long *buf1,
                                                      const int64_t *K_dev, PsControl *ctl, PsBucket *list,
                                                      uint32_t list_cap, const PsBucket *__restrict__ over) {
    extern __shared__ uint32_t smem[];
    __shared__ uint32_t big[kPsW / (kPsRank + 1) + 1];  // bins too large to rank: start | size << 16
    __shared__ uint32_t bigs, next_sh, low_min, low_max;
    const int b = key_bits(*K_dev), s1 = fine_shift(b);
    const uint32_t splits = kSplit ? ctl->over : 0u, planned = ctl->planned;
    const uint32_t count = kSplit ? splits + min(planned, list_cap) : min(ctl->buckets, list_cap) - min(planned, list_cap);
    while (true) {
        if (threadIdx.x == 0) {
            // a split in another block may set the guard at any time: one thread
            // reads it, so that a block goes on or ends as a whole
            const bool off = *static_cast<volatile uint32_t *>(&ctl->guard) != 0u;
            next_sh = off ? 0xFFFFFFFFu : atomicAdd(kSplit ? &ctl->split_ticket : &ctl->ticket, 1u);
            bigs = 0u;
            low_min = 0xFFFFFFFFu;
            low_max = 0u;
        }
        __syncthreads();
        uint32_t q = next_sh;
        if (q >= count) return;
        if (kSplit && q < splits) {
            ps_split(over[q], b, buf1, buf0, ctl, list, list_cap, smem);
            continue;
        }
        q = kSplit ? q - splits : q + planned;
        const PsBucket e = list[q];
        const unsigned long long *in = ((e.flags & kSrcSplit) ? buf0 : buf1) + e.start;
        unsigned long long *out = buf0 + e.start;
        const int n = int(e.count);
        if (e.flags & kEqual) {
            for (int i = threadIdx.x; i < n; i += kThreads) out[i] = in[i];
            __syncthreads();
            continue;
        }
        if (e.count > kPsW) {  // only buckets of the split: their keys are in buf0
            ps_count_out(e, buf0, buf1, smem);
            continue;
        }
        // primary = high part of the key inside the bucket: its row, or a part of
        // a row when bins are smaller than rows
        int p = b;
        if ((e.flags & kSrcSplit) || s1 < b) {
            p = 0;
            while (((e.span - 1) >> p) + 1 > kPsMaxPrim) ++p;  // at most 30: ids have at most kPairSortBits bits
        }
        const int P = int((e.span - 1) >> p) + 1, P2 = (P + 1023) & ~1023;
        uint32_t *sec = smem;                                        // [n] low parts of the keys, in bin order
        uint16_t *prim = reinterpret_cast<uint16_t *>(smem + n);     // [n] their primaries
        uint32_t *pcnt = reinterpret_cast<uint32_t *>(prim + n + (n & 1));  // [P2] keys per primary, then its bins
        uint32_t *bins = pcnt + P2;                                  // [n / 2 + P]
        const uint32_t mask = uint32_t((1ull << p) - 1ull);
        constexpr int kIn = 8;
        // f(primary, low part) of every key; the second and third pass find the
        // keys in L2
        auto each_key = [&](auto f) {
            for (int i0 = threadIdx.x; i0 < n; i0 += kThreads * kIn) {
                unsigned long long k[kIn];
#pragma unroll
                for (int r = 0; r < kIn; ++r) k[r] = i0 + r * kThreads < n ? in[i0 + r * kThreads] - e.lo : 0ull;
#pragma unroll
                for (int r = 0; r < kIn; ++r)
                    if (i0 + r * kThreads < n) f(min(uint32_t(k[r] >> p), uint32_t(P - 1)), uint32_t(k[r]) & mask);
            }
        };
        for (int i = threadIdx.x; i < P2; i += kThreads) pcnt[i] = 0u;
        __syncthreads();
        // the range of the low parts: ids that keep to their neighbourhood (graphs side
        // by side, crawls) leave most of the 2^p values out
        uint32_t least = 0xFFFFFFFFu, most = 0u;
        each_key([&](uint32_t pr, uint32_t low) {
            atomicAdd(&pcnt[swz(pr)], 1u);
            least = min(least, low);
            most = max(most, low);
        });
        least = __reduce_min_sync(0xFFFFFFFFu, least);
        most = __reduce_max_sync(0xFFFFFFFFu, most);
        if ((threadIdx.x & 31) == 0) {
            atomicMin(&low_min, least);
            atomicMax(&low_max, most);
        }
        __syncthreads();
        least = low_min;
        const int lb = low_max > least ? 32 - __clz(low_max - least) : 0;  // bits of the range, at most p
        // bins of a primary with c keys: 2^k, about c / 4 (at most c / 2)
        int NB;
        {
            const int per = (P + kThreads - 1) / kThreads;
            const int i0 = min(int(threadIdx.x) * per, P), i1 = min(i0 + per, P);
            uint32_t sum = 0, all;
            for (int i = i0; i < i1; ++i) {
                const uint32_t c = pcnt[swz(i)];
                const int k = c > 4 ? min(32 - __clz((c - 1) >> 2), lb) : 0;
                pcnt[swz(i)] = uint32_t(k) << 24;
                sum += 1u << k;
            }
            uint32_t run = ps_scan<uint32_t>(sum, &all);
            for (int i = i0; i < i1; ++i) {
                const uint32_t k = pcnt[swz(i)] >> 24;
                pcnt[swz(i)] |= run;
                run += 1u << k;
            }
            NB = int(all);
        }
        for (int i = threadIdx.x; i < NB; i += kThreads) bins[i] = 0u;
        __syncthreads();
        auto bin_of = [&](uint32_t pr, uint32_t low, int *k) {
            const uint32_t x = pcnt[swz(pr)];
            *k = int(x >> 24);
            return (x & 0xFFFFFFu) + (*k ? (low - least) >> (lb - *k) : 0u);
        };
        each_key([&](uint32_t pr, uint32_t low) {
            int k;
            atomicAdd(&bins[bin_of(pr, low, &k)], 1u);
        });
        __syncthreads();
        {
            const int per = (NB + kThreads - 1) / kThreads;
            const int i0 = min(int(threadIdx.x) * per, NB), i1 = min(i0 + per, NB);
            uint32_t sum = 0, all;
            for (int i = i0; i < i1; ++i) sum += bins[i];
            uint32_t run = ps_scan<uint32_t>(sum, &all);
            for (int i = i0; i < i1; ++i) {
                const uint32_t c = bins[i];
                bins[i] = run;
                run += c;
            }
        }
        __syncthreads();
        each_key([&](uint32_t pr, uint32_t low) {
            int k;
            const uint32_t s = atomicAdd(&bins[bin_of(pr, low, &k)], 1u);
            sec[s] = low;
            prim[s] = uint16_t(pr);
        });
        __syncthreads();
        // bins[j] is now the end of bin j: rank every key inside its bin (a bin
        // holds one primary, so the low parts decide)
        auto key_of = [&](uint32_t pr, uint32_t low) { return e.lo + (static_cast<unsigned long long>(pr) << p) + low; };
        for (int s = threadIdx.x; s < n; s += kThreads) {
            const uint32_t pr = prim[s], mine = sec[s];
            int k;
            const uint32_t j = bin_of(pr, mine, &k);
            const int lo = j ? int(bins[j - 1]) : 0, hi = int(bins[j]);
            int pos = s;
            if (k < lb) {  // else the bin is one key value
                if (hi - lo > kPsRank) {
                    if (s == lo) big[atomicAdd(&bigs, 1u)] = uint32_t(lo) | (uint32_t(hi - lo) << 16);
                    continue;
                }
                pos = lo;
                for (int t = lo; t < hi; ++t) {
                    const uint32_t o = sec[t];
                    pos += (o < mine || (o == mine && t < s)) ? 1 : 0;
                }
            }
            out[pos] = key_of(pr, mine);
        }
        __syncthreads();
        const uint32_t nb = bigs;
        for (uint32_t w = threadIdx.x >> 5; w < nb; w += kThreads / 32) {
            const int lo = int(big[w] & 0xFFFFu), c = int(big[w] >> 16);
            if (c > kPsWarpBin) continue;
            ps_bitonic<true>(sec + lo, c);
            for (int t = threadIdx.x & 31; t < c; t += 32) out[lo + t] = key_of(prim[lo + t], sec[lo + t]);
        }
        __syncthreads();
        for (uint32_t w = 0; w < nb; ++w) {
            const int lo = int(big[w] & 0xFFFFu), c = int(big[w] >> 16);
            if (c <= kPsWarpBin) continue;
            ps_bitonic<false>(sec + lo, c);
            for (int t = threadIdx.x; t < c; t += kThreads) out[lo + t] = key_of(prim[lo + t], sec[lo + t]);
            __syncthreads();
        }
        __syncthreads();
    }
}

constexpr size_t kHistSmem = size_t(kFine) * sizeof(uint32_t);
// sec and prim (6 bytes a key), bins (2 bytes a key and 4 a primary), pcnt (4 a
// primary, rounded up to 1,024): keys + primaries <= kPsW, or kPsMaxPrim
// primaries besides kPsW keys
constexpr size_t kSortSmem = size_t(kPsW) * 8 + size_t(kPsMaxPrim) * 8 + 4096 + 64;
static_assert(kPsW <= 65536 / 2, "bin starts and sizes in 16 bits");
static_assert(kSortSmem >= kHistSmem + 2 * kSplitGroups * sizeof(uint32_t), "splits and ps_count_out work in the same memory");
}  // namespace

void carve_pair_sort(Carver &c, int64_t m, int32_t n, PairSortScratch &s) {
    const int64_t weight = 2 * (m > 0 ? m : 1) + n;
    s.total = c.take<uint32_t>(kFine);
    s.bstart = c.take<uint32_t>(kFine);
    s.bfine = c.take<uint32_t>(kFine);
    s.cursor = c.take<uint32_t>(kFine);
    s.run_cursor = c.take<uint32_t>(kCoarse);
    s.bmap = c.take<uint16_t>(kFine);
    s.ctl = c.take<PsControl>(1);
    s.over_cap = uint32_t(weight / kPsT + 64);
    s.over = c.take<PsBucket>(s.over_cap);
    // groups: at most 3 per kPsT of weight and 4 more, once for the fine bins
    // and once for every oversize bucket; pieces of equal keys
    s.list_cap = uint32_t(12 * (weight / kPsT) + kFine + 64);
    s.list = c.take<PsBucket>(s.list_cap);
}

int pair_sort(const int32_t *edges, int64_t m, int32_t n, const int32_t *node_map, const int64_t *K_dev,
              const uint32_t *moved, const PairSortScratch &s, unsigned long long *buf0, unsigned long long *buf1,
              unsigned long long *nkeys, uint32_t *status, cudaStream_t st) {
    const int64_t pairs = (m + 1) / 2;
    const int sms = sm_count();  // one block per SM, two of the moves
    const int64_t cap = 2 * m;
    BGV_CUDA(cudaFuncSetAttribute(k_ps_hist, cudaFuncAttributeMaxDynamicSharedMemorySize, int(kHistSmem)));
    BGV_CUDA(cudaFuncSetAttribute(k_ps_plan, cudaFuncAttributeMaxDynamicSharedMemorySize, int(kHistSmem)));
    BGV_CUDA(cudaFuncSetAttribute(k_ps_coarse, cudaFuncAttributeMaxDynamicSharedMemorySize, int(kCoarseSmem)));
    BGV_CUDA(cudaFuncSetAttribute(k_ps_place, cudaFuncAttributeMaxDynamicSharedMemorySize, int(kPlaceSmem)));
    BGV_CUDA(cudaFuncSetAttribute(k_ps_sort<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, int(kSortSmem)));
    BGV_CUDA(cudaFuncSetAttribute(k_ps_sort<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, int(kSortSmem)));
    BGV_CUDA(cudaMemsetAsync(s.total, 0, sizeof(uint32_t) * kFine, st));
    BGV_CUDA(cudaMemsetAsync(s.ctl, 0, sizeof(PsControl), st));
    int4 *mapped = reinterpret_cast<int4 *>(buf1);  // the mapped edges, until their keys are in buf0
    note_launch(), k_ps_hist<<<grid_for(pairs, kThreads * 4, sms), kThreads, kHistSmem, st>>>(
        edges, m, n, node_map, K_dev, moved, mapped, s.total, status);
    BGV_TRY(launch_status());
    note_launch(), k_ps_plan<<<1, kThreads, kHistSmem, st>>>(s.total, K_dev, s.ctl, s.bstart, s.bfine, s.bmap, s.cursor,
                                                     s.run_cursor, s.list, s.list_cap, s.over, s.over_cap, nkeys);
    BGV_TRY(launch_status());
    note_launch(), k_ps_coarse<<<grid_for(pairs, kMoveKeys / 4, 2 * sms), kMoveThreads, kCoarseSmem, st>>>(
        edges, m, n, K_dev, moved, mapped, s.bmap, s.run_cursor, s.ctl, buf0, cap);
    BGV_TRY(launch_status());
    note_launch(), k_ps_place<<<grid_for(2 * m, kMoveKeys, 2 * sms), kMoveThreads, kPlaceSmem, st>>>(
        buf0, K_dev, s.bmap, s.bstart, s.run_cursor, s.ctl, s.cursor, buf1, cap);
    BGV_TRY(launch_status());
    const int blocks = grid_for(2 * m, int(kPsT), sms);
    note_launch(), k_ps_sort<true><<<blocks, kThreads, kSortSmem, st>>>(buf0, buf1, K_dev, s.ctl, s.list, s.list_cap, s.over);
    BGV_TRY(launch_status());
    note_launch(), k_ps_sort<false><<<blocks, kThreads, kSortSmem, st>>>(buf0, buf1, K_dev, s.ctl, s.list, s.list_cap, s.over);
    return launch_status();
}

}  // namespace bgv
