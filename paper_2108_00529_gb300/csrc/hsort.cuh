// hsort.cuh -- sort of (key, id) pairs into (key, id) order, given a hint:
// an order of the ids that is already close to the sorted one.
//
// ForceAtlas2 moves every body a little per iteration, so the previous
// iteration's Morton order of the bodies is such a hint for the next one:
// on the 3.2 M-body rmat22x supergraph, 98.3 % (first iterations) to 99.8 %
// (iteration 500) of the bodies end within 4,096 places of where the
// previous order had them.  The LSD radix sort ignores that; this sort uses
// it to cut the global passes to two (count, scatter) and to sort the rest
// in shared memory, with kernels that need no grid-wide residency.
//
// Method: a bucket sort whose buckets follow the hint.
//   1. Splitters.  ForceAtlas2 still holds the previous iteration's sorted
//      (key, id) pairs: every kHsBucket-th of them is a splitter (HsPrevious), in
//      order already, with about as many new pairs between two as old ones.
//      The public entry point has no earlier keys, and a first or single step of
//      up to kHsFirstMax bodies not even a hint (id order serves as one): they
//      take the ids at ns evenly spaced places and their keys, rank them by
//      counting (equal pairs by sample index), and every s-th is a splitter
//      (HsSampled).  Bucket u holds the pairs x with splitter(u) <= x <
//      splitter(u+1), splitter(0) = -inf, splitter(nb) = +inf.
//   2. Count: every pair's key and bucket (the search starts at the bucket
//      its place in the hint would have, so a good hint needs one or two
//      probes), counted per bucket with one atomic per bucket per warp; the
//      last block turns the counts into bucket starts.  When the keys have
//      moved as a whole (a caller's own start that expands, a frame that a few
//      bodies stretch), many of them lie between two of the previous splitters:
//      with a bucket of more than hs_poor pairs the step takes samples of its
//      own keys after all and counts again.  Those two kernels follow every count
//      and return at once as a rule.
//   3. Scatter: every pair to its bucket (one atomic per bucket per warp).
//   4. Bucket sort: one block per bucket.  Up to kHsCap pairs it sorts in
//      shared memory, as single words of its key above the least one and its id
//      (or its place, when the keys span too many bits): words go to bins by their high bits
//      (shared-memory atomics) and are ranked inside their bins, which hold a
//      word or two; a bin too full for that (keys crowded in a corner of the
//      bucket), or keys too far apart for one word, take a merge sort in
//      shared memory.  A larger bucket (a poor hint) is sorted in chunks and
//      merged in global memory by the same block.
// The result is the (key, id) order for any hint: a poor hint only makes the
// buckets uneven.  A hint entry >= K raises BGV_DEV_BADHINT and is read as
// id 0 (a hint that is not a permutation gives an unspecified result but
// never an access outside the arrays).
#pragma once

#include "bgv_internal.cuh"

namespace bgv {

constexpr int kHsBucket = 1024;         // target pairs per bucket
constexpr int kHsMaxBuckets = 4096;     // so at most 4096 * 1024 pairs
constexpr int kHsMaxSamples = 4096;     // ns <= this
constexpr int kHsMaxPerBucket = 8;      // s <= this
constexpr int kHsThreads = 256;         // bucket-sort block
constexpr int kHsItems = 8;             // pairs (or words) per thread
constexpr int kHsPairCap = kHsThreads * kHsItems;  // 2048: a chunk of the pair sort
constexpr int kHsCap = kHsPairCap;      // larger buckets take the chunked path
constexpr int kHsCapBits = 11;
static_assert(kHsCap == 1 << kHsCapBits, "places of a bucket");
constexpr int kHsRankSlices = 16;       // slices of the samples per ranking thread
constexpr int kHsAgainSlices = 8;       // the same of the ranking that returns at once as a rule: fewer blocks
constexpr int kHsBins = 2048;           // bins of a bucket's words
constexpr uint32_t kHsRankBin = 32;     // largest bin ranked by counting
constexpr int kHsSmem = kHsCap + kHsCap / 16;  // skewed shared-memory slots
// The sort counts again with a larger bucket than this: where the second count has eight
// samples a bucket, nearly all its buckets stay in shared memory, and a bucket of one
// block's chunks and merges costs more than that count (80 us for 2,049 to 4,096 pairs,
// 27 for the rest; 10 steps of 140,000 bodies at scales e^0 to e^14 2,283 us with a line
// of 4,096 and 2,105 so).  With four samples or two some of its buckets are larger too.
__host__ __device__ constexpr uint32_t hs_poor(int nb) { return nb <= 512 ? kHsCap : 2 * kHsCap; }

inline int64_t hs_max_keys() { return int64_t(kHsMaxBuckets) * kHsBucket; }

// Small device arrays of the sort (the large ones are the caller's).
struct HsBuffers {
    unsigned long long *smp_key;  // [kHsMaxSamples] samples in hint order (sampled splitters only)
    uint32_t *smp_id;             // [kHsMaxSamples]
    unsigned long long *spl_key;  // [nb] splitter u at u - 1
    uint32_t *spl_id;             // [nb]
    uint32_t *count;              // [nb] pairs per bucket; zero between sorts, with all that follows:
    uint32_t *cursor;             // [nb] scatter cursors
    uint32_t *ticket;             // [3] last-block tickets of the ranking, the count and the second count
    uint32_t *poor;               // [1] the sort counts again
    uint32_t *smp_rank;           // [hs_shape(nb).ns] ranks of the samples
    uint32_t *start;              // [nb + 1] bucket starts
};

// Up to this many bodies the kernels of a step are short, and each may take its
// place while the one before drains (launch_chained): single steps of 60,000,
// 100,000 and 130,000 bodies 141, 158 and 163 us without and 127, 143 and 150 with
// it.  In the later steps of a run, beside a longer attraction, the waiting blocks
// keep the attraction's off the SMs: 30 steps of 60,000 bodies 2,993 us without and
// 2,952 with it, of 130,000 equal, of 145,000 3,367 and 3,473, of 240,000 4,093 and
// 4,211, 500 steps of 1 M bodies 190 and 214 ms.  A first or single step is shorter
// with it up to its line (145,000 bodies 162 and 155 us, 240,000 184 and 178).
inline bool hs_early(int64_t K, bool first) { return K <= int64_t(1) << (first ? 18 : 17); }
inline int hs_buckets(int64_t K) { return K > kHsBucket ? int((K + kHsBucket - 1) / kHsBucket) : 1; }
// Without a hint (bodies in id order) only the samples tell where the keys lie,
// and a bucket between sampled splitters may hold twice its share: half the
// share keeps it in shared memory.  A bucket may also span far-apart clusters
// of keys, crowded in few of its bins, and is merged then, 30 us more for the
// whole sort.  Single steps with the radix sort and with this: 30,000 bodies 132 us
// and 114, 60,000 140 and 127 (crowded 156), 80,000 143 and 142, 100,000 145 and
// 143, 115,000 (crowded) 146 and 173, 160,000 158 and 199.
constexpr int kHsFirstBucket = kHsBucket / 2;
constexpr int64_t kHsFirstMax = int64_t(1) << 16;
static_assert(kHsFirstMax / kHsFirstBucket * kHsMaxPerBucket <= kHsMaxSamples, "eight samples a bucket");
inline int hs_first_buckets(int64_t K) { return K > kHsFirstBucket ? int((K + kHsFirstBucket - 1) / kHsFirstBucket) : 1; }
// Samples per bucket for K pairs in nb buckets (ns = 0: no splitters).  The ranking
// compares all pairs of samples: 8 a bucket up to 512 buckets, 4 up to 2,048 and 2
// above keep it shorter than the count.
struct HsShape {
    int s, ns;
};
inline HsShape hs_shape(int nb) {
    HsShape h;
    h.s = nb <= 512 ? kHsMaxPerBucket : nb <= 2048 ? kHsMaxPerBucket / 2 : kHsMaxPerBucket / 4;
    h.ns = nb > 1 ? nb * h.s : 0;  // nb > 1 means K > 512 (nb - 1) >= 8 nb, so ns < K
    return h;
}
// The shape of a sort whose splitters are always samples.
inline HsShape hs_shape_sampled(int nb) {
    HsShape h;
    h.s = kHsMaxSamples / nb;
    if (h.s > kHsMaxPerBucket) h.s = kHsMaxPerBucket;
    if (h.s < 1) h.s = 1;
    h.ns = nb > 1 ? nb * h.s : 0;
    return h;
}

// Words from `count` on that are zero before a sort into nb buckets (and after it).
inline int64_t hs_counter_words(int nb) { return 2 * int64_t(nb) + 4 + hs_shape(nb).ns; }

inline void carve_hs(Carver &c, int nb, bool sampled, HsBuffers &h) {
    h = HsBuffers{};
    if (sampled) {
        h.smp_key = c.take<unsigned long long>(kHsMaxSamples);
        h.smp_id = c.take<uint32_t>(kHsMaxSamples);
    }
    h.spl_key = c.take<unsigned long long>(size_t(nb));
    h.spl_id = c.take<uint32_t>(size_t(nb));
    h.count = c.take<uint32_t>(size_t(hs_counter_words(nb)));
    h.start = c.take<uint32_t>(size_t(nb) + 1);
}
// The same buffers for a sort into nb buckets (no more than they were carved for).
inline HsBuffers hs_for(HsBuffers h, int nb) {
    h.cursor = h.count + nb;
    h.ticket = h.cursor + nb;
    h.poor = h.ticket + 3;
    h.smp_rank = h.poor + 1;
    return h;
}

// Splitter u + 1 (the least pair of bucket u + 1).
struct HsSampled {
    const unsigned long long *key;
    const uint32_t *id;
    __device__ unsigned long long key_at(int u) const { return key[u]; }
    __device__ uint32_t id_at(int u) const { return id[u]; }
};
struct HsPrevious {  // the sorted pairs of the previous iteration
    const unsigned long long *key;
    const uint32_t *id;
    __device__ unsigned long long key_at(int u) const { return __ldg(&key[int64_t(u + 1) * kHsBucket]); }
    __device__ uint32_t id_at(int u) const { return __ldg(&id[int64_t(u + 1) * kHsBucket]); }
};

// Extra words the first kernel clears (for the kernels after the sort).
struct HsClears {
    uint32_t *u32 = nullptr;
    int64_t n_u32 = 0;
};

// The kernels are private to each translation unit that includes this
// header (each instantiates its own key source).
namespace {

__device__ __forceinline__ bool hs_less(unsigned long long ak, uint32_t ai, unsigned long long bk, uint32_t bi) {
    return ak < bk || (ak == bk && ai < bi);
}

__device__ __forceinline__ uint32_t hs_id(const uint32_t *__restrict__ hint, int64_t p, int64_t K,
                                          uint32_t *status) {
    uint32_t id = hint ? hint[p] : uint32_t(p);  // no hint: id order
    if (id >= uint64_t(K)) {
        raise_status(status, BGV_DEV_BADHINT);
        id = 0u;
    }
    return id;
}

// 1a. Sample keys; clears the counters of the later kernels.
template <class KeyOf>
__global__ void __launch_bounds__(256) k_hs_sample(KeyOf key_of, const uint32_t *__restrict__ hint, int64_t K,
                                                   int64_t counter_words, int ns, HsBuffers h, HsClears clr,
                                                   uint32_t *status) {
    chain_wait();
    const int64_t stride = int64_t(gridDim.x) * blockDim.x;
    const int64_t t0 = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
    for (int64_t t = t0; t < ns; t += stride) {
        const int64_t p = ((2 * t + 1) * K) / (2 * int64_t(ns));
        const uint32_t id = hs_id(hint, p, K, status);
        h.smp_key[t] = key_of(id);
        h.smp_id[t] = id;
    }
    for (int64_t t = t0; t < counter_words; t += stride) h.count[t] = 0u;
    for (int64_t t = t0; t < clr.n_u32; t += stride) clr.u32[t] = 0u;
}

// The samples that k_hs_sample left.
struct HsStored {
    static constexpr bool kAgain = false;
    const unsigned long long *key_;
    const uint32_t *id_;
    __device__ void get(int t, unsigned long long *key, uint32_t *id) const {
        *key = key_[t];
        *id = id_[t];
    }
};
// Samples of the keys that the first count left, in hint order.
struct HsCounted {
    static constexpr bool kAgain = true;
    const unsigned long long *key_;
    const uint32_t *hint;
    int64_t K;
    int ns;
    __device__ void get(int t, unsigned long long *key, uint32_t *id) const {
        const int64_t p = ((2 * int64_t(t) + 1) * K) / (2 * int64_t(ns));
        const uint32_t i = hint ? hint[p] : uint32_t(p);
        *key = key_[p];
        *id = i < uint64_t(K) ? i : 0u;  // reported by the count kernel
    }
};

// 1b. Ranks of the samples by counting, one slice of the others per block
// row; the last block places every s-th one as a splitter, and leaves the ranks
// at zero.
template <class Samples>
__global__ void __launch_bounds__(256) k_hs_rank(Samples samples, int ns, int s, HsBuffers h) {  // 256 threads
    chain_wait();  // with no samples in a block's slice too: its tickets are the kernel's before to clear
    if (Samples::kAgain && *h.poor == 0u) return;
    __shared__ unsigned long long sk[256];
    __shared__ uint32_t si[256];
    __shared__ bool last;
    const int per = (ns + int(gridDim.y) - 1) / int(gridDim.y);
    const int j0 = blockIdx.y * per;
    const int j1 = min(ns, j0 + per);
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    unsigned long long ki = 0ull;
    uint32_t ii = 0u, c = 0u;
    if (i < ns) samples.get(i, &ki, &ii);
    for (int b0 = j0; b0 < j1; b0 += 256) {
        const int n = min(256, j1 - b0);
        if (int(threadIdx.x) < n) samples.get(b0 + threadIdx.x, &sk[threadIdx.x], &si[threadIdx.x]);
        __syncthreads();
        for (int j = 0; j < n; ++j) {
            const unsigned long long kj = sk[j];
            const uint32_t ij = si[j];
            c += (hs_less(kj, ij, ki, ii) || (kj == ki && ij == ii && b0 + j < i)) ? 1u : 0u;
        }
        __syncthreads();
    }
    if (i < ns && c) atomicAdd(&h.smp_rank[i], c);
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        last = atomicAdd(&h.ticket[0], 1u) == gridDim.x * gridDim.y - 1;
    }
    __syncthreads();
    if (!last) return;
    __threadfence();
    // every load of a round first (one round trip to L2), then the placements
    constexpr int kPer = 16;
    for (int t0 = threadIdx.x; t0 < ns; t0 += 256 * kPer) {
        uint32_t r[kPer], id[kPer];
        unsigned long long key[kPer];
#pragma unroll
        for (int q = 0; q < kPer; ++q) {
            const int t = t0 + 256 * q;
            r[q] = id[q] = 0u;
            key[q] = 0ull;
            if (t < ns) {
                r[q] = __ldcg(&h.smp_rank[t]);
                samples.get(t, &key[q], &id[q]);
            }
        }
#pragma unroll
        for (int q = 0; q < kPer; ++q) {
            if (t0 + 256 * q < ns) h.smp_rank[t0 + 256 * q] = 0u;
            if (r[q] >= uint32_t(s) && r[q] % uint32_t(s) == 0u && r[q] < uint32_t(ns)) {
                const uint32_t u = r[q] / uint32_t(s);
                h.spl_key[u - 1] = key[q];
                h.spl_id[u - 1] = id[q];
            }
        }
    }
}

// Bucket of pair x: the smallest u in [0, nb) with u == nb - 1 or
// x < splitter(u + 1) (stored at u), searched outwards from the guess g.
template <class Split>
__device__ __forceinline__ int hs_bucket(unsigned long long xk, uint32_t xi, const Split &split, int nb, int g) {
    auto above = [&](int u) { return u >= nb - 1 || hs_less(xk, xi, split.key_at(u), split.id_at(u)); };
    int lo, hi;  // the answer is in [lo, hi]; above(hi); lo == 0 or !above(lo - 1)
    if (above(g)) {
        hi = g;
        for (int d = 1;; d <<= 1) {
            const int u = g - d;
            if (u < 0) {
                lo = 0;
                break;
            }
            if (!above(u)) {
                lo = u + 1;
                break;
            }
            hi = u;
        }
    } else {
        lo = g + 1;
        for (int d = 1;; d <<= 1) {
            const int u = g + d;
            if (u >= nb - 1) {
                hi = nb - 1;
                break;
            }
            if (above(u)) {
                hi = u;
                break;
            }
            lo = u + 1;
        }
    }
    while (lo < hi) {
        const int mid = (lo + hi) >> 1;
        if (above(mid))
            hi = mid;
        else
            lo = mid + 1;
    }
    return lo;
}

// The keys of the second count: by place in the hint, as the first one left them.
struct HsAgain {};

// 2. Keys and buckets in hint order, counts per bucket; the last block
// writes the bucket starts, or, with previous splitters and a bucket of more than
// hs_poor pairs, asks for the second count (KeyOf = HsAgain).
template <class KeyOf, class Split>
__global__ void __launch_bounds__(256) k_hs_count(KeyOf key_of, Split split, const uint32_t *__restrict__ hint,
                                                  int64_t K, int nb, HsBuffers h, unsigned long long *tmp_key,
                                                  uint32_t *__restrict__ tmp_bucket, uint32_t *status) {
    chain_wait();
    constexpr bool kAgain = std::is_same<KeyOf, HsAgain>::value, kWatch = std::is_same<Split, HsPrevious>::value;
    if (kAgain && *h.poor == 0u) return;
    __shared__ bool last;
    __shared__ uint32_t part[8];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    // the bucket a hint place would have if the buckets split the hint
    // evenly: the search starts there
    const float g_scale = float(nb) / float(K);
    const int64_t stride = int64_t(gridDim.x) * blockDim.x;
    for (int64_t p0 = int64_t(blockIdx.x) * blockDim.x + (threadIdx.x & ~31); p0 < K; p0 += stride) {
        const int64_t p = p0 + lane;
        int u = -1;
        if (p < K) {
            const uint32_t id = hs_id(hint, p, K, status);
            unsigned long long k;
            if constexpr (kAgain) {
                k = tmp_key[p];
            } else {
                k = key_of(id);
                tmp_key[p] = k;
            }
            const int g = min(nb - 1, int(float(p) * g_scale));
            u = nb > 1 ? hs_bucket(k, id, split, nb, g) : 0;
            tmp_bucket[p] = uint32_t(u);
        }
        const unsigned peers = __match_any_sync(0xFFFFFFFFu, u);
        if (u >= 0 && lane == __ffs(peers) - 1) atomicAdd(&h.count[u], uint32_t(__popc(peers)));
    }
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        last = atomicAdd(&h.ticket[kAgain ? 2 : 1], 1u) == gridDim.x - 1;
    }
    __syncthreads();
    if (!last) return;
    __threadfence();
    // exclusive scan of the counts, 1,024 at a time
    uint32_t carry = 0u, most = 0u;
    for (int b0 = 0; b0 < nb; b0 += 1024) {
        const int b = b0 + 4 * int(threadIdx.x);
        uint32_t c[4], sum = 0u;
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            c[q] = b + q < nb ? __ldcg(&h.count[b + q]) : 0u;
            sum += c[q];
            most = max(most, c[q]);
        }
        uint32_t inc = sum;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, inc, d);
            if (lane >= d) inc += y;
        }
        if (lane == 31) part[warp] = inc;
        __syncthreads();
        uint32_t run = carry + inc - sum, all = 0u;
        for (int w = 0; w < 8; ++w) {
            if (w < warp) run += part[w];
            all += part[w];
        }
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            if (b + q < nb) h.start[b + q] = run;
            run += c[q];
        }
        carry += all;
        __syncthreads();
    }
    if (threadIdx.x == 0) h.start[nb] = uint32_t(K);
    if (kAgain && threadIdx.x == 0) *h.poor = 0u;
    if (kWatch && __syncthreads_or(most > hs_poor(nb))) {
        for (int b = threadIdx.x; b < nb; b += blockDim.x) h.count[b] = 0u;
        if (threadIdx.x == 0) *h.poor = 1u;
    }
}

// 3. Every pair to its bucket.
__global__ void __launch_bounds__(256) k_hs_scatter(const uint32_t *__restrict__ hint, int64_t K, HsBuffers h,
                                                    const unsigned long long *tmp_key, const uint32_t *tmp_bucket,
                                                    unsigned long long *__restrict__ slot_key,
                                                    uint32_t *__restrict__ slot_id) {
    chain_wait();
    const int lane = threadIdx.x & 31;
    const unsigned lt_mask = (1u << lane) - 1u;
    const int64_t stride = int64_t(gridDim.x) * blockDim.x;
    for (int64_t p0 = int64_t(blockIdx.x) * blockDim.x + (threadIdx.x & ~31); p0 < K; p0 += stride) {
        const int64_t p = p0 + lane;
        int u = -1;
        unsigned long long k = 0ull;
        uint32_t id = 0u;
        if (p < K) {
            u = int(tmp_bucket[p]);
            k = tmp_key[p];
            id = hint ? hint[p] : uint32_t(p);
            if (id >= uint64_t(K)) id = 0u;  // reported by the count kernel
        }
        const unsigned peers = __match_any_sync(0xFFFFFFFFu, u);
        const int leader = __ffs(peers) - 1;
        uint32_t base = 0u;
        if (u >= 0 && lane == leader) base = atomicAdd(&h.cursor[u], uint32_t(__popc(peers)));
        base = __shfl_sync(0xFFFFFFFFu, base, leader);
        if (u >= 0) {
            const uint32_t q = h.start[u] + base + uint32_t(__popc(peers & lt_mask));
            slot_key[q] = k;
            slot_id[q] = id;
        }
    }
}

// 4. Bucket sort.
__device__ __forceinline__ int hs_sw(int i) { return i + (i >> 4); }

__device__ __forceinline__ void hs_ce(unsigned long long (&k)[kHsItems], uint32_t (&v)[kHsItems], int a, int b) {
    if (hs_less(k[b], v[b], k[a], v[a])) {
        const unsigned long long tk = k[a];
        k[a] = k[b];
        k[b] = tk;
        const uint32_t tv = v[a];
        v[a] = v[b];
        v[b] = tv;
    }
}

// Sorts n <= kHsPairCap pairs from (ik, iv) into (ok, ov) (which may alias
// them); every thread of the block calls it.
__device__ void hs_block_sort(const unsigned long long *ik, const uint32_t *iv, int n, unsigned long long *ok,
                              uint32_t *ov, unsigned long long *shk, uint32_t *shv) {
    int P = kHsItems;
    while (P < n) P <<= 1;
    const int t = threadIdx.x;
    const bool act = kHsItems * t < P;
    unsigned long long k[kHsItems];
    uint32_t v[kHsItems];
#pragma unroll
    for (int j = 0; j < kHsItems; ++j) {
        const int q = kHsItems * t + j;
        const bool in = act && q < n;
        k[j] = in ? __ldcg(&ik[q]) : ~0ull;
        v[j] = in ? __ldcg(&iv[q]) : ~0u;
    }
    // Batcher's odd-even merge network for 8 inputs (19 comparators)
    hs_ce(k, v, 0, 1); hs_ce(k, v, 2, 3); hs_ce(k, v, 4, 5); hs_ce(k, v, 6, 7);
    hs_ce(k, v, 0, 2); hs_ce(k, v, 1, 3); hs_ce(k, v, 4, 6); hs_ce(k, v, 5, 7);
    hs_ce(k, v, 1, 2); hs_ce(k, v, 5, 6);
    hs_ce(k, v, 0, 4); hs_ce(k, v, 1, 5); hs_ce(k, v, 2, 6); hs_ce(k, v, 3, 7);
    hs_ce(k, v, 2, 4); hs_ce(k, v, 3, 5);
    hs_ce(k, v, 1, 2); hs_ce(k, v, 3, 4); hs_ce(k, v, 5, 6);
    for (int w = kHsItems; w < P; w <<= 1) {
        __syncthreads();  // the previous round's reads are done
        if (act) {
#pragma unroll
            for (int j = 0; j < kHsItems; ++j) {
                shk[hs_sw(kHsItems * t + j)] = k[j];
                shv[hs_sw(kHsItems * t + j)] = v[j];
            }
        }
        __syncthreads();
        if (act) {
            const int o0 = kHsItems * t;
            const int a0 = o0 & ~(2 * w - 1), b0 = a0 + w;
            const int o = o0 - a0;
            int lo = max(0, o - w), hi = min(o, w);
            while (lo < hi) {  // merge path: A's share of the first o outputs
                const int mid = (lo + hi) >> 1;
                const int bi = hs_sw(b0 + o - mid - 1), ai = hs_sw(a0 + mid);
                if (!hs_less(shk[bi], shv[bi], shk[ai], shv[ai]))
                    lo = mid + 1;
                else
                    hi = mid;
            }
            int ia = a0 + lo, ib = b0 + (o - lo);
            const int ae = a0 + w, be = b0 + w;
#pragma unroll
            for (int j = 0; j < kHsItems; ++j) {
                bool take_a;
                if (ia >= ae)
                    take_a = false;
                else if (ib >= be)
                    take_a = true;
                else
                    take_a = !hs_less(shk[hs_sw(ib)], shv[hs_sw(ib)], shk[hs_sw(ia)], shv[hs_sw(ia)]);
                const int q = hs_sw(take_a ? ia : ib);
                k[j] = shk[q];
                v[j] = shv[q];
                ia += take_a ? 1 : 0;
                ib += take_a ? 0 : 1;
            }
        }
    }
    __syncthreads();  // every read of (ik, iv) and of shared memory is done
    if (act) {
#pragma unroll
        for (int j = 0; j < kHsItems; ++j) {
            const int q = kHsItems * t + j;
            if (q < n) {
                ok[q] = k[j];
                ov[q] = v[j];
            }
        }
    }
    __syncthreads();
}

template <int I>
__device__ __forceinline__ void hs_ce64(unsigned long long (&c)[I], int a, int b) {
    const unsigned long long x = c[a], y = c[b];
    c[a] = x < y ? x : y;
    c[b] = x < y ? y : x;
}

// The same sort on single 64-bit words (no equal words but the padding):
// c holds the thread's I words of a P-word array (P a power of two >= I,
// at most I * blockDim.x); on return they are the thread's words of the
// sorted array.  The thread's words are sorted in registers, then merged.
template <int I>
__device__ void hs_sort_words(unsigned long long (&c)[I], int P, unsigned long long *sh) {
    static_assert(I == 4 || I == 8, "4 or 8 words a thread");
    const int t = threadIdx.x;
    const bool act = I * t < P;
    if constexpr (I == 4) {  // 5 comparators
        hs_ce64(c, 0, 1); hs_ce64(c, 2, 3);
        hs_ce64(c, 0, 2); hs_ce64(c, 1, 3);
        hs_ce64(c, 1, 2);
    } else {  // Batcher's odd-even merge network, 19 comparators
        hs_ce64(c, 0, 1); hs_ce64(c, 2, 3); hs_ce64(c, 4, 5); hs_ce64(c, 6, 7);
        hs_ce64(c, 0, 2); hs_ce64(c, 1, 3); hs_ce64(c, 4, 6); hs_ce64(c, 5, 7);
        hs_ce64(c, 1, 2); hs_ce64(c, 5, 6);
        hs_ce64(c, 0, 4); hs_ce64(c, 1, 5); hs_ce64(c, 2, 6); hs_ce64(c, 3, 7);
        hs_ce64(c, 2, 4); hs_ce64(c, 3, 5);
        hs_ce64(c, 1, 2); hs_ce64(c, 3, 4); hs_ce64(c, 5, 6);
    }
    for (int w = I; w < P; w <<= 1) {  // runs of w words; 2w > I, so a thread's outputs lie in one pair
        __syncthreads();  // the previous round's reads are done
        if (act) {
#pragma unroll
            for (int j = 0; j < I; ++j) sh[hs_sw(I * t + j)] = c[j];
        }
        __syncthreads();
        if (act) {
            const int o0 = I * t;
            const int a0 = o0 & ~(2 * w - 1), b0 = a0 + w;
            const int o = o0 - a0;
            int lo = max(0, o - w), hi = min(o, w);
            while (lo < hi) {  // merge path: A's share of the first o outputs
                const int mid = (lo + hi) >> 1;
                if (sh[hs_sw(a0 + mid)] <= sh[hs_sw(b0 + o - mid - 1)])
                    lo = mid + 1;
                else
                    hi = mid;
            }
            int ia = a0 + lo, ib = b0 + (o - lo);
            const int ae = a0 + w, be = b0 + w;
            unsigned long long va = ia < ae ? sh[hs_sw(ia)] : 0ull, vb = ib < be ? sh[hs_sw(ib)] : 0ull;
#pragma unroll
            for (int j = 0; j < I; ++j) {  // the heads stay in registers
                const bool take_a = ia < ae && (ib >= be || va <= vb);
                c[j] = take_a ? va : vb;
                if (take_a) {
                    ++ia;
                    va = ia < ae ? sh[hs_sw(ia)] : 0ull;
                } else {
                    ++ib;
                    vb = ib < be ? sh[hs_sw(ib)] : 0ull;
                }
            }
        }
    }
}

// n > kHsPairCap pairs (a wide or oversized bucket): chunks sorted in shared
// memory into (dk, dv), then merges of sorted runs in global memory,
// alternating between (dk, dv) and (sk, sv); the result ends in (dk, dv).
// Every thread of the block calls it.
__device__ void hs_pairs_chunked(unsigned long long *sk, uint32_t *sv, int64_t n, unsigned long long *dk,
                                 uint32_t *dv, unsigned long long *shk, uint32_t *shv) {
    for (int64_t c = 0; c < n; c += kHsPairCap)
        hs_block_sort(sk + c, sv + c, int(min(int64_t(kHsPairCap), n - c)), dk + c, dv + c, shk, shv);
    unsigned long long *srck = dk, *dstk = sk;
    uint32_t *srcv = dv, *dstv = sv;
    for (int64_t w = kHsPairCap; w < n; w <<= 1) {
        for (int64_t o0 = int64_t(threadIdx.x) * kHsItems; o0 < n; o0 += int64_t(blockDim.x) * kHsItems) {
            const int64_t a0 = o0 / (2 * w) * (2 * w), b0r = a0 + w;
            const int64_t alen = min(w, n - a0), blen = max(int64_t(0), min(w, n - b0r));
            const int64_t o = o0 - a0;
            int64_t lo = max(int64_t(0), o - blen), hi = min(o, alen);
            while (lo < hi) {
                const int64_t mid = (lo + hi) >> 1;
                const int64_t bi = b0r + o - mid - 1, ai = a0 + mid;
                if (!hs_less(__ldcg(&srck[bi]), __ldcg(&srcv[bi]), __ldcg(&srck[ai]), __ldcg(&srcv[ai])))
                    lo = mid + 1;
                else
                    hi = mid;
            }
            int64_t ia = a0 + lo, ib = b0r + (o - lo);
            const int64_t ae = a0 + alen, be = b0r + blen;
            for (int j = 0; j < kHsItems && o0 + j < n; ++j) {
                bool take_a;
                if (ia >= ae)
                    take_a = false;
                else if (ib >= be)
                    take_a = true;
                else
                    take_a = !hs_less(__ldcg(&srck[ib]), __ldcg(&srcv[ib]), __ldcg(&srck[ia]), __ldcg(&srcv[ia]));
                const int64_t q = take_a ? ia : ib;
                dstk[o0 + j] = __ldcg(&srck[q]);
                dstv[o0 + j] = __ldcg(&srcv[q]);
                ia += take_a ? 1 : 0;
                ib += take_a ? 0 : 1;
            }
        }
        __syncthreads();
        unsigned long long *tk = srck;
        srck = dstk;
        dstk = tk;
        uint32_t *tv = srcv;
        srcv = dstv;
        dstv = tv;
    }
    if (srck != dk) {
        for (int64_t q = threadIdx.x; q < n; q += blockDim.x) {
            dk[q] = __ldcg(&srck[q]);
            dv[q] = __ldcg(&srcv[q]);
        }
    }
}

// A bucket of n <= I * blockDim.x pairs, sorted as single words.  If its keys
// span less than 2^(63 - idbits), the words (key - kmin) << idbits | id (ids <
// 2^idbits) order exactly as (key, id).  Wider keys (up to 2^52: a batch's graph
// ids and Morton bits) take the pair's place in the bucket instead of its id, and
// equal keys look their ids up; that keeps the block at 8 bytes a pair, which
// matters beside its own time (keys and ids apart, 34 KB for 26 a block, slowed
// the attraction that shares the L1: 500 steps at 1 M bodies 191.4 for 188.7 ms).
// Words go to kHsBins bins by the high bits of the span, are ranked inside their
// bins and written to their places; with a bin of more than kHsRankBin words they
// are merged instead, and words with places as pairs.  Every thread of the block
// calls it.
// Bound by instruction issue: about 140 instructions per pair, 720 with the
// merge rounds (34 and 152 us for 3.2 M bodies).  Keys too wide for an id used to
// be sorted as pairs by merging, 302 us a step for 160 graphs of 6.0 M bodies; 300
// steps of them 456.6 -> 424.6 ms.
template <int I>
__device__ void hs_bucket_small(unsigned long long *sk, uint32_t *sv, int n, unsigned long long *dk,
                                uint32_t *dv, int idbits, unsigned long long *shk, uint32_t *shv,
                                unsigned long long *wmin, unsigned long long *wmax) {
    static_assert(kHsBins == 8 * kHsThreads && kHsBins <= kHsSmem, "eight bins a thread, in the ids' memory");
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    uint32_t *bins = shv;
    unsigned long long c[I];
    uint32_t id[I];
    unsigned long long kmin = ~0ull, kmax = 0ull;
#pragma unroll
    for (int j = 0; j < I; ++j) {
        const int q = j * kHsThreads + t;
        c[j] = q < n ? __ldcg(&sk[q]) : 0ull;
        id[j] = q < n ? __ldcg(&sv[q]) : 0u;
    }
#pragma unroll
    for (int j = 0; j < I; ++j) {
        if (j * kHsThreads + t < n) {
            kmin = c[j] < kmin ? c[j] : kmin;
            kmax = c[j] > kmax ? c[j] : kmax;
        }
    }
    for (int b = t; b < kHsBins; b += kHsThreads) bins[b] = 0u;
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) {
        const unsigned long long a = __shfl_xor_sync(0xFFFFFFFFu, kmin, d);
        const unsigned long long b = __shfl_xor_sync(0xFFFFFFFFu, kmax, d);
        kmin = a < kmin ? a : kmin;
        kmax = b > kmax ? b : kmax;
    }
    if (lane == 0) {
        wmin[warp] = kmin;
        wmax[warp] = kmax;
    }
    __syncthreads();
    kmin = wmin[0];
    kmax = wmax[0];
    for (int w = 1; w < kHsThreads / 32; ++w) {
        kmin = wmin[w] < kmin ? wmin[w] : kmin;
        kmax = wmax[w] > kmax ? wmax[w] : kmax;
    }
    const bool local = ((kmax - kmin) >> (63 - idbits)) != 0ull;  // ids do not fit
    const int low = local ? kHsCapBits : idbits;
    if (((kmax - kmin) >> (63 - low)) != 0ull) {  // too wide for one word
        __syncthreads();
        hs_block_sort(sk, sv, n, dk, dv, shk, shv);
        return;
    }
    const int bits = kmax > kmin ? 64 - __clzll(static_cast<long long>(kmax - kmin)) : 0;
    const int sh = bits > 11 ? bits - 11 : 0;
    uint32_t rank[I];
#pragma unroll
    for (int j = 0; j < I; ++j) {
        const bool in = j * kHsThreads + t < n;
        rank[j] = in ? atomicAdd(&bins[uint32_t((c[j] - kmin) >> sh)], 1u) : 0u;
        c[j] = in ? ((c[j] - kmin) << low) | (local ? uint32_t(j * kHsThreads + t) : id[j]) : ~0ull;
    }
    __syncthreads();
    // bins -> starts, eight bins per thread
    uint4 *b4 = reinterpret_cast<uint4 *>(bins) + 2 * t;
    uint4 x = b4[0], y = b4[1];
    const uint32_t most = max(max(max(x.x, x.y), max(x.z, x.w)), max(max(y.x, y.y), max(y.z, y.w)));
    const uint32_t sum = x.x + x.y + x.z + x.w + y.x + y.y + y.z + y.w;
    uint32_t inc = sum;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const uint32_t z = __shfl_up_sync(0xFFFFFFFFu, inc, d);
        if (lane >= d) inc += z;
    }
    if (lane == 31) wmin[warp] = inc;  // kmin is in registers
    if (__syncthreads_or(most > kHsRankBin)) {
        // words crowded in few bins: sorted by merging
        if (local) {
            hs_block_sort(sk, sv, n, dk, dv, shk, shv);
            return;
        }
#pragma unroll
        for (int j = 0; j < I; ++j) {
            const int q = j * kHsThreads + t;
            if (q < n) shk[hs_sw(q)] = c[j];
        }
        __syncthreads();
#pragma unroll
        for (int j = 0; j < I; ++j) c[j] = I * t + j < n ? shk[hs_sw(I * t + j)] : ~0ull;
        int P = I;
        while (P < n) P <<= 1;
        hs_sort_words<I>(c, P, shk);
        __syncthreads();  // the last round's reads are done
#pragma unroll
        for (int j = 0; j < I; ++j)
            if (I * t + j < n) shk[hs_sw(I * t + j)] = c[j];
        __syncthreads();
        const unsigned long long mask = (1ull << idbits) - 1ull;
        for (int q = t; q < n; q += kHsThreads) {
            const unsigned long long w = shk[hs_sw(q)];
            dk[q] = (w >> idbits) + kmin;
            dv[q] = uint32_t(w & mask);
        }
        return;
    }
    uint32_t run = inc - sum;
    for (int w = 0; w < warp; ++w) run += uint32_t(wmin[w]);
    const uint32_t r1 = run + x.x, r2 = r1 + x.y, r3 = r2 + x.z, r4 = r3 + x.w, r5 = r4 + y.x, r6 = r5 + y.y,
                   r7 = r6 + y.z;
    b4[0] = make_uint4(run, r1, r2, r3);
    b4[1] = make_uint4(r4, r5, r6, r7);
    __syncthreads();
#pragma unroll
    for (int j = 0; j < I; ++j)
        if (j * kHsThreads + t < n) shk[bins[uint32_t((c[j] >> low) >> sh)] + rank[j]] = c[j];
    __syncthreads();
    const unsigned long long mask = (1ull << low) - 1ull;
    for (int q = t; q < n; q += kHsThreads) {
        const unsigned long long w = shk[q], k = w >> low;
        const uint32_t b = uint32_t(k >> sh);
        const int lo = int(bins[b]), hi = b + 1 < uint32_t(kHsBins) ? int(bins[b + 1]) : n;
        const uint32_t i = local ? __ldcg(&sv[w & mask]) : uint32_t(w & mask);
        int at = lo;
        for (int z = lo; z < hi; ++z) at += shk[z] < w ? 1 : 0;
        if (local)  // equal keys so far in the order of their places
            for (int z = lo; z < hi; ++z) {
                const unsigned long long o = shk[z];
                if ((o >> low) != k || o == w) continue;
                at += (__ldcg(&sv[o & mask]) < i ? 1 : 0) - (o < w ? 1 : 0);
            }
        dk[at] = k + kmin;
        dv[at] = i;
    }
}

// One block per bucket: sorts its pairs from the slots into the output, and
// leaves the bucket's counters at zero for the next sort.
__global__ void __launch_bounds__(kHsThreads) k_hs_bucket(HsBuffers h, unsigned long long *__restrict__ slot_key,
                                                          uint32_t *__restrict__ slot_id,
                                                          unsigned long long *__restrict__ out_key,
                                                          uint32_t *__restrict__ out_id, int idbits) {
    chain_wait();
    __shared__ unsigned long long shk[kHsSmem];
    __shared__ __align__(16) uint32_t shv[kHsSmem];
    __shared__ unsigned long long wmin[kHsThreads / 32], wmax[kHsThreads / 32];
    const int u = blockIdx.x;
    if (threadIdx.x == 0) {
        h.count[u] = 0u;
        h.cursor[u] = 0u;
        if (u == 0) h.ticket[0] = h.ticket[1] = h.ticket[2] = 0u;
    }
    const int64_t b0 = h.start[u];
    const int64_t n = int64_t(h.start[u + 1]) - b0;
    if (n <= 0) return;
    unsigned long long *sk = slot_key + b0, *dk = out_key + b0;
    uint32_t *sv = slot_id + b0, *dv = out_id + b0;
    if (n <= kHsCap / 2)  // every thread busy at 4 words
        hs_bucket_small<4>(sk, sv, int(n), dk, dv, idbits, shk, shv, wmin, wmax);
    else if (n <= kHsCap)
        hs_bucket_small<8>(sk, sv, int(n), dk, dv, idbits, shk, shv, wmin, wmax);
    else
        hs_pairs_chunked(sk, sv, n, dk, dv, shk, shv);
}

}  // namespace

// The sort into nb buckets on stream `st`; key_of(id) gives the key of id, a null
// hint is id order.  tmp_key/tmp_bucket and slot_key/slot_id hold K entries each
// and may not alias the hint, the splitters or the output.  The counters of `h`
// are zero before it, and after.
template <class KeyOf, class Split>
int hinted_sort_place(KeyOf key_of, Split split, const uint32_t *hint, int64_t K, int nb, const HsBuffers &buffers,
                      unsigned long long *tmp_key, uint32_t *tmp_bucket, unsigned long long *slot_key,
                      uint32_t *slot_id, unsigned long long *out_key, uint32_t *out_id, uint32_t *status,
                      cudaStream_t st) {
    if (K <= 0) return BGV_OK;
    const HsBuffers h = hs_for(buffers, nb);
    constexpr bool kSampled = std::is_same<Split, HsSampled>::value;
    const bool early = hs_early(K, kSampled);
    // after the samples' kernels it follows in the chain; else an event precedes it
    BGV_TRY(launch_chained(kSampled && early, k_hs_count<KeyOf, Split>,
                           grid_for(K, 256, sm_count() * 8), 256, st, key_of, split, hint, K, nb, h, tmp_key, tmp_bucket,
                           status));
    // The second count, which returns at once as a rule: few blocks, launched beside
    // the ranking, as the scatter is beside them (500 steps of 1 M bodies 171.2 ms
    // without the two kernels, 172.8 so, 174.8 with 16 slices, 4 blocks an SM and
    // plain launches).  What it is for: 20 steps of 1 M bodies, ten of them far off,
    // 65 ms without and 9.1 with it; three steps from a tight start 12.3 and 1.5.
    const bool again = !kSampled && nb > 1;
    if (again) {
        const HsShape sh = hs_shape(nb);
        const dim3 g((sh.ns + 255) / 256, kHsAgainSlices);
        BGV_TRY(launch_chained(early, k_hs_rank<HsCounted>, g, 256, st, HsCounted{tmp_key, hint, K, sh.ns}, sh.ns, sh.s,
                               h));
        BGV_TRY(launch_chained(true, k_hs_count<HsAgain, HsSampled>, grid_for(K, 256, sm_count() * 2), 256, st,
                               HsAgain{}, HsSampled{h.spl_key, h.spl_id}, hint, K, nb, h, tmp_key, tmp_bucket, status));
    }
    BGV_TRY(launch_chained(early || again, k_hs_scatter, grid_for(K, 256, sm_count() * 8), 256, st, hint, K, h, tmp_key, tmp_bucket,
                           slot_key, slot_id));
    int idbits = 0;  // bits of the largest id
    while (idbits < 32 && (int64_t(1) << idbits) < K) ++idbits;
    return launch_chained(early, k_hs_bucket, nb, kHsThreads, st, h, slot_key, slot_id, out_key, out_id, idbits);
}

// The same with splitters from samples of the hint, nb <= kHsMaxBuckets; clears
// the counters first.
template <class KeyOf>
int hinted_sort_sampled(KeyOf key_of, const uint32_t *hint, int64_t K, int nb, const HsBuffers &buffers,
                        unsigned long long *tmp_key, uint32_t *tmp_bucket, unsigned long long *slot_key,
                        uint32_t *slot_id, unsigned long long *out_key, uint32_t *out_id, uint32_t *status,
                        cudaStream_t st, const HsClears &clr = HsClears()) {
    if (K <= 0) return BGV_OK;
    if (nb > kHsMaxBuckets) return BGV_EINVAL;
    const HsBuffers h = hs_for(buffers, nb);
    const HsShape sh = hs_shape_sampled(nb);
    const int64_t words = hs_counter_words(nb);
    int64_t work = sh.ns;
    for (const int64_t w : {words, clr.n_u32})
        if (w > work) work = w;
    note_launch(), k_hs_sample<KeyOf><<<grid_for(work, 256, sm_count() * 4), 256, 0, st>>>(key_of, hint, K, words,
                                                                                          sh.ns, h, clr, status);
    BGV_TRY(launch_status());
    if (sh.ns > 0) {
        const dim3 g((sh.ns + 255) / 256, kHsRankSlices);
        BGV_TRY(launch_chained(hs_early(K, true), k_hs_rank<HsStored>, g, 256, st, HsStored{h.smp_key, h.smp_id},
                               sh.ns, sh.s, h));
    }
    return hinted_sort_place(key_of, HsSampled{h.spl_key, h.spl_id}, hint, K, nb, h, tmp_key, tmp_bucket, slot_key,
                             slot_id, out_key, out_id, status, st);
}

}  // namespace bgv
