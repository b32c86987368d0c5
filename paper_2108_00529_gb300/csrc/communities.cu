// communities.cu -- streaming community rounds (Algorithm 3, Section 3.2.1).
//
// Each round streams the edge list (int4 loads, two edges per load), gathers
// the start-of-round (degree, label) pair of both endpoints as one 8-byte load
// each, applies the rule and offers the move to the joining node with a 64-bit
// atomicMin of (edge index << 32 | label): the lowest edge index wins whatever
// order the threads run in, so labels are bit-identical to the sequential
// oracle.  Then every node that received a proposal is updated and its proposal
// slot reset for the next round.  No state is written while edges are read, so
// every edge reads the snapshot of the round.
//
// Edges whose endpoints are not both at or below the threshold move nothing,
// and on skewed graphs (whose sketched degrees are high) that is nearly every
// edge.  The random state gathers bound the pass (about 160 to 280 G gathers/s),
// so each block first tests both endpoints on a bit map of the nodes that pass
// the threshold, kept in its shared memory; only the edges that pass gather
// anything.  With more nodes than bits, a bit stands for 2^shift neighbouring
// ids and is set if any of them passes; the exact test follows on the gathered
// degrees either way.  Measured: 3 rounds over 10 M R-MAT edges on 2^20 nodes
// 114 us with the map, 386 with the gathers alone.
//
// Gathers in flight need room in the L1 that the map takes away: a map of 200 KB per
// SM halved the rate of rounds in which nearly all edges pass (3 rounds over 10 M
// uniform edges on 3.2 M nodes 1,115 us, 427 with the gathers alone), so a block's
// map is 64 KB at most, two blocks share an SM (batched, whose words are twice as
// wide, one), and from the round on in which nearly all edges would pass there is no
// map: 443 us.
//
// Batched form: each node also carries its graph's threshold, (degree,
// label, threshold) in one 16-byte word, so a propose still gathers one
// 32-byte sector per endpoint and graphs with different thresholds share a
// launch.  Edge indices and labels are global but ordered as inside each
// graph, so the winners are those of G separate runs.
#include "bgv_internal.cuh"

namespace bgv {
namespace {
constexpr int kThreads = 256;
constexpr int kRoundThreads = 1024;
constexpr int kMapBytes = 64 * 1024;
constexpr unsigned long long kNone = ~0ull;

// Ids per bit of the map, as a shift: the finest that fits.
inline int map_shift(int64_t n) {
    int s = 0;
    while (((n - 1) >> s) >= int64_t(kMapBytes) * 8) ++s;
    return s;
}
inline int64_t map_words(int64_t n, int s) { return ((((n - 1) >> s) >> 5) + 4) / 4 * 4; }  // whole uint4s

// The rule of one edge on the round's snapshot: returns the joining node w
// and the label it is offered, or -1 when the edge moves nothing.
__device__ __forceinline__ int32_t edge_rule(int32_t u, int32_t v, uint32_t du, uint32_t lu, uint32_t dv, uint32_t lv,
                                             uint32_t D, int tie_mode, uint32_t *lab) {
    if (du > D || dv > D) return -1;
    if (lu == lv) return -1;
    if (du > dv) {
        *lab = lu;
        return v;
    }
    if (dv > du) {
        *lab = lv;
        return u;
    }
    if (!tie_mode) return -1;
    *lab = u < v ? lv : lu;
    return u < v ? u : v;
}

__device__ __forceinline__ bool endpoints_ok(int32_t u, int32_t v, int32_t n, uint32_t *status) {
    if (static_cast<uint32_t>(u) >= static_cast<uint32_t>(n) || static_cast<uint32_t>(v) >= static_cast<uint32_t>(n)) {
        raise_status(status, BGV_DEV_BADEDGE);
        return false;
    }
    return u != v;
}

// The offers of two edges: each joins best[w] (w < 0: none) as (edge index, label).
// Both slots are read before either is written, so their round trips overlap.  A
// slot only decreases, so a stale read can only be larger than the current value:
// skipping when the offer is not below it is always safe.
__device__ __forceinline__ void offer_two(unsigned long long *best, const int32_t (&w)[2], const uint32_t (&e)[2],
                                          const uint32_t (&lab)[2]) {
    unsigned long long now[2];
#pragma unroll
    for (int j = 0; j < 2; ++j) now[j] = w[j] >= 0 ? __ldcg(&best[w[j]]) : 0ull;
#pragma unroll
    for (int j = 0; j < 2; ++j) {
        const unsigned long long cand = (static_cast<unsigned long long>(e[j]) << 32) | lab[j];
        if (cand < now[j]) atomicMin(&best[w[j]], cand);
    }
}

// Edges from which a round filters them by the map.  Below, the map's way through
// L2 costs more than the gathers it saves: ten rounds over 11,000 edges 160 us with
// it and 136 without, four over 180,000 109 and 108, eight over 247,000 of an R-MAT
// graph 132 and 159.
constexpr int64_t kMapMin = int64_t(1) << 17;
// Largest share of the degrees that lies in nodes below the threshold, for a map: with
// 0.9 about 0.8 of the edges pass it.  Seven rounds over 582,515 edges of an R-MAT graph
// 132 us with 0.9, 143 with 0.7 and 158 with three quarters of the nodes, most of which
// have few edges; three over 5 M uniform edges 166, 169 and 178.
constexpr float kMapShare = 0.9f;

// All rounds in one persistent kernel (cooperative launch, every block
// resident): initial state and bit map, then per round the map into shared
// memory, the proposals over the edge list, a grid barrier, the winning
// proposals applied (and the thresholds advanced, and the next round's map
// made), a barrier, the pointer-jumping steps (read, barrier, write, barrier),
// and at the end the labels.  Reads of what other blocks wrote since the last
// barrier go to L2 (L1 is not coherent).  From the second round on, a round in
// which no node passes the threshold reads no edges (the first round has
// checked their endpoints).  The barrier waits are bounded and report
// BGV_DEV_TIMEOUT.  kB: the batched form.
template <bool kB>
__global__ void __launch_bounds__(kRoundThreads, kB ? 1 : 2) k_comm_rounds(
    const int32_t *__restrict__ edges, int64_t m, int32_t n, const uint32_t *__restrict__ deg_est,
    const int32_t *__restrict__ node_graph, const uint32_t *__restrict__ D0, int32_t passes, uint32_t threshold,
    uint32_t growth, int tie_mode, int32_t jumps, uint2 *state, uint4 *bstate, unsigned long long *best, uint32_t *jump,
    uint32_t *map, int shift, int words, int filter, float2 *weight, int32_t *__restrict__ labels, uint32_t *__restrict__ deg_out,
    uint32_t *status, WsHeader *hdr, int spin_limit) {
    extern __shared__ uint4 map_sh4[];
    const uint32_t *map_sh = reinterpret_cast<const uint32_t *>(map_sh4);
    const int64_t stride = int64_t(gridDim.x) * blockDim.x;
    const int64_t t0 = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
    const int lane = threadIdx.x & 31;
    __shared__ float2 part[kRoundThreads / 32];
    // A warp takes the 2^shift rows of 32 nodes of one map word (lane t: the rows'
    // votes of bit t); `pass(v, d)` brings node v to the next round and says whether
    // it passes that round's threshold, and its degree d.  Adds the degrees (each
    // plus one) of the nodes that pass, and of all, to weight[slot].
    auto each_node = [&](int slot, auto pass) {
        float passing = 0.0f, all = 0.0f;
        for (int64_t w = t0 >> 5; w < words; w += stride >> 5) {
            bool bit = false;
            for (int j = 0; j < 1 << shift; ++j) {
                const int64_t v = (((w << shift) + j) << 5) + lane;
                uint32_t d = 0u;
                const bool ok = v < n && pass(v, d);
                if (!filter) continue;
                const float dw = v < n ? __uint2float_rn(d) + 1.0f : 0.0f;
                passing += ok ? dw : 0.0f;
                all += dw;
                const uint32_t row = __ballot_sync(0xFFFFFFFFu, ok);
                if (shift >= 5) {  // rows lie inside one bit
                    bit |= row != 0u && (j >> (shift - 5)) == lane;
                } else {           // 32 >> shift bits in a row
                    const int per = 32 >> shift, first = (lane & (per - 1)) << shift;
                    bit |= lane / per == j && ((row >> first) & ((2u << ((1 << shift) - 1)) - 1u)) != 0u;
                }
            }
            if (!filter) continue;
            const uint32_t word = __ballot_sync(0xFFFFFFFFu, bit);
            if (lane == 0) map[w] = word;
        }
        if (!filter) return;
        auto warp_sum = [&]() {
#pragma unroll
            for (int k = 16; k > 0; k >>= 1) {
                passing += __shfl_xor_sync(0xFFFFFFFFu, passing, k);
                all += __shfl_xor_sync(0xFFFFFFFFu, all, k);
            }
        };
        warp_sum();
        if (lane == 0) part[threadIdx.x >> 5] = make_float2(passing, all);
        __syncthreads();
        if (threadIdx.x >= 32) return;
        passing = part[lane].x;
        all = part[lane].y;
        warp_sum();
        if (lane == 0 && all > 0.0f) {
            atomicAdd(&weight[slot].x, passing);
            atomicAdd(&weight[slot].y, all);
        }
    };
    each_node(0, [&](int64_t v, uint32_t &d) {
        d = deg_est[v];
        best[v] = kNone;
        if (kB) {
            const uint32_t d0 = D0[node_graph[v]];
            bstate[v] = make_uint4(d, uint32_t(v), d0, d0);
            return d <= d0;
        }
        state[v] = make_uint2(d, uint32_t(v));
        return d <= threshold;
    });
    if (!grid_barrier(&hdr->bar, spin_limit, status)) return;
    const int4 *e2 = reinterpret_cast<const int4 *>(edges);
    const int64_t pairs = m >> 1;
    bool use = false;  // the round's map
    auto passes_map = [&](int32_t x) {
        const uint32_t b = uint32_t(x) >> shift;
        return !use || ((map_sh[b >> 5] >> (b & 31u)) & 1u) != 0u;
    };
    // both endpoints in range (else reported), not a loop, and both on the map
    auto wanted = [&](int32_t u, int32_t v) { return endpoints_ok(u, v, n, status) && passes_map(u) && passes_map(v); };
    unsigned long long D = threshold;
    const unsigned long long factor = growth ? growth : threshold;
    for (int32_t p = 0; p < passes; ++p) {
        const float2 wt = filter ? __ldcg(&weight[p & 1]) : make_float2(1.0f, 1.0f);
        use = filter && wt.x <= kMapShare * wt.y;
        // thresholds do not fall: nearly all edges pass from here on (all blocks read
        // the same sums)
        if (!use) filter = 0;
        if (p == 0 || wt.x > 0.0f) {
            const uint4 *src = reinterpret_cast<const uint4 *>(map);
            if (use) {
                for (int i = threadIdx.x; i < words / 4; i += kRoundThreads) map_sh4[i] = __ldcg(src + i);
                __syncthreads();
            }
            // two edges and the gathers of both at once
            auto edge_pair = [&](const int4 e, const bool (&go)[2], const uint32_t (&index)[2]) {
                uint2 su[2], sv[2];
                uint32_t thr[2];
#pragma unroll
                for (int j = 0; j < 2; ++j) {
                    const int32_t u = j ? e.z : e.x, v = j ? e.w : e.y;
                    thr[j] = uint32_t(D);
                    su[j] = sv[j] = make_uint2(0xFFFFFFFFu, 0u);
                    if (go[j] && kB) {  // both endpoints belong to one graph: u's threshold is the graph's
                        const uint4 a = __ldcg(&bstate[u]), b = __ldcg(&bstate[v]);
                        su[j] = make_uint2(a.x, a.y);
                        sv[j] = make_uint2(b.x, b.y);
                        thr[j] = a.z;
                    } else if (go[j]) {
                        su[j] = __ldcg(&state[u]);
                        sv[j] = __ldcg(&state[v]);
                    }
                }
                int32_t w[2];
                uint32_t lab[2] = {0u, 0u};
#pragma unroll
                for (int j = 0; j < 2; ++j)
                    w[j] = go[j] ? edge_rule(j ? e.z : e.x, j ? e.w : e.y, su[j].x, su[j].y, sv[j].x, sv[j].y, thr[j],
                                             tie_mode, &lab[j])
                                 : -1;
                offer_two(best, w, index, lab);
            };
            for (int64_t q = t0; q < pairs; q += stride) {
                const int4 e = __ldcs(e2 + q);
                const bool go[2] = {wanted(e.x, e.y), wanted(e.z, e.w)};
                const uint32_t index[2] = {uint32_t(2 * q), uint32_t(2 * q + 1)};
                if (go[0] || go[1]) edge_pair(e, go, index);
            }
            if ((m & 1) && t0 == 0) {
                const int4 e = make_int4(edges[2 * (m - 1)], edges[2 * (m - 1) + 1], 0, 0);
                const bool go[2] = {wanted(e.x, e.y), false};
                const uint32_t index[2] = {uint32_t(m - 1), 0u};
                edge_pair(e, go, index);
            }
        }
        if (!grid_barrier(&hdr->bar, spin_limit, status)) return;
        D *= factor;
        if (D > 0xFFFFFFFFull) D = 0xFFFFFFFFull;
        if (t0 == 0) weight[p & 1] = make_float2(0.0f, 0.0f);  // read by every block before the barrier; written next after the one below
        each_node((p + 1) & 1, [&](int64_t v, uint32_t &d) {
            const unsigned long long b = __ldcg(&best[v]);
            if (kB) {
                uint4 st = __ldcg(&bstate[v]);
                if (b != kNone) {
                    st.y = static_cast<uint32_t>(b & 0xFFFFFFFFull);
                    if (st.x != 0xFFFFFFFFu) st.x += 1;
                    best[v] = kNone;
                }
                const unsigned long long nd = static_cast<unsigned long long>(st.z) * (growth ? growth : st.w);
                st.z = nd > 0xFFFFFFFFull ? 0xFFFFFFFFu : uint32_t(nd);
                bstate[v] = st;
                d = st.x;
                return st.x <= st.z;
            }
            uint2 st = __ldcg(&state[v]);
            if (b != kNone) {
                st.y = static_cast<uint32_t>(b & 0xFFFFFFFFull);
                if (st.x != 0xFFFFFFFFu) st.x += 1;
                state[v] = st;
                best[v] = kNone;
            }
            d = st.x;
            return st.x <= uint32_t(D);
        });
        if (!grid_barrier(&hdr->bar, spin_limit, status)) return;
        for (int32_t j = 0; j < jumps; ++j) {
            for (int64_t v = t0; v < n; v += stride)
                jump[v] = kB ? __ldcg(&bstate[__ldcg(&bstate[v].y)].y) : __ldcg(&state[__ldcg(&state[v].y)].y);
            if (!grid_barrier(&hdr->bar, spin_limit, status)) return;
            for (int64_t v = t0; v < n; v += stride) {
                if (kB) bstate[v].y = __ldcg(&jump[v]);
                else state[v].y = __ldcg(&jump[v]);
            }
            if (!grid_barrier(&hdr->bar, spin_limit, status)) return;
        }
    }
    for (int64_t v = t0; v < n; v += stride) {
        const uint32_t d = kB ? __ldcg(&bstate[v].x) : __ldcg(&state[v].x);
        const uint32_t l = kB ? __ldcg(&bstate[v].y) : __ldcg(&state[v].y);
        labels[v] = int32_t(l);
        if (deg_out) deg_out[v] = d;
    }
}

// Mode degree (Section 4.2.2): the keys (graph << 32 | degree) are sorted;
// the end of every run of equal nonzero keys finds the run's start by binary
// search and offers (run length, complement of the degree) to its graph, so
// the longest run wins and ties go to the smaller degree.
__global__ void __launch_bounds__(kThreads) k_mode_keys(const uint32_t *__restrict__ deg, int32_t n,
                                                        const int32_t *__restrict__ node_graph,
                                                        unsigned long long *__restrict__ keys) {
    const int64_t stride = int64_t(gridDim.x) * blockDim.x;
    for (int64_t v = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; v < n; v += stride) {
        const unsigned long long g = node_graph ? static_cast<unsigned long long>(node_graph[v]) : 0ull;
        keys[v] = (g << 32) | deg[v];
    }
}

__global__ void __launch_bounds__(kThreads) k_mode_runs(const unsigned long long *__restrict__ sorted, int32_t n,
                                                        unsigned long long *best) {
    const int64_t stride = int64_t(gridDim.x) * blockDim.x;
    for (int64_t i = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; i < n; i += stride) {
        const unsigned long long k = sorted[i];
        const uint32_t value = static_cast<uint32_t>(k & 0xFFFFFFFFull);
        if (value == 0 || (i + 1 < n && sorted[i + 1] == k)) continue;
        int64_t lo = 0, hi = i;  // first position holding k
        while (lo < hi) {
            const int64_t mid = (lo + hi) >> 1;
            if (sorted[mid] < k) lo = mid + 1; else hi = mid;
        }
        const unsigned long long len = static_cast<unsigned long long>(i - lo + 1);
        atomicMax(&best[k >> 32], (len << 32) | (0xFFFFFFFFull - value));
    }
}

__global__ void k_mode_out(const unsigned long long *__restrict__ best, int32_t G, uint32_t *__restrict__ mode) {
    for (int32_t g = blockIdx.x * blockDim.x + threadIdx.x; g < G; g += gridDim.x * blockDim.x)
        mode[g] = best[g] ? uint32_t(0xFFFFFFFFull - (best[g] & 0xFFFFFFFFull)) : 0u;
}
}  // namespace

void carve_comm(Carver &c, int64_t m, int32_t n, CommScratch &s, bool batched) {
    (void)m;
    s.state = batched ? nullptr : c.take<uint2>(size_t(n));
    s.bstate = batched ? c.take<uint4>(size_t(n)) : nullptr;
    s.best = c.take<unsigned long long>(size_t(n));
    s.jump = c.take<uint32_t>(size_t(n));
    s.map = c.take<uint32_t>(size_t(map_words(n, map_shift(n))));
    s.weight = c.take<float2>(2);
}

void carve_mode(Carver &c, int32_t n, int32_t G, ModeScratch &s) {
    carve_sort(c, n, false, s.sort);
    s.best = c.take<unsigned long long>(size_t(G > 0 ? G : 1));
}

int run_mode_degree(const uint32_t *deg, int32_t n, const BatchView *batch, uint32_t *mode_dev,
                    const ModeScratch &s, uint32_t *status, cudaStream_t st) {
    const int32_t G = batch ? batch->G : 1;
    const int gn = grid_for(n, kThreads, sm_count() * 8);
    BGV_CUDA(cudaMemsetAsync(s.best, 0, sizeof(unsigned long long) * size_t(G), st));
    note_launch(), k_mode_keys<<<gn, kThreads, 0, st>>>(deg, n, batch ? batch->node_graph : nullptr,
                                                        s.sort.keys[0]);
    BGV_TRY(launch_status());
    SortBuffers sb = s.sort;
    int res = 0;
    BGV_TRY(radix_sort(sb, n, nullptr, 32 + (batch ? bits_for(G) : 0), st, &res, status));
    note_launch(), k_mode_runs<<<gn, kThreads, 0, st>>>(sb.keys[res], n, s.best);
    note_launch(), k_mode_out<<<grid_for(G, kThreads, sm_count()), kThreads, 0, st>>>(s.best, G, mode_dev);
    return launch_status();
}

int run_communities(const int32_t *edges, int64_t m, int32_t n, const uint32_t *deg_est, int32_t passes,
                    uint32_t threshold, uint32_t growth, int32_t tie_mode, int32_t jumps, int32_t *labels,
                    uint32_t *deg_out, const CommScratch &s, uint32_t *status, cudaStream_t st,
                    const BatchView *batch, WsHeader *hdr) {
    const int32_t *node_graph = batch ? batch->node_graph : nullptr;
    const uint32_t *D0 = batch ? batch->D0 : nullptr;
    uint2 *state = s.state;
    uint4 *bstate = s.bstate;
    unsigned long long *best = s.best;
    uint32_t *jump = s.jump;
    int tmode = tie_mode, limit = spin_limit();
    uint32_t *map = s.map;
    float2 *weight = s.weight;
    int filter = m >= kMapMin ? 1 : 0;
    int shift = filter ? map_shift(n) : 0, words = int(map_words(n, shift));
    BGV_CUDA(cudaMemsetAsync(weight, 0, 2 * sizeof(float2), st));
    void *args[] = {&edges, &m, &n, &deg_est, &node_graph, &D0, &passes, &threshold, &growth, &tmode, &jumps,
                    &state, &bstate, &best, &jump, &map, &shift, &words, &filter, &weight, &labels, &deg_out, &status, &hdr, &limit};
    const void *kernel = batch ? reinterpret_cast<const void *>(k_comm_rounds<true>)
                               : reinterpret_cast<const void *>(k_comm_rounds<false>);
    const size_t smem = filter ? size_t(words) * sizeof(uint32_t) : 0;
    BGV_CUDA(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kMapBytes));
    // no more blocks than there is work for (two edges a thread): a barrier over
    // few blocks is shorter; with four a thread ten rounds over 11,000 edges took 136
    // us, with two 110
    const int64_t work = int64_t(n) > m / 2 ? int64_t(n) : m / 2;
    const int blocks = coop_blocks(kernel, kRoundThreads, grid_for(work, kRoundThreads, sm_count() * (batch ? 1 : 2)), smem);
    return launch_coop(kernel, blocks, kRoundThreads, args, st, smem);
}

}  // namespace bgv
