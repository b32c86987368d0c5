// sketch.cu -- degree count-min sketch (Algorithm 2, Section 3.3).
//
// Algorithm 2 adds 1 to M[i][h_i(x)] for every event x; the events here are
// the 2m edge endpoints.  Integer addition commutes, so the same matrix is
// built from exact per-node degrees: one edge pass counts degrees (L2
// atomics on an n-entry array, aggregated per warp over equal node ids),
// then every node with degree d adds d to its r cells.  That turns 2 r m
// scattered sketch updates into at most 2m + r n.
//
// Edges are read as int4 (two edges per 16-byte load) with a grid-stride
// loop over a grid sized to fill the GPU.
//
// The 2m atomics bound the small form of that edge pass (139 G/s at 3.2 M nodes;
// 51 G/s at 1 M nodes with the hubs of a = 0.57 R-MAT).  From kDegSplitMin
// edges up the endpoints are first sorted out by node range, as 16-bit offsets
// inside ranges of 32,768 nodes whose counters fit in shared memory:
//   k_deg_ranges   endpoints per range
//   k_deg_place    every endpoint's offset to its range's list (coalesced runs
//                  out of shared memory)
//   k_deg_count    lists counted with shared-memory atomics, one range's
//                  counters per block, and added to the degrees
// Degree sketch of 34 M edges on 3.2 M nodes: 608 us before, 431 with the ranges.
#include <mutex>

#include "bgv_internal.cuh"
#include "pieces.cuh"

namespace bgv {

HashFamily make_hash_family(uint64_t seed, int rows, uint32_t width) {
    HashFamily h{};
    const unsigned long long p = 2147483647ull;
    for (int i = 0; i < rows && i < kMaxRows; ++i) {
        unsigned long long st = seed + static_cast<unsigned long long>(i);
        unsigned long long z[2];
        for (int k = 0; k < 2; ++k) {
            st += 0x9E3779B97F4A7C15ull;
            unsigned long long x = st;
            x = (x ^ (x >> 30)) * 0xBF58476D1CE4E5B9ull;
            x = (x ^ (x >> 27)) * 0x94D049BB133111EBull;
            z[k] = x ^ (x >> 31);
        }
        h.a[i] = 1 + z[0] % (p - 1);
        h.b[i] = z[1] % p;
    }
    h.rows = rows;
    h.width = width;
    return h;
}

namespace {
constexpr int kThreads = 256;

// One endpoint per lane: lanes holding the same node id are found with
// __match_any_sync and only the lowest of them adds their number, so a hub
// that shows up several times in a warp's 32 endpoints costs one atomic.
__device__ __forceinline__ void count_endpoints_warp(bool have, int32_t x, int32_t n, uint32_t *deg,
                                                     uint32_t *status) {
    const bool ok = have && static_cast<uint32_t>(x) < static_cast<uint32_t>(n);
    if (have && !ok) raise_status(status, BGV_DEV_BADEDGE);
    const unsigned peers = __match_any_sync(0xFFFFFFFFu, ok ? x : -1);
    const int lane = threadIdx.x & 31;
    if (ok && (peers & ((1u << lane) - 1u)) == 0u) atomicAdd(&deg[x], uint32_t(__popc(peers)));
}

// Whole warps iterate together (the exit test uses the warp's first index)
// so every __match_any_sync sees all 32 lanes.  Each lane loads two int4
// (four edges) before counting, so the loads are in flight together.
constexpr int kDegLoads = 2;
__global__ void __launch_bounds__(kThreads) k_degree_count(const int32_t *__restrict__ edges, int64_t m, int32_t n,
                                                           uint32_t *__restrict__ deg, uint32_t *status) {
    const int4 *e2 = reinterpret_cast<const int4 *>(edges);
    const int64_t pairs = m >> 1;
    const int lane = threadIdx.x & 31;
    const int64_t warp = (int64_t(blockIdx.x) * blockDim.x + threadIdx.x) >> 5;
    const int64_t warps = (int64_t(gridDim.x) * blockDim.x) >> 5;
    for (int64_t base = warp * 32 * kDegLoads; base < pairs; base += warps * 32 * kDegLoads) {
        int4 e[kDegLoads];
        bool have[kDegLoads];
#pragma unroll
        for (int r = 0; r < kDegLoads; ++r) {
            const int64_t p = base + int64_t(r) * 32 + lane;
            have[r] = p < pairs;
            e[r] = have[r] ? __ldcs(e2 + p) : make_int4(0, 0, 0, 0);
        }
#pragma unroll
        for (int r = 0; r < kDegLoads; ++r) {
            count_endpoints_warp(have[r], e[r].x, n, deg, status);
            count_endpoints_warp(have[r], e[r].y, n, deg, status);
            count_endpoints_warp(have[r], e[r].z, n, deg, status);
            count_endpoints_warp(have[r], e[r].w, n, deg, status);
        }
    }
    if ((m & 1) && blockIdx.x == 0 && threadIdx.x < 32) {  // the odd last edge, one warp
        count_endpoints_warp(lane == 0, edges[2 * (m - 1)], n, deg, status);
        count_endpoints_warp(lane == 0, edges[2 * (m - 1) + 1], n, deg, status);
    }
}

// ------------------------------------------------ degrees by node ranges
constexpr int kDegThreads = 1024;
constexpr int kRangeBits = 15;
constexpr int kRange = 1 << kRangeBits;
constexpr int kMaxRanges = 512;                    // n <= 16,777,216
// Edges; below, one kernel is shorter than three.  The sketch takes 81 us at 2^20
// R-MAT edges with the ranges and 67 without, 89 and 89 at 2^21, 110 and 129 at
// 2^22; with uniform endpoints 87 and 75 at 2.2 M edges.
constexpr int64_t kDegSplitMin = int64_t(1) << 22;
constexpr int kDegIn = 4;                          // int4 loads per thread and tile
constexpr int kPlaceThreads = 512;  // of k_deg_place, two blocks per SM: their phases overlap (437 us with one of 1,024)
constexpr int kDegTile = kPlaceThreads * kDegIn * 4; // endpoints per tile
constexpr uint32_t kDegPiece = 1u << 18;           // endpoints a block counts at a time

inline int deg_ranges(int32_t n) { return (n + kRange - 1) / kRange; }
// With few endpoints a node the ranges' runs are short: uniform endpoints, 4.2 M edges on
// 4 M nodes 197 us with the ranges and 208 without, 5 M on 8 M 318 and 316, 8 M on 8 M
// 373 and 386; 8 M on 16 M 579 and 557, 16 M on 16 M 753 and 746, 32 M on 16 M 994 and
// 1,009.
inline bool split_degrees(int64_t m, int32_t n) {
    return m >= kDegSplitMin && m >= n && (deg_ranges(n) <= kMaxRanges / 2 || 2 * m >= 3 * int64_t(n)) &&
           deg_ranges(n) <= kMaxRanges;
}

// Endpoint j (0..3) of int4 pair e; an odd last edge is half a pair.
__device__ __forceinline__ int32_t endpoint(const int4 &e, int j) { return j == 0 ? e.x : j == 1 ? e.y : j == 2 ? e.z : e.w; }
__device__ __forceinline__ int4 load_pair(const int32_t *__restrict__ edges, int64_t m, int64_t q, int *have) {
    const int64_t full = m >> 1;
    *have = q < full ? 4 : (q == full && (m & 1) ? 2 : 0);
    if (*have == 4) return __ldcs(reinterpret_cast<const int4 *>(edges) + q);
    if (*have == 2) return make_int4(edges[2 * (m - 1)], edges[2 * (m - 1) + 1], 0, 0);
    return make_int4(0, 0, 0, 0);
}

__global__ void __launch_bounds__(kDegThreads, 2) k_deg_ranges(const int32_t *__restrict__ edges, int64_t m, int32_t n,
                                                               int ranges, uint32_t *__restrict__ count,
                                                               uint32_t *status) {
    constexpr int kHistIn = 2;  // 32 registers: two blocks per SM
    extern __shared__ uint32_t h[];  // [warps][ranges]: a warp's own counters
    uint32_t *mine = h + (threadIdx.x >> 5) * ranges;
    for (int i = threadIdx.x; i < (kDegThreads / 32) * ranges; i += kDegThreads) h[i] = 0u;
    __syncthreads();
    const int64_t pairs = (m + 1) >> 1, stride = int64_t(gridDim.x) * kDegThreads;
    for (int64_t q0 = int64_t(blockIdx.x) * kDegThreads + threadIdx.x; q0 < pairs; q0 += stride * kHistIn) {
        int4 e[kHistIn];
        int have[kHistIn];
#pragma unroll
        for (int r = 0; r < kHistIn; ++r) e[r] = load_pair(edges, m, q0 + r * stride, &have[r]);
#pragma unroll
        for (int r = 0; r < kHistIn; ++r)
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                if (j >= have[r]) continue;
                const uint32_t x = uint32_t(endpoint(e[r], j));
                if (x < uint32_t(n))
                    atomicAdd(&mine[x >> kRangeBits], 1u);
                else
                    raise_status(status, BGV_DEV_BADEDGE);
            }
    }
    __syncthreads();
    for (int b = threadIdx.x; b < ranges; b += kDegThreads) {
        uint32_t c = 0;
        for (int w = 0; w < kDegThreads / 32; ++w) c += h[w * ranges + b];
        if (c) atomicAdd(&count[b], c);
    }
}

// Exclusive scan of v[0, kMaxRanges) into out[0, kMaxRanges]; the first
// kMaxRanges threads of the block hold one value each, every thread calls it.
__device__ __forceinline__ void scan_ranges(uint32_t v, uint32_t *out) {
    __shared__ uint32_t wsum[kMaxRanges / 32];
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    uint32_t inc = v;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, inc, d);
        if (lane >= d) inc += y;
    }
    if (lane == 31 && warp < kMaxRanges / 32) wsum[warp] = inc;
    __syncthreads();
    if (t < kMaxRanges) {
        uint32_t before = 0;
        for (int w = 0; w < warp; ++w) before += wsum[w];
        out[t] = before + inc - v;
        if (t == kMaxRanges - 1) out[kMaxRanges] = before + inc;
    }
    __syncthreads();
}

__global__ void __launch_bounds__(kPlaceThreads, 2) k_deg_place(const int32_t *__restrict__ edges, int64_t m, int32_t n,
                                                              int ranges, const uint32_t *__restrict__ count,
                                                              uint32_t *cursor, uint16_t *__restrict__ local) {
    __shared__ uint16_t stage[kDegTile];
    __shared__ uint32_t cnt[kMaxRanges], lstart[kMaxRanges + 1], start[kMaxRanges + 1], gbase[kMaxRanges];
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    scan_ranges(t < ranges ? count[t] : 0u, start);
    const int64_t pairs = (m + 1) >> 1, tile_pairs = kPlaceThreads * kDegIn;
    for (int64_t p0 = int64_t(blockIdx.x) * tile_pairs; p0 < pairs; p0 += int64_t(gridDim.x) * tile_pairs) {
        if (t < kMaxRanges) cnt[t] = 0u;
        int4 e[kDegIn];
        int have[kDegIn];
#pragma unroll
        for (int r = 0; r < kDegIn; ++r) e[r] = load_pair(edges, m, p0 + r * kPlaceThreads + t, &have[r]);
        __syncthreads();
        uint32_t rank[kDegIn * 4];
#pragma unroll
        for (int r = 0; r < kDegIn; ++r)
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const uint32_t x = uint32_t(endpoint(e[r], j));
                rank[4 * r + j] = j < have[r] && x < uint32_t(n) ? atomicAdd(&cnt[x >> kRangeBits], 1u) : 0xFFFFFFFFu;
            }
        __syncthreads();
        const uint32_t c = t < kMaxRanges ? cnt[t] : 0u;
        if (c) gbase[t] = start[t] + atomicAdd(&cursor[t], c);
        scan_ranges(c, lstart);
#pragma unroll
        for (int r = 0; r < kDegIn; ++r)
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const uint32_t x = uint32_t(endpoint(e[r], j));
                if (rank[4 * r + j] != 0xFFFFFFFFu)
                    stage[lstart[x >> kRangeBits] + rank[4 * r + j]] = uint16_t(x & (kRange - 1));
            }
        __syncthreads();
        for (int b = warp; b < ranges; b += kPlaceThreads / 32) {  // a warp per run
            const uint32_t s = lstart[b], k = lstart[b + 1] - s;
            uint16_t *dst = local + (k ? gbase[b] : 0u);
            for (uint32_t i = lane; i < k; i += 32) dst[i] = stage[s + i];
        }
        __syncthreads();
    }
}

__global__ void __launch_bounds__(kDegThreads, 1) k_deg_count(const uint16_t *__restrict__ local, int32_t n, int ranges,
                                                              const uint32_t *__restrict__ count,
                                                              uint32_t *__restrict__ deg) {
    extern __shared__ uint32_t h[];  // [kRange]
    __shared__ uint32_t start[kMaxRanges + 1], pieces[kMaxRanges + 1];
    const int t = threadIdx.x;
    const uint32_t c = t < ranges ? count[t] : 0u;
    scan_ranges(c, start);
    scan_ranges(pieces_of(c, kDegPiece), pieces);
    const uint32_t total = pieces[kMaxRanges];
    for (uint32_t q = blockIdx.x; q < total; q += gridDim.x) {
        int lo = 0, hi = kMaxRanges;  // the range whose pieces hold q
        while (hi - lo > 1) {
            const int mid = (lo + hi) >> 1;
            if (pieces[mid] <= q) lo = mid; else hi = mid;
        }
        for (int i = t; i < kRange; i += kDegThreads) h[i] = 0u;
        __syncthreads();
        const uint32_t a = start[lo] + (q - pieces[lo]) * kDegPiece;
        const uint32_t b = a + piece_size(a, start[lo + 1], kDegPiece);
        // whole 16-byte words between the ragged ends
        const uint32_t a8 = a + ragged_head(a, b, 8u), b8 = max(b & ~7u, a8);
        if (t < a8 - a) atomicAdd(&h[swz(local[a + t] & (kRange - 1))], 1u);
        if (t < b - b8) atomicAdd(&h[swz(local[b8 + t] & (kRange - 1))], 1u);
        const uint4 *words = reinterpret_cast<const uint4 *>(local);
        for (uint32_t w = a8 / 8 + t; w < b8 / 8; w += kDegThreads) {
            const uint4 v = __ldcs(words + w);
            const uint32_t x[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                atomicAdd(&h[swz(x[k] & (kRange - 1))], 1u);
                atomicAdd(&h[swz((x[k] >> 16) & (kRange - 1))], 1u);
            }
        }
        __syncthreads();
        const int64_t v0 = int64_t(lo) << kRangeBits;
        for (int i = t; i < kRange; i += kDegThreads)
            if (h[swz(i)] && v0 + i < n) atomicAdd(&deg[v0 + i], h[swz(i)]);
        __syncthreads();
    }
}

// Batched form: node v of graph g = node_graph[v] hashes its local id
// v - node_off[g] into graph g's own rows x width matrix.
__device__ __forceinline__ uint32_t *sketch_of(uint32_t *sketch, const HashFamily &h, int64_t v,
                                               const int32_t *node_graph, const int32_t *node_off, uint32_t *x) {
    if (!node_graph) {
        *x = uint32_t(v);
        return sketch;
    }
    const int32_t g = node_graph[v];
    *x = uint32_t(v - node_off[g]);
    return sketch + size_t(g) * size_t(h.rows) * h.width;
}

__global__ void __launch_bounds__(kThreads) k_sketch_fill(const uint32_t *__restrict__ deg, int32_t n,
                                                          const __grid_constant__ HashFamily h,
                                                          uint32_t *__restrict__ sketch,
                                                          const int32_t *__restrict__ node_graph,
                                                          const int32_t *__restrict__ node_off) {
    const int64_t stride = int64_t(gridDim.x) * blockDim.x;
    for (int64_t v = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; v < n; v += stride) {
        uint32_t d = deg[v];
        if (d == 0) continue;
        uint32_t x;
        uint32_t *M = sketch_of(sketch, h, v, node_graph, node_off, &x);
        for (int i = 0; i < h.rows; ++i) atomicAdd(&M[size_t(i) * h.width + hash_eval(h.a[i], h.b[i], x, h.width)], d);
    }
}

__global__ void __launch_bounds__(kThreads) k_sketch_query(const uint32_t *__restrict__ sketch, int32_t n,
                                                           const __grid_constant__ HashFamily h,
                                                           uint32_t *__restrict__ deg_est,
                                                           const int32_t *__restrict__ node_graph,
                                                           const int32_t *__restrict__ node_off) {
    const int64_t stride = int64_t(gridDim.x) * blockDim.x;
    for (int64_t v = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; v < n; v += stride) {
        uint32_t x;
        const uint32_t *M = sketch_of(const_cast<uint32_t *>(sketch), h, v, node_graph, node_off, &x);
        uint32_t best = 0xFFFFFFFFu;
        for (int i = 0; i < h.rows; ++i) {
            uint32_t c = M[size_t(i) * h.width + hash_eval(h.a[i], h.b[i], x, h.width)];
            best = c < best ? c : best;
        }
        deg_est[v] = best;
    }
}
}  // namespace

void carve_sketch(Carver &c, int64_t m, int32_t n, int32_t rows, int32_t width, SketchScratch &s) {
    (void)rows; (void)width;
    s.deg = c.take<uint32_t>(size_t(n));
    const bool split = split_degrees(m, n);
    s.local = split ? c.take<uint16_t>(2 * size_t(m) + 8) : nullptr;
    s.ranges = split ? c.take<uint32_t>(2 * kMaxRanges) : nullptr;
}

int run_sketch(const int32_t *edges, int64_t m, int32_t n, const HashFamily &h, uint32_t *sketch,
               uint32_t *deg_est, const SketchScratch &s, uint32_t *status, cudaStream_t st, const BatchView *batch) {
    const int32_t *node_graph = batch ? batch->node_graph : nullptr;
    const int32_t *node_off = batch ? batch->node_off : nullptr;
    const size_t mats = batch ? size_t(batch->G) : 1;
    BGV_CUDA(cudaMemsetAsync(s.deg, 0, sizeof(uint32_t) * size_t(n), st));
    BGV_CUDA(cudaMemsetAsync(sketch, 0, sizeof(uint32_t) * size_t(h.rows) * h.width * mats, st));
    if (s.local) {
        const int R = deg_ranges(n);
        const size_t hist = sizeof(uint32_t) * (kDegThreads / 32) * size_t(R), counters = sizeof(uint32_t) * kRange;
        uint32_t *count = s.ranges, *cursor = s.ranges + kMaxRanges;
        BGV_CUDA(cudaFuncSetAttribute(k_deg_ranges, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                      int(sizeof(uint32_t) * (kDegThreads / 32) * kMaxRanges)));
        BGV_CUDA(cudaFuncSetAttribute(k_deg_count, cudaFuncAttributeMaxDynamicSharedMemorySize, int(counters)));
        BGV_CUDA(cudaMemsetAsync(s.ranges, 0, sizeof(uint32_t) * 2 * kMaxRanges, st));
        const int64_t pairs = (m + 1) / 2;
        note_launch(), k_deg_ranges<<<grid_for(pairs, kDegThreads * kDegIn, sm_count() * 2), kDegThreads, hist, st>>>(
            edges, m, n, R, count, status);
        BGV_TRY(launch_status());
        note_launch(), k_deg_place<<<grid_for(pairs, kPlaceThreads * kDegIn, sm_count() * 2), kPlaceThreads, 0, st>>>(
            edges, m, n, R, count, cursor, s.local);
        BGV_TRY(launch_status());
        note_launch(), k_deg_count<<<grid_for(2 * m / kDegPiece + R, 1, sm_count()), kDegThreads, counters, st>>>(
            s.local, n, R, count, s.deg);
        BGV_TRY(launch_status());
    } else if (m > 0) {
        note_launch(), k_degree_count<<<grid_for((m / 2 + kDegLoads - 1) / kDegLoads, kThreads, sm_count() * 8), kThreads, 0, st>>>(edges, m, n, s.deg, status);
        BGV_TRY(launch_status());
    }
    note_launch(), k_sketch_fill<<<grid_for(n, kThreads, sm_count() * 8), kThreads, 0, st>>>(s.deg, n, h, sketch, node_graph,
                                                                                       node_off);
    BGV_TRY(launch_status());
    note_launch(), k_sketch_query<<<grid_for(n, kThreads, sm_count() * 8), kThreads, 0, st>>>(sketch, n, h, deg_est, node_graph,
                                                                                        node_off);
    return launch_status();
}

}  // namespace bgv

// ------------------------------------------------------------------------
// bgv_sketch_degrees_noalloc: the degree sketch for callers that cannot
// allocate device memory.
//
// Some callers may not call cudaMalloc at all: a plugin running inside a
// host application whose device memory is owned by another allocator, code
// that runs while a stream is being captured (cudaMalloc is not allowed
// there), or real-time callers that must not allocate on their hot path.
// They cannot hand this library a workspace, so this entry point keeps the
// one scratch array the sketch needs -- the per-node degree counters -- in a
// fixed-size array of device memory that is part of the library image.  The
// caller still provides the edges, the sketch and the estimates.
//
// Size limit: n <= kNoAllocMaxNodes (4,194,304 nodes, 16 MiB of counters).
// Every GPU that loads the library holds that array until the process exits.
// All calls on a device share it and it keeps the last call's contents; the
// counters are cleared at the start of every call.  Calls whose work
// overlaps on the GPU (different streams, no ordering between them) race on
// the shared counters and give wrong results: order them on one stream.
namespace bgv {
namespace {
constexpr int32_t kNoAllocMaxNodes = 1 << 22;
constexpr int kNoAllocMaxDevices = 64;

// Degree counters followed by one status word used when the caller passes
// no status pointer (cleared by every such call and read back at its end).
static __device__ __align__(256) uint32_t g_noalloc_scratch[kNoAllocMaxNodes + 64];

std::mutex g_noalloc_mutex;
uint32_t *g_noalloc_ptr[kNoAllocMaxDevices] = {};

// The array's name is a host-side stand-in in host code, not a device
// address: the address a kernel may use is looked up once per device, with
// that device current, on the first call.
int noalloc_scratch(uint32_t **out) {
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kNoAllocMaxDevices) return BGV_ECUDA;
    std::lock_guard<std::mutex> lock(g_noalloc_mutex);
    if (!g_noalloc_ptr[dev]) {
        void *p = nullptr;
        if (cudaGetSymbolAddress(&p, g_noalloc_scratch) != cudaSuccess || !p) return BGV_ECUDA;
        g_noalloc_ptr[dev] = static_cast<uint32_t *>(p);
    }
    *out = g_noalloc_ptr[dev];
    return BGV_OK;
}
}  // namespace

}  // namespace bgv

extern "C" int bgv_sketch_degrees_noalloc(const int32_t *edges, int64_t m, int32_t n, int32_t rows, int32_t width,
                                          uint64_t seed, uint32_t *sketch, uint32_t *deg_est, uint32_t *status,
                                          void *stream) {
    using namespace bgv;
    if (n < 1 || m < 0 || m >= (int64_t(1) << 31)) return BGV_EINVAL;
    if (m > 0 && (!edges || reinterpret_cast<uintptr_t>(edges) % 16 != 0)) return BGV_EINVAL;
    if (rows < 1 || rows > kMaxRows || width < 1 || !sketch || !deg_est) return BGV_EINVAL;
    if (n > kNoAllocMaxNodes) return BGV_ELIMIT;
    uint32_t *scratch = nullptr;
    BGV_TRY(noalloc_scratch(&scratch));
    SketchScratch s{};  // the counters alone: no room to sort the endpoints by range
    s.deg = scratch;
    cudaStream_t cs = static_cast<cudaStream_t>(stream);
    const HashFamily h = make_hash_family(seed, rows, uint32_t(width));
    if (status) return run_sketch(edges, m, n, h, sketch, deg_est, s, status, cs);
    // No status word from the caller: use the one after the counters, cleared
    // on every call, and report what the device found before returning.
    uint32_t *own = scratch + kNoAllocMaxNodes;
    BGV_CUDA(cudaMemsetAsync(own, 0, sizeof(uint32_t), cs));
    BGV_TRY(run_sketch(edges, m, n, h, sketch, deg_est, s, own, cs));
    uint32_t seen = 0;
    BGV_CUDA(cudaMemcpyAsync(&seen, own, sizeof(uint32_t), cudaMemcpyDeviceToHost, cs));
    BGV_CUDA(cudaStreamSynchronize(cs));
    return seen ? BGV_EDEVICE : BGV_OK;
}

