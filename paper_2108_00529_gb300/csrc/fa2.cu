// fa2.cu -- ForceAtlas2 on the supergraph (Section 3.1, Algorithm 1).
//
// One iteration is a fixed chain of kernels with no host round trip:
//   k_frame     bounding square of the positions (last-block finalise); the
//               later steps of a run find it made by the tail before them
//   k_hs_*      (key, body) pairs -> Morton order: fixed-point coordinates U and
//               2L-bit Morton keys, to buckets between the previous step's
//               pairs (a first step: between sampled ones), sorted there
//               (hsort.cuh).  First steps of more than 65,536 bodies take k_keys
//               and the radix sort: LSD passes on the bits above 24, then each
//               run of equal high bits ordered locally
//   k_tile*     bodies in Morton order, quadtree cells with FP32 centres from
//               exact integer moments, and the depth-first pre-order with skip
//               indices (tree.cuh)
//   k_repulse   Barnes-Hut repulsion: one thread per body walks the
//               pre-order array without a stack (accept -> skip past the
//               subtree, open -> next element); every body takes its own
//               opening decisions, so its interaction set is exactly the
//               one the definition gives
//   k_att_*     attraction, rows by length class: short rows one lane
//               each, medium rows one warp each, long rows one block each
//               (the class lists are made once per CSR).  They run on a
//               second stream while the tree is built and walked.
//   k_tail      one persistent kernel (cooperative launch, bounded grid
//               barriers): per node gravity, total force, swing and
//               traction, summed exactly (integer accumulation); the global
//               speed (per graph in the batched form); per node the local
//               speed, the displacement and Fprev = F; the next step's frame
//   (k_node gives the forces alone, without a step)
//
// The opening test and the centre it uses are computed with explicit
// round-to-nearest FP32 operations (no contraction) from the exact integer
// moments, so the decisions do not depend on thread scheduling and equal
// the oracle's decisions on the same positions.
#include <atomic>

#include "bgv_internal.cuh"
#include "forces.cuh"
#include "hsort.cuh"
#include "tree.cuh"
#include "small.cuh"

namespace bgv {

namespace {
constexpr int kThreads = 256;
constexpr int kMaxFrameBlocks = 1024;  // frame-kernel grid: 2 blocks per SM, at most this many
constexpr int kMaxNodeBlocks = 2048;   // node-kernel and tail grids: at most this many blocks
inline int frame_blocks() { return sm_count() * 2 < kMaxFrameBlocks ? sm_count() * 2 : kMaxFrameBlocks; }
// Bodies per warp when `blocks` blocks share K of them, in whole rows of 32.
inline int64_t warp_share(int64_t K, int blocks) {
    const int64_t warps = int64_t(blocks) * (kThreads / 32);
    return ((K + warps - 1) / warps + 31) / 32 * 32;
}
inline int node_blocks() { return sm_count() * 4 < kMaxNodeBlocks ? sm_count() * 4 : kMaxNodeBlocks; }

// ----------------------------------------------------------------- frame
// Block-wide box; every thread calls it, thread 0 receives the result.
__device__ __forceinline__ void box_block(float4 &b) {
    __shared__ float4 wbox[kThreads / 32];
    box_warp(b);
    if ((threadIdx.x & 31) == 0) wbox[threadIdx.x >> 5] = b;
    __syncthreads();
    if (threadIdx.x == 0)
        for (int w = 1; w < kThreads / 32; ++w) box_merge(b, wbox[w]);
    __syncthreads();
}

// The frame of all blocks' boxes: block partials, then the last block reduces
// them, all threads at once (min and max do not depend on the order).  Every
// thread of every block calls it.
__device__ __forceinline__ void box_to_frame(float4 b, float4 *part, float4 *frame, unsigned int *ticket) {
    __shared__ bool last;
    box_block(b);
    if (threadIdx.x == 0) {
        part[blockIdx.x] = b;
        __threadfence();
        last = atomicAdd(ticket, 1u) == gridDim.x - 1;
    }
    __syncthreads();
    if (!last) return;
    __threadfence();
    b = box_empty();
    for (unsigned k = threadIdx.x; k < gridDim.x; k += blockDim.x) box_merge(b, __ldcg(&part[k]));
    box_block(b);
    if (threadIdx.x == 0) {
        *frame = frame_of(b.x, b.y, b.z, b.w);
        *ticket = 0u;
    }
}

// First step of a run, and single steps: later steps of a run find the frame
// made by the step before (k_tail).
__global__ void __launch_bounds__(kThreads) k_frame(const float2 *__restrict__ pos, int64_t K, float4 *part,
                                                    float4 *frame, unsigned int *ticket) {
    float4 b = box_empty();
    const int64_t stride = int64_t(gridDim.x) * blockDim.x;
    for (int64_t i = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; i < K; i += stride) box_add(b, pos[i]);
    box_to_frame(b, part, frame, ticket);
}

// Bounding boxes of the batched form: four ordered integers per graph (a
// float's bits, flipped so that unsigned order is float order), so a box is
// the atomic min and max of its parts, whatever their order.
__device__ __forceinline__ uint32_t box_key(float f) {
    const uint32_t b = __float_as_uint(f);
    return (b & 0x80000000u) ? ~b : b | 0x80000000u;
}
__device__ __forceinline__ float box_val(uint32_t k) {
    return __uint_as_float((k & 0x80000000u) ? k & 0x7FFFFFFFu : ~k);
}
__device__ __forceinline__ uint4 box_keys_empty() {
    return make_uint4(box_key(INFINITY), box_key(INFINITY), box_key(-INFINITY), box_key(-INFINITY));
}
__device__ __forceinline__ void box_publish(uint4 *box, const float4 &b) {
    atomicMin(&box->x, box_key(b.x));
    atomicMin(&box->y, box_key(b.y));
    atomicMax(&box->z, box_key(b.z));
    atomicMax(&box->w, box_key(b.w));
}

__global__ void __launch_bounds__(kThreads) k_box_init(int32_t G, uint4 *__restrict__ box) {
    for (int32_t g = blockIdx.x * blockDim.x + threadIdx.x; g < G; g += gridDim.x * blockDim.x)
        box[g] = box_keys_empty();
}

// Frames from the finished boxes, which are emptied for the next step.
__global__ void __launch_bounds__(kThreads) k_frame_fin(int32_t G, uint4 *__restrict__ box,
                                                        float4 *__restrict__ frames) {
    for (int32_t g = blockIdx.x * blockDim.x + threadIdx.x; g < G; g += gridDim.x * blockDim.x) {
        const uint4 b = box[g];
        frames[g] = frame_of(box_val(b.x), box_val(b.y), box_val(b.z), box_val(b.w));
        box[g] = box_keys_empty();
    }
}

// Graph of body i: the largest g with koff[g] <= i.
__device__ __forceinline__ int32_t body_graph(const int64_t *__restrict__ koff, int32_t G, int64_t i) {
    int32_t lo = 0, hi = G;
    while (hi - lo > 1) {
        const int32_t mid = (lo + hi) >> 1;
        if (koff[mid] <= i) lo = mid; else hi = mid;
    }
    return lo;
}

// Batched form, first step of a run: the graph of every body and the boxes.
// Warp w takes bodies [w per, (w + 1) per) and walks the graphs in them (one
// block per graph left most of the GPU idle behind the largest graphs: 110 us
// for 6.0 M bodies in 160 graphs).
__global__ void __launch_bounds__(kThreads) k_frame_seg(const float2 *__restrict__ pos, int64_t K, int64_t per,
                                                        const int64_t *__restrict__ koff, int32_t G,
                                                        uint4 *__restrict__ box, int32_t *__restrict__ bgraph) {
    const int lane = threadIdx.x & 31;
    int64_t lo = ((int64_t(blockIdx.x) * blockDim.x + threadIdx.x) >> 5) * per;
    if (lo >= K) return;
    const int64_t end = lo + per < K ? lo + per : K;
    for (int32_t g = body_graph(koff, G, lo); lo < end; ++g) {
        const int64_t hi = koff[g + 1] < end ? koff[g + 1] : end;
        float4 b = box_empty();
        for (int64_t i = lo + lane; i < hi; i += 32) {
            box_add(b, pos[i]);
            bgraph[i] = g;
        }
        box_warp(b);
        if (lane == 0) box_publish(&box[g], b);
        lo = hi;
    }
}

// ------------------------------------------------------------------ keys
// Morton key of the body's fixed-point position in its graph's frame; in the
// batched form the graph id sits above the 2L Morton bits, so each graph's
// bodies stay together and form their own subtree.
__device__ __forceinline__ unsigned long long morton_key(const float2 *__restrict__ pos,
                                                         const float4 *__restrict__ frames,
                                                         const int32_t *__restrict__ bgraph, int L, int64_t i) {
    const int g = bgraph ? bgraph[i] : 0;
    const uint2 U = fixed_point(pos[i], frames[g]);
    const uint32_t qx = U.x >> (32 - L), qy = U.y >> (32 - L);
    return (static_cast<unsigned long long>(g) << (2 * L)) | (spread_bits(qx) << 1) | spread_bits(qy);
}

// The same key by body id, for the hinted sort.
struct MortonOf {
    const float2 *pos;
    const float4 *frames;
    const int32_t *bgraph;
    int L;
    __device__ unsigned long long operator()(uint32_t id) const { return morton_key(pos, frames, bgraph, L, id); }
};

// Also clears, for the kernels after it, the step's counters (2 words), the
// tiles' flags and the sort's digit counters: the launches that
// would otherwise clear them sit on the step's dependency chain.
__global__ void __launch_bounds__(kThreads) k_keys(const float2 *__restrict__ pos, int64_t K,
                                                   const float4 *__restrict__ frames,
                                                   const int32_t *__restrict__ bgraph, int L,
                                                   unsigned long long *__restrict__ keys,
                                                   uint32_t *__restrict__ vals,
                                                   unsigned long long *__restrict__ step_counters,
                                                   uint32_t *__restrict__ clear_a, int64_t n_a,
                                                   uint32_t *__restrict__ clear_b, int64_t n_b) {
    const int64_t stride = int64_t(gridDim.x) * blockDim.x;
    for (int64_t t = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; t < n_a || t < n_b || t < 2; t += stride) {
        if (t < 2) step_counters[t] = 0ull;
        if (t < n_a) clear_a[t] = 0u;
        if (t < n_b) clear_b[t] = 0u;
    }
    for (int64_t i = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; i < K; i += stride) {
        keys[i] = morton_key(pos, frames, bgraph, L, i);
        vals[i] = uint32_t(i);
    }
}

// -------------------------------------------------------------- repulsion
// Barnes-Hut traversal, one body per thread (bh_walk).  Each body sees exactly
// its own interaction set in depth-first order; threads of a warp are Morton
// neighbours, so they mostly read the same elements.
template <int kRT>
__global__ void __launch_bounds__(kRT) k_repulse(const float4 *geo, const int32_t *skip, const uint32_t *T,
                                                      const int64_t *__restrict__ koff,
                                                      const int32_t *__restrict__ bgraph,
                                                      const float4 *__restrict__ body, int64_t K, float kr,
                                                      float theta2, float2 *__restrict__ Frep,
                                                      unsigned long long *inter_step,
                                                      unsigned long long *inter_total) {
    chain_wait();
    const int64_t s = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
    unsigned inter = 0;
    if (s < K) {
        const float4 bi = body[s];
        const float kmi = kr * bi.z;
        const uint32_t self = uint32_t(s + T[s + 1]);
        // the body's own graph: its subtree spans [start, end) in pre-order
        uint32_t cur = 0, end = uint32_t(K + T[K]);
        if (bgraph) {
            const int g = bgraph[s];
            const int64_t a = koff[g], b = koff[g + 1];
            cur = uint32_t(a + T[a]);
            end = uint32_t(b + T[b]);
        }
        Frep[__float_as_int(bi.w)] = bh_walk(geo, skip, bi, kmi, theta2, self, cur, end, inter);
    }
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) inter += __shfl_xor_sync(0xFFFFFFFFu, inter, d);
    if ((threadIdx.x & 31) == 0 && inter) {
        atomicAdd(inter_step, static_cast<unsigned long long>(inter));
        atomicAdd(inter_total, static_cast<unsigned long long>(inter));
    }
}

// ------------------------------------------------------------ attraction
// F^a_i = sum over row i's CSR entries (j, w) of w (p_j - p_i), in FP32.
// Every row is summed by one worker in an order that depends only on the
// row's own entries (deterministic, and the same whatever else the CSR
// holds).  The plan, made once per CSR, lists the rows by length: short rows
// (at most `att_short` entries) take one lane each, 32 rows to a warp, and
// add their entries in order; medium rows (up to kAttMedium entries) take
// one warp each, two rows at a time: lane l adds entries l, l + 32, ... in order, then a fixed
// butterfly; long rows take one block each (thread t adds t, t + 256, ...,
// then a fixed tree).  Every worker first issues kAttIn loads of neighbour
// ids and weights, then their position gathers, so they are in flight
// together.  An empty row is a short row of sum 0.
// loads in flight per worker; with 5 blocks of 256 per SM (at most 51
// registers) that is 320 outstanding gathers per SM
constexpr int kAttIn = 8;

// Block-aggregated append of row r to the list of class c (one atomic per
// class per block).
__global__ void __launch_bounds__(kThreads) k_att_plan(int64_t K, const int32_t *__restrict__ off, int att_short,
                                                       int32_t *__restrict__ rows_short, int32_t *__restrict__ rows_med,
                                                       int32_t *__restrict__ rows_long, uint32_t *counts) {
    __shared__ uint32_t wn[3][kThreads / 32], base[3];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int64_t r0 = int64_t(blockIdx.x) * blockDim.x; r0 < K; r0 += int64_t(gridDim.x) * blockDim.x) {
        const int64_t r = r0 + threadIdx.x;
        int c = -1;
        if (r < K) {
            const int64_t len = int64_t(off[r + 1]) - off[r];
            c = len <= att_short ? 0 : (len <= kAttMedium ? 1 : 2);
        }
        unsigned m[3];
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            m[k] = __ballot_sync(0xFFFFFFFFu, c == k);
            if (lane == 0) wn[k][warp] = uint32_t(__popc(m[k]));
        }
        __syncthreads();
        if (threadIdx.x < 3) {
            const int k = threadIdx.x;
            uint32_t t = 0;
            for (int w = 0; w < kThreads / 32; ++w) {
                const uint32_t x = wn[k][w];
                wn[k][w] = t;
                t += x;
            }
            base[k] = t ? atomicAdd(&counts[k], t) : 0u;
        }
        __syncthreads();
        if (c >= 0) {
            int32_t *list = c == 0 ? rows_short : (c == 1 ? rows_med : rows_long);
            list[base[c] + wn[c][warp] + __popc(m[c] & ((1u << lane) - 1u))] = int32_t(r);
        }
        __syncthreads();
    }
}

// Short rows: one lane each, by up to 64 blocks per SM: blocks that end early leave
// their places to the main chain (500 steps of 1 M bodies with uniform rows 175.4 ms
// with 16 per SM, 170.6 with 64).  Where there is a medium row, whose launch follows,
// for every 32 short ones or more, only `wave` blocks work, 16 per SM (150 steps of
// 3.2 M bodies of an R-MAT graph 161.7 ms with 16, 169 with 64).
__global__ void __launch_bounds__(kThreads, 5) k_att_short(int64_t K, const int32_t *__restrict__ off,
                                                        const int32_t *__restrict__ adj,
                                                        const uint32_t *__restrict__ w,
                                                        const float2 *__restrict__ pos,
                                                        const int32_t *__restrict__ rows, const uint32_t *counts,
                                                        unsigned wave, float2 *__restrict__ full) {
    const int64_t count = counts[0];
    const unsigned blocks = int64_t(counts[1]) * 32 >= count && wave < gridDim.x ? wave : gridDim.x;
    if (blockIdx.x >= blocks) return;
    const int64_t stride = int64_t(blocks) * blockDim.x;
    for (int64_t q = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; q < count; q += stride) {
        const int32_t r = rows[q];
        const int64_t b = off[r], e = off[r + 1];
        const float2 pi = pos[r];
        float ax = 0.0f, ay = 0.0f;
        for (int64_t e0 = b; e0 < e; e0 += kAttIn) {
            int32_t j[kAttIn];
            uint32_t wt[kAttIn];
#pragma unroll
            for (int k = 0; k < kAttIn; ++k) {
                j[k] = e0 + k < e ? __ldcs(adj + e0 + k) : -1;
                wt[k] = e0 + k < e ? __ldcs(w + e0 + k) : 0u;
            }
            float2 pj[kAttIn];
#pragma unroll
            for (int k = 0; k < kAttIn; ++k) pj[k] = valid_row(j[k], K) ? pos[j[k]] : pi;
#pragma unroll
            for (int k = 0; k < kAttIn; ++k) {
                const float wf = valid_row(j[k], K) ? __uint2float_rn(wt[k]) : 0.0f;
                ax += wf * (pj[k].x - pi.x);
                ay += wf * (pj[k].y - pi.y);
            }
        }
        full[r] = make_float2(ax, ay);
    }
}

// Medium rows: one warp each, two rows at a time (each lane keeps
// kAttIn / 2 loads in flight per row, so a warp waits on two rows' round
// trips at once).  Lane l adds entries l, l + 32, ... of a row in order, then
// a fixed butterfly: the sums do not depend on how the rows are paired.
__global__ void __launch_bounds__(kThreads, 4) k_att_medium(int64_t K, const int32_t *__restrict__ off,
                                                         const int32_t *__restrict__ adj,
                                                         const uint32_t *__restrict__ w,
                                                         const float2 *__restrict__ pos,
                                                         const int32_t *__restrict__ rows, const uint32_t *counts,
                                                         float2 *__restrict__ full) {
    constexpr int kIn = kAttIn / 2;
    const int lane = threadIdx.x & 31;
    const int64_t count = counts[1];
    const int64_t warps = (int64_t(gridDim.x) * blockDim.x) >> 5;
    for (int64_t q = ((int64_t(blockIdx.x) * blockDim.x + threadIdx.x) >> 5) * 2; q < count; q += warps * 2) {
        const bool two = q + 1 < count;
        const int32_t r0 = rows[q], r1 = two ? rows[q + 1] : r0;
        const int64_t b0 = off[r0], len0 = int64_t(off[r0 + 1]) - b0;
        const int64_t b1 = off[r1], len1 = two ? int64_t(off[r1 + 1]) - b1 : 0;
        const float2 p0 = pos[r0], p1 = pos[r1];
        float ax0 = 0.0f, ay0 = 0.0f, ax1 = 0.0f, ay1 = 0.0f;
        const int64_t len = len0 > len1 ? len0 : len1;
        for (int64_t t0 = lane; t0 < len; t0 += 32 * kIn) {
            int32_t j0[kIn], j1[kIn];
            uint32_t w0[kIn], w1[kIn];
#pragma unroll
            for (int k = 0; k < kIn; ++k) {
                const int64_t t = t0 + 32 * k;
                j0[k] = t < len0 ? __ldcs(adj + b0 + t) : -1;
                w0[k] = t < len0 ? __ldcs(w + b0 + t) : 0u;
                j1[k] = t < len1 ? __ldcs(adj + b1 + t) : -1;
                w1[k] = t < len1 ? __ldcs(w + b1 + t) : 0u;
            }
            float2 q0[kIn], q1[kIn];
#pragma unroll
            for (int k = 0; k < kIn; ++k) {
                q0[k] = valid_row(j0[k], K) ? pos[j0[k]] : p0;
                q1[k] = valid_row(j1[k], K) ? pos[j1[k]] : p1;
            }
#pragma unroll
            for (int k = 0; k < kIn; ++k) {
                const float wf0 = valid_row(j0[k], K) ? __uint2float_rn(w0[k]) : 0.0f;
                const float wf1 = valid_row(j1[k], K) ? __uint2float_rn(w1[k]) : 0.0f;
                ax0 += wf0 * (q0[k].x - p0.x);
                ay0 += wf0 * (q0[k].y - p0.y);
                ax1 += wf1 * (q1[k].x - p1.x);
                ay1 += wf1 * (q1[k].y - p1.y);
            }
        }
#pragma unroll
        for (int d = 16; d > 0; d >>= 1) {
            ax0 += __shfl_xor_sync(0xFFFFFFFFu, ax0, d);
            ay0 += __shfl_xor_sync(0xFFFFFFFFu, ay0, d);
            ax1 += __shfl_xor_sync(0xFFFFFFFFu, ax1, d);
            ay1 += __shfl_xor_sync(0xFFFFFFFFu, ay1, d);
        }
        if (lane == 0) {
            full[r0] = make_float2(ax0, ay0);
            if (two) full[r1] = make_float2(ax1, ay1);
        }
    }
}

// Long rows: one block each.
__global__ void __launch_bounds__(kThreads) k_att_long(int64_t K, const int32_t *__restrict__ off,
                                                       const int32_t *__restrict__ adj, const uint32_t *__restrict__ w,
                                                       const float2 *__restrict__ pos, const int32_t *__restrict__ rows,
                                                       const uint32_t *counts, float2 *__restrict__ full) {
    __shared__ float2 wsum[kThreads / 32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t count = counts[2];
    for (int64_t q = blockIdx.x; q < count; q += gridDim.x) {
        const int32_t r = rows[q];
        const int64_t b = off[r], e = off[r + 1];
        const float2 pi = pos[r];
        float ax = 0.0f, ay = 0.0f;
        for (int64_t e0 = b + threadIdx.x; e0 < e; e0 += int64_t(kThreads) * kAttIn) {
            int32_t j[kAttIn];
            uint32_t wt[kAttIn];
#pragma unroll
            for (int k = 0; k < kAttIn; ++k) {
                const int64_t x = e0 + int64_t(kThreads) * k;
                j[k] = x < e ? __ldcs(adj + x) : -1;
                wt[k] = x < e ? __ldcs(w + x) : 0u;
            }
            float2 pj[kAttIn];
#pragma unroll
            for (int k = 0; k < kAttIn; ++k) pj[k] = valid_row(j[k], K) ? pos[j[k]] : pi;
#pragma unroll
            for (int k = 0; k < kAttIn; ++k) {
                const float wf = valid_row(j[k], K) ? __uint2float_rn(wt[k]) : 0.0f;
                ax += wf * (pj[k].x - pi.x);
                ay += wf * (pj[k].y - pi.y);
            }
        }
#pragma unroll
        for (int d = 16; d > 0; d >>= 1) {
            ax += __shfl_xor_sync(0xFFFFFFFFu, ax, d);
            ay += __shfl_xor_sync(0xFFFFFFFFu, ay, d);
        }
        if (lane == 0) wsum[warp] = make_float2(ax, ay);
        __syncthreads();
        if (threadIdx.x == 0) {
            float2 t = wsum[0];
            for (int k = 1; k < kThreads / 32; ++k) {
                t.x += wsum[k].x;
                t.y += wsum[k].y;
            }
            full[r] = t;
        }
        __syncthreads();
    }
}

// ------------------------------------------------- node forces and tail
// Forces only (no state change): repulsion, attraction and gravity per node.
__global__ void __launch_bounds__(kThreads) k_node(int64_t K, const float2 *__restrict__ att,
                                                   const uint32_t *__restrict__ mass, const float2 *__restrict__ pos,
                                                   const float2 *__restrict__ Frep, float kg, int strong,
                                                   float2 *__restrict__ Fr_out, float2 *__restrict__ Fa_out,
                                                   float2 *__restrict__ Fg_out) {
    const int64_t stride = int64_t(gridDim.x) * blockDim.x;
    for (int64_t i = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; i < K; i += stride) {
        const float m = __uint2float_rn(mass[i]);
        const float2 pi = pos[i];
        if (Fr_out) Fr_out[i] = Frep[i];
        if (Fa_out) Fa_out[i] = att ? att[i] : make_float2(0.0f, 0.0f);
        if (Fg_out) Fg_out[i] = node_force(i, nullptr, m, pi, make_float2(0.0f, 0.0f), kg, strong);
    }
}

// The step's tail in one persistent kernel (all blocks resident at once,
// cooperative launch): per node the total force and the swing and traction
// products, summed exactly; a grid barrier; the global speed; then per node
// the local speed and the displacement, Fprev = F, and the bounding box of the
// new positions, so that the next step of a run starts with its frame.  The
// barrier waits are bounded and report BGV_DEV_TIMEOUT.
// Warp w takes nodes [w per, (w + 1) per), four to a lane and pass, and the
// grid has no more blocks than it takes to give every thread kTailItems nodes:
// a barrier over hundreds of blocks cost more than the work of a few thousand
// nodes (measured at K = 60,013: 21.4 us with 608 blocks).
// Batched (kB): a warp walks the graphs in its nodes and leaves one exact
// partial per graph, at slot w + g (every step along the walk raises one of the
// two, so slots are distinct); after the barrier a warp per graph merges its
// partials and sets its speed; a second barrier.  (One block per graph summing
// that graph's rows took 569 us for 6.0 M nodes in 160 graphs; with this split
// and the frames from the tail, 300 steps of that batch take 556.9 ms instead
// of 689.2, and 200 steps of a 1,000-node layout 12.4 ms instead of 14.7.)
// att == nullptr: no CSR entries, no attraction.
constexpr int kTailItems = 4;  // nodes a lane takes per pass, every load issued before the arithmetic

template <bool kB>
__global__ void __launch_bounds__(kThreads, 3) k_tail(int64_t K, int64_t per, const float2 *__restrict__ att,
                                                   const uint32_t *__restrict__ mass, float2 *__restrict__ pos,
                                                   const float2 *__restrict__ Frep, float kg, int strong,
                                                   float2 *__restrict__ F, float2 *__restrict__ Fprev, XPart *part,
                                                   double *speed, float tau, float ks, float ksmax, WsHeader *hdr,
                                                   const int64_t *__restrict__ koff, int32_t G, uint4 *box,
                                                   float4 *frame_part, float4 *frame, int spin_limit) {
    __shared__ double sp_sh;
    const int lane = threadIdx.x & 31;
    const int64_t warp = (int64_t(blockIdx.x) * blockDim.x + threadIdx.x) >> 5;
    const int64_t warps = (int64_t(gridDim.x) * blockDim.x) >> 5;
    const int64_t c_lo = warp * per < K ? warp * per : K;
    const int64_t c_hi = c_lo + per < K ? c_lo + per : K;
    const double sp_old = kB ? 0.0 : *speed;  // read by every block before anyone writes it
    const float2 z = make_float2(0.0f, 0.0f);
    const int32_t g_first = kB && c_lo < c_hi ? body_graph(koff, G, c_lo) : 0;
    XSum S = xsum_zero(), T = xsum_zero();
    auto sum_forces = [&](int64_t lo, int64_t hi) {
        for (int64_t i0 = lo + lane; i0 < hi; i0 += 32 * kTailItems) {
            uint32_t mk[kTailItems];
            float2 pk[kTailItems], rk[kTailItems], ak[kTailItems], qk[kTailItems];
#pragma unroll
            for (int k = 0; k < kTailItems; ++k) {
                const int64_t i = i0 + 32 * k;
                const bool in = i < hi;
                mk[k] = in ? mass[i] : 0u;
                pk[k] = in ? pos[i] : z;
                rk[k] = in ? Frep[i] : z;
                ak[k] = in && att ? att[i] : z;
                qk[k] = in ? Fprev[i] : z;
            }
#pragma unroll
            for (int k = 0; k < kTailItems; ++k) {
                const int64_t i = i0 + 32 * k;
                if (i >= hi) continue;
                const float m = __uint2float_rn(mk[k]);
                const float2 f = force_sum(ak[k], m, pk[k], rk[k], kg, strong);
                F[i] = f;
                const float2 st = swing_traction(m, f.x, f.y, qk[k].x, qk[k].y);
                xsum_add(S, st.x);
                xsum_add(T, st.y);
            }
        }
    };
    if (!kB) {
        sum_forces(c_lo, c_hi);
        xsum_block<kThreads>(S, T);
        if (threadIdx.x == 0) {
            part[2 * blockIdx.x] = xsum_pack(S);
            part[2 * blockIdx.x + 1] = xsum_pack(T);
        }
        if (!grid_barrier(&hdr->bar, spin_limit, &hdr->status)) return;
        // every block merges the block partials, so all hold the same speed
        S = xsum_zero();
        T = xsum_zero();
        for (unsigned bk = threadIdx.x; bk < gridDim.x; bk += blockDim.x) {
            S = xsum_merge(S, xsum_unpack(&part[2 * bk]));
            T = xsum_merge(T, xsum_unpack(&part[2 * bk + 1]));
        }
        xsum_block<kThreads>(S, T);
        if (threadIdx.x == 0) {
            const double Ssum = xsum_value(S), Tsum = xsum_value(T);
            sp_sh = speed_update(sp_old, Ssum, Tsum, tau);
            if (blockIdx.x == 0) {
                *speed = sp_sh;
                hdr->S = Ssum;
                hdr->T = Tsum;
                hdr->steps_total += 1;
            }
        }
        __syncthreads();
    } else {
        int32_t g = g_first;
        for (int64_t lo = c_lo; lo < c_hi; ++g) {
            const int64_t hi = koff[g + 1] < c_hi ? koff[g + 1] : c_hi;
            S = xsum_zero();
            T = xsum_zero();
            sum_forces(lo, hi);
            xsum_warp(S, T);
            if (lane == 0) {
                part[2 * (warp + g)] = xsum_pack(S);
                part[2 * (warp + g) + 1] = xsum_pack(T);
            }
            lo = hi;
        }
        if (!grid_barrier(&hdr->bar, spin_limit, &hdr->status)) return;
        for (int64_t q = warp; q < G; q += warps) {  // a warp per graph: the warps its nodes lie in
            const int64_t w0 = koff[q] / per, w1 = (koff[q + 1] - 1) / per;
            S = xsum_zero();
            T = xsum_zero();
            for (int64_t w = w0 + lane; w <= w1; w += 32) {
                S = xsum_merge(S, xsum_unpack(&part[2 * (w + q)]));
                T = xsum_merge(T, xsum_unpack(&part[2 * (w + q) + 1]));
            }
            xsum_warp(S, T);
            if (lane == 0) {
                const double Ssum = xsum_value(S), Tsum = xsum_value(T);
                speed[q] = speed_update(speed[q], Ssum, Tsum, tau);
                if (q == 0) {
                    hdr->S = Ssum;
                    hdr->T = Tsum;
                    hdr->steps_total += 1;
                }
            }
        }
        if (!grid_barrier(&hdr->bar, spin_limit, &hdr->status)) return;
    }
    float4 b = box_empty();
    auto move = [&](int64_t lo, int64_t hi, float sp) {
        for (int64_t i0 = lo + lane; i0 < hi; i0 += 32 * kTailItems) {
            float2 fk[kTailItems], qk[kTailItems], pk[kTailItems];
#pragma unroll
            for (int k = 0; k < kTailItems; ++k) {
                const int64_t i = i0 + 32 * k;
                const bool in = i < hi;
                fk[k] = in ? F[i] : z;  // written by this thread before the barrier
                qk[k] = in ? Fprev[i] : z;
                pk[k] = in ? pos[i] : z;
            }
#pragma unroll
            for (int k = 0; k < kTailItems; ++k) {
                const int64_t i = i0 + 32 * k;
                if (i >= hi) continue;
                const float2 p = displaced(pk[k], fk[k], qk[k], sp, ks, ksmax);
                pos[i] = p;
                Fprev[i] = fk[k];
                box_add(b, p);
            }
        }
    };
    if (!kB) {
        move(c_lo, c_hi, float(sp_sh));
        box_to_frame(b, frame_part, frame, &hdr->bbox_ticket);
    } else {
        int32_t g = g_first;
        for (int64_t lo = c_lo; lo < c_hi; ++g) {
            const int64_t hi = koff[g + 1] < c_hi ? koff[g + 1] : c_hi;
            b = box_empty();
            move(lo, hi, float(__ldcg(&speed[g])));
            box_warp(b);
            if (lane == 0) box_publish(&box[g], b);
            lo = hi;
        }
    }
}

// -------------------------------------------------------------------- init
__global__ void __launch_bounds__(kThreads) k_init(int64_t K, unsigned long long seed, float R, float2 *pos,
                                                   float2 *Fprev) {
    const int64_t stride = int64_t(gridDim.x) * blockDim.x;
    const float R2 = __fmul_rn(R, 2.0f);
    for (int64_t i = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; i < K; i += stride) {
        float c[2];
#pragma unroll
        for (int axis = 0; axis < 2; ++axis) {
            unsigned long long z = seed + 2ull * static_cast<unsigned long long>(i) + unsigned(axis);
            z += 0x9E3779B97F4A7C15ull;
            z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
            z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
            z ^= z >> 31;
            const float U = __fmul_rn(__uint2float_rn(uint32_t(z >> 40)), 5.9604644775390625e-08f);  // 2^-24
            c[axis] = __fsub_rn(__fmul_rn(U, R2), R);
        }
        pos[i] = make_float2(c[0], c[1]);
        Fprev[i] = make_float2(0.0f, 0.0f);
    }
}

__global__ void k_set_speed(double *speed) { *speed = 1.0; }

// Batched form: graph g starts exactly as it would alone (local index, its
// own square of side 2 sqrt(K_g)) with speed 1.
__global__ void __launch_bounds__(kThreads) k_init_seg(const int64_t *__restrict__ koff, unsigned long long seed,
                                                       float2 *pos, float2 *Fprev, double *speed) {
    const int g = blockIdx.x;
    const int64_t a = koff[g], b = koff[g + 1];
    const float R = sqrtf(float(b - a));
    const float R2 = __fmul_rn(R, 2.0f);
    for (int64_t i = a + threadIdx.x; i < b; i += blockDim.x) {
        const int64_t local = i - a;
        float c[2];
#pragma unroll
        for (int axis = 0; axis < 2; ++axis) {
            unsigned long long z = seed + 2ull * static_cast<unsigned long long>(local) + unsigned(axis);
            z += 0x9E3779B97F4A7C15ull;
            z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
            z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
            z ^= z >> 31;
            const float U = __fmul_rn(__uint2float_rn(uint32_t(z >> 40)), 5.9604644775390625e-08f);  // 2^-24
            c[axis] = __fsub_rn(__fmul_rn(U, R2), R);
        }
        pos[i] = make_float2(c[0], c[1]);
        Fprev[i] = make_float2(0.0f, 0.0f);
    }
    if (threadIdx.x == 0) speed[g] = 1.0;
}
}  // namespace

// ------------------------------------------------------------- scratch
struct Fa2Scratch {
    float4 *frame;         // frames: one per graph
    float4 *frame_part;
    int32_t *bgraph;       // batched form: graph of each body
    uint4 *box;            // batched form: bounding box of each graph (ordered integers)
    SortBuffers sort;
    RunFixBuffers runfix;
    float4 *body;          // sorted bodies: x, y, mass, index
    TileArrays tree;
    uint32_t *T;           // cells whose first body precedes each body, K + 1 entries
    float4 *geo;           // pre-order elements (cells and bodies)
    int32_t *skip;         // pre-order index after each element's subtree
    float2 *Frep;
    float2 *full;          // attraction per row
    int32_t *rows_short, *rows_med, *rows_long;  // plan: rows by length class
    uint32_t *att_counts;  // plan: the three list lengths
    XPart *part;  // exact S and T partials: per tail block; batched: per warp and graph (slot warp + graph)
    HsBuffers hs;  // hinted sort of the Morton keys
};

static void carve_fa2(Carver &c, int64_t K, int64_t nnz, int32_t G, Fa2Scratch &s) {
    const size_t k = size_t(K > 0 ? K : 1);
    const bool batched = G > 1;
    s.frame = c.take<float4>(size_t(G > 1 ? G : 1));
    s.frame_part = c.take<float4>(kMaxNodeBlocks);
    s.bgraph = batched ? c.take<int32_t>(k) : nullptr;
    s.box = batched ? c.take<uint4>(size_t(G)) : nullptr;
    carve_sort(c, int64_t(k), true, s.sort);
    carve_run_fix(c, int64_t(k), s.runfix);
    s.body = c.take<float4>(k);
    carve_tiles(c, int64_t(k), s.tree);
    s.T = c.take<uint32_t>(k + 1);
    s.geo = c.take<float4>(2 * k);
    s.skip = c.take<int32_t>(2 * k);
    s.Frep = c.take<float2>(k);
    s.full = c.take<float2>(k);
    s.rows_short = c.take<int32_t>(k);
    s.rows_med = c.take<int32_t>(k);
    s.rows_long = c.take<int32_t>(k);
    s.att_counts = c.take<uint32_t>(4);
    s.part = c.take<XPart>(2 * (batched ? size_t(kMaxNodeBlocks) * (kThreads / 32) + size_t(G) : size_t(kMaxNodeBlocks)));
    carve_hs(c, K <= kHsFirstMax ? hs_first_buckets(K) : hs_buckets(K), K <= kHsFirstMax, s.hs);
}

size_t fa2_scratch_bytes(int64_t K, int64_t nnz, int32_t G) {
    Carver c(nullptr, 0);
    Fa2Scratch s;
    carve_fa2(c, K, nnz, G, s);
    return c.used();
}

int fa2_check_params(const bgv_fa2_params *p) {
    if (!p) return BGV_EINVAL;
    if (!(p->theta >= 0.0f) || !(p->kr >= 0.0f) || !(p->kg >= 0.0f) || !(p->tau > 0.0f) || !(p->ks >= 0.0f) ||
        !(p->ksmax > 0.0f))
        return BGV_EINVAL;
    if (p->strong_gravity != 0 && p->strong_gravity != 1) return BGV_EINVAL;
    if (p->leaf_cap < 1 || p->max_depth < 1 || p->max_depth > 24 || p->reserved != 0) return BGV_EINVAL;
    return BGV_OK;
}

int run_fa2_init(int64_t K, const bgv_fa2_params &p, float *pos, float *Fprev, double *speed, cudaStream_t st,
                 int32_t G, const int64_t *koff) {
    if (G > 1) {
        note_launch(), k_init_seg<<<G, kThreads, 0, st>>>(koff, p.seed, reinterpret_cast<float2 *>(pos),
                                                          reinterpret_cast<float2 *>(Fprev), speed);
        return launch_status();
    }
    if (K > 0) {
        const float R = __builtin_sqrtf(float(K));
        note_launch(), k_init<<<grid_for(K, kThreads, sm_count() * 8), kThreads, 0, st>>>(
            K, p.seed, R, reinterpret_cast<float2 *>(pos), reinterpret_cast<float2 *>(Fprev));
        BGV_TRY(launch_status());
    }
    note_launch(), k_set_speed<<<1, 1, 0, st>>>(speed);
    return launch_status();
}

// Bounded-wait self check of the moment look-back: one k_tile block as tile 1 of
// two tiles of bodies (all at the origin, body 0 everywhere, mass 0, frame side
// 1) whose tile 0 never runs, so its look-back must give up at the spin limit.
// Equal keys make no cells, and every write stays within the two tiles' arrays.
namespace {
struct WaitCheckMoments {
    unsigned long long *keys;
    uint32_t *perm, *mass;
    float2 *pos;
    float4 *frame, *body;
    TileArrays tree;
};
void carve_wait_check_moments(Carver &c, WaitCheckMoments &w) {
    const size_t K = 2 * kTile;
    w.keys = c.take<unsigned long long>(K);
    w.perm = c.take<uint32_t>(K);
    w.mass = c.take<uint32_t>(K);
    w.pos = c.take<float2>(K);
    w.frame = c.take<float4>(1);
    w.body = c.take<float4>(K);
    carve_tiles(c, int64_t(K), w.tree);
}
}  // namespace

size_t wait_check_moments_bytes() {
    Carver c(nullptr, 0);
    WaitCheckMoments w;
    carve_wait_check_moments(c, w);
    return c.used();
}

int wait_check_moments(void *scratch, uint32_t *dev_status, cudaStream_t st) {
    Carver c(scratch, 0);
    WaitCheckMoments w;
    carve_wait_check_moments(c, w);
    BGV_CUDA(cudaMemsetAsync(scratch, 0, wait_check_moments_bytes(), st));
    const float4 frame = make_float4(0.0f, 0.0f, 1.0f, 0.0f);
    const uint32_t one = 1u;  // the tile counter (after the two tiles' flags)
    BGV_CUDA(cudaMemcpyAsync(w.frame, &frame, sizeof(frame), cudaMemcpyHostToDevice, st));
    BGV_CUDA(cudaMemcpyAsync(w.tree.flags + 2, &one, sizeof(one), cudaMemcpyHostToDevice, st));
    note_launch(), k_tile<<<1, kTileThreads, 0, st>>>(w.keys, w.perm, 2 * kTile, w.pos, w.mass, w.frame, nullptr, 24, 0,
                                                      1, w.body, w.tree, dev_status, spin_limit());
    BGV_TRY(launch_status());
    return cudaStreamSynchronize(st) == cudaSuccess ? BGV_OK : BGV_ECUDA;
}

// Launch shapes of the step, process wide (bgv_autotune_fa2 picks them):
// the longest rows the attraction sums one lane each, threads per block of
// the traversal, blocks per SM of the persistent tail.  Packed in one word so a
// step reads a consistent set.
static std::atomic<uint32_t> g_fa2_tune{(32u << 16) | (128u << 4) | 4u};  // measured best on GB300 (rmat22x)
Fa2Tune fa2_tune() {
    const uint32_t w = g_fa2_tune.load(std::memory_order_relaxed);
    return Fa2Tune{int(w >> 16), int((w >> 4) & 0xFFFu), int(w & 0xFu)};
}
int set_fa2_tune(const Fa2Tune &t) {
    if ((t.att_short != 8 && t.att_short != 16 && t.att_short != 32) ||
        (t.repulse_threads != 128 && t.repulse_threads != 256) || t.tail_blocks_per_sm < 1 ||
        t.tail_blocks_per_sm > 8)
        return BGV_EINVAL;
    g_fa2_tune.store((uint32_t(t.att_short) << 16) | (uint32_t(t.repulse_threads) << 4) | uint32_t(t.tail_blocks_per_sm),
                     std::memory_order_relaxed);
    return BGV_OK;
}

// How a step finds the Morton order, process wide: 1 (default) by buckets, from the
// previous step's order or, in a first or single step of up to kHsFirstMax bodies,
// between sampled keys; 0 by the radix sort in every step.  Both give the same order.
static std::atomic<int> g_fa2_order{1};
int fa2_order() { return g_fa2_order.load(std::memory_order_relaxed); }
int set_fa2_order(int method) {
    if (method != 0 && method != 1) return -1;
    return g_fa2_order.exchange(method, std::memory_order_relaxed);
}

// A second stream per host thread and device, made on first use.
cudaStream_t aux_stream() {
    static thread_local cudaStream_t streams[64] = {};
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return nullptr;
    if (!streams[dev] && cudaStreamCreateWithFlags(&streams[dev], cudaStreamNonBlocking) != cudaSuccess)
        streams[dev] = nullptr;
    return streams[dev];
}

// A stream at the device's highest priority per host thread and device,
// made on first use.
cudaStream_t priority_stream() {
    static thread_local cudaStream_t streams[64] = {};
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return nullptr;
    if (!streams[dev]) {
        int least = 0, greatest = 0;
        if (cudaDeviceGetStreamPriorityRange(&least, &greatest) != cudaSuccess ||
            cudaStreamCreateWithPriority(&streams[dev], cudaStreamNonBlocking, greatest) != cudaSuccess)
            streams[dev] = nullptr;
    }
    return streams[dev];
}

// The two events of a fork onto the second stream and the join back,
// destroyed when the step's work has been enqueued (work already enqueued
// keeps them valid).
struct ForkJoin {
    cudaEvent_t fork = nullptr, join = nullptr;
    cudaError_t make() {
        cudaError_t e = cudaEventCreateWithFlags(&fork, cudaEventDisableTiming);
        if (e == cudaSuccess) e = cudaEventCreateWithFlags(&join, cudaEventDisableTiming);
        return e;
    }
    ~ForkJoin() {
        if (fork) cudaEventDestroy(fork);
        if (join) cudaEventDestroy(join);
    }
};

static int run_fa2_body(int mode, int64_t K, int64_t nnz, const int32_t *csr_off, const int32_t *csr_adj,
                        const uint32_t *csr_w, const uint32_t *mass, const bgv_fa2_params &p, float *pos_f, float *F_f,
                        float *Fprev_f, double *speed, float *Fr, float *Fa, float *Fg, WsHeader *hdr, void *scratch,
                        cudaStream_t st, cudaEvent_t *marks, bool build_plan, int32_t G, const int64_t *koff,
                        bool hinted) {
    if (K <= 0) return BGV_OK;
    const bool batched = G > 1;
    if (!fa2_batch_fits(G, p.max_depth)) return BGV_EINVAL;
    Carver c(scratch, 0);
    Fa2Scratch s;
    carve_fa2(c, K, nnz, G, s);
    float2 *pos = reinterpret_cast<float2 *>(pos_f);
    float2 *F = reinterpret_cast<float2 *>(F_f);
    float2 *Fprev = reinterpret_cast<float2 *>(Fprev_f);
    const int L = p.max_depth;
    const int gbits = batched ? bits_for(G) : 0;
    const Fa2Tune tune = fa2_tune();
    auto mark = [&](int i) -> int {
        if (marks && cudaEventRecord(marks[i], st) != cudaSuccess) return BGV_ECUDA;
        return BGV_OK;
    };

    // Of the per-step counters, k_tile_cross writes tree_nodes whole and k_tile_emit
    // clears the interactions before the traversal counts them; S and T are
    // written whole by the tail; the last-block tickets are reset by their last
    // blocks (the header starts zeroed, see bgv_ws_init).
    BGV_TRY(mark(0));
    ForkJoin ev;
    cudaStream_t aux = nullptr;
    if (nnz > 0) {
        aux = aux_stream();
        if (!aux || ev.make() != cudaSuccess) return BGV_ECUDA;
    }
    // Once the second stream is forked, every way out of this function joins
    // it back into `st` (so `st` stays ordered after the attraction, and a
    // capture never ends with an unjoined fork).
    struct JoinGuard {
        cudaEvent_t ev = nullptr;
        cudaStream_t from = nullptr, into = nullptr;
        int join() {
            if (!ev) return BGV_OK;
            const cudaError_t a = cudaEventRecord(ev, from);
            const cudaError_t b = cudaStreamWaitEvent(into, ev, 0);
            ev = nullptr;
            return a == cudaSuccess && b == cudaSuccess ? BGV_OK : BGV_ECUDA;
        }
        ~JoinGuard() { join(); }
    } guard;
    // The attraction needs only the positions and the CSR: it runs on a
    // second stream while the tree is built and traversed, and k_node waits
    // for it.
    if (nnz > 0) {
        BGV_CUDA(cudaEventRecord(ev.fork, st));
        BGV_CUDA(cudaStreamWaitEvent(aux, ev.fork, 0));
        guard.ev = ev.join;
        guard.from = aux;
        guard.into = st;
        if (build_plan) {
            BGV_CUDA(cudaMemsetAsync(s.att_counts, 0, 4 * sizeof(uint32_t), aux));
            note_launch(), k_att_plan<<<grid_for(K, kThreads), kThreads, 0, aux>>>(
                K, csr_off, tune.att_short, s.rows_short, s.rows_med, s.rows_long, s.att_counts);
            BGV_TRY(launch_status());
        }
        note_launch(), k_att_short<<<grid_for(K, kThreads, sm_count() * 64), kThreads, 0, aux>>>(
            K, csr_off, csr_adj, csr_w, pos, s.rows_short, s.att_counts, unsigned(sm_count() * 16), s.full);
        BGV_TRY(launch_status());
        // as many blocks as fit at once (4 per SM): 3.2 M bodies of an R-MAT graph, 150 steps, 167.2 ms with
        // 16 per SM and 161.7 with 4
        note_launch(), k_att_medium<<<grid_for(K * 32, kThreads, sm_count() * 4), kThreads, 0, aux>>>(
            K, csr_off, csr_adj, csr_w, pos, s.rows_med, s.att_counts, s.full);
        BGV_TRY(launch_status());
        note_launch(), k_att_long<<<sm_count() * 2, kThreads, 0, aux>>>(K, csr_off, csr_adj, csr_w, pos, s.rows_long,
                                                                        s.att_counts, s.full);
        BGV_TRY(launch_status());
    }
    // the tail of the previous step of a run left the frame (batched: the
    // boxes) of the positions it wrote
    if (batched) {
        const int gg = grid_for(G, kThreads, sm_count());
        if (!hinted) {
            const int fb = grid_for(K, kThreads * kTailItems, node_blocks());
            note_launch(), k_box_init<<<gg, kThreads, 0, st>>>(G, s.box);
            BGV_TRY(launch_status());
            note_launch(), k_frame_seg<<<fb, kThreads, 0, st>>>(pos, K, warp_share(K, fb), koff, G, s.box, s.bgraph);
            BGV_TRY(launch_status());
        }
        note_launch(), k_frame_fin<<<gg, kThreads, 0, st>>>(G, s.box, s.frame);
        BGV_TRY(launch_status());
    } else if (!hinted) {
        note_launch(), k_frame<<<grid_for(K, kThreads, frame_blocks()), kThreads, 0, st>>>(pos, K, s.frame_part,
                                                                                         s.frame, &hdr->bbox_ticket);
        BGV_TRY(launch_status());
    }
    // the sorted order lands in the buffer pair the radix sort ends in, so
    // the next iteration finds its hint there whichever sort made it
    const int res = radix_sort_high_result(K, 2 * L + gbits);
    if (fa2_order() == 1 && (hinted || K <= kHsFirstMax)) {
        BGV_TRY(mark(1));
        const MortonOf key_of{pos, s.frame, s.bgraph, L};
        // the pre-order arrays are free until k_tile_emit: the buckets' slots
        unsigned long long *slot_key = reinterpret_cast<unsigned long long *>(s.geo);
        uint32_t *slot_id = reinterpret_cast<uint32_t *>(slot_key + K);
        if (hinted) {
            // the previous iteration's sorted pairs are the hint and the splitters
            const uint32_t *hint = s.sort.vals[res];
            BGV_TRY(hinted_sort_place(key_of, HsPrevious{s.sort.keys[res], hint}, hint, K, hs_buckets(K), s.hs,
                                      s.sort.keys[res ^ 1], s.sort.vals[res ^ 1], slot_key, slot_id, s.sort.keys[res],
                                      s.sort.vals[res], &hdr->status, st));
        } else {
            // a first or single step: from id order, with sampled splitters (five
            // launches; the radix sort, with its local finish, takes nine); also
            // clears what later steps find cleared
            HsClears clr;
            clr.u32 = s.tree.flags;
            clr.n_u32 = tile_flag_words(K);
            BGV_TRY(hinted_sort_sampled(key_of, nullptr, K, hs_first_buckets(K), s.hs, s.sort.keys[res ^ 1],
                                        s.sort.vals[res ^ 1], slot_key, slot_id, s.sort.keys[res], s.sort.vals[res],
                                        &hdr->status, st, clr));
        }
    } else {
        // the first step also clears what the later ones find cleared
        if (!hinted)
            BGV_CUDA(cudaMemsetAsync(s.hs.count, 0, sizeof(uint32_t) * size_t(hs_counter_words(hs_buckets(K))), st));
        const int gk = grid_for(K, kThreads, sm_count() * 16);
        note_launch(), k_keys<<<gk, kThreads, 0, st>>>(pos, K, s.frame, s.bgraph, L, s.sort.keys[0], s.sort.vals[0],
                                                       &hdr->interactions, s.tree.flags, tile_flag_words(K), s.sort.counts,
                                                       sort_counter_words());
        BGV_TRY(launch_status());
        BGV_TRY(mark(1));
        int got = 0;
        BGV_TRY(radix_sort_high(s.sort, s.runfix, K, nullptr, 2 * L + gbits, st, &got, &hdr->status, true));
        if (got != res) return BGV_EINVAL;  // radix_sort_high_result disagrees with the sort
    }
    BGV_TRY(mark(2));
    if (K >= 2) {
        const unsigned tiles = unsigned(tile_count(K));
        const bool early = hs_early(K, !hinted);
        BGV_TRY(launch_chained(early, k_tile, tiles, kTileThreads, st, s.sort.keys[res], s.sort.vals[res], K, pos, mass, s.frame,
                               s.bgraph, L, gbits, p.leaf_cap, s.body, s.tree, &hdr->status, spin_limit()));
        BGV_TRY(mark(3));
        const unsigned per = kTileThreads / 32;  // tiles per block
        BGV_TRY(launch_chained(early, k_tile_cross, (tiles + per - 1) / per, kTileThreads, st, K, L, p.leaf_cap, s.frame,
                               s.bgraph, s.tree, &hdr->tree_nodes));
        BGV_TRY(mark(4));
        BGV_TRY(launch_chained(early, k_tile_emit, tiles, kTileThreads, st, K, s.body, s.tree, s.T, s.geo, s.skip,
                               &hdr->interactions));
        BGV_TRY(mark(5));
        const float theta2 = p.theta * p.theta;
        const unsigned rt = tune.repulse_threads == 128 ? 128u : unsigned(kThreads);
        BGV_TRY(launch_chained(early, rt == 128 ? k_repulse<128> : k_repulse<kThreads>, unsigned((K + rt - 1) / rt), rt, st, s.geo,
                               s.skip, s.T, koff, s.bgraph, s.body, K, p.kr, theta2, s.Frep, &hdr->interactions,
                               &hdr->interactions_total));
    } else {
        // no tree kernels, which leave the step's counters (interactions, tree_nodes)
        BGV_CUDA(cudaMemsetAsync(s.Frep, 0, sizeof(float2), st));
        BGV_CUDA(cudaMemsetAsync(&hdr->interactions, 0, 2 * sizeof(unsigned long long), st));
        BGV_TRY(mark(3));
        BGV_TRY(mark(4));
        BGV_TRY(mark(5));
    }
    BGV_TRY(mark(6));
    BGV_TRY(guard.join());  // the attraction ran alongside on the second stream
    BGV_TRY(mark(7));
    const float2 *att = nnz > 0 ? s.full : nullptr;
    if (mode == 0) {
        note_launch(), k_node<<<grid_for(K, kThreads, node_blocks()), kThreads, 0, st>>>(
            K, att, mass, pos, s.Frep, p.kg, p.strong_gravity, reinterpret_cast<float2 *>(Fr),
            reinterpret_cast<float2 *>(Fa), reinterpret_cast<float2 *>(Fg));
        BGV_TRY(launch_status());
    } else {
        int32_t g_count = G;
        float kg = p.kg, tau = p.tau, ks = p.ks, ksmax = p.ksmax;
        int strong = p.strong_gravity, limit = spin_limit();
        const void *tail = batched ? reinterpret_cast<const void *>(k_tail<true>)
                                   : reinterpret_cast<const void *>(k_tail<false>);
        const int want = grid_for(K, kThreads * kTailItems, sm_count() * tune.tail_blocks_per_sm);
        const int blocks = coop_blocks(tail, kThreads, want);
        int64_t k_count = K, per = warp_share(K, blocks);
        XPart *part = s.part;
        const float2 *frep = s.Frep;
        void *args[] = {&k_count, &per, &att, &mass, &pos, &frep, &kg, &strong, &F, &Fprev, &part, &speed, &tau, &ks,
                        &ksmax, &hdr, &koff, &g_count, &s.box, &s.frame_part, &s.frame, &limit};
        BGV_TRY(launch_coop(tail, blocks, kThreads, args, st));
    }
    BGV_TRY(mark(8));
    return BGV_OK;
}

// The iteration's main chain runs on a high-priority stream forked from the
// caller's and joined back at the end: when SMs free up, its blocks go before
// those of the attraction, which runs beside it at the default priority.
int run_fa2(int mode, int64_t K, int64_t nnz, const int32_t *csr_off, const int32_t *csr_adj, const uint32_t *csr_w,
            const uint32_t *mass, const bgv_fa2_params &p, float *pos_f, float *F_f, float *Fprev_f, double *speed,
            float *Fr, float *Fa, float *Fg, WsHeader *hdr, void *scratch, cudaStream_t st, cudaEvent_t *marks,
            bool build_plan, int32_t G, const int64_t *koff, bool hinted) {
    if (K <= 0) return BGV_OK;
    cudaStream_t hp = priority_stream();
    ForkJoin ev;
    if (!hp || ev.make() != cudaSuccess) return BGV_ECUDA;
    BGV_CUDA(cudaEventRecord(ev.fork, st));
    BGV_CUDA(cudaStreamWaitEvent(hp, ev.fork, 0));
    const int rc = run_fa2_body(mode, K, nnz, csr_off, csr_adj, csr_w, mass, p, pos_f, F_f, Fprev_f, speed, Fr, Fa, Fg,
                                hdr, scratch, hp, marks, build_plan, G, koff, hinted);
    BGV_CUDA(cudaEventRecord(ev.join, hp));
    BGV_CUDA(cudaStreamWaitEvent(st, ev.join, 0));
    return rc;
}

// Steps of graphs that a cluster of blocks keeps in shared memory (small.cuh):
// G graphs of at most Kmax bodies, koff on the device (null for one graph).
// A cluster takes its SMs whole, so a batch of more clusters than two rounds of
// the GPU's SMs runs faster side by side in the general path's launches (50 steps of
// 38 graphs of 2,000 bodies, two rounds, 3.6 ms here and 6.2 there), and with two
// rounds half as many entries a graph pay.
bool small_fits(int64_t Kmax, int64_t nnz, int32_t G) {
    const int64_t graphs = G > 1 ? G : 1, blocks = graphs * small_cluster(Kmax), sms = sm_count();
    const int64_t rounds = blocks > sms ? 2 : 1;
    return Kmax <= kSmallMax && nnz * rounds <= kSmallEntries * graphs && blocks <= 2 * sms;
}

int run_fa2_small(int64_t K, int64_t Kmax, int64_t nnz, const int32_t *csr_off, const int32_t *csr_adj,
                  const uint32_t *csr_w, const uint32_t *mass, const bgv_fa2_params &p, int32_t iterations, float *pos,
                  float *F, float *Fprev, double *speed, WsHeader *hdr, cudaStream_t st, int32_t G,
                  const int64_t *koff) {
    SmallArgs a{};
    a.K = K;
    a.koff = G > 1 ? koff : nullptr;
    a.off = nnz > 0 ? csr_off : nullptr;
    a.adj = csr_adj;
    a.w = csr_w;
    a.mass = mass;
    a.pos = reinterpret_cast<float2 *>(pos);
    a.F = reinterpret_cast<float2 *>(F);
    a.Fprev = reinterpret_cast<float2 *>(Fprev);
    a.speed = speed;
    a.hdr = hdr;
    a.theta2 = p.theta * p.theta;
    a.kr = p.kr;
    a.kg = p.kg;
    a.tau = p.tau;
    a.ks = p.ks;
    a.ksmax = p.ksmax;
    a.strong = p.strong_gravity;
    a.L = p.max_depth;
    a.leaf_cap = p.leaf_cap;
    a.att_short = fa2_tune().att_short;
    const int C = small_cluster(Kmax);
    BGV_CUDA(cudaFuncSetAttribute(k_small, cudaFuncAttributeMaxDynamicSharedMemorySize, int(sizeof(SmallMem))));
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(unsigned((G > 1 ? G : 1) * C));
    cfg.blockDim = dim3(kSmallThreads);
    cfg.dynamicSmemBytes = sizeof(SmallMem);
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = unsigned(C);
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    for (int32_t done = 0; done < iterations; done += kSmallChunk) {
        a.iterations = iterations - done < kSmallChunk ? iterations - done : kSmallChunk;
        BGV_CUDA(cudaMemsetAsync(&hdr->interactions, 0, 2 * sizeof(unsigned long long), st));  // and tree_nodes
        note_launch();
        BGV_CUDA(cudaLaunchKernelEx(&cfg, k_small, a));
    }
    return BGV_OK;
}

}  // namespace bgv
