// style.cu -- supernode colour groups (Section 4.3) and drawing the discs
// into an image (Section 4.1 radii, Section 4.3 colours).
//
// Communities are ordered by size (a stable radix sort of (size, id), so
// ties keep id order).  With alpha the total size, the longest prefix of
// that order whose sizes sum to at most alpha / 2 is group 0 (drawn brown);
// the remaining R communities get group 1 + floor(10 * rank / R), from small
// to big.  One pass sums tiles of the sorted sizes (64-bit); its last block
// scans the tile sums and counts the brown prefix inside the tile where it
// ends; a second pass writes the groups.
#include "bgv_internal.cuh"

namespace bgv {
namespace {
constexpr int kStyleThreads = 1024;

// The sort's keys and values; also clears the ticket of k_size_prefix.
__global__ void k_size_keys(const uint32_t *__restrict__ size, int64_t K, unsigned long long *__restrict__ keys,
                            uint32_t *__restrict__ vals, unsigned int *ticket) {
    if (blockIdx.x == 0 && threadIdx.x == 0) *ticket = 0u;
    for (int64_t k = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; k < K; k += int64_t(gridDim.x) * blockDim.x) {
        keys[k] = size[k];
        vals[k] = uint32_t(k);
    }
}

__device__ unsigned long long block_exclusive_u64(unsigned long long x, unsigned long long *total) {
    __shared__ unsigned long long warp_sums[kStyleThreads / 32 + 1];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    unsigned long long inc = x;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const unsigned long long y = __shfl_up_sync(0xFFFFFFFFu, inc, d);
        if (lane >= d) inc += y;
    }
    if (lane == 31) warp_sums[warp] = inc;
    __syncthreads();
    if (warp == 0) {
        const unsigned long long w = warp_sums[lane];
        unsigned long long run = w;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const unsigned long long y = __shfl_up_sync(0xFFFFFFFFu, run, d);
            if (lane >= d) run += y;
        }
        warp_sums[lane] = run - w;
        if (lane == 31) warp_sums[32] = run;
    }
    __syncthreads();
    const unsigned long long r = warp_sums[warp] + inc - x;
    *total = warp_sums[kStyleThreads / 32];
    __syncthreads();
    return r;
}

// Length of the brown prefix: the places r whose running size, their own
// included, stays within half of the total (a prefix, as sizes are not
// negative).  One tile of kStyleTile sorted sizes per block and its sum; the
// last block finds the tile in which the prefix ends and counts inside it.
// One block over all K sizes took 399 us for K = 248,188 (each thread read a
// contiguous chunk, so no load was coalesced, three times over).  With this, the
// image frame on the whole GPU and a lane per small disc, grouping 248,188
// communities, colouring 3.2 M nodes and drawing 2048 x 2048 pixels takes
// 125.5 us instead of 573.9.
constexpr int kStyleTile = 4096;
constexpr int kStyleItems = kStyleTile / kStyleThreads;
__global__ void __launch_bounds__(kStyleThreads) k_size_prefix(const unsigned long long *__restrict__ sizes, int64_t K,
                                                               unsigned long long *__restrict__ sums,
                                                               unsigned int *ticket, int64_t *__restrict__ half) {
    __shared__ bool last;
    __shared__ unsigned long long base_sh;
    __shared__ long long tile_sh;
    const int64_t tiles = gridDim.x;
    unsigned long long mine = 0, total;
#pragma unroll
    for (int q = 0; q < kStyleItems; ++q) {
        const int64_t r = int64_t(blockIdx.x) * kStyleTile + q * kStyleThreads + threadIdx.x;
        mine += r < K ? sizes[r] : 0ull;
    }
    block_exclusive_u64(mine, &total);
    if (threadIdx.x == 0) {
        sums[blockIdx.x] = total;
        __threadfence();
        last = atomicAdd(ticket, 1u) == gridDim.x - 1;
        tile_sh = tiles;
    }
    __syncthreads();
    if (!last) return;
    __threadfence();
    mine = 0;
    for (int64_t t = threadIdx.x; t < tiles; t += kStyleThreads) mine += __ldcg(&sums[t]);
    unsigned long long all;
    block_exclusive_u64(mine, &all);
    // the first tile whose end lies past half of the total
    unsigned long long carry = 0;
    for (int64_t t0 = 0; t0 < tiles; t0 += kStyleThreads) {
        const int64_t t = t0 + threadIdx.x;
        const unsigned long long x = t < tiles ? __ldcg(&sums[t]) : 0ull;
        unsigned long long chunk;
        const unsigned long long before = carry + block_exclusive_u64(x, &chunk);
        if (t < tiles && 2 * (before + x) > all && 2 * before <= all) {  // one tile at most: sums grow past it
            tile_sh = t;
            base_sh = before;
        }
        carry += chunk;
        __syncthreads();
        if (tile_sh < tiles) break;
    }
    if (tile_sh < tiles) {
        const int64_t r0 = int64_t(tile_sh) * kStyleTile + int64_t(threadIdx.x) * kStyleItems;
        unsigned long long v[kStyleItems], sum = 0;
#pragma unroll
        for (int q = 0; q < kStyleItems; ++q) {
            v[q] = r0 + q < K ? sizes[r0 + q] : 0ull;
            sum += v[q];
        }
        unsigned long long tot;
        unsigned long long cum = base_sh + block_exclusive_u64(sum, &tot);
        unsigned long long brown = 0;
#pragma unroll
        for (int q = 0; q < kStyleItems; ++q) {
            cum += v[q];
            brown += (r0 + q < K && 2 * cum <= all) ? 1ull : 0ull;
        }
        unsigned long long n;
        block_exclusive_u64(brown, &n);
        if (threadIdx.x == 0) *half = int64_t(tile_sh) * kStyleTile + int64_t(n);
    } else if (threadIdx.x == 0) {
        *half = K;  // every size is 0
    }
}

// Up to this many communities one block finds the prefix and writes the groups: grouping
// 4,000 communities and colouring 10,001 nodes 60.5 us in two launches and 51.1 so,
// 8,000 61.5 and 57.3.
constexpr int64_t kStyleOne = 8192;
__device__ __forceinline__ uint8_t group_of(int64_t r, int64_t half, int64_t rest) {
    return r < half ? uint8_t(0) : uint8_t(1 + (10 * (r - half)) / rest);
}
__global__ void __launch_bounds__(kStyleThreads) k_colour_few(const unsigned long long *__restrict__ sizes,
                                                              const uint32_t *__restrict__ order, int K,
                                                              uint8_t *__restrict__ group) {
    constexpr int kMost = int(kStyleOne) / kStyleThreads;
    const int per = (K + kStyleThreads - 1) / kStyleThreads, r0 = int(threadIdx.x) * per;
    unsigned long long v[kMost], sum = 0, all;
    uint32_t id[kMost];
#pragma unroll
    for (int q = 0; q < kMost; ++q) {
        const bool in = q < per && r0 + q < K;
        v[q] = in ? sizes[r0 + q] : 0ull;
        id[q] = in ? order[r0 + q] : 0u;
        sum += v[q];
    }
    unsigned long long cum = block_exclusive_u64(sum, &all);
    int brown = 0;
#pragma unroll
    for (int q = 0; q < kMost; ++q) {
        cum += v[q];
        brown += q < per && r0 + q < K && 2 * cum <= all ? 1 : 0;
    }
    __shared__ int half_sh;
    if (threadIdx.x == 0) half_sh = 0;
    __syncthreads();
    brown = __reduce_add_sync(0xFFFFFFFFu, brown);
    if ((threadIdx.x & 31) == 0 && brown) atomicAdd(&half_sh, brown);
    __syncthreads();
    const int half = half_sh, rest = K - half;
#pragma unroll
    for (int q = 0; q < kMost; ++q)
        if (q < per && r0 + q < K) group[id[q]] = group_of(r0 + q, half, rest);
}

__global__ void __launch_bounds__(kStyleThreads) k_colour_groups(const uint32_t *__restrict__ order, int64_t K,
                                                                 const int64_t *__restrict__ half_dev,
                                                                 uint8_t *__restrict__ group) {
    const int64_t half = *half_dev, rest = K - half;
    for (int64_t r = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; r < K; r += int64_t(gridDim.x) * blockDim.x)
        group[order[r]] = group_of(r, half, rest);
}

// Whole-graph drawing (Section 4.3): every node takes its supernode's colour.
__device__ __forceinline__ uint8_t colour_of(int32_t k, int64_t K, const uint8_t *__restrict__ group) {
    return (k >= 0 && k < K) ? group[k] : uint8_t(0);
}
__global__ void k_node_colours(int32_t n, const int32_t *__restrict__ node_map, int64_t K,
                               const uint8_t *__restrict__ group, uint8_t *__restrict__ node_colour) {
    const int64_t t0 = int64_t(blockIdx.x) * blockDim.x + threadIdx.x, stride = int64_t(gridDim.x) * blockDim.x;
    int64_t done = 0;
    // four nodes per thread and pass where both arrays allow whole words
    if (reinterpret_cast<uintptr_t>(node_map) % 16 == 0 && reinterpret_cast<uintptr_t>(node_colour) % 4 == 0) {
        const int64_t quads = n >> 2;
        for (int64_t q = t0; q < quads; q += stride) {
            const int4 k = reinterpret_cast<const int4 *>(node_map)[q];
            reinterpret_cast<uchar4 *>(node_colour)[q] = make_uchar4(colour_of(k.x, K, group), colour_of(k.y, K, group),
                                                                     colour_of(k.z, K, group), colour_of(k.w, K, group));
        }
        done = quads << 2;
    }
    for (int64_t v = done + t0; v < n; v += stride) node_colour[v] = colour_of(node_map[v], K, group);
}
}  // namespace

}  // namespace bgv

using namespace bgv;

namespace {
struct StyleScratch {
    SortBuffers sort;
    unsigned long long *sums;  // per tile of sorted sizes
    int64_t *half;             // length of the brown prefix
    unsigned int *ticket;
};
int64_t style_tiles(int64_t K) { return (K + kStyleTile - 1) / kStyleTile; }
void carve_style(Carver &c, int64_t K, StyleScratch &s) {
    carve_sort(c, K > 0 ? K : 1, true, s.sort);
    s.sums = c.take<unsigned long long>(size_t(style_tiles(K)));
    s.half = c.take<int64_t>(1);
    s.ticket = c.take<unsigned int>(1);
}
}  // namespace

extern "C" size_t bgv_colour_groups_ws_size(int64_t K) {
    Carver c(nullptr, kHeaderBytes);
    StyleScratch s;
    carve_style(c, K, s);
    return c.used();
}

extern "C" int bgv_colour_groups(int64_t K, const uint32_t *sizes, uint8_t *group, int32_t n,
                                 const int32_t *node_map, uint8_t *node_colour, void *ws, size_t ws_bytes,
                                 void *stream) {
    if (K < 0 || K >= 0x7FFFFFFF || (K > 0 && (!sizes || !group))) return BGV_EINVAL;
    if (node_colour && (n < 0 || (n > 0 && !node_map))) return BGV_EINVAL;
    if (!ws || reinterpret_cast<uintptr_t>(ws) % kAlign) return BGV_EINVAL;
    if (ws_bytes < bgv_colour_groups_ws_size(K)) return BGV_ENOSPC;
    if (K == 0) return BGV_OK;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    Carver c(ws, kHeaderBytes);
    StyleScratch s;
    carve_style(c, K, s);
    note_launch(), k_size_keys<<<grid_for(K, 256, sm_count() * 8), 256, 0, st>>>(sizes, K, s.sort.keys[0],
                                                                                 s.sort.vals[0], s.ticket);
    BGV_TRY(launch_status());
    int res = 0;
    BGV_TRY(radix_sort(s.sort, K, nullptr, 32, st, &res, status_ptr(ws)));
    if (K <= kStyleOne) {
        note_launch(), k_colour_few<<<1, kStyleThreads, 0, st>>>(s.sort.keys[res], s.sort.vals[res], int(K), group);
        BGV_TRY(launch_status());
    } else {
        note_launch(), k_size_prefix<<<unsigned(style_tiles(K)), kStyleThreads, 0, st>>>(s.sort.keys[res], K, s.sums,
                                                                                        s.ticket, s.half);
        BGV_TRY(launch_status());
        note_launch(), k_colour_groups<<<grid_for(K, kStyleThreads, sm_count() * 4), kStyleThreads, 0, st>>>(
            s.sort.vals[res], K, s.half, group);
        BGV_TRY(launch_status());
    }
    if (node_colour && n > 0) {
        note_launch(), k_node_colours<<<grid_for((int64_t(n) + 3) / 4, 256, sm_count() * 8), 256, 0, st>>>(
            n, node_map, K, group, node_colour);
        BGV_TRY(launch_status());
    }
    return BGV_OK;
}

// ------------------------------------------------------------- drawing
// Discs of radius r (sqrt of the size, Section 4.1) in the colour of their
// group (Section 4.3), splatted into an RGBA image: the discs' bounding box
// maps to the pixels with one scale s = min(W, H) / largest extent; pixel
// (px, py) shows the disc whose scaled circle covers its centre (px + 0.5,
// py + 0.5); overlaps keep the smaller radius, then the smaller id.  The
// covered pixels are marked with an atomicMax of (priority, id); a second
// pass shades.  Most discs of a big graph's picture span a few pixels: a lane
// takes a disc of up to kLaneCells candidate pixels by itself, and the warp
// takes its lanes' larger discs together, one after the other.  A warp has as
// many discs as still leave every warp slot of the GPU busy (one, for few
// discs, which are large ones).  FP32 with explicit round-to-nearest
// operations, so the coverage equals the plain definition's.
namespace bgv {
namespace {
__constant__ uint8_t c_palette[11][3] = {
    {177, 89, 40},   {202, 178, 214}, {106, 61, 154}, {253, 191, 111}, {255, 127, 0}, {251, 154, 153},
    {227, 26, 28},   {178, 223, 138}, {51, 160, 44},  {166, 206, 227}, {31, 120, 180}};

constexpr int kRenderThreads = 256;
constexpr int kRenderBlocks = 304;  // blocks (and block partials) of the frame pass, at most
constexpr int kLaneCells = 36;

struct Box {
    float lx, ly, hx, hy;
};
__device__ __forceinline__ void box_join(Box &b, const Box &o) {
    b.lx = fminf(b.lx, o.lx); b.ly = fminf(b.ly, o.ly);
    b.hx = fmaxf(b.hx, o.hx); b.hy = fmaxf(b.hy, o.hy);
}
// Block-wide join; thread 0 receives the result.
__device__ __forceinline__ void box_join_block(Box &b) {
    __shared__ Box part[kStyleThreads / 32];
    const int warps = int(blockDim.x) / 32;
#pragma unroll
    for (int d = 16; d > 0; d >>= 1)
        box_join(b, Box{__shfl_xor_sync(0xFFFFFFFFu, b.lx, d), __shfl_xor_sync(0xFFFFFFFFu, b.ly, d),
                        __shfl_xor_sync(0xFFFFFFFFu, b.hx, d), __shfl_xor_sync(0xFFFFFFFFu, b.hy, d)});
    if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = b;
    __syncthreads();
    if (threadIdx.x == 0)
        for (int w = 1; w < warps; ++w) box_join(b, part[w]);
    __syncthreads();
}

// The image frame: block boxes, joined by the last block (one block over all
// discs took 42 us at K = 248,188).  Few discs are left to one block of
// kStyleThreads, without the other blocks' fence and ticket.
__global__ void __launch_bounds__(kStyleThreads) k_render_frame(const float2 *__restrict__ xy,
                                                                 const float *__restrict__ radius, int64_t K,
                                                                 int32_t W, int32_t H, Box *parts,
                                                                 unsigned int *ticket, float4 *frame) {
    __shared__ bool last;
    Box b{INFINITY, INFINITY, -INFINITY, -INFINITY};
    for (int64_t k = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; k < K; k += int64_t(gridDim.x) * blockDim.x) {
        const float2 p = xy[k];
        const float r = radius[k];
        box_join(b, Box{__fsub_rn(p.x, r), __fsub_rn(p.y, r), __fadd_rn(p.x, r), __fadd_rn(p.y, r)});
    }
    box_join_block(b);
    if (gridDim.x > 1) {
        if (threadIdx.x == 0) {
            parts[blockIdx.x] = b;
            __threadfence();
            last = atomicAdd(ticket, 1u) == gridDim.x - 1;
        }
        __syncthreads();
        if (!last) return;
        __threadfence();
        b = Box{INFINITY, INFINITY, -INFINITY, -INFINITY};
        for (unsigned t = threadIdx.x; t < gridDim.x; t += blockDim.x)
            box_join(b, Box{__ldcg(&parts[t].lx), __ldcg(&parts[t].ly), __ldcg(&parts[t].hx), __ldcg(&parts[t].hy)});
        box_join_block(b);
    }
    if (threadIdx.x != 0) return;
    const float ex = __fsub_rn(b.hx, b.lx), ey = __fsub_rn(b.hy, b.ly);
    const float ext = ex > ey ? ex : ey;
    const float s = (K > 0 && ext > 0.0f) ? __fdiv_rn(float(W < H ? W : H), ext) : 1.0f;
    *frame = make_float4(b.lx, b.ly, s, 0.0f);
}

__device__ __forceinline__ void splat_pixel(unsigned long long *zbuf, int32_t W, int px, int py, float u, float v,
                                            float rs2, unsigned long long key) {
    const float dx = __fsub_rn(__fadd_rn(float(px), 0.5f), u), dy = __fsub_rn(__fadd_rn(float(py), 0.5f), v);
    const float d2 = __fadd_rn(__fmul_rn(dx, dx), __fmul_rn(dy, dy));
    if (d2 <= rs2) atomicMax(&zbuf[size_t(py) * W + px], key);
}

__global__ void __launch_bounds__(kRenderThreads) k_render_splat(const float2 *__restrict__ xy,
                                                                 const float *__restrict__ radius, int64_t K,
                                                                 int32_t W, int32_t H, const float4 *frame,
                                                                 int per_warp, unsigned long long *__restrict__ zbuf) {
    const int lane = threadIdx.x & 31;
    const float4 f = *frame;
    const int64_t warps = (int64_t(gridDim.x) * blockDim.x) >> 5;
    for (int64_t q = (int64_t(blockIdx.x) * blockDim.x + threadIdx.x) >> 5; q * per_warp < K; q += warps) {
        const int64_t k = lane < per_warp ? q * per_warp + lane : K;
        float u = 0.0f, v = 0.0f, rs2 = -1.0f;
        int x0 = 0, x1 = -1, y0 = 0, y1 = -1;
        unsigned long long key = 0ull;
        if (k < K) {
            const float2 p = xy[k];
            const float r = radius[k];
            u = __fmul_rn(__fsub_rn(p.x, f.x), f.z);
            v = __fmul_rn(__fsub_rn(p.y, f.y), f.z);
            const float rs = __fmul_rn(r, f.z);
            rs2 = __fmul_rn(rs, rs);
            // pixels whose centre can lie within rs of (u, v), one pixel of slack
            x0 = max(0, int(floorf(u - rs)) - 1);
            x1 = min(W - 1, int(ceilf(u + rs)) + 1);
            y0 = max(0, int(floorf(v - rs)) - 1);
            y1 = min(H - 1, int(ceilf(v + rs)) + 1);
            if (!(rs >= 0.0f)) x1 = x0 - 1;
            key = (static_cast<unsigned long long>(0xFFFFFFFFu - __float_as_uint(r)) << 32) |
                  (0xFFFFFFFFull - uint64_t(k));
        }
        const bool any = x0 <= x1 && y0 <= y1;
        const bool wide = any && (per_warp == 1 || int64_t(x1 - x0 + 1) * (y1 - y0 + 1) > kLaneCells);
        if (any && !wide)
            for (int py = y0; py <= y1; ++py)
                for (int px = x0; px <= x1; ++px) splat_pixel(zbuf, W, px, py, u, v, rs2, key);
        for (unsigned todo = __ballot_sync(0xFFFFFFFFu, wide); todo; todo &= todo - 1u) {
            const int src = __ffs(todo) - 1;
            const float su = __shfl_sync(0xFFFFFFFFu, u, src), sv = __shfl_sync(0xFFFFFFFFu, v, src);
            const float sr = __shfl_sync(0xFFFFFFFFu, rs2, src);
            const int a0 = __shfl_sync(0xFFFFFFFFu, x0, src), a1 = __shfl_sync(0xFFFFFFFFu, x1, src);
            const int b0 = __shfl_sync(0xFFFFFFFFu, y0, src), b1 = __shfl_sync(0xFFFFFFFFu, y1, src);
            const unsigned long long sk = __shfl_sync(0xFFFFFFFFu, key, src);
            const int bw = a1 - a0 + 1, cells = bw * (b1 - b0 + 1);  // at most 2^30: W, H <= 32768
            for (int c = lane; c < cells; c += 32) splat_pixel(zbuf, W, a0 + c % bw, b0 + c / bw, su, sv, sr, sk);
        }
    }
}

__global__ void __launch_bounds__(kStyleThreads) k_render_shade(const unsigned long long *__restrict__ zbuf,
                                                                int64_t pixels, int64_t K,
                                                                const uint8_t *__restrict__ group,
                                                                uchar4 *__restrict__ rgba) {
    for (int64_t i = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; i < pixels;
         i += int64_t(gridDim.x) * blockDim.x) {
        const unsigned long long z = zbuf[i];
        uchar4 o = make_uchar4(255, 255, 255, 255);
        if (z) {
            const int64_t k = int64_t(0xFFFFFFFFull - (z & 0xFFFFFFFFull));
            const uint8_t g = k < K ? group[k] : 0;
            const int c = g <= 10 ? g : 0;
            o = make_uchar4(c_palette[c][0], c_palette[c][1], c_palette[c][2], 255);
        }
        rgba[i] = o;
    }
}
}  // namespace
}  // namespace bgv

namespace {
struct RenderScratch {
    float4 *frame;
    Box *parts;
    unsigned int *ticket;      // just before the z-buffer: one memset clears both
    unsigned long long *zbuf;
};
void carve_render(Carver &c, int64_t pixels, RenderScratch &s) {
    s.frame = c.take<float4>(1);
    s.parts = c.take<Box>(kRenderBlocks);
    s.ticket = c.take<unsigned int>(1);
    s.zbuf = c.take<unsigned long long>(size_t(pixels));
}
}  // namespace

extern "C" size_t bgv_render_ws_size(int32_t W, int32_t H) {
    Carver c(nullptr, kHeaderBytes);
    RenderScratch s;
    carve_render(c, int64_t(W > 0 ? W : 1) * (H > 0 ? H : 1), s);
    return c.used();
}

extern "C" int bgv_render(int64_t K, const float *xy, const float *radius, const uint8_t *group, int32_t W, int32_t H,
                          uint8_t *rgba, void *ws, size_t ws_bytes, void *stream) {
    if (K < 0 || K >= 0xFFFFFFFFll || W < 1 || H < 1 || W > 32768 || H > 32768 || !rgba) return BGV_EINVAL;
    if (K > 0 && (!xy || !radius || !group || reinterpret_cast<uintptr_t>(xy) % 8)) return BGV_EINVAL;
    if (reinterpret_cast<uintptr_t>(rgba) % 4) return BGV_EINVAL;
    if (!ws || reinterpret_cast<uintptr_t>(ws) % kAlign) return BGV_EINVAL;
    if (ws_bytes < bgv_render_ws_size(W, H)) return BGV_ENOSPC;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    Carver c(ws, kHeaderBytes);
    RenderScratch s;
    const int64_t pixels = int64_t(W) * H;
    carve_render(c, pixels, s);
    const size_t clear = size_t(reinterpret_cast<char *>(s.zbuf + pixels) - reinterpret_cast<char *>(s.ticket));
    BGV_CUDA(cudaMemsetAsync(s.ticket, 0, clear, st));
    const float2 *p = reinterpret_cast<const float2 *>(xy);
    const bool few = K <= kStyleOne;
    note_launch(), k_render_frame<<<few ? 1 : grid_for(K, kRenderThreads, kRenderBlocks),
                                    few ? kStyleThreads : kRenderThreads, 0, st>>>(p, radius, K, W, H, s.parts, s.ticket,
                                                                                   s.frame);
    BGV_TRY(launch_status());
    if (K > 0) {
        int per_warp = 1;  // discs per warp: a power of two up to 32
        while (per_warp < 32 && K >= int64_t(sm_count()) * 64 * 2 * per_warp) per_warp *= 2;
        const int64_t warps = (K + per_warp - 1) / per_warp;
        note_launch(), k_render_splat<<<grid_for(warps * 32, kRenderThreads, sm_count() * 16), kRenderThreads, 0, st>>>(
            p, radius, K, W, H, s.frame, per_warp, s.zbuf);
        BGV_TRY(launch_status());
    }
    note_launch(), k_render_shade<<<grid_for(pixels, kStyleThreads, sm_count() * 8), kStyleThreads, 0, st>>>(
        s.zbuf, pixels, K, group, reinterpret_cast<uchar4 *>(rgba));
    return launch_status();
}
