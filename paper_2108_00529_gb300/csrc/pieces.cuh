// pieces.cuh -- shares of lists whose places take all of 32 bits.  A graph of nearly
// 2^31 edges has nearly 2^32 endpoints and pairs, so no place past a list's end, and
// no count rounded up, may be formed in 32 bits.  (Host and device; no CUDA needed.)
#pragma once

#include <stdint.h>

#ifdef __CUDACC__
#define BGV_HD __host__ __device__ __forceinline__
#else
#define BGV_HD inline
#endif

namespace bgv {

// Pieces of `piece` entries in `count`.
BGV_HD uint32_t pieces_of(uint32_t count, uint32_t piece) { return count / piece + (count % piece ? 1u : 0u); }
// Entries of the piece that starts at `at`, in a list that ends at `end` >= at.
BGV_HD uint32_t piece_size(uint32_t at, uint32_t end, uint32_t piece) { return end - at < piece ? end - at : piece; }
// Of [at, end): the entries before the first multiple of `unit` (a power of two).
BGV_HD uint32_t ragged_head(uint32_t at, uint32_t end, uint32_t unit) {
    const uint32_t to = (0u - at) & (unit - 1u);
    return to < end - at ? to : end - at;
}

}  // namespace bgv
