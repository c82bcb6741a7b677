// Loads that the score and window kernels share.
#pragma once

#include "kvec_internal.cuh"
#include "sm100_ptx.cuh"

namespace kvec {

// The R window query rows of KV head h of sequence s, as two halves of 64 columns
// (128-byte swizzled rows, `half` bytes apart); 2 * R * 128 bytes arrive on `bar`.
// G.jm: one box per query head, so that a tile's rows are ordered by query head
// (w is a multiple of 8, the swizzle's row period); else one box of all rows.
__device__ __forceinline__ void load_queries(uint8_t* dst, uint32_t half, const CUtensorMap* map, uint64_t* bar,
                                             const Geometry& G, int h, int s) {
    if (G.jm) {
        for (int j = 0; j < G.g; ++j) {
            uint8_t* d = dst + j * G.w * 128;
            ptx::tma_load_4d(d, map, bar, 0, h * G.g + j, 0, s);
            ptx::tma_load_4d(d + half, map, bar, 64, h * G.g + j, 0, s);
        }
    } else {
        ptx::tma_load_4d(dst, map, bar, 0, h * G.g, 0, s);
        ptx::tma_load_4d(dst + half, map, bar, 64, h * G.g, 0, s);
    }
}

}  // namespace kvec
