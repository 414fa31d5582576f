// elt_tile.cuh -- the entries of a layer's ELTs in one tile of catalog events,
// for the builders that take a tile per block (tile_rows.cu, folded.cu).
#pragma once

#include <cuda_runtime.h>

#include "are_internal.cuh"

namespace are {

struct EltTile {
    uint32_t start[kMaxElts + 1];          // entries before ELT j's, and all
    int32_t from[kMaxElts];                // ELT j's first entry of the tile
    uint32_t base;                         // entries of all ELTs in the tiles before this

    // Called by one warp (in shared memory; a block barrier before the rest).
    __device__ __forceinline__ void find(const ScatterArgs &a, int tile, int lane)
    {
        static_assert(kMaxElts == 32, "a lane per ELT");
        int32_t first = 0, cnt = 0;
        if (lane < a.n_elts) {
            const int32_t tiles = a.tiles[lane];
            const int32_t *off = a.off[lane];
            first = tile < tiles ? __ldg(off + tile) : a.n[lane];
            cnt = tile < tiles ? __ldg(off + tile + 1) - first : 0;
        }
        uint32_t incl = (uint32_t)cnt, before = (uint32_t)first;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const uint32_t o = __shfl_up_sync(0xffffffffu, incl, d);
            if (lane >= d) incl += o;
            before += __shfl_xor_sync(0xffffffffu, before, d);
        }
        from[lane] = first;
        start[lane] = incl - (uint32_t)cnt;
        if (lane == 31) {
            start[32] = incl;
            base = before;
        }
    }
    // Entry i of the tile: its event less e0, its ELT, and its place in the
    // ELT's arrays.
    __device__ __forceinline__ int32_t entry(const ScatterArgs &a, uint32_t i, uint32_t e0, uint32_t &e, int &j) const
    {
        j = 0;
#pragma unroll
        for (int s = 16; s; s >>= 1)
            if (start[j + s] <= i) j += s;
        const int32_t at = from[j] + (int32_t)(i - start[j]);
        e = (uint32_t)a.ids[j][at] - e0;
        return at;
    }
};

}  // namespace are
