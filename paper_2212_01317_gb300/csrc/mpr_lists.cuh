// Gap-list entries: the description of one gap site that every half-step
// reads (where it lies, its block, which of its four neighbours exist and
// are gaps, and which of its bonds another block owns). The flags are shared
// by the block-major lists (gap_item, mpr_kernels.cu) and the tile-major lists
// of the staged half-step (gap_entry, mpr_tile.cu).
#pragma once
#include <cuda_runtime.h>

#include <cstdint>

#include "mpr_internal.h"

namespace mpr {

// A block's sites [x0, x1) x [y0, y1) (clipped to the canvas) and whether the
// block across each edge belongs to the same slice (no bond joins two slices).
struct BlockFrame {
    int b, x0, x1, y0, y1, slice;
    bool l_ok, r_ok, u_ok, d_ok;
};

__device__ __forceinline__ BlockFrame block_frame(const Geom& g, const int32_t* __restrict__ of_block,
                                                  int b) {
    BlockFrame fr;
    fr.b = b;
    const int by = b / g.nbx, bx = b % g.nbx;
    fr.y0 = by * g.lb;
    fr.x0 = bx * g.lb;
    fr.y1 = min(g.H, fr.y0 + g.lb);
    fr.x1 = min(g.W, fr.x0 + g.lb);
    fr.slice = of_block[b];
    fr.l_ok = bx > 0 && of_block[b - 1] == fr.slice;
    fr.r_ok = bx + 1 < g.nbx && of_block[b + 1] == fr.slice;
    fr.u_ok = by > 0 && of_block[b - g.nbx] == fr.slice;
    fr.d_ok = by + 1 < g.nby && of_block[b + g.nbx] == fr.slice;
    return fr;
}

// The site's left or up bond is owned by the neighbouring block.
__device__ __forceinline__ bool block_edge(const BlockFrame& fr, int y, int x) {
    return (x == fr.x0 && fr.l_ok) || (y == fr.y0 && fr.u_ok);
}

// The entry of gap site (y, x) of block fr: .x = y << 16 | x,
// .y = b << META_SHIFT | flags (NB_*: the neighbour exists, i.e. lies in the
// canvas, in the same slice and is not absent; GAP_*: it is a gap site;
// EDGE_L / EDGE_U: the left / up bond belongs to the block on that side).
__device__ __forceinline__ uint2 gap_entry(const Geom& g, const uint8_t* __restrict__ mask,
                                           const BlockFrame& fr, int y, int x) {
    const int64_t i = (int64_t)y * g.W + x;
    uint32_t f = 0;
    const bool hl = (x > fr.x0 || fr.l_ok) && mask[i - 1] != MASK_ABSENT;
    const bool hr = (x + 1 < fr.x1 || fr.r_ok) && mask[i + 1] != MASK_ABSENT;
    const bool hu = (y > fr.y0 || fr.u_ok) && mask[i - g.W] != MASK_ABSENT;
    const bool hd = (y + 1 < fr.y1 || fr.d_ok) && mask[i + g.W] != MASK_ABSENT;
    if (hl) { f |= NB_L; if (mask[i - 1] == MASK_GAP) f |= GAP_L; }
    if (hr) { f |= NB_R; if (mask[i + 1] == MASK_GAP) f |= GAP_R; }
    if (hu) { f |= NB_U; if (mask[i - g.W] == MASK_GAP) f |= GAP_U; }
    if (hd) { f |= NB_D; if (mask[i + g.W] == MASK_GAP) f |= GAP_D; }
    if (hl && x == fr.x0) f |= EDGE_L;
    if (hu && y == fr.y0) f |= EDGE_U;
    return make_uint2(((uint32_t)y << 16) | (uint32_t)x, ((uint32_t)fr.b << META_SHIFT) | f);
}

// The block-major lists' entry of gap site (y, x): everything the sweep would
// otherwise compute for every realization pair it updates the site in, worked
// out once. .x = half index y Wh + x / 2 (below 2^29), .y = gap_entry's .y,
// .z = the Philox counter word (the site's index within its field), .w = the
// left neighbour's half index (the right one's is one more; -1 at the grid's
// first site).
__device__ __forceinline__ uint4 gap_item(const Geom& g, const int4& rect,
                                          const uint8_t* __restrict__ mask,
                                          const BlockFrame& fr, int y, int x) {
    const uint2 e = gap_entry(g, mask, fr, y, x);
    const uint32_t hs = (uint32_t)y * (uint32_t)g.Wh + (uint32_t)(x >> 1);
    return make_uint4(hs, e.y, local_index(rect, y, x), hs + (uint32_t)(x & 1) - 1u);
}

}  // namespace mpr
