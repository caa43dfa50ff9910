// Growth of bit regions in a slice held in shared memory (hull diagnostics, the
// hysteresis of the SM edge detection).  Word (y, w) = y * rw + w holds voxels
// x = 32 w .. 32 w + 31 of row y (bit x & 31).
#pragma once

#include <cstdint>

namespace hd {
namespace {

// Bits of g reachable from g through set bits of p, moving toward higher
// bits (left) and toward lower bits (right) inside one word (Kogge-Stone).
__device__ __forceinline__ uint32_t fill_word(uint32_t g, uint32_t p)
{
    uint32_t l = g, pl = p;
    l |= pl & (l << 1);
    pl &= pl << 1;
    l |= pl & (l << 2);
    pl &= pl << 2;
    l |= pl & (l << 4);
    pl &= pl << 4;
    l |= pl & (l << 8);
    pl &= pl << 8;
    l |= pl & (l << 16);
    uint32_t r = g, pr = p;
    r |= pr & (r >> 1);
    pr &= pr >> 1;
    r |= pr & (r >> 2);
    pr &= pr >> 2;
    r |= pr & (r >> 4);
    pr &= pr >> 4;
    r |= pr & (r >> 8);
    pr &= pr >> 8;
    r |= pr & (r >> 16);
    return l | r;
}

// Row y's word w of E, with the neighbouring bits in x when kDiagonal.
template <bool kDiagonal>
__device__ __forceinline__ uint32_t row_reach(const uint32_t *E, int k, int w, int rw)
{
    const uint32_t e = E[k];
    if (!kDiagonal) return e;
    uint32_t g = e | (e << 1) | (e >> 1);
    if (w > 0) g |= E[k - 1] >> 31;
    if (w + 1 < rw) g |= E[k + 1] << 31;
    return g;
}

// Grows the region E inside P (E a part of P) to everything connected to it,
// 4-connected or, kDiagonal, 8-connected; the whole block.  A warp takes a tile
// of 32 rows (one per lane) of one word and grows it in registers until nothing
// changes, so a block barrier is paid per tile crossed and not per row: with a
// barrier per row the fill of a head-sized volume took 111 us and its
// hysteresis most of 224 (now 49, and 59 with the rest of the slice kernel).
// Warps may read a neighbour's word old or new, both inside the region; a sweep
// that changes nothing has read nothing old.  Every sweep but the last adds a
// voxel, so at most voxels + 1 run.
template <bool kDiagonal>
__device__ __forceinline__ void grow_region(const uint32_t *P, uint32_t *E, int rw, int ny,
                                            long long voxels)
{
    const int lane = static_cast<int>(threadIdx.x & 31u);
    const int warp = static_cast<int>(threadIdx.x >> 5), nwarps = static_cast<int>(blockDim.x >> 5);
    const int tiles = ((ny + 31) >> 5) * rw;
    for (long long it = 0; it < voxels + 1; ++it) {
        int changed = 0;
        for (int t = warp; t < tiles; t += nwarps) {
            const int rb = t / rw, w = t - rb * rw, y = 32 * rb + lane;
            const int k = y * rw + w;
            const bool in = y < ny;
            const uint32_t p = in ? P[k] : 0u;
            if (!__any_sync(0xffffffffu, p != 0u)) continue;
            const uint32_t e0 = in ? E[k] : 0u;
            uint32_t side = 0u;  // from the words beside
            if (in && w > 0) side |= E[k - 1] >> 31;
            if (in && w + 1 < rw) side |= E[k + 1] << 31;
            uint32_t above = 0u, below = 0u;  // from the rows beyond the tile
            if (lane == 0 && y > 0) above = row_reach<kDiagonal>(E, k - rw, w, rw);
            if (lane == 31 && y + 1 < ny) below = row_reach<kDiagonal>(E, k + rw, w, rw);
            uint32_t e = e0;
            for (;;) {
                const uint32_t h = e | (e << 1) | (e >> 1) | side;
                const uint32_t v = kDiagonal ? h : e;
                const uint32_t up = __shfl_up_sync(0xffffffffu, v, 1);
                const uint32_t down = __shfl_down_sync(0xffffffffu, v, 1);
                const uint32_t g = h | (lane == 0 ? above : up) | (lane == 31 ? below : down);
                const uint32_t n = fill_word(g & p, p) | e;
                const bool more = n != e;
                e = n;
                if (!__any_sync(0xffffffffu, more)) break;
            }
            if (e != e0) {
                E[k] = e;
                changed = 1;
            }
        }
        if (!__syncthreads_or(changed)) break;
    }
}

}  // namespace
}  // namespace hd
