// Growth of bit regions in a slice held in shared memory (hull diagnostics, the
// hysteresis of the SM edge detection).  Word (y, w) = y * rw + w holds voxels
// x = 32 w .. 32 w + 31 of row y (bit x & 31).
#pragma once

#include <cstdint>

namespace hd {
namespace {

// Rows of words: the row of word k (a division by the words per row, k below 2^21:
// (k + 1/2) / rw lies at least 1 / (2 rw) from a whole number, its float error is
// at most k 2^-22 / rw).
struct WordRows {
    float r;
    __device__ __forceinline__ explicit WordRows(int rw) : r(1.0f / static_cast<float>(rw)) {}
    __device__ __forceinline__ int operator()(int k) const
    {
        return static_cast<int>((static_cast<float>(k) + 0.5f) * r);
    }
};

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

// Bits of e reachable from e through set bits of p along the columns of a warp's 32
// rows, one row per lane.
__device__ __forceinline__ uint32_t fill_columns(uint32_t e, uint32_t p)
{
    const int lane = static_cast<int>(threadIdx.x & 31u);
    uint32_t a = e, pa = p, b = e, pb = p;  // downwards and upwards
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t ga = __shfl_up_sync(0xffffffffu, a, o), qa = __shfl_up_sync(0xffffffffu, pa, o);
        const uint32_t gb = __shfl_down_sync(0xffffffffu, b, o), qb = __shfl_down_sync(0xffffffffu, pb, o);
        a |= lane >= o ? pa & ga : 0u;
        pa = lane >= o ? pa & qa : 0u;
        b |= lane + o < 32 ? pb & gb : 0u;
        pb = lane + o < 32 ? pb & qb : 0u;
    }
    return a | b;
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

// Grows row y of E along the row by a warp, 32 words at a time in either
// direction: a word passes on what reaches its end, a full one also what
// enters it, which an addition carries through the words at once.  Returns
// whether the lane's words changed.
__device__ __forceinline__ bool fill_row(const uint32_t *P, uint32_t *E, int rw)
{
    const int lane = static_cast<int>(threadIdx.x & 31u);
    bool changed = false;
    // the carries into the words of a chunk, and out of it (in `carry`)
    auto carries = [&](uint32_t out, uint32_t full, uint32_t &carry) {
        const unsigned g = __ballot_sync(0xffffffffu, out != 0u);
        const unsigned a = __ballot_sync(0xffffffffu, full == 0xffffffffu) | g;
        const unsigned long long sum = static_cast<unsigned long long>(a) + g + carry;
        carry = static_cast<uint32_t>(sum >> 32);
        return static_cast<uint32_t>(sum) ^ a ^ g;
    };
    uint32_t carry = 0u;
    for (int w0 = 0; w0 < rw; w0 += 32) {
        const int w = w0 + lane;
        const uint32_t p = w < rw ? P[w] : 0u, e = w < rw ? E[w] : 0u;
        uint32_t n = fill_word(e, p);
        const uint32_t in = carries(n >> 31, p, carry);
        if ((in >> lane) & 1u) n |= p & ~(p + 1u);  // the word's first bits
        if (n != e) E[w] = n;
        changed = changed || n != e;
    }
    __syncwarp();
    carry = 0u;
    for (int w0 = (rw - 1) & ~31; w0 >= 0; w0 -= 32) {
        const int w = w0 + 31 - lane;  // lanes in the direction of the carry
        const uint32_t p = w < rw ? P[w] : 0u, e = w < rw ? E[w] : 0u;
        const uint32_t in = carries(e & 1u, p, carry), q = __brev(p);
        uint32_t n = e;
        if ((in >> lane) & 1u) n |= __brev(q & ~(q + 1u));  // its last bits
        if (n != e) E[w] = n;
        changed = changed || n != e;
    }
    return changed;
}

// Words of a row from which it is also filled as a whole in every sweep, and rows
// below which a sweep takes a word per thread (a tile would leave its warp's lanes
// idle).
constexpr int kLongRow = 20, kFewRows = 16;

// Grows the region E inside P (E a part of P) to everything connected to it,
// 4-connected or, kDiagonal, 8-connected; the whole block.  A warp takes a tile
// of 32 rows (one per lane) of one word and grows it in registers until nothing
// changes, so a block barrier is paid per tile crossed and not per row: with a
// barrier per row the fill of a head-sized volume took 111 us and its
// hysteresis most of 224 (now 31, and 52 with the rest of the slice kernel).
// Across the words of long rows a region advanced by one a sweep (a corridor of
// 4096 x 32 voxels 617 us, with whole rows filled between the sweeps 58).
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
    const WordRows row_of(rw);
    for (long long it = 0; it < voxels + 1; ++it) {
        int changed = 0;
        for (int k = static_cast<int>(threadIdx.x); ny < kFewRows && k < ny * rw;
             k += static_cast<int>(blockDim.x)) {
            const int y = row_of(k), w = k - y * rw;
            const uint32_t p = P[k], e = E[k];
            if ((p & ~e) == 0u) continue;
            uint32_t g = row_reach<true>(E, k, w, rw);
            if (y > 0) g |= row_reach<kDiagonal>(E, k - rw, w, rw);
            if (y + 1 < ny) g |= row_reach<kDiagonal>(E, k + rw, w, rw);
            const uint32_t n = fill_word(g & p, p) | e;
            if (n != e) {
                E[k] = n;
                changed = 1;
            }
        }
        for (int t = warp; ny >= kFewRows && t < tiles; t += nwarps) {
            const int rb = row_of(t), w = t - rb * rw, y = 32 * rb + lane;
            const int k = y * rw + w;
            const bool in = y < ny;
            const uint32_t p = in ? P[k] : 0u;
            const uint32_t e0 = in ? E[k] : 0u;
            if (!__any_sync(0xffffffffu, (p & ~e0) != 0u)) continue;  // nothing left to grow into
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
                if (!__any_sync(0xffffffffu, (g & p & ~e) != 0u)) break;
                e |= fill_word(g & p, p);
                if (!kDiagonal) e = fill_columns(e, p);
            }
            if (e != e0) {
                E[k] = e;
                changed = 1;
            }
        }
        if (rw > kLongRow) {
            __syncthreads();
            for (int y = warp; y < ny; y += nwarps)
                if (fill_row(P + y * rw, E + y * rw, rw)) changed = 1;
        }
        if (!__syncthreads_or(changed)) break;
    }
}

}  // namespace
}  // namespace hd
