// General-walk traversal in global memory: histories (or tile pieces of
// them) whose walk has no closed form or does not fit the tiled pass.
#pragma once

#include "hd_geom.cuh"

namespace hd {
namespace {

// Global-memory voxel update of one history: one atomic add into N or M.
struct GlobalVisit {
    uint32_t *vol;  // N or M
    __device__ __forceinline__ void operator()(uint32_t v) const { atomicAdd(vol + v, 1u); }
};

// A lane's part of a segment in a box of dx x dy voxels (in-plane), for walks
// shared by `lanes` lanes of a warp (a power of two): the box becomes the lane's
// strip of it along the segment's longer in-plane axis, (ox, oy) its corner, and a, b the segment relative to
// that.  The strips' parts are a partition of the segment's voxels in the box
// (A_i is a set of points).  False when the lane has no strip.  (With a lane
// per segment instead the last walks alone took 0.1 ms at the end of the
// head-sized traversal.)
__device__ __forceinline__ bool warp_strip(const int32_t gi[3], const int32_t go[3], int &dx,
                                           int &dy, int &ox, int &oy, int32_t a[3], int32_t b[3],
                                           int lanes = 32)
{
    const bool along_y = abs(go[1] - gi[1]) > abs(go[0] - gi[0]);
    const int n = along_y ? dy : dx;
    const int strip = (n + lanes - 1) / lanes;
    const int s0 = (static_cast<int>(threadIdx.x) & (lanes - 1)) * strip, len = min(strip, n - s0);
    if (len <= 0) return false;
    ox = along_y ? 0 : s0;
    oy = along_y ? s0 : 0;
    (along_y ? dy : dx) = len;
    a[0] = gi[0] - (ox << 16);
    a[1] = gi[1] - (oy << 16);
    a[2] = gi[2];
    b[0] = go[0] - (ox << 16);
    b[1] = go[1] - (oy << 16);
    b[2] = go[2];
    return true;
}

// The voxels of a segment clipped to one tile of tp (gi, go relative to the
// tile's origin, grid Q16), by `lanes` lanes with the general run walk, visited with
// global indices.
__device__ void walk_tile_global(const TilePlan &tp, const int32_t gi[3], const int32_t go[3],
                                 int tile, int lanes, const GlobalVisit &visit)
{
    const int tix = tile % tp.ntx;
    const int tiy = (tile / tp.ntx) % tp.nty;
    const int tiz = tile / (tp.ntx * tp.nty);
    int x0 = tix * tp.tx, y0 = tiy * tp.ty;
    const int z0 = tiz * tp.tz;
    int dx = min(tp.tx, tp.nx - x0), dy = min(tp.ty, tp.ny - y0);
    const int dz = min(tp.tz, tp.nz - z0);
    int ox, oy;
    int32_t a[3], b[3];
    if (!warp_strip(gi, go, dx, dy, ox, oy, a, b, lanes)) return;
    x0 += ox;
    y0 += oy;
    RunWalk w;
    if (!run_begin(w, a, b, dx, dy, dz)) return;
    const bool ymaj = (w.flags >> 5) & 1;
    int row, lo, hi;
    while (run_next(w, row, lo, hi)) {
        // x-major rows are y + dy z, y-major rows x + dx z (box-local)
        const int ra = ymaj ? row % dx : row % dy;
        const int lz = ymaj ? row / dx : row / dy;
        for (int m = lo; m <= hi; ++m) {
            const uint32_t X = static_cast<uint32_t>(x0 + (ymaj ? ra : m));
            const uint32_t Y = static_cast<uint32_t>(y0 + (ymaj ? m : ra));
            const uint32_t Z = static_cast<uint32_t>(z0 + lz);
            visit(X + static_cast<uint32_t>(tp.nx) * (Y + static_cast<uint32_t>(tp.ny) * Z));
        }
    }
}

// A pair slot holding a general walk instead of an event walk: the segment's
// tile-local endpoints, and 2 tile + class in word 7, marked empty for the
// tiled pass there (bit 31, event_pack).
__device__ __forceinline__ void general_pack(const int32_t gi[3], const int32_t go[3], int tile,
                                             int cls, uint32_t o[kLeanWords])
{
    o[0] = static_cast<uint32_t>(gi[0]);
    o[1] = static_cast<uint32_t>(gi[1]);
    o[2] = static_cast<uint32_t>(gi[2]);
    o[3] = static_cast<uint32_t>(go[0]);
    o[4] = static_cast<uint32_t>(go[1]);
    o[5] = static_cast<uint32_t>(go[2]);
    o[6] = 0;
    o[7] = 0x80000000u + 2u * static_cast<uint32_t>(tile) + static_cast<uint32_t>(cls);
}

// The general walk held by pair slot pos: its endpoints, and 2 tile + class.
__device__ __forceinline__ uint32_t load_general(const Pairs &pairs, uint32_t pos, int32_t gi[3],
                                                 int32_t go[3])
{
    const uint4 a = pairs.v[2 * static_cast<size_t>(pos)];
    const uint4 b = pairs.v[2 * static_cast<size_t>(pos) + 1];
    gi[0] = static_cast<int32_t>(a.x);
    gi[1] = static_cast<int32_t>(a.y);
    gi[2] = static_cast<int32_t>(a.z);
    go[0] = static_cast<int32_t>(a.w);
    go[1] = static_cast<int32_t>(b.x);
    go[2] = static_cast<int32_t>(b.y);
    return b.w & 0x7fffffffu;
}

}  // namespace
}  // namespace hd
