// Bucketing of the (record, tile) pairs of a chunk for the tiled traversal,
// after the ingest blocks have reserved their places in each bucket
// (reserve_buckets): a counting sort of the pairs by bucket, block b writing
// those of ingest block b from its places on, with each pair's walk set-up.
#include <cooperative_groups.h>
#include "hd_admit.cuh"
#include "hd_fallback.cuh"

namespace cg = cooperative_groups;

namespace hd {

namespace {

constexpr unsigned kFull = 0xffffffffu;
constexpr int kScatterThreads = 512;
// Buckets whose events a block sums in shared memory: with more of them, beside the
// positions, only one block per SM would be resident, and two updates of one bucket
// are then rare (64 x 64 x 2000: 160 us).
constexpr int kLocalEvents = 12 * 1024;

// The general set-up of one (record, tile) pair: its packed event walk, an
// empty walk, or (returns true) the general form for the fallback list.
__device__ __noinline__ bool general_setup(const int32_t gi[3], const int32_t go[3], int dx,
                                           int dy, int dz, int thick, int tile, int cls,
                                           uint4 &p0, uint4 &p1)
{
    RunWalk w;
    LeanWalk L;
    uint32_t pk[kLeanWords];
    bool fallback = false;
    if (!run_begin(w, gi, go, dx, dy, dz)) {
        event_pack_empty(pk);
    } else if (lean_of(w, L)) {
        const bool ymaj = (L.fl >> 2) & 1;
        event_pack(L, ymaj ? dy : dx, ymaj ? dx : dy, thick, pk);
    } else {
        // walked from the fallback list by the general run walk
        general_pack(gi, go, tile, cls, pk);
        fallback = true;
    }
    p0 = make_uint4(pk[0], pk[1], pk[2], pk[3]);
    p1 = make_uint4(pk[4], pk[5], pk[6], pk[7]);
    return fallback;
}

// Counting sort of (record, tile) pairs by bucket.  Block b takes the pairs
// ingest block b listed, one per thread, and writes those of a bucket from its
// places there on (a shared-memory cursor per bucket orders them).
__global__ void __launch_bounds__(kScatterThreads, 2) scatter_kernel(
    TilePlan tp, Records rec, int64_t per_block, Buckets buckets, const uint32_t *block_base,
    const uint32_t *block_pairs, Ctrl *ctrl, Pairs pairs)
{
    extern __shared__ uint32_t s_mem[];
    const int nt = kGroups * tp.ntiles;
    uint32_t *s_next = s_mem;         // this block's next position in each bucket
    uint32_t *s_events = s_mem + nt;  // the events of the walks written there
    const bool local = nt <= kLocalEvents;
    for (int t = threadIdx.x; local && t < nt; t += blockDim.x) s_events[t] = 0;
    after_previous();
    bucket_places<kScatterThreads>(nt, buckets, block_base, s_next);
    const int64_t h0 = static_cast<int64_t>(blockIdx.x) * per_block;
    const unsigned npairs = block_pairs[blockIdx.x];
    unsigned runs = 0;
    const uint32_t *list = pairs.stage + static_cast<int64_t>(blockIdx.x) * per_block * tp.pairs_per_record;
    for (unsigned e = threadIdx.x; e < npairs; e += kScatterThreads) {
        const uint32_t code = list[e];
        const int64_t slot = h0 + (code >> kRecordTileBits);
        const int j = static_cast<int>(code & (kMaxRecordTiles - 1u));
        const int32_t stw = rec.status[slot];
        const int cls = status_cls(stw);
        int32_t q[6];
#pragma unroll
        for (int a = 0; a < 6; ++a) q[a] = rec.g[a][slot];
        // the j-th tile of the record's box, x fastest; with whole-plane
        // tiles the box is the record's slices alone (in its status word)
        int x = 0, y = 0, z;
        if (tp.ntx == 1 && tp.nty == 1) {
            const unsigned zl = static_cast<unsigned>(status_zlo(stw));
            z = (tp.mtz ? static_cast<int>(umulhi32(zl, tp.mtz)) : static_cast<int>(zl)) + j;
        } else {
            int lo[3], hi[3];
            tile_range_z(tp, q, status_zlo(stw), status_zhi(stw), lo, hi);
            const int ex = hi[0] - lo[0] + 1, ey = hi[1] - lo[1] + 1;
            x = lo[0] + j % ex;
            y = lo[1] + (j / ex) % ey;
            z = lo[2] + j / (ex * ey);
        }
        const int tile = x + tp.ntx * (y + tp.nty * z);
        const int t = status_group(stw) * tp.ntiles + tile;
        const uint32_t pos = atomicAdd(&s_next[t], 1u);
        // set up the walk of this record clipped to this tile
        const int x0 = x * tp.tx, y0 = y * tp.ty, z0 = z * tp.tz;
        const int dx = min(tp.tx, tp.nx - x0), dy = min(tp.ty, tp.ny - y0),
                  dz = min(tp.tz, tp.nz - z0);
        const int32_t gi[3] = {q[0] - (x0 << 16), q[1] - (y0 << 16), q[2] - (z0 << 16)};
        const int32_t go[3] = {q[3] - (x0 << 16), q[4] - (y0 << 16), q[5] - (z0 << 16)};
        // one-slice tiles (the default plan): the direct set-up; the
        // walks it declines (ties at the start, no in-plane motion) go to
        // the fallback list, whose general run walk is exact for any walk.
        // Deeper slabs: the general set-up (out of line).
        uint4 p0, p1;
        bool fallback = false;
        if (dz == 1) {
            LeanWalk L;
            const int rl = slab_lean(gi, go, dx, dy, L);
            uint32_t pk[kLeanWords];
            if (rl == 1) {
                const bool ymaj = (L.fl >> 2) & 1;
                event_pack(L, ymaj ? dy : dx, ymaj ? dx : dy, tp.thick, pk);
            } else if (rl == 0) {
                event_pack_empty(pk);
            } else {
                general_pack(gi, go, tile, cls, pk);
                fallback = true;
            }
            p0 = make_uint4(pk[0], pk[1], pk[2], pk[3]);
            p1 = make_uint4(pk[4], pk[5], pk[6], pk[7]);
        } else {
            fallback = general_setup(gi, go, dx, dy, dz, tp.thick, tile, cls, p0, p1);
        }
        if (static_cast<int>(p1.w) >= 0) {
            runs += p1.w + 1u;  // a walk's runs: one more than its events
            if (p1.w != 0u) {
                if (local) atomicAdd(&s_events[t], p1.w);
                else atomicAdd(&buckets.events[t], static_cast<unsigned long long>(p1.w));
            }
        }
        pairs.v[2 * static_cast<size_t>(pos)] = p0;
        pairs.v[2 * static_cast<size_t>(pos) + 1] = p1;
        if (fallback) {
            // append to the fallback list, one counter update per group of
            // lanes arriving together
            cg::coalesced_group grp = cg::coalesced_threads();
            unsigned at = 0;
            if (grp.thread_rank() == 0) {
                at = atomicAdd(&ctrl->n_pair_fallback, grp.size());
                atomicAdd(&ctrl->pairs_general, static_cast<unsigned long long>(grp.size()));
            }
            at = grp.shfl(at, 0) + grp.thread_rank();
            pairs.fb[at] = make_uint2(pos, 0u);
        }
    }
    // runs of the chunk's thin walks, for the statistics
    unsigned long long all = tp.thick > 0 ? 0u : runs;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) all += __shfl_xor_sync(kFull, all, o);
    if ((threadIdx.x & 31u) == 0 && all) atomicAdd(&ctrl->runs, all);
    __syncthreads();
    for (int t = threadIdx.x; local && t < nt; t += blockDim.x)
        if (s_events[t])
            atomicAdd(&buckets.events[t], static_cast<unsigned long long>(s_events[t]));
}

}  // namespace

cudaError_t init_scatter()
{
    return cudaFuncSetAttribute(scatter_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                static_cast<int>(sizeof(uint32_t)) * 2 * kGroups * kMaxTiles);
}

cudaError_t launch_scatter(const TilePlan &tp, const Records &rec, int64_t n, Ctrl *ctrl,
                           const Buckets &buckets, const uint32_t *block_base,
                           const uint32_t *block_pairs, const Pairs &pairs, int sm_count,
                           cudaStream_t s)
{
    if (n <= 0) return cudaSuccess;
    const ChunkSplit sp = chunk_split(n, sm_count, tp.ntiles);
    const size_t nt = kGroups * static_cast<size_t>(tp.ntiles);
    const size_t smem = sizeof(uint32_t) * (nt <= kLocalEvents ? 2 * nt : nt);
    return launch_chained(scatter_kernel, static_cast<unsigned>(sp.blocks), kScatterThreads, smem, s, tp,
                          rec, sp.per_block, buckets, block_base, block_pairs, ctrl, pairs);
}

}  // namespace hd
