// Admission of records to the tiled path, shared by the ingest kernels: the
// pair budget of a block, its tile histogram, its pair list, and the records at
// their histories' slots.
#pragma once

#include "hd_geom.cuh"

namespace hd {
namespace {

__device__ __forceinline__ unsigned warp_sum_u32(unsigned v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

__device__ __forceinline__ unsigned warp_incl_scan(unsigned v)
{
    const unsigned lane = threadIdx.x & 31u;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const unsigned t = __shfl_up_sync(0xffffffffu, v, o);
        if (lane >= static_cast<unsigned>(o)) v += t;
    }
    return v;
}

// Decide the path of each lane's record (tiled within the block's pair
// budget, else global; ok false: no record), count its tiles in the block
// histogram, list its pairs in the block's share of stage, and write it at its
// history's slot i (when i < i1).  tcount: its tiles (-1: not for the tiled
// path); tiles(lo, hi) gives their box.  Budget reservations are per warp on a
// shared-memory counter, so the block never waits at a barrier.  The pairs
// the budget admits fill the list from its start without gaps: the
// reservations tile [0, total) in the order of their ends, and only the one
// record that straddles the budget, and the records after it, are turned
// away (they take the global path, exact either way).
template <class TilesT>
__device__ __forceinline__ void reserve_and_write(const TilePlan &tp, const Records &rec, Ctrl *ctrl,
                                                  uint32_t *s_hist, unsigned *s_demand,
                                                  unsigned budget, int64_t h0, int64_t i,
                                                  int64_t i1, uint32_t *stage, int cls, int type,
                                                  bool ok, int tcount, int zlo, int zhi,
                                                  const int32_t r[6], const TilesT &tiles)
{
    const unsigned demand = ok && tcount > 0 ? static_cast<unsigned>(tcount) : 0u;
    const unsigned lane = threadIdx.x & 31u;
    const unsigned incl = warp_incl_scan(demand);
    const unsigned tot = __shfl_sync(0xffffffffu, incl, 31);
    unsigned wbase = 0;
    if (lane == 31 && tot) wbase = atomicAdd(s_demand, tot);
    wbase = __shfl_sync(0xffffffffu, wbase, 31);
    const unsigned long long end = static_cast<unsigned long long>(wbase) + incl;
    const int path = ok ? (demand > 0 && end <= budget ? 1 : 2) : 0;
    if (rec.glist) {
        // the global path's list: one counter update per warp
        const unsigned gm = __ballot_sync(0xffffffffu, path == 2);
        if (gm) {
            const int lead = __ffs(gm) - 1;
            unsigned gb = 0;
            if (static_cast<int>(lane) == lead) gb = atomicAdd(&ctrl->n_global, __popc(gm));
            gb = __shfl_sync(0xffffffffu, gb, lead);
            if (path == 2) rec.glist[gb + __popc(gm & ((1u << lane) - 1u))] = static_cast<int32_t>(i);
        }
    }
    if (i >= i1) return;
    int32_t st = 0;
    if (ok) {
        st = record_status(path, cls, type, zlo, zhi);
        if (path == 1) {
            int lo[3], hi[3];
            tiles(lo, hi);
            uint32_t *const hist = s_hist + (cls + 2 * type) * tp.ntiles;
            // the record's pairs hold positions end - c .. end - 1 of the
            // block's list (all below its budget)
            const uint32_t code = static_cast<uint32_t>(i - h0) << kRecordTileBits;
            uint32_t *const list = stage + (static_cast<unsigned>(end) - demand);
            if (tp.ntx == 1 && tp.nty == 1) {  // whole planes: the tiles are consecutive
                for (int j = 0; j < tcount; ++j) {
                    atomicAdd(hist + lo[2] + j, 1u);
                    list[j] = code | static_cast<uint32_t>(j);
                }
            } else {
                for (int z = lo[2]; z <= hi[2]; ++z)
                    for (int y = lo[1]; y <= hi[1]; ++y)
                        for (int x = lo[0]; x <= hi[0]; ++x)
                            atomicAdd(hist + x + tp.ntx * (y + tp.nty * z), 1u);
                for (int j = 0; j < tcount; ++j) list[j] = code | static_cast<uint32_t>(j);
            }
        }
#pragma unroll
        for (int a = 0; a < 6; ++a) rec.g[a][i] = r[a];
    }
    rec.status[i] = st;
}

// The end of an ingest block: it reserves its pairs' places in every bucket
// (block_base[b nh + t], by block b's atomic on the bucket's count; the order of
// the blocks inside a bucket is the order they end in, which no count depends
// on) and leaves its pairs in all.
__device__ __forceinline__ void reserve_buckets(int nh, const uint32_t *s_hist, unsigned *s_total,
                                                uint32_t *bucket_count, uint32_t *block_base,
                                                uint32_t *block_pairs)
{
    __syncthreads();
    unsigned mine = 0;
    for (int t = threadIdx.x; t < nh; t += blockDim.x) {
        const unsigned c = s_hist[t];
        if (c == 0) continue;
        block_base[static_cast<size_t>(blockIdx.x) * nh + t] = atomicAdd(bucket_count + t, c);
        mine += c;
    }
    mine = warp_sum_u32(mine);
    if ((threadIdx.x & 31u) == 0 && mine) atomicAdd(s_total, mine);
    __syncthreads();
    if (threadIdx.x == 0) block_pairs[blockIdx.x] = *s_total;
}

// The start of a scatter block: s_base[t], its first place in each of the nt
// buckets it has pairs in, from the exclusive scan of the buckets' counts and
// its reservations; block 0 also writes the buckets' first pairs.
template <int kThreads>
__device__ __forceinline__ void bucket_places(int nt, const Buckets &buckets,
                                              const uint32_t *block_base, uint32_t *s_base)
{
    __shared__ unsigned s_warp[kThreads / 32];
    const unsigned lane = threadIdx.x & 31u, wid = threadIdx.x >> 5;
    for (int t = threadIdx.x; t < nt; t += kThreads) s_base[t] = buckets.count[t];
    __syncthreads();
    const int per = (nt + kThreads - 1) / kThreads;
    const int t0 = min(static_cast<int>(threadIdx.x) * per, nt), t1 = min(t0 + per, nt);
    unsigned mine = 0;
    for (int t = t0; t < t1; ++t) mine += s_base[t];
    const unsigned incl = warp_incl_scan(mine);
    if (lane == 31) s_warp[wid] = incl;
    __syncthreads();
    unsigned at = incl - mine;
    for (unsigned w = 0; w < kThreads / 32; ++w) at += w < wid ? s_warp[w] : 0u;
    for (int t = t0; t < t1; ++t) {
        const unsigned c = s_base[t];
        s_base[t] = at;
        at += c;
    }
    __syncthreads();
    for (int t = threadIdx.x; t < nt; t += kThreads) {
        const unsigned first = s_base[t];
        if (blockIdx.x == 0) buckets.first[t] = first;
        // nothing was reserved (and none of these is used) where the block has no pair
        s_base[t] = first + block_base[static_cast<size_t>(blockIdx.x) * nt + t];
    }
    __syncthreads();
}

}  // namespace
}  // namespace hd
