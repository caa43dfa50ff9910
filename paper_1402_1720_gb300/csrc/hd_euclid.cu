// Thick rays by the Euclidean distance of Eq. 3.2 (d_0 > 0, d the distance
// from a voxel's centre to the closed segment L_i, Sec. 2.1): A_i(d_0) = the
// voxels whose centre lies within d_0 mm of L_i.  Counted into N and M like
// the thin paths, once per history for every voxel of its A_i(d_0).  The
// exact membership test, its float filter and the row search are in
// hd_euclid.cuh.
//
// A scan whose tiles are one slice deep counts them on the tiled path, like the
// thin paths (launch_euclid_scan): records with world endpoints, a pair per
// record and tile its capsule can reach, sorted by tile and major axis, each
// pair's rows of one slice by a closed form with certified float bounds
// (SliceRows in hd_euclid.cuh) into shared-memory difference arrays; the few
// rows the bounds leave open go to the exact search, a thread each, and the
// records without the closed form (trackers inside the grid, axis-parallel
// paths, too many tiles) to the kernel below, which the standalone
// accumulation and other plans use for every history.  Head-sized scan,
// 2.7e6 histories, d_0 = 2.5 mm, all hulls: 12.46 -> 1.33 ms.
//
// euclid_kernel.  A warp takes groups of 32 consecutive histories (so each lane's
// gantry cos/sin rarely change); each lane classifies one history and sets
// its capsule up (endpoints, index box, the float part) in shared memory.  Then the
// warp takes the group's histories one at a time: its lanes take the rows of
// voxels along the segment's major in-plane axis that cross the box bounding
// the capsule (segment grown by d_0).  Each nonempty row adds +1 / -1 to a
// difference array along the major axis (the thick rays' workspace), and row
// prefix sums add them to N and M.
#include <cmath>
#include <cstdint>

#include "hd_admit.cuh"
#include "hd_euclid.cuh"
#include "hd_thick.cuh"

namespace hd {
namespace {

constexpr int kEuThreads = 256;
constexpr int kEuBlocksPerSm = 2;  // resident blocks per SM (the launch bounds)
constexpr int kEuGroup = 32;  // consecutive histories a warp takes at once, one per lane

struct EuCounts {
    unsigned n_in = 0, n_miss = 0, n_hit = 0, n_none = 0, n_reject = 0;
};

// One history of a warp's group, as the lane that set it up left it.
struct EuSlot {
    long long A[3], B[3];  // doubled endpoints in the capsule's frame
    CapF cf;               // the float part of its capsule
    int16_t blo1, bhi1, blo2, bhi2;  // index box of the rows on axes 1 and 2
    int flags;             // bit 0: hit class, bit 1: rows along y, bit 2: has rows
};

__global__ void __launch_bounds__(kEuThreads, kEuBlocksPerSm) euclid_kernel(Inputs in, int64_t n, GeomQ g,
                                                            Cordic cd, float tau_l, float tau_h,
                                                            int use_miss, int use_hit,
                                                            long long R2, ThickDiff td,
                                                            unsigned long long *stats,
                                                            unsigned long long *next,
                                                            const int32_t *__restrict__ list,
                                                            const unsigned *__restrict__ listed)
{
    // with a list: its histories only
    if (list != nullptr) n = static_cast<int64_t>(*listed);
    if (n == 0) return;
    const unsigned lane = threadIdx.x & 31u;
    const int warp = static_cast<int>(threadIdx.x >> 5);
    // per warp: a queue of rows to process (at most 31 left + 32 new), the
    // group's histories, and the exact part of the current one's capsule
    __shared__ int s_queue[kEuThreads / 32][64];
    __shared__ EuSlot s_slot[kEuThreads / 32][kEuGroup];
    __shared__ CapX s_cx[kEuThreads / 32];
    int *const queue = s_queue[warp];
    EuSlot *const slot = s_slot[warp];
    CapX *const cxs = &s_cx[warp];
    EuCounts nc;
    unsigned long long vox[2] = {0, 0}, rows = 0;
    bool tc_valid = false;
    float tc_ang = 0.0f;
    long long tc_c = 0, tc_s = 0;
    for (;;) {
        unsigned long long base = 0;
        if (lane == 0) base = atomicAdd(next, static_cast<unsigned long long>(kEuGroup));
        base = __shfl_sync(0xffffffffu, base, 0);
        if (base >= static_cast<unsigned long long>(n)) break;
        // each lane sets one history of the group up: class, endpoints
        // (rejected by the thin rule like the thin paths), capsule frame
        const int64_t at = static_cast<int64_t>(base) + lane;
        EuSlot &e = slot[lane];
        __syncwarp();  // the previous group is done with the slots
        int flags = 0;
        if (at < n) {
            const int64_t i = list != nullptr ? static_cast<int64_t>(list[at]) : at;
            const float w = in.wepl[i];
            const int cls = w < tau_l ? 0 : (w > tau_h ? 1 : -1);
            nc.n_in += 1;
            nc.n_miss += cls == 0;
            nc.n_hit += cls == 1;
            nc.n_none += cls < 0;
            if (!(cls < 0 || (cls == 0 && !use_miss) || (cls == 1 && !use_hit))) {
                const float ang = in.angle[i];
                const float ui = in.u_in[i], vi = in.v_in[i], uo = in.u_out[i], vo = in.v_out[i];
                bool ok = fabsf(ang) < 1048576.0f;
                int32_t G[6];
                if (ok) {
                    if (!tc_valid || ang != tc_ang) {
                        cordic_cs(q16_of(ang), cd, tc_c, tc_s);
                        tc_ang = ang;
                        tc_valid = true;
                    }
                    ok = endpoints_cs(g, tc_c, tc_s, ui, vi, uo, vo, G);  // the thin rule
                }
                if (!ok) {
                    nc.n_reject += 1;
                } else {
                    long long W[6];
                    world_cs(g, tc_c, tc_s, ui, vi, uo, vo, W);
                    bool ymaj;
                    int blo[3], bhi[3];
                    float S;
                    long long A[3], B[3];
                    if (capsule_frame(g, W, R2, A, B, ymaj, blo, bhi, S)) {
#pragma unroll
                        for (int q = 0; q < 3; ++q) {
                            e.A[q] = A[q];
                            e.B[q] = B[q];
                        }
                        CapX cx;
                        capx_of(g, A, B, ymaj, R2, cx);
                        e.cf = capf_of(cx, S, R2);
                        e.blo1 = static_cast<int16_t>(blo[1]);
                        e.bhi1 = static_cast<int16_t>(bhi[1]);
                        e.blo2 = static_cast<int16_t>(blo[2]);
                        e.bhi2 = static_cast<int16_t>(bhi[2]);
                        flags = cls | (ymaj ? 2 : 0) | 4;
                    }
                }
            }
        }
        e.flags = flags;
        __syncwarp();
        // the group's histories one at a time, all lanes on the rows of each
        for (int j = 0; j < kEuGroup; ++j) {
            const int fl = slot[j].flags;
            if (!(fl & 4)) continue;
            const int cls = fl & 1;
            const bool ymaj = (fl & 2) != 0;
            __syncwarp();  // the previous history is done with *cxs
            if (lane == 0) capx_of(g, slot[j].A, slot[j].B, ymaj, R2, *cxs);
            __syncwarp();
            const CapF cf = slot[j].cf;
            const int blo1 = slot[j].blo1, bhi1 = slot[j].bhi1;
            const int blo2 = slot[j].blo2, bhi2 = slot[j].bhi2;
            int32_t *diff = ymaj ? td.dy[cls] : td.dx[cls];
            const int n1 = ymaj ? g.nx : g.ny;
            // the rows that can meet the capsule queue up in shared memory;
            // whenever 32 are queued all lanes take one each, so the interval
            // search runs with full warps
            int qn = 0;
            auto drain = [&](int keep) {
                while (qn > keep) {
                    __syncwarp();
                    int lo, hi;
                    if (static_cast<int>(lane) < qn &&
                        row_interval(cf, *cxs, queue[lane] & 0xffff, queue[lane] >> 16, lo, hi)) {
                        const int ra = queue[lane] & 0xffff, rk = queue[lane] >> 16;
                        // x-major rows: (nx + 1) entries per (y, z); y-major:
                        // (ny + 1) per (x, z)
                        int32_t *row = diff + (static_cast<int64_t>(ra) +
                                               static_cast<int64_t>(n1) * rk) *
                                                  (cf.n0 + 1);
                        atomicAdd(row + lo, 1);
                        atomicAdd(row + hi + 1, -1);
                        vox[cls] += static_cast<unsigned>(hi - lo + 1);
                        rows += 1;
                    }
                    __syncwarp();
                    // keep what did not fit (fewer than 32 entries)
                    const int rest = qn > 32 ? qn - 32 : 0;
                    const int moved = static_cast<int>(lane) < rest ? queue[32 + lane] : 0;
                    __syncwarp();
                    if (static_cast<int>(lane) < rest) queue[lane] = moved;
                    __syncwarp();
                    qn = rest;
                }
            };
            // each lane one index a of the box, with the band of k whose rows
            // can meet the capsule
            for (int ab = blo1; ab <= bhi1; ab += 32) {
                const int a = ab + static_cast<int>(lane);
                int klo = 1, khi = 0;
                if (a <= bhi1) k_range(cf, a, blo2, bhi2, klo, khi);
                const int cnt = khi >= klo ? khi - klo + 1 : 0;
                const int most = __reduce_max_sync(0xffffffffu, cnt);
                for (int t = 0; t < most; ++t) {
                    const int k = klo + t;
                    // inside the band nearly every row meets the capsule, and
                    // the row search is exact for any row: the band's rows go
                    // to it directly; a whole box is filtered first
                    const bool meets = t < cnt && (cf.kband || row_meets_at(cf, *cxs, a, k));
                    const unsigned bal = __ballot_sync(0xffffffffu, meets);
                    if (meets) queue[qn + __popc(bal & ((1u << lane) - 1u))] = a | (k << 16);
                    qn += __popc(bal);
                    drain(31);
                }
            }
            drain(0);
        }
    }
    const unsigned long long part[8] = {nc.n_in, nc.n_miss, nc.n_hit, nc.n_none, nc.n_reject,
                                        vox[0], vox[1], rows};
#pragma unroll
    for (int q = 0; q < 8; ++q) {
        unsigned long long e = part[q];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) e += __shfl_xor_sync(0xffffffffu, e, o);
        if (lane == 0 && e != 0) atomicAdd(stats + q, e);
    }
}

// ------------------------------------------------------------- tiled path

constexpr int kSetupThreads = 512;

// Out of line, like ingest's: it runs when a thread meets a new angle.
__device__ __noinline__ void euclid_trig(float ang, const Cordic &cd, long long &c, long long &s)
{
    cordic_cs(q16_of(ang), cd, c, s);
}

// The tiles of a record: slices klo .. khi, and along y the strips that its
// part of the grid can reach.
__device__ __forceinline__ void euclid_tiles(const TilePlan &tp, int klo, int khi, int ylo, int yhi,
                                             int lo[3], int hi[3])
{
    lo[0] = hi[0] = 0;
    lo[1] = tp.mty ? static_cast<int>(umulhi32(static_cast<unsigned>(ylo), tp.mty)) : ylo;
    hi[1] = tp.mty ? static_cast<int>(umulhi32(static_cast<unsigned>(yhi), tp.mty)) : yhi;
    lo[2] = klo;
    hi[2] = khi;
}

// The strips along y of a record's tiles, as its status word holds them in place of
// its last slice (euclid_setup_kernel names the tiles from there: computed twice, in
// float, the two kernels' strips would have to agree to the bit).
__device__ __forceinline__ int strips_code(int lo, int hi) { return lo | ((hi - lo + 1) << 4); }
static_assert(kOpenStrips <= 16 && (kOpenStrips << 4 | (kOpenStrips - 1)) < 4096, "12 bits");

// Classification and records of a chunk (see ingest_kernel): world endpoints
// at the histories' slots, the walk type 2 for rows along y.
__global__ void __launch_bounds__(kIngestThreads, 4) euclid_ingest_kernel(
    Inputs in, int64_t n, int64_t per_block, GeomQ g, Cordic cd, float tau_l, float tau_h,
    int use_miss, int use_hit, long long R, TilePlan tp, Records rec, Ctrl *ctrl,
    uint32_t *bucket_count, uint32_t *block_base, uint32_t *block_pairs, uint32_t *stage)
{
    extern __shared__ uint32_t s_hist[];  // kGroups * ntiles counters
    __shared__ unsigned s_demand, s_total;
    const int nh = kGroups * tp.ntiles;
    for (int t = threadIdx.x; t < nh; t += blockDim.x) s_hist[t] = 0;
    if (threadIdx.x == 0) {
        s_demand = 0;
        s_total = 0;
    }
    __syncthreads();
    after_previous();
    EuCounts nc;
    bool tc_valid = false;
    float tc_ang = 0.0f;
    long long tc_c = 0, tc_s = 0;
    const int64_t h0 = static_cast<int64_t>(blockIdx.x) * per_block;
    const int64_t h1 = h0 + per_block < n ? h0 + per_block : n;
    const unsigned budget =
        h1 > h0 ? static_cast<unsigned>(h1 - h0) * static_cast<unsigned>(tp.pairs_per_record) : 0u;
    uint32_t *const list = stage + static_cast<int64_t>(blockIdx.x) * per_block * tp.pairs_per_record;
    for (int64_t base = h0; base < h1; base += blockDim.x) {
        const int64_t i = base + threadIdx.x;
        int cls = -1;
        bool ok = false, closed = false;
        int klo = 0, khi = -1, ylo = 0, yhi = 0, type = 0;
        int32_t w6[6] = {0, 0, 0, 0, 0, 0};
        if (i < h1) {
            const float w = in.wepl[i];
            cls = w < tau_l ? 0 : (w > tau_h ? 1 : -1);
            nc.n_in += 1;
            nc.n_miss += cls == 0;
            nc.n_hit += cls == 1;
            nc.n_none += cls < 0;
            if ((cls == 0 && use_miss) || (cls == 1 && use_hit)) {
                const float ang = in.angle[i];
                const float ui = in.u_in[i], vi = in.v_in[i], uo = in.u_out[i], vo = in.v_out[i];
                ok = fabsf(ang) < 1048576.0f;
                if (ok) {
                    if (!tc_valid || ang != tc_ang) {
                        euclid_trig(ang, cd, tc_c, tc_s);
                        tc_ang = ang;
                        tc_valid = true;
                    }
                    int32_t G[6];
                    ok = endpoints_cs(g, tc_c, tc_s, ui, vi, uo, vo, G);  // the thin rule
                }
                if (!ok) {
                    nc.n_reject += 1;
                } else {
                    long long W[6];
                    world_cs(g, tc_c, tc_s, ui, vi, uo, vo, W);
                    ok = euclid_range(g, W, R, klo, khi, ylo, yhi, closed);
#pragma unroll
                    for (int q = 0; q < 6; ++q) w6[q] = static_cast<int32_t>(W[q]);
                    type = abs(w6[4] - w6[1]) > abs(w6[3] - w6[0]) ? 2 : 0;
                }
            }
        }
        int c = 0, strips = 0;
        if (ok) {
            int lo[3], hi[3];
            euclid_tiles(tp, klo, khi, ylo, yhi, lo, hi);
            c = (hi[1] - lo[1] + 1) * (hi[2] - lo[2] + 1);
            strips = strips_code(lo[1], hi[1]);
        }
        reserve_and_write(tp, rec, ctrl, s_hist, &s_demand, budget, h0, i, h1, list, cls, type, ok,
                          closed && c <= tp.max_tiles ? c : -1, klo, strips, w6,
                          [&](int lo[3], int hi[3]) { euclid_tiles(tp, klo, khi, ylo, yhi, lo, hi); });
    }
    const unsigned sums[5] = {nc.n_in, nc.n_miss, nc.n_hit, nc.n_none, nc.n_reject};
    unsigned long long *const to[5] = {&ctrl->n_in, &ctrl->n_miss, &ctrl->n_hit, &ctrl->n_none,
                                       &ctrl->n_reject};
#pragma unroll
    for (int q = 0; q < 5; ++q) {
        const unsigned v = warp_sum_u32(sums[q]);
        if ((threadIdx.x & 31u) == 0 && v) atomicAdd(to[q], static_cast<unsigned long long>(v));
    }
    reserve_buckets(nh, s_hist, &s_total, bucket_count, block_base, block_pairs);
}

// Counting sort of the pairs (see scatter_kernel) with each pair's slice rows.
__global__ void __launch_bounds__(kSetupThreads, 2) euclid_setup_kernel(
    TilePlan tp, RowsArgs ra, int64_t per_block, Buckets buckets, const uint32_t *block_base,
    const uint32_t *block_pairs, Pairs pairs)
{
    extern __shared__ uint32_t s_mem[];
    const int nt = kGroups * tp.ntiles;
    uint32_t *s_base = s_mem;          // this block's first position in each bucket
    uint32_t *s_next = s_mem + nt;     // pairs written per bucket so far
    uint32_t *s_events = s_next + nt;  // and their rows
    for (int t = threadIdx.x; t < nt; t += blockDim.x) s_next[t] = s_events[t] = 0;
    after_previous();
    bucket_places<kSetupThreads>(nt, buckets, block_base, s_base);
    const int64_t h0 = static_cast<int64_t>(blockIdx.x) * per_block;
    const unsigned npairs = block_pairs[blockIdx.x];
    const uint32_t *list = pairs.stage + static_cast<int64_t>(blockIdx.x) * per_block * tp.pairs_per_record;
    for (unsigned e = threadIdx.x; e < npairs; e += kSetupThreads) {
        const uint32_t code = list[e];
        const int64_t slot = h0 + (code >> kRecordTileBits);
        const int j = static_cast<int>(code & (kMaxRecordTiles - 1u));
        const int32_t stw = ra.rec.status[slot];
        int32_t w[6];
#pragma unroll
        for (int a = 0; a < 6; ++a) w[a] = ra.rec.g[a][slot];
        const int klo = status_zlo(stw);
        int y = 0, k = klo + j;
        if (tp.nty > 1) {
            const int strips = status_zhi(stw), ey = strips >> 4;
            y = (strips & 15) + j % ey;
            k = klo + j / ey;
        }
        const int t = status_group(stw) * tp.ntiles + y + tp.nty * k;
        const uint32_t pos = s_base[t] + atomicAdd(&s_next[t], 1u);
        const int y0 = y * tp.ty, dy = min(tp.ty, tp.ny - y0);
        const bool ymaj = ((stw >> 4) & 1) != 0;
        const int rows = ymaj ? tp.nx : dy, len = ymaj ? dy : tp.nx;
        const int a0 = ymaj ? 0 : y0, m0 = ymaj ? y0 : 0;
        SliceRows r{};
        if (!slice_rows(ra.g, w, ra.R, k, a0, rows, m0, len, r)) r.n = 0;
        const int W = tile_row_words(len, rows);
        const unsigned long long open = open_code(static_cast<uint32_t>(slot), a0 + r.row, k, 0, y);
        uint4 *out = pairs.v + (kSliceWords / 4) * static_cast<size_t>(pos);
        out[0] = make_uint4(__float_as_uint(r.e0), __float_as_uint(r.ea), __float_as_uint(r.f0),
                            __float_as_uint(r.fa));
        out[1] = make_uint4(__float_as_uint(r.Kr), __float_as_uint(r.E0), __float_as_uint(r.Kd),
                            __float_as_uint(r.dq));
        out[2] = make_uint4(static_cast<uint32_t>(r.row * W) | (static_cast<uint32_t>(r.n) << 16),
                            static_cast<uint32_t>(len) | (static_cast<uint32_t>(W) << 16),
                            static_cast<uint32_t>(open),
                            static_cast<uint32_t>(open >> 32));
        if (r.n > 0) atomicAdd(&s_events[t], static_cast<uint32_t>(r.n));
    }
    __syncthreads();
    for (int t = threadIdx.x; t < nt; t += blockDim.x)
        if (s_events[t])
            atomicAdd(&buckets.events[t], static_cast<unsigned long long>(s_events[t]));
}

// What the tiled pass left open, a thread each: kOpenParts blocks per part of the
// list (a block's of that pass).
constexpr int kOpenParts = 8;

__global__ void __launch_bounds__(128) euclid_open_kernel(const ScanDesc *__restrict__ dp, RowsArgs ra)
{
    after_previous();
    const ScanDesc &d = *dp;
    const unsigned part = blockIdx.x / kOpenParts;
    const unsigned listed = d.pairs.fb_count[part];
    const unsigned n = listed < d.pairs.fb_cap ? listed : d.pairs.fb_cap;
    const uint2 *list = d.pairs.fb + static_cast<size_t>(part) * d.pairs.fb_cap;
    for (unsigned k = (blockIdx.x % kOpenParts) * blockDim.x + threadIdx.x; k < n;
         k += kOpenParts * blockDim.x) {
        const uint2 e = list[k];
        settle_open(ra, d, e.x, static_cast<int>(e.y));
    }
}

}  // namespace

cudaError_t launch_euclid(const Inputs &in, int64_t n, const hd_geometry *geom, const GeomQ &g,
                          const Cordic &cd, float tau_l, float tau_h, int use_miss, int use_hit,
                          float d0, void *workspace, uint32_t *N, uint32_t *M,
                          unsigned long long *stats, int64_t *rows, int sm_count,
                          cudaStream_t st)
{
    const size_t need = thick_workspace_bytes(geom);
    cudaError_t e = cudaMemsetAsync(workspace, 0, need, st);
    if (e == cudaSuccess && n > 0) {
        const long long R2 = 2 * q16_of(d0);
        const ThickDiff td = thick_diff_of(geom, workspace);
        unsigned long long *cnt = thick_counters_of(geom, workspace);
        // persistent warps
        int64_t blocks = int64_t(sm_count > 0 ? sm_count : 1) * kEuBlocksPerSm;
        const int64_t want = (n + kEuGroup * (kEuThreads / 32) - 1) /
                             (kEuGroup * (kEuThreads / 32));
        if (blocks > want) blocks = want;
        count_kernels(1);
        euclid_kernel<<<static_cast<unsigned>(blocks), kEuThreads, 0, st>>>(
            in, n, g, cd, tau_l, tau_h, use_miss, use_hit, R2, td, cnt, cnt + 8, nullptr, nullptr);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess)
        e = launch_thick_finish(geom, workspace, use_miss ? N : nullptr, use_hit ? M : nullptr,
                                stats, rows, st);
    return e;
}

cudaError_t init_euclid()
{
    cudaError_t e = cudaFuncSetAttribute(euclid_ingest_kernel,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         static_cast<int>(sizeof(uint32_t)) * kGroups * kMaxTiles);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(euclid_setup_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 static_cast<int>(sizeof(uint32_t)) * 3 * kGroups * kMaxTiles);
    return e;
}

int euclid_pairs_per_record(const hd_geometry *geom, float d0, const TilePlan &tp)
{
    const double k = std::ceil(2.0 * d0 / geom->sz) + 2.0;  // slices of a nearly flat path
    const double p = k * (tp.nty > 2 ? 2 : tp.nty);
    if (tp.ntiles <= 0 || tp.ntx != 1 || tp.tz != 1 || tp.nty > kOpenStrips || 2 * q16_of(d0) < 2 ||
        p > kMaxRecordTiles)
        return 0;
    return static_cast<int>(p);
}

cudaError_t launch_euclid_scan(const ScanDesc *desc_dev, const ScanDesc &desc, const Inputs &in,
                               int64_t n, const hd_geometry *geom, const GeomQ &g,
                               const Cordic &cd, float tau_l, float tau_h, int use_miss,
                               int use_hit, float d0, const Records &rec, uint32_t *block_base,
                               uint32_t *block_pairs, void *workspace, int grid, int sm_count,
                               cudaStream_t st)
{
    const TilePlan &tp = desc.tp;
    RowsArgs ra;
    ra.g = g;
    ra.R = 2 * q16_of(d0);
    ra.rec = rec;
    const ChunkSplit sp = chunk_split(n, sm_count, tp.ntiles);
    const size_t cols = kGroups * static_cast<size_t>(tp.ntiles);
    cudaError_t e = launch_chunk_begin(desc.ctrl, desc.buckets, tp.ntiles, st);
    if (e != cudaSuccess) return e;
    e = launch_chained(euclid_ingest_kernel, static_cast<unsigned>(sp.blocks), kIngestThreads, 4 * cols,
                       st, in, n, sp.per_block, g, cd, tau_l, tau_h, use_miss, use_hit, ra.R, tp,
                       rec, desc.ctrl, desc.buckets.count, block_base, block_pairs,
                       desc.pairs.stage);
    if (e != cudaSuccess) return e;
    e = launch_chained(euclid_setup_kernel, static_cast<unsigned>(sp.blocks), kSetupThreads, 12 * cols,
                       st, tp, ra, sp.per_block, desc.buckets, block_base, block_pairs, desc.pairs);
    if (e != cudaSuccess) return e;
    e = launch_trace_rows(desc_dev, tp.tile_words, tp.threads, grid, ra, st);
    if (e != cudaSuccess) return e;
    e = launch_chained(euclid_open_kernel, static_cast<unsigned>(grid * kOpenParts), 128, 0, st, desc_dev,
                       ra);
    if (e != cudaSuccess) return e;
    // the records of the global path, when there are any
    e = launch_thick_clear(geom, workspace, desc.ctrl, sm_count, st);
    if (e != cudaSuccess) return e;
    unsigned long long *cnt = thick_counters_of(geom, workspace);
    count_kernels(1);
    euclid_kernel<<<static_cast<unsigned>((sm_count > 0 ? sm_count : 1) * kEuBlocksPerSm), kEuThreads, 0,
                    st>>>(in, n, g, cd, tau_l, tau_h, use_miss, use_hit, ra.R,
                          thick_diff_of(geom, workspace), cnt, cnt + 8, rec.glist,
                          &desc.ctrl->n_global);
    e = cudaGetLastError();
    if (e == cudaSuccess)
        e = launch_thick_left(geom, workspace, use_miss ? desc.N : nullptr,
                              use_hit ? desc.M : nullptr, desc.ctrl, st);
    return e;
}

}  // namespace hd

extern "C" {

hd_status hd_accumulate_euclid(const hd_geometry *geom, const hd_params *params, float d0_mm,
                               const float *angle_deg, const float *u_in, const float *v_in,
                               const float *u_out, const float *v_out, const float *wepl,
                               int64_t n, uint32_t *N, uint32_t *M, void *workspace,
                               size_t workspace_bytes, int64_t *rows, void *stream)
{
    if (!geom || !params || n < 0 || !workspace) return HD_ERR_ARG;
    if (!(d0_mm >= 0.0f && d0_mm <= 64.0f)) return HD_ERR_RANGE;
    const hd_status gs = hd::check_geometry(geom);
    if (gs != HD_OK) return gs;
    if (std::isnan(params->wepl_miss_lt) || std::isnan(params->wepl_hit_gt) ||
        params->wepl_miss_lt > params->wepl_hit_gt)
        return HD_ERR_ARG;
    const uint32_t m = params->methods;
    if (m == 0 || (m & ~uint32_t(HD_SC | HD_MSC | HD_SM))) return HD_ERR_ARG;
    const int use_miss = (m & (HD_SC | HD_MSC)) ? 1 : 0;
    const int use_hit = (m & HD_SM) ? 1 : 0;
    if ((use_miss && !N) || (use_hit && !M)) return HD_ERR_ARG;
    if (n > 0 && (!angle_deg || !u_in || !v_in || !u_out || !v_out || !wepl)) return HD_ERR_ARG;
    if (workspace_bytes < hd::thick_workspace_bytes(geom) ||
        (reinterpret_cast<uintptr_t>(workspace) & 255) != 0)
        return HD_ERR_ARG;
    hd::Cordic cd{};
    if (!hd::make_cordic_table(cd)) return HD_ERR_RANGE;
    int dev = 0, sms = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) {
        cudaGetLastError();
        return HD_ERR_CUDA;
    }
    const hd::GeomQ gq = hd::make_geomq(geom->nx, geom->ny, geom->nz, geom->sx, geom->sy,
                                        geom->sz, geom->tracker_half_sep_mm);
    const hd::Inputs in{angle_deg, u_in, v_in, u_out, v_out, wepl};
    const cudaError_t e = hd::launch_euclid(in, n, geom, gq, cd, params->wepl_miss_lt,
                                            params->wepl_hit_gt, use_miss, use_hit, d0_mm,
                                            workspace, N, M, nullptr, rows, sms,
                                            static_cast<cudaStream_t>(stream));
    if (e != cudaSuccess) {
        hd::note_cuda_error(e, "hd_accumulate_euclid");
        return HD_ERR_CUDA;
    }
    return HD_OK;
}

}  // extern "C"
