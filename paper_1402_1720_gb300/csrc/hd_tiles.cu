// Shared-memory privatised traversal: the grid is cut into tiles whose
// counters fit in one block's shared memory, every (record, tile) pair is
// walked with the exact traversal clipped to the tile, and each block adds
// its private tile into N or M once per part of a bucket (the pairs of one
// group and tile, sorted in hd_scatter.cu) that it has walked; warps refill
// idle lanes from the parts' pairs, so lanes do not wait for the longest path.
#include <type_traits>

#include "hd_euclid.cuh"
#include "hd_fallback.cuh"

namespace hd {

namespace {

constexpr unsigned kFull = 0xffffffffu;
constexpr int kEventsPerStep = 8;  // events a traversal lane walks between refill checks

// ---------------------------------------------------------------- traversal
//
// A block's private tile holds one 32-bit word per voxel of the tile box in
// the layout of event walks (hd_geom.cuh): all walks of a bucket have one type,
// so the tile's fast axis is their major axis, the low half of a word counts
// the row changes that leave a run there and the high half the walks' first
// and last marks.  A part has at most 32767 pairs, so every prefix sum of
// either half stays inside 16 bits.
//
// Bound: integer issue of the event loop and the refills, one shared atomic
// per run (3.4 voxels on the head-sized scan).  The form before, +1 and -1 at
// the two ends of each run, took two and about three times the integer steps
// per run: head-sized scan (9e6 histories) 0.683 -> 0.407 ms, large streamed
// scan 0.288 -> 0.186 ms per chunk, with the balance and the flush below.

// What the kernel of the thin and dilated walks needs besides the scans: nothing.
struct NoRows {
    static constexpr bool kRows = false, kCells = false;
};
// The same for launches that look for cells to join (see Cell): a bucket per thread
// where there are threads enough, else a cell per thread, or several.
enum PlanBy { kByBucket, kByCell, kByCells };
template <PlanBy kPlanBy>
struct Cells {
    static constexpr bool kRows = false, kCells = true;
    static constexpr PlanBy kBy = kPlanBy;
};

template <class RowsT>
constexpr PlanBy plan_by()
{
    if constexpr (RowsT::kCells) return RowsT::kBy;
    else return kByBucket;
}

// Shared-memory reduction (no value returned) at a shared-space byte address.
__device__ __forceinline__ void smem_red_add(int addr, uint32_t v)
{
    asm volatile("red.shared.add.u32 [%0], %1;" ::"r"(addr), "r"(v));
}

// Event u of a step of cnt events: counted at the cursor, which then moves on
// (event_next without the count of events left); nothing when u >= cnt.
// Predicated by hand: the loop the compiler made of "leave when the walk ends"
// took about 16 instructions and a reconvergence per event, this takes 7.
__device__ __forceinline__ void event_step(EventCursor &c, int u, int cnt)
{
    asm volatile(
        "{\n\t"
        ".reg .pred p, q;\n\t"
        "setp.gt.s32 p, %3, %4;\n\t"
        "@p red.shared.add.u32 [%0], 1;\n\t"
        "@p add.u32 %1, %1, %5;\n\t"
        "setp.ge.and.u32 q, %1, %2, p;\n\t"
        "@p add.s32 %0, %0, %6;\n\t"
        "@q sub.u32 %1, %1, %2;\n\t"
        "@q add.s32 %0, %0, 4;\n\t"
        "}"
        : "+r"(c.addr), "+r"(c.rem)
        : "r"(c.ad), "r"(cnt), "r"(u), "r"(c.Ru), "r"(c.step)
        : "memory");
}

// One block's part of a bucket.  Pairs lie in the order of their histories (by
// gantry angle), so the lengths of their walks drift along a bucket; slots
// take them in pieces of 32 (a warp's walks stay alike) from kCols places of
// the bucket in turn, so that a range of slots samples all of it and ranges
// of equal size cost about the same: slot p is pair
// 32 ((v % kCols) rows + v / kCols) + p % 32, v = p / 32 (none when that is
// past the bucket's count).
//
// Parts are walked in groups: as many consecutive ones as have room for their
// tiles side by side in shared memory are walked together and then flushed, so
// that the block waits for its last walks once per group (about 14 000 cycles,
// as long as the walks of 1 300 pairs) and not once per part.
constexpr int kCols = 16;
struct TilePart {
    const uint4 *pairs;  // the scan's pairs
    uint32_t first;      // the bucket's first one
    int tile;    // tile id within its group
    int count;   // the bucket's pairs
    int start;   // slots [start, end)
    int end;
    int words;   // of its tile
    int offset;  // of the tile in the block's shared memory, in words
    int slot0;   // slots of the group before this part's
    int16_t scan;
    int8_t group;   // bit 0 the class (missed: N, hit: M), bits 1-2 the walk type
    int8_t form;    // kOwn, kJoined or kSame
    JoinedBox box;  // unless kOwn
};
// A part's walks: in a tile of their type's layout; in a joined one; in the joined
// one of the part before, which is flushed once for both.
constexpr int8_t kOwn = 0, kJoined = 1, kSame = 2;

struct TileBox {
    int x0, y0, z0, dx, dy, dz;
};

__device__ __forceinline__ TileBox tile_box(const TilePlan &tp, int tile)
{
    TileBox b;
    b.x0 = tile % tp.ntx * tp.tx;
    b.y0 = (tile / tp.ntx) % tp.nty * tp.ty;
    b.z0 = tile / (tp.ntx * tp.nty) * tp.tz;
    b.dx = min(tp.tx, tp.nx - b.x0);
    b.dy = min(tp.ty, tp.ny - b.y0);
    b.dz = min(tp.tz, tp.nz - b.z0);
    return b;
}

__device__ __forceinline__ int slot_rows(int count) { return (count + 32 * kCols - 1) / (32 * kCols); }

// A lane's next walk, loaded ahead: kVec 16-byte words per pair.
template <int kVec>
struct NextWalk {
    uint4 v[kVec];
    int base;      // its tile's offset in bytes
    int part;      // its part in the group
    uint32_t pos;  // the pair
    bool have;
    bool walk;  // false: a slot past its bucket's pairs
};

// The walk in slot r of the group of `n` parts: none past the pairs of a part.
template <int kVec>
__device__ __forceinline__ void load_slot(const TilePart *parts, int n, int r, NextWalk<kVec> &nw)
{
    int j = 0;
    while (j + 1 < n && r >= parts[j + 1].slot0) ++j;
    const TilePart &t = parts[j];
    const int p = t.start + r - t.slot0;
    const int v = p >> 5;
    const int k = 32 * ((v & (kCols - 1)) * slot_rows(t.count) + v / kCols) + (p & 31);
    nw.base = 4 * t.offset;
    nw.part = j;
    nw.walk = k < t.count;
    if (nw.walk) {
        nw.pos = t.first + static_cast<uint32_t>(k);
#pragma unroll
        for (int q = 0; q < kVec; ++q) nw.v[q] = t.pairs[kVec * static_cast<size_t>(nw.pos) + q];
    }
}

// The first walks of a group of `total` slots, a lane its own slot.  Loaded
// before the flush that precedes them, which hides their latency.
template <int kVec>
__device__ __forceinline__ void first_walks(const TilePart *parts, int n, int total,
                                            NextWalk<kVec> &nw)
{
    nw.have = static_cast<int>(threadIdx.x) < total;
    if (nw.have) load_slot(parts, n, static_cast<int>(threadIdx.x), nw);
}

// Walks the `total` slots of a group of parts into the block's tiles: each
// lane walks one pair and holds the packed walk of its next one (loaded a
// refill ahead, so starting a walk never waits on memory).  A refill happens
// once enough lanes are idle: they mark the ends of their finished walks, and
// those with a prefetched pair start it and fetch another, the slot coming
// from the block's counter *s_next (blockDim.x at the start: the first walks
// are the lanes' own, see first_walks).  Between refills the warp only counts
// events.  Out of line, so that nothing else in the kernel takes its registers.
__device__ __noinline__ void walk_parts(uint32_t *tiles, int thick, const TilePart *parts, int n,
                                        int total, int refill, unsigned *s_next,
                                        NextWalk<2> nw)
{
    const unsigned lane = threadIdx.x & 31u;
    const int sbase = static_cast<int>(__cvta_generic_to_shared(tiles));
    const int thick4 = 4 * (thick + 1);
    EventCursor c;
    c.ad = c.Ru = c.rem = 0u;
    c.addr = c.step = c.left = c.endl = 0;
    bool unmarked = false;  // the walk's end is still to be marked
    for (;;) {
        const unsigned idle = __ballot_sync(kFull, c.left == 0);
        if (__popc(idle) >= refill) {
            const unsigned want = __ballot_sync(kFull, c.left == 0 && nw.have);
            if (c.left == 0) {
                if (unmarked) smem_red_add(event_end(c, thick4), 0xffff0000u);
                unmarked = false;
                if (nw.have) {
                    const uint32_t o[kLeanWords] = {nw.v[0].x, nw.v[0].y, nw.v[0].z, nw.v[0].w,
                                                    nw.v[1].x, nw.v[1].y, nw.v[1].z, nw.v[1].w};
                    int first = 0;
                    if (nw.walk) unmarked = event_start(o, sbase + nw.base, c, first);
                    if (unmarked) smem_red_add(first, 65536u);
                    nw.have = false;
                }
            }
            if (want != 0) {
                unsigned base = 0;
                if (lane == 0) base = atomicAdd(s_next, __popc(want));
                base = __shfl_sync(kFull, base, 0);
                if (want & (1u << lane)) {
                    const unsigned r = base + __popc(want & ((1u << lane) - 1u));
                    nw.have = r < static_cast<unsigned>(total);
                    if (nw.have) load_slot(parts, n, static_cast<int>(r), nw);
                }
            } else if (idle == kFull) {
                break;
            }
        }
        const int cnt = min(c.left, kEventsPerStep);
#pragma unroll
        for (int u = 0; u < kEventsPerStep; ++u) event_step(c, u, cnt);
        c.left -= cnt;
    }
}

// event_step in a joined tile: the event's two updates.
__device__ __forceinline__ void joined_step(JoinedCursor &c, int u, int cnt)
{
    asm volatile(
        "{\n\t"
        ".reg .pred p, q;\n\t"
        ".reg .b32 e, s, n;\n\t"
        "setp.gt.s32 p, %3, %4;\n\t"
        "add.s32 e, %0, %7;\n\t"
        "add.s32 s, %0, %8;\n\t"
        "neg.s32 n, %9;\n\t"
        "@p red.shared.add.u32 [e], n;\n\t"
        "@p red.shared.add.u32 [s], %9;\n\t"
        "@p add.u32 %1, %1, %5;\n\t"
        "setp.ge.and.u32 q, %1, %2, p;\n\t"
        "@p add.s32 %0, %0, %6;\n\t"
        "@q sub.u32 %1, %1, %2;\n\t"
        "@q add.s32 %0, %0, %7;\n\t"
        "}"
        : "+r"(c.addr), "+r"(c.rem)
        : "r"(c.ad), "r"(cnt), "r"(u), "r"(c.Ru), "r"(c.step), "r"(c.major), "r"(c.minor), "r"(c.v)
        : "memory");
}

// walk_parts for joined tiles.
__device__ __noinline__ void walk_joined(uint32_t *tiles, const TilePart *parts, int n, int total,
                                         int refill, unsigned *s_next, NextWalk<2> nw)
{
    const unsigned lane = threadIdx.x & 31u;
    const int sbase = static_cast<int>(__cvta_generic_to_shared(tiles));
    JoinedCursor c{};
    bool unmarked = false;  // the walk's end is still to be marked
    for (;;) {
        const unsigned idle = __ballot_sync(kFull, c.left == 0);
        if (__popc(idle) >= refill) {
            const unsigned want = __ballot_sync(kFull, c.left == 0 && nw.have);
            if (c.left == 0) {
                if (unmarked) smem_red_add(joined_end(c), 0u - c.v);
                unmarked = false;
                if (nw.have) {
                    const uint32_t o[kLeanWords] = {nw.v[0].x, nw.v[0].y, nw.v[0].z, nw.v[0].w,
                                                    nw.v[1].x, nw.v[1].y, nw.v[1].z, nw.v[1].w};
                    int first = 0;
                    if (nw.walk) unmarked = joined_start(o, parts[nw.part].box, sbase + nw.base, c, first);
                    if (unmarked) smem_red_add(first, c.v);
                    nw.have = false;
                }
            }
            if (want != 0) {
                unsigned base = 0;
                if (lane == 0) base = atomicAdd(s_next, __popc(want));
                base = __shfl_sync(kFull, base, 0);
                if (want & (1u << lane)) {
                    const unsigned r = base + __popc(want & ((1u << lane) - 1u));
                    nw.have = r < static_cast<unsigned>(total);
                    if (nw.have) load_slot(parts, n, static_cast<int>(r), nw);
                }
            } else if (idle == kFull) {
                break;
            }
        }
        const int cnt = min(c.left, kEventsPerStep);
#pragma unroll
        for (int u = 0; u < kEventsPerStep; ++u) joined_step(c, u, cnt);
        c.left -= cnt;
    }
}

// One row of a slice walk (slice_row): its interval's +1 and -1 in the row at
// `at` (a byte address less 4 kWhole's bits, so that the whole_up form of an
// index is added to it directly); nothing unless `on`.
__device__ __forceinline__ void row_step(int at, float lo, float hi, bool on)
{
    asm volatile(
        "{\n\t"
        ".reg .pred p;\n\t"
        ".reg .b32 a, b;\n\t"
        "setp.ne.s32 p, %3, 0;\n\t"
        "shl.b32 a, %1, 2;\n\t"
        "shl.b32 b, %2, 2;\n\t"
        "add.s32 a, a, %0;\n\t"
        "add.s32 b, b, %0;\n\t"
        "@p red.shared.add.u32 [a], 1;\n\t"
        "@p red.shared.add.u32 [b+4], -1;\n\t"
        "}" ::"r"(at),
        "r"(__float_as_int(lo)), "r"(__float_as_int(hi)), "r"(on ? 1 : 0)
        : "memory");
}

constexpr int kRowsPerStep = 8;  // rows a lane takes between refill checks (4: 6 % slower)

// walk_parts for Euclidean thick rays: a lane takes the rows of one history in
// one slice, one after the other, each a closed form of about 35 instructions
// (slice_row) and two shared atomics.  What the closed form leaves open goes to
// the scan's list, or is settled at once when that is full.
__device__ __noinline__ void walk_parts(uint32_t *tiles, const TilePart *parts, int n, int total,
                                        int refill, unsigned *s_next, NextWalk<3> nw,
                                        const ScanDesc &d, const RowsArgs &ra)
{
    const unsigned lane = threadIdx.x & 31u;
    const int sbase = static_cast<int>(__cvta_generic_to_shared(tiles)) -
                      static_cast<int>(0x4B400000u << 2);
    SliceRows c{};
    float i = 0.0f, top = 0.0f;
    int left = 0, at = 0, step = 0;
    uint32_t pos = 0;  // the pair
    for (;;) {
        const unsigned idle = __ballot_sync(kFull, left == 0);
        if (__popc(idle) >= refill) {
            const unsigned want = __ballot_sync(kFull, left == 0 && nw.have);
            if (left == 0 && nw.have) {
                if (nw.walk) {
                    unsigned long long code;
                    slice_unpack(nw.v, c, top, code);
                    left = c.n;
                    pos = nw.pos;
                    at = sbase + nw.base + 4 * static_cast<int>(nw.v[2].x & 0xffffu);
                    step = 4 * static_cast<int>(nw.v[2].y >> 16);
                    i = 0.0f;
                }
                nw.have = false;
            }
            if (want != 0) {
                unsigned base = 0;
                if (lane == 0) base = atomicAdd(s_next, __popc(want));
                base = __shfl_sync(kFull, base, 0);
                if (want & (1u << lane)) {
                    const unsigned r = base + __popc(want & ((1u << lane) - 1u));
                    nw.have = r < static_cast<unsigned>(total);
                    if (nw.have) load_slot(parts, n, static_cast<int>(r), nw);
                }
            } else if (idle == kFull) {
                break;
            }
        }
        const int cnt = min(left, kRowsPerStep);
        unsigned open = 0;  // rows of this step with something left open
#pragma unroll
        for (int u = 0; u < kRowsPerStep; ++u) {
            float x0, x1, y0, y1;
            const float q = slice_row(c, i, x0, x1, y0, y1);
            const float lo = fmaxf(x1, kWhole), hi = fminf(y0, top);
            const bool on = u < cnt, closed = q > 4.0f * c.dq;
            row_step(at, lo, hi, on && closed && lo <= hi);
            if (on && !((closed && x0 == x1 && y0 == y1) || q < -c.dq)) open |= 1u << u;
            i += 1.0f;
            at += step;
        }
        left -= cnt;
        while (open != 0) {
            const int u = __ffs(open) - 1;
            open &= open - 1;
            // to the block's list, or settled at once when that is full
            const int row = static_cast<int>(i) + u - kRowsPerStep;
            const unsigned n = atomicAdd(s_next + 1, 1u);
            if (n < d.pairs.fb_cap)
                d.pairs.fb[static_cast<size_t>(blockIdx.x) * d.pairs.fb_cap + n] =
                    make_uint2(pos, static_cast<uint32_t>(row));
            else
                settle_open(ra, d, pos, row);
        }
    }
}

// A warp's inclusive prefix sums of a row of W <= 32 kPer words: word
// lane kPer + i in v[i] (kPer odd: the lanes read from 32 banks).  `after`:
// the tile's words from the row's start on.  When there are 32 kPer of them,
// those past the row's end are read too: they come after the row's and are
// dropped.
template <int kPer>
__device__ __forceinline__ void row_prefix(const uint32_t *row, int W, int after,
                                           uint32_t (&v)[kPer])
{
    const int lane = static_cast<int>(threadIdx.x & 31u);
    const int b = lane * kPer;
    if (after >= 32 * kPer) {
#pragma unroll
        for (int i = 0; i < kPer; ++i) v[i] = row[b + i];
    } else {
#pragma unroll
        for (int i = 0; i < kPer; ++i) v[i] = b + i < W ? row[b + i] : 0u;
    }
#pragma unroll
    for (int i = 1; i < kPer; ++i) v[i] += v[i - 1];
    uint32_t incl = v[kPer - 1];
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t t = __shfl_up_sync(kFull, incl, o);
        if (lane >= o) incl += t;
    }
    const uint32_t before = incl - v[kPer - 1];
#pragma unroll
    for (int i = 0; i < kPer; ++i) v[i] += before;
}

// Adds a count to a voxel unless it is zero (predicated: no branch).
__device__ __forceinline__ void add_count(uint32_t *v, uint32_t c)
{
    asm volatile(
        "{\n\t"
        ".reg .pred p;\n\t"
        "setp.ne.u32 p, %1, 0;\n\t"
        "@p red.global.add.u32 [%0], %1;\n\t"
        "}" ::"l"(v),
        "r"(c)
        : "memory");
}

// Where a tile's counts go: the volume's voxel (0, 0, 0) of the tile, and its
// grid's extents.
struct FlushTo {
    uint32_t *vol;
    int nx, ny;
    __device__ __forceinline__ uint32_t *line(int y, int z) const
    {
        return vol + static_cast<long long>(nx) * (y + static_cast<long long>(ny) * z);
    }
};

// Flush of thin walks whose rows fit 32 kPer words.  A warp takes a band of
// rows in walk order and keeps each row's prefix sums in registers for the
// next one, so a word is read once for its count (modulo 2^16, where counts
// lie, SP + SE' - SE is one three-operand sum of the words), written back as a
// count, and read, cleared and added to the volume by lanes along x: about 100
// instructions per 200-voxel row, where separate prefix, decode and clear
// passes took 240.  kPlain: the words are difference counts along the rows, and
// their prefix sums the counts (Euclidean thick rays).
template <int kPer, bool kPlain>
__device__ __noinline__ void flush_rows(uint32_t *tile, int dx, int dy, int dz, bool ymaj, int s,
                                        int W, FlushTo to)
{
    const int lane = static_cast<int>(threadIdx.x & 31u);
    const int warp = static_cast<int>(threadIdx.x >> 5), nwarps = static_cast<int>(blockDim.x >> 5);
    const int nmaj = ymaj ? dy : dx, nminor = ymaj ? dx : dy;
    const int rows = nminor * dz;
    const int band = (rows + nwarps - 1) / nwarps;
    const int a = min(warp * band, rows), e = min(a + band, rows);
    const int i0 = s > 0 ? 0 : nminor - 1;  // a slice's first row in walk order
    int r = s > 0 ? a : e - 1;
    int z = dz == 1 ? 0 : r / nminor, i = r - z * nminor;
    uint32_t pv[kPer];
#pragma unroll
    for (int k = 0; k < kPer; ++k) pv[k] = 0u;
    // the row before the band belongs to another warp, which overwrites it
    if (!kPlain && a < e && i != i0) row_prefix<kPer>(tile + W * (r - s), W, W * (rows - (r - s)), pv);
    __syncthreads();
    for (int n = a; n < e; ++n, r += s) {
        uint32_t *row = tile + W * r;
        if (i == i0) {
#pragma unroll
            for (int k = 0; k < kPer; ++k) pv[k] = 0u;
        }
        uint32_t v[kPer];
        // what follows the row may be rewritten meanwhile: harmless, it is dropped
        row_prefix<kPer>(row, W, W * (rows - r), v);
        uint32_t left = __shfl_up_sync(kFull, v[kPer - 1], 1);
        if (lane == 0) left = 0u;
        __syncwarp();
#pragma unroll
        for (int k = 0; k < kPer; ++k) {
            const int m = lane * kPer + k;
            const uint32_t c = kPlain ? v[k] : ((v[k] >> 16) + pv[k] - left) & 0xffffu;
            left = v[k];
            pv[k] = v[k];
            if (m < W) row[m] = m < nmaj ? c : 0u;
        }
        if (!ymaj) {
            __syncwarp();
            uint32_t *out = to.line(i, z) + lane;
            uint32_t c[kPer];
#pragma unroll
            for (int k = 0; k < kPer; ++k) c[k] = lane + 32 * k < dx ? row[lane + 32 * k] : 0u;
#pragma unroll
            for (int k = 0; k < kPer; ++k) {
                if (lane + 32 * k < dx) row[lane + 32 * k] = 0u;
                add_count(out + 32 * k, c[k]);
            }
        }
        // the next row in walk order
        i += s;
        if (i < 0) {
            i = nminor - 1;
            --z;
        } else if (i == nminor) {
            i = 0;
            ++z;
        }
    }
    if (ymaj) {
        __syncthreads();
        for (int l = warp; l < dy * dz; l += nwarps) {
            const int zz = dz == 1 ? 0 : l / dy, y = l - zz * dy;
            uint32_t *out = to.line(y, zz) + lane;
            uint32_t *line = tile + y + W * nminor * zz + W * lane;
            for (int x = lane; x - lane < dx; x += 128, out += 128, line += 128 * W) {
                uint32_t c[4];
#pragma unroll
                for (int k = 0; k < 4; ++k) c[k] = x + 32 * k < dx ? line[32 * k * W] : 0u;
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    if (x + 32 * k < dx) line[32 * k * W] = 0u;
                    add_count(out + 32 * k, c[k]);
                }
            }
        }
    }
}

// Flush of a group's n parts in joined tiles, all tiles at once (small ones leave
// most warps without a column).  A thread per column turns the high halves into
// their sums along y (lanes along x); then a warp per row sums the low halves along
// x, kPer words a lane at a time, and adds both to the volume, clearing the row.
__device__ __noinline__ void flush_joined(uint32_t *tiles, const TilePart *parts, int n,
                                          const ScanDesc *__restrict__ descs)
{
    constexpr int kPer = 7, kAhead = 8;
    const int lane = static_cast<int>(threadIdx.x & 31u);
    const int warp = static_cast<int>(threadIdx.x >> 5), nwarps = static_cast<int>(blockDim.x >> 5);
    int mine = warp;  // this warp's next piece of 32 columns, or row, of the tile at hand
    for (int t = 0; t < n; ++t) {
        const TilePart &j = parts[t];
        if (j.form == kSame) continue;
        const TileBox b = tile_box(descs[j.scan].tp, j.tile);
        const int P = b.dx + 1, slice = P * (b.dy + 1), pieces = (b.dx * b.dz + 31) >> 5;
        for (; mine < pieces; mine += nwarps) {
            const int q = 32 * mine + lane;
            if (q >= b.dx * b.dz) continue;
            const int z = b.dz == 1 ? 0 : q / b.dx;
            uint32_t *col = tiles + j.offset + slice * z + q - z * b.dx;
            uint32_t sum = 0u;
            for (int y = 0; y < b.dy; y += kAhead, col += kAhead * P) {
                uint32_t w[kAhead];
#pragma unroll
                for (int k = 0; k < kAhead; ++k) w[k] = y + k < b.dy ? col[k * P] : 0u;
#pragma unroll
                for (int k = 0; k < kAhead; ++k) {
                    sum += joined_high(w[k]);
                    if (y + k < b.dy) col[k * P] = (w[k] & 0xffffu) | (sum << 16);
                }
            }
        }
        mine -= pieces;
    }
    __syncthreads();
    mine = warp;
    for (int t = 0; t < n; ++t) {
        const TilePart &j = parts[t];
        if (j.form == kSame) continue;
        const ScanDesc &d = descs[j.scan];
        const TileBox b = tile_box(d.tp, j.tile);
        uint32_t *const tile = tiles + j.offset;
        const int P = b.dx + 1, slice = P * (b.dy + 1), rows = b.dy * b.dz;
        const FlushTo to{((j.group & 1) == 0 ? d.N : d.M) + b.x0 +
                             static_cast<long long>(d.tp.nx) *
                                 (b.y0 + static_cast<long long>(d.tp.ny) * b.z0),
                         d.tp.nx, d.tp.ny};
        for (; mine < rows; mine += nwarps) {
            const int z = b.dz == 1 ? 0 : mine / b.dy, y = mine - z * b.dy;
            uint32_t *row = tile + slice * z + P * y;
            uint32_t *out = to.line(y, z);
            uint32_t carry = 0u;
            for (int m0 = 0; m0 < b.dx; m0 += 32 * kPer) {
                const int a = m0 + lane * kPer;
                uint32_t v[kPer], hi[kPer];
#pragma unroll
                for (int k = 0; k < kPer; ++k) v[k] = a + k < b.dx ? row[a + k] : 0u;
#pragma unroll
                for (int k = 0; k < kPer; ++k) hi[k] = v[k] >> 16;
#pragma unroll
                for (int k = 1; k < kPer; ++k) v[k] += v[k - 1];
                uint32_t incl = v[kPer - 1];
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const uint32_t u = __shfl_up_sync(kFull, incl, o);
                    if (lane >= o) incl += u;
                }
                const uint32_t before = incl - v[kPer - 1] + carry;
                carry += __shfl_sync(kFull, incl, 31);
#pragma unroll
                for (int k = 0; k < kPer; ++k)
                    if (a + k < b.dx) row[a + k] = ((v[k] + before) & 0xffffu) + hi[k];
                __syncwarp();
#pragma unroll
                for (int k = 0; k < kPer; ++k) {
                    const int x = m0 + lane + 32 * k;
                    if (x < b.dx) {
                        add_count(out + x, row[x]);
                        row[x] = 0u;
                    }
                }
            }
            if (lane == 0) row[b.dx] = 0u;
        }
        mine -= rows;
        for (int q = static_cast<int>(threadIdx.x); q < P * b.dz; q += blockDim.x) {
            const int z = b.dz == 1 ? 0 : q / P;
            tile[slice * z + P * b.dy + q - z * P] = 0u;
        }
    }
}

// In-place inclusive prefix sum of a row of any length by a warp.
__device__ __forceinline__ void prefix_row(uint32_t *row, int W)
{
    const int lane = static_cast<int>(threadIdx.x & 31u);
    uint32_t carry = 0;
    for (int w0 = 0; w0 < W; w0 += 32) {
        uint32_t v = w0 + lane < W ? row[w0 + lane] : 0u;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t t = __shfl_up_sync(kFull, v, o);
            if (lane >= o) v += t;
        }
        v += carry;
        if (w0 + lane < W) row[w0 + lane] = v;
        carry = __shfl_sync(kFull, v, 31);
    }
}

// The count of voxel m of a dilated row from the prefix-summed tile (see the
// event walks in hd_geom.cuh); i is the row's minor index, s the walks' row
// direction, `row` its first word.
__device__ __forceinline__ int thick_count(const uint32_t *row, int W, int m, int nmaj, int i,
                                           int nminor, int s, int thick)
{
    int v = 0;
    const int j0 = max(-thick, -i), j1 = min(thick, nminor - 1 - i);
    for (int j = j0; j <= j1; ++j) v += static_cast<int>(row[m + j * W]) >> 16;
    const int ia = i - (thick + 1) * s, ib = i + thick * s;
    if (ia >= 0 && ia < nminor)
        v += static_cast<int>(row[min(m + thick, nmaj) - (thick + 1) * s * W] & 0xffffu);
    if (ib >= 0 && ib < nminor && m - thick > 0)
        v -= static_cast<int>(row[m - thick - 1 + thick * s * W] & 0xffffu);
    return v;
}

// Flush of dilated walks, and of rows longer than flush_rows takes: prefix
// sums in place, each voxel's count from its neighbours' words (or its own,
// kPlain), then clearing.
template <bool kPlain>
__device__ __noinline__ void flush_general(uint32_t *tile, int dx, int dy, int dz, bool ymaj, int s,
                                           int W, int thick, FlushTo to)
{
    const int lane = static_cast<int>(threadIdx.x & 31u);
    const int warp = static_cast<int>(threadIdx.x >> 5), nwarps = static_cast<int>(blockDim.x >> 5);
    const int nmaj = ymaj ? dy : dx, nminor = ymaj ? dx : dy;
    for (int r = warp; r < nminor * dz; r += nwarps) prefix_row(tile + W * r, W);
    __syncthreads();
    // a warp per line of voxels along x; mx, my: words from a voxel to the next
    const int mx = ymaj ? W : 1, my = ymaj ? 1 : W;
    for (int l = warp; l < dy * dz; l += nwarps) {
        const int z = dz == 1 ? 0 : l / dy, y = l - z * dy;
        uint32_t *out = to.line(y, z);
        const uint32_t *line = tile + my * y + W * nminor * z;
        for (int x = lane; x < dx; x += 32) {
            const int i = ymaj ? x : y, m = ymaj ? y : x;
            add_count(out + x, kPlain ? line[mx * x]
                                      : static_cast<uint32_t>(thick_count(
                                            line + mx * x - m, W, m, nmaj, i, nminor, s, thick)));
        }
    }
    __syncthreads();
    // the tile starts on a 16-byte boundary and is planned in whole vectors
    uint4 *t4 = reinterpret_cast<uint4 *>(tile);
    for (int w = static_cast<int>(threadIdx.x); w < (W * nminor * dz + 3) >> 2; w += blockDim.x)
        t4[w] = make_uint4(0u, 0u, 0u, 0u);
}

// Adds the tile's counts to the volume (one global atomic per nonzero voxel,
// lanes along x whichever axis the rows follow) and clears it for the next part.
template <bool kPlain>
__device__ __forceinline__ void flush_tile(uint32_t *tile, int dx, int dy, int dz, int type,
                                           int thick, uint32_t *vol, int nx, int ny, int x0,
                                           int y0, int z0)
{
    const bool ymaj = (type & 2) != 0;
    const int s = (type & 1) ? -1 : 1;
    const int nmaj = ymaj ? dy : dx, nminor = ymaj ? dx : dy;
    const int W = tile_row_words(nmaj, nminor);
    const FlushTo to{vol + x0 + static_cast<long long>(nx) * (y0 + static_cast<long long>(ny) * z0),
                     nx, ny};
    if ((!kPlain && thick > 0) || W > 32 * 13) flush_general<kPlain>(tile, dx, dy, dz, ymaj, s, W, thick, to);
    else if (W <= 32 * 3) flush_rows<3, kPlain>(tile, dx, dy, dz, ymaj, s, W, to);
    else if (W <= 32 * 5) flush_rows<5, kPlain>(tile, dx, dy, dz, ymaj, s, W, to);
    else if (W <= 32 * 7) flush_rows<7, kPlain>(tile, dx, dy, dz, ymaj, s, W, to);
    else if (W <= 32 * 9) flush_rows<9, kPlain>(tile, dx, dy, dz, ymaj, s, W, to);
    else flush_rows<13, kPlain>(tile, dx, dy, dz, ymaj, s, W, to);
}

// The pairs without an event walk (the fallback lists), walked with the general
// run walk in global memory by the blocks as they run out of parts: a warp per
// pair while there are no more of them than warps (the last walks end sooner), else
// fewer lanes for each, whose strips are set up fewer times (deep slabs list every
// walk that crosses z inside one: 64 x 64 x 64 in slabs of four, 1e6 histories 275
// -> 248 us, 250 with a lane for each, which ends 0.1 ms late where they are few).
// Out of line, so its registers do not weigh on
// the event loop.
__device__ __noinline__ void walk_fallback_lists(const ScanDesc *__restrict__ descs, int nscans)
{
    const unsigned lane = threadIdx.x & 31u;
    const unsigned warps = gridDim.x * (blockDim.x >> 5);
    for (int k = 0; k < nscans; ++k) {
        const ScanDesc &d = descs[k];
        if (d.tp.thick > 0) continue;  // dilated by a kernel of their own
        const unsigned nf = d.ctrl->n_pair_fallback;
        if (nf == 0) continue;
        const int lanes = nf <= warps ? 32 : (nf <= 4u * warps ? 8 : 2);
        for (;;) {
            unsigned i = 0;
            if (lane == 0) i = atomicAdd(&d.ctrl->fb_next, 32u / lanes);
            i = __shfl_sync(kFull, i, 0);
            if (i >= nf) break;
            i += lane / lanes;
            if (i < nf) {
                int32_t gi[3], go[3];
                const uint32_t id = load_general(d.pairs, d.pairs.fb[i].x, gi, go);
                GlobalVisit v;
                v.vol = (id & 1u) == 0 ? d.N : d.M;
                walk_tile_global(d.tp, gi, go, static_cast<int>(id >> 1), lanes, v);
            }
            __syncwarp();
        }
    }
}

// Cost of a bucket in event units: its events, kPairCost per walk (its start,
// marks and loads), and for its flush kFlushCost per word of the tile and
// kPartCost besides (fits over the parts of the head-sized and the large
// streamed scan).
// For Euclidean thick rays the events are rows, each about five times the work.
constexpr unsigned kPairCost = 9, kFlushCost = 4, kPartCost = 10000;
constexpr int kPartList = 32;  // parts a block lists at a time

__device__ __forceinline__ unsigned long long flush_cost(int tile_words)
{
    return kPartCost + static_cast<unsigned long long>(kFlushCost) * static_cast<unsigned>(tile_words);
}

// A cell is one tile of one class with its four buckets, by walk type (bucket
// (class + 2 type) ntiles + tile).  Each bucket with pairs is walked and flushed for
// itself, or, joined, all of them into one tile that is flushed once.  An event
// costs more there (two updates and a conversion of the walk) and so does the
// flush (columns, then rows), but a cell of few walks in several directions
// (histories of many angles, or in no order of angle, on many tiles) pays for
// one flush instead of four.  400 x 400 x 128, 9e6 histories in no order: in 20
// chunks 11.4 -> 6.8 ms (8.2 before walks were sorted by type), 2e5 of them in one
// 765 -> 510 us (592); 236 x 236 x 60, 1e5 histories 167 -> 119 us.  Costs in event
// units: kJoinedEvent quarters of one per event, kJoinedPair per walk, a quarter
// more per flush.  What a flush saves is far less than what one costs (it also
// waits while others walk): kSavedPart and kSavedWord, with four types joined up to
// 3.7 events per word of the tile.  In 17 grids at four chunk sizes joined takes 0.5
// to 0.9 of the time at one event per word, and the forms are alike at 8; but
// joined up to 11, 48 head-sized scans in one launch of this kernel took 27.2 ms,
// and 25.6 up to 3.7 or not joined at all.
constexpr unsigned kJoinedEvent = 7, kJoinedPair = 16, kSavedPart = 1000, kSavedWord = 1;

// Launches of fewer cells than three to four blocks do not look at it
// (launch_trace_tiles): their cells are cut into parts, each with a flush, and the
// four flushes of a cell are spread over blocks that would have little else to do
// (64 x 64 x 50 joined takes 1.1 times as long at any chunk size); and a small scan
// waits for every instruction before its walks.  Nor do those of too many histories
// per cell, which the host knows: 3 to 5 us of 140 to 300 (1e6 histories on 100 x 100
// x 100 to 400 x 400 x 64, nine chunks 2 % slower with it).
struct Cell {
    unsigned long long cost[4];  // of the parts made of each bucket (joined: cost[0], of all)
    unsigned count[4];           // pairs
    bool joined;
};

// Pieces of 32 slots of a bucket.
__device__ __forceinline__ int pieces_of(unsigned count) { return kCols * slot_rows(static_cast<int>(count)); }

template <bool kRows>
__device__ __forceinline__ unsigned long long bucket_cost(unsigned count, unsigned long long events,
                                                          int tile_words)
{
    return count == 0 ? 0ull
                      : (kRows ? 5ull : 1ull) * events + static_cast<unsigned long long>(kPairCost) * count +
                            flush_cost(tile_words);
}

__device__ __forceinline__ Cell cell_of(const ScanDesc &d, int cell)
{
    const int step = 2 * d.tp.ntiles, words = d.tp.tile_words;
    const unsigned long long flush = flush_cost(words);
    unsigned long long e[4], events = 0, pairs = 0;
    int types = 0;
    Cell c;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        c.count[j] = d.buckets.count[cell + step * j];
        e[j] = d.buckets.events[cell + step * j];
    }
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        c.cost[j] = bucket_cost<false>(c.count[j], e[j], words);
        pairs += c.count[j];
        events += e[j];
        types += c.count[j] != 0u ? 1 : 0;
    }
    const unsigned long long all = kJoinedEvent * events / 4ull + kJoinedPair * pairs + flush + flush / 4ull;
    const unsigned long long more = (kJoinedEvent - 4u) * events + 4u * (kJoinedPair - kPairCost) * pairs;
    const unsigned long long saved = kSavedPart + static_cast<unsigned long long>(kSavedWord) *
                                                      static_cast<unsigned>(words);
    c.joined = types > 1 && more < static_cast<unsigned>(4 * types - 5) * saved;  // quarters
    if (c.joined) {
        c.cost[0] = all;
        c.cost[1] = c.cost[2] = c.cost[3] = 0ull;
    }
    return c;
}

// Blocks of its own for that cost, about two flushes' worth of work each.
__device__ __forceinline__ unsigned long long own_blocks(unsigned long long cost, int tile_words)
{
    const unsigned long long f = 2ull * flush_cost(tile_words);
    return (cost + f - 1ull) / f;
}

// Where the boundary at cost x of the launch falls in `pieces` pieces of 32 slots
// whose cost begins at p: slots before it (0 .. all).  A part worth less
// than its own flush goes to the neighbour (tile_words -1: costs are blocks,
// and a boundary stays where it falls).
__device__ __forceinline__ int boundary_slot(unsigned long long cost, int pieces, int tile_words,
                                             unsigned long long p, unsigned long long x)
{
    const unsigned long long f = tile_words < 0 ? 0ull : flush_cost(tile_words);
    if (x <= p + f) return 0;
    if (x + f >= p + cost) return 32 * pieces;
    return 32 * static_cast<int>((x - p) * static_cast<unsigned long long>(pieces) / cost);
}

// Exclusive block scan of one 64-bit value per thread (blockDim.x <= 1024).
__device__ __forceinline__ unsigned long long block_excl_scan64(unsigned long long v,
                                                                unsigned long long *s_warp,
                                                                unsigned long long &total)
{
    const unsigned lane = threadIdx.x & 31u, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
    unsigned long long incl = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const unsigned long long t = __shfl_up_sync(kFull, incl, o);
        if (lane >= static_cast<unsigned>(o)) incl += t;
    }
    __syncthreads();  // the last use of s_warp is over
    if (lane == 31) s_warp[wid] = incl;
    __syncthreads();
    // every warp scans the warps' sums for itself
    unsigned long long w = lane < nw ? s_warp[lane] : 0ull;
    const unsigned long long own = w;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const unsigned long long t = __shfl_up_sync(kFull, w, o);
        if (lane >= static_cast<unsigned>(o)) w += t;
    }
    total = __shfl_sync(kFull, w, 31);
    return __shfl_sync(kFull, w - own, wid) + incl - v;
}

// The block's stretch [x0, x1) of the launch's costs, in blocks when `own`.
struct Stretch {
    unsigned long long before;  // of the thread's first bucket
    unsigned long long x0, x1;
    bool own;
};

__device__ __forceinline__ void fill_part(TilePart &j, const ScanDesc &d, int k, int t, int count,
                                          int s0, int s1, int8_t form)
{
    j.pairs = d.pairs.v;
    j.first = d.buckets.first[t];
    j.scan = static_cast<int16_t>(k);
    j.tile = t % d.tp.ntiles;
    j.group = static_cast<int8_t>(t / d.tp.ntiles);
    j.count = count;
    j.start = s0;
    j.end = s1;
    j.words = d.tp.tile_words;
    j.form = form;
}

// Passes over a thread's cells i0 .. i1 - 1 (of scan k those from s_first[k] / 4
// on): the sums of their costs by type, or of the blocks of their own.
template <bool kBlocks>
__device__ __forceinline__ void cell_sums(const ScanDesc *__restrict__ descs, const int *s_first,
                                          int i0, int i1, unsigned long long sum[4])
{
#pragma unroll
    for (int j = 0; j < 4; ++j) sum[j] = 0ull;
    int k = 0;
    for (int i = i0; i < i1; ++i) {
        while (4 * i >= s_first[k + 1]) ++k;
        const ScanDesc &d = descs[k];
        const Cell c = cell_of(d, i - s_first[k] / 4);
#pragma unroll
        for (int j = 0; j < 4; ++j)
            sum[j] += kBlocks ? own_blocks(c.cost[j], d.tp.tile_words) : c.cost[j];
    }
}

// Exclusive block scan of them in the order of the launch's costs, with four words
// of s for each warp.  Many cells: all buckets of type 0, then of type 1, and so on.
// With a cell's types close together, blocks beside one another go through the same
// tiles in step and their flushes meet (a batch of 48 scans 27.3 ms, 26.5 so).  At
// most a cell per thread: of the cells of a warp all of type 0, then of type 1, ..,
// a scan instead of four (1 us of a chunk of the large streamed scan).
template <bool many>
__device__ __forceinline__ void scan_types(const unsigned long long sum[4], unsigned long long *s,
                                           unsigned long long before[4], unsigned long long &total)
{
    const unsigned lane = threadIdx.x & 31u, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
    unsigned long long types = 0;  // of the warp's types so far
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        unsigned long long incl = sum[j];
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const unsigned long long t = __shfl_up_sync(kFull, incl, o);
            if (lane >= static_cast<unsigned>(o)) incl += t;
        }
        before[j] = incl - sum[j] + (many ? 0ull : types);
        types += __shfl_sync(kFull, incl, 31);
        if (lane == 31) s[4 * wid + j] = many ? incl : types;
    }
    __syncthreads();
    total = 0ull;
    // every warp scans the warps' sums for itself
#pragma unroll
    for (int j = many ? 0 : 3; j < 4; ++j) {
        unsigned long long w = lane < nw ? s[4 * lane + j] : 0ull;
        const unsigned long long own = w;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const unsigned long long t = __shfl_up_sync(kFull, w, o);
            if (lane >= static_cast<unsigned>(o)) w += t;
        }
        const unsigned long long base = total + __shfl_sync(kFull, w - own, wid);
        total += __shfl_sync(kFull, w, 31);
#pragma unroll
        for (int q = 0; q < 4; ++q)
            if (!many || q == j) before[q] += base;
    }
    __syncthreads();  // s is free again
}

// The parts of bucket j of cell t0 of scan k (cost c.cost[j], beginning at p) in the
// block's stretch, counted in n, or listed (kList: the thread's next has number
// rank, list begins at number j0): each at most job_size pairs, of a joined cell in
// up to four, one to a bucket.
template <bool kList>
struct PartTaker {
    const Stretch &st;
    unsigned long long rank, j0;
    TilePart *list;
    unsigned long long n = 0;

    __device__ __forceinline__ void put(const ScanDesc &d, int k, const Cell &c, int t0, int u, int s0,
                                        int s1, bool same)
    {
        if (kList && rank >= j0 && rank < j0 + kPartList) {
            TilePart &j = list[rank - j0];
            fill_part(j, d, k, t0 + 2 * d.tp.ntiles * u, static_cast<int>(c.count[u]), s0, s1,
                      !c.joined ? kOwn : (same ? kSame : kJoined));
            if (c.joined) {
                const TileBox b = tile_box(d.tp, j.tile);
                j.box = joined_box(u, b.dx, b.dy);
            }
        }
        ++rank;
        ++n;
    }
    // (j a constant after unrolling)
    __device__ __forceinline__ void take(const ScanDesc &d, int k, const Cell &c, int t0, int j,
                                         unsigned long long cost, unsigned long long p)
    {
        if (cost == 0 || p >= st.x1 || p + cost <= st.x0) return;
        const int words = st.own ? -1 : d.tp.tile_words, most = d.tp.job_size & ~31;
        const int all = c.joined ? pieces_of(c.count[0]) + pieces_of(c.count[1]) +
                                       pieces_of(c.count[2]) + pieces_of(c.count[3])
                                 : pieces_of(c.count[j]);
        const int s0 = st.x0 > p ? boundary_slot(cost, all, words, p, st.x0) : 0;
        const int s1 = st.x1 < p + cost ? boundary_slot(cost, all, words, p, st.x1) : 32 * all;
        for (int s = s0; s < s1; s += most) {
            const int e = min(s + most, s1);
            if (!c.joined) {
                put(d, k, c, t0, j, s, e, false);
                continue;
            }
            int off = 0;
            bool same = false;
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int len = 32 * pieces_of(c.count[u]);
                const int a = max(s - off, 0), z = min(e - off, len);
                if (a < z) put(d, k, c, t0, u, a, z, same);
                same = same || a < z;
                off += len;
            }
        }
    }
};

// The parts of a thread's cells i0 .. i1 - 1; before: of the first, by type.
template <bool kList>
__device__ __forceinline__ unsigned long long cell_parts(const ScanDesc *__restrict__ descs,
                                                         const int *s_first, int i0, int i1,
                                                         const Stretch &st,
                                                         const unsigned long long before[4],
                                                         unsigned long long rank,
                                                         unsigned long long j0, TilePart *list)
{
    PartTaker<kList> taker{st, rank, j0, list};
    unsigned long long p[4] = {before[0], before[1], before[2], before[3]};
    int k = 0;
    for (int i = i0; i < i1; ++i) {
        while (4 * i >= s_first[k + 1]) ++k;
        const ScanDesc &d = descs[k];
        const int t0 = i - s_first[k] / 4;
        const Cell c = cell_of(d, t0);
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const unsigned long long cost = st.own ? own_blocks(c.cost[j], d.tp.tile_words) : c.cost[j];
            taker.take(d, k, c, t0, j, cost, p[j]);
            p[j] += cost;
        }
    }
    return taker.n;
}

// Bucket i of the launch with its cell; visit(scan's number, scan, cell, its number, type).
template <class VisitT>
__device__ __forceinline__ void with_bucket(const ScanDesc *__restrict__ descs, const int *s_first,
                                            int i, VisitT visit)
{
    int k = 0;
    while (i >= s_first[k + 1]) ++k;
    const ScanDesc &d = descs[k];
    const int t = i - s_first[k], type = t / (2 * d.tp.ntiles), t0 = t - 2 * d.tp.ntiles * type;
    visit(k, d, cell_of(d, t0), t0, type);
}

__device__ __forceinline__ unsigned long long cost_of(const Cell &c, int type)
{
    const unsigned long long a = type & 1 ? c.cost[1] : c.cost[0], b = type & 1 ? c.cost[3] : c.cost[2];
    return type & 2 ? b : a;
}

}  // namespace

// The traversal: the buckets of all scans laid end to end by cost, one equal
// stretch per block (static: the costs are counted, not estimated, so the
// blocks end within a few per cent of each other, and a bucket is flushed once
// per block that has a part of it; a queue of four pieces per SM flushed twice
// as often and left the SMs 10 % apart).  Each part is walked into the block's
// shared-memory tile and flushed; then the blocks walk the fallback lists.
// smem_words: the dynamic shared memory of the launch, at least the
// largest tile of the scans.
template <int kThreads, class RowsT>
__global__ void __launch_bounds__(kThreads, 1) trace_tiles_kernel(
    const ScanDesc *__restrict__ descs, int nscans, int smem_words, const RowsT ra)
{
    constexpr bool kRows = RowsT::kRows, kCells = RowsT::kCells;
    constexpr int kVec = kRows ? kSliceWords / 4 : kLeanWords / 4;
    extern __shared__ __align__(16) uint32_t tile[];
    __shared__ unsigned s_next[2];  // the next slot; entries of the block's list of open rows
    __shared__ int s_first[kMaxBatch + 1];
    __shared__ TilePart s_parts[kPartList];
    __shared__ int s_group[kPartList + 1];  // first part of each group
    __shared__ int s_slots[kPartList];      // slots of each group
    __shared__ int s_ngroups;
    __shared__ unsigned long long s_warp[32];
    // each flush clears its box: the tile starts cleared once
    for (int w = threadIdx.x; w < smem_words >> 2; w += blockDim.x)
        reinterpret_cast<uint4 *>(tile)[w] = make_uint4(0u, 0u, 0u, 0u);
    after_previous();
    // buckets of scan k are the launch's buckets [s_first[k], s_first[k + 1])
    if (threadIdx.x == 0) {
        s_next[0] = s_next[1] = 0;
        int acc = 0;
        for (int k = 0; k < nscans; ++k) {
            s_first[k] = acc;
            acc += kGroups * descs[k].tp.ntiles;
        }
        s_first[nscans] = acc;
    }
    __syncthreads();
    const int nb = s_first[nscans];
    // the thread's buckets, or its cells (see cell_parts)
    constexpr bool kByBuckets = plan_by<RowsT>() == kByBucket;
    const int ni = kByBuckets ? nb : nb / 4, per = (ni + kThreads - 1) / kThreads;
    const int i0 = min(static_cast<int>(threadIdx.x) * per, ni), i1 = min(i0 + per, ni);
    // visit(scan, bucket within it, its cost and pairs)
    auto each = [&](auto visit) {
        int k = 0;
        for (int i = i0; i < i1; ++i) {
            while (i >= s_first[k + 1]) ++k;
            const ScanDesc &d = descs[k];
            const int t = i - s_first[k];
            const unsigned count = d.buckets.count[t];
            visit(k, t, bucket_cost<kRows>(count, d.buckets.events[t], d.tp.tile_words), count);
        }
    };
    Stretch st{};
    unsigned long long total, before[4];  // before: of a cell's types
    if constexpr (!kByBuckets) {
        unsigned long long mine[4];
        cell_sums<false>(descs, s_first, i0, i1, mine);
        scan_types<plan_by<RowsT>() == kByCells>(mine, reinterpret_cast<unsigned long long *>(s_parts),
                                                 before, total);
    } else {
        unsigned long long mine = 0;
        if constexpr (kCells) {
            if (i0 < i1)
                with_bucket(descs, s_first, i0,
                            [&](int, const ScanDesc &, const Cell &c, int, int type) {
                                mine = cost_of(c, type);
                            });
        } else {
            each([&](int, int, unsigned long long cost, unsigned) { mine += cost; });
        }
        st.before = block_excl_scan64(mine, s_warp, total);
    }
    // the block's stretch: an equal share, but worth about two flushes
    unsigned long long blocks = total / (2ull * flush_cost(descs[0].tp.tile_words)) + 1ull;
    unsigned long long share = 0;
    // a launch too small for that on every block: whole blocks for each bucket
    // instead, one for about two flushes' worth (a block of two small buckets
    // flushes twice, 11 000 cycles each)
    st.own = blocks < gridDim.x;  // the same in all blocks and threads
    if (st.own) {
        unsigned long long m = 0, all, b = 0, bs[4];
        if constexpr (!kByBuckets) {
            unsigned long long ms[4];
            cell_sums<true>(descs, s_first, i0, i1, ms);
            scan_types<plan_by<RowsT>() == kByCells>(ms, reinterpret_cast<unsigned long long *>(s_parts),
                                                     bs, all);
        } else if constexpr (kCells) {
            if (i0 < i1)
                with_bucket(descs, s_first, i0,
                            [&](int, const ScanDesc &d, const Cell &c, int, int type) {
                                m = own_blocks(cost_of(c, type), d.tp.tile_words);
                            });
            b = block_excl_scan64(m, s_warp, all);
        } else {
            each([&](int k, int, unsigned long long cost, unsigned) {
                m += own_blocks(cost, descs[k].tp.tile_words);
            });
            b = block_excl_scan64(m, s_warp, all);
        }
        st.own = all <= gridDim.x;
        if (st.own) {
            st.before = b;
            if constexpr (!kByBuckets)
                for (int j = 0; j < 4; ++j) before[j] = bs[j];
            share = 1ull;
        }
    }
    if (!st.own) {
        if (blocks > gridDim.x) blocks = gridDim.x;
        share = (total + blocks - 1ull) / blocks;
    }
    st.x0 = share * blockIdx.x;
    st.x1 = st.x0 + share;
    // the parts of the thread's buckets in that stretch, each at most job_size
    // pairs (in whole pieces): count, then list
    auto parts = [&](auto take) {
        unsigned long long p = st.before;
        each([&](int k, int t, unsigned long long cost, unsigned count) {
            const ScanDesc &d = descs[k];
            if (st.own) cost = own_blocks(cost, d.tp.tile_words);
            if (cost != 0 && p < st.x1 && p + cost > st.x0) {
                const int words = st.own ? -1 : d.tp.tile_words, all = pieces_of(count);
                const int s0 = st.x0 > p ? boundary_slot(cost, all, words, p, st.x0) : 0;
                const int s1 = st.x1 < p + cost ? boundary_slot(cost, all, words, p, st.x1) : 32 * all;
                const int most = d.tp.job_size & ~31;
                for (int s = s0; s < s1; s += most) take(k, t, static_cast<int>(count), s, min(s + most, s1));
            }
            p += cost;
        });
    };
    // the same of launches that join cells
    auto planned = [&](auto list, unsigned long long rank, unsigned long long j0) {
        constexpr bool kList = decltype(list)::value;
        if constexpr (!kByBuckets) {
            return cell_parts<kList>(descs, s_first, i0, i1, st, before, rank, j0, s_parts);
        } else {
            PartTaker<kList> taker{st, rank, j0, s_parts};
            if (i0 < i1)
                with_bucket(descs, s_first, i0,
                            [&](int k, const ScanDesc &d, const Cell &c, int t0, int type) {
                                unsigned long long cost = cost_of(c, type);
                                if (st.own) cost = own_blocks(cost, d.tp.tile_words);
#pragma unroll
                                for (int j = 0; j < 4; ++j)
                                    if (j == type) taker.take(d, k, c, t0, j, cost, st.before);
                            });
            return taker.n;
        }
    };
    unsigned long long nmine = 0, nparts, rank0 = 0;
    if constexpr (kCells) {
        // (the order of the parts does not matter: numbers from a counter, no scan)
        nmine = planned(std::false_type{}, 0, 0);
        if (nmine != 0) rank0 = atomicAdd(&s_next[0], static_cast<unsigned>(nmine));
        __syncthreads();
        nparts = s_next[0];
    } else {
        parts([&](int, int, int, int, int) { ++nmine; });
        rank0 = block_excl_scan64(nmine, s_warp, nparts);
    }
    for (unsigned long long j0 = 0; j0 < nparts; j0 += kPartList) {
        if (nmine != 0) {
            unsigned long long r = rank0;
            if constexpr (kCells) planned(std::true_type{}, r, j0);
            else
                parts([&](int k, int t, int count, int s0, int s1) {
                    if (r >= j0 && r < j0 + kPartList)
                        fill_part(s_parts[r - j0], descs[k], k, t, count, s0, s1, kOwn);
                    ++r;
                });
        }
        __syncthreads();
        if (threadIdx.x == 0) {
            const int here = static_cast<int>(nparts - j0 < kPartList ? nparts - j0 : kPartList);
            int g = 0, words = 0, slots = 0;
            s_group[0] = 0;
            for (int q = 0; q < here; ++q) {
                TilePart &j = s_parts[q];
                const int form = kCells ? j.form : kOwn;
                j.slot0 = slots;
                slots += j.end - j.start;
                if (form == kSame && q > 0) {
                    j.offset = s_parts[q - 1].offset;
                    continue;
                }
                // (the first part of a list begins a tile in any case)
                if (form == kSame) j.form = kJoined;
                if (q > s_group[g] && (words + j.words > smem_words ||
                                       (kCells && (form == kOwn) != (s_parts[q - 1].form == kOwn)))) {
                    s_slots[g] = j.slot0;
                    s_group[++g] = q;
                    slots -= j.slot0;
                    j.slot0 = words = 0;
                }
                j.offset = words;
                words += j.words;
            }
            s_slots[g] = slots;
            s_group[++g] = here;
            s_ngroups = g;
        }
        __syncthreads();
        const int ngroups = s_ngroups;
        NextWalk<kVec> nw{};
        first_walks(s_parts, s_group[1], s_slots[0], nw);
        for (int g = 0; g < ngroups; ++g) {
            const int q0 = s_group[g], q1 = s_group[g + 1];
            if (threadIdx.x == 0) s_next[0] = blockDim.x;
            __syncthreads();
            const TilePlan &tp0 = descs[s_parts[q0].scan].tp;
            bool joined = false;
            if constexpr (kCells) {
                joined = s_parts[q0].form != kOwn;
                if (joined) walk_joined(tile, s_parts + q0, q1 - q0, s_slots[g], tp0.refill, s_next, nw);
            }
            if constexpr (kRows)
                walk_parts(tile, s_parts + q0, q1 - q0, s_slots[g], tp0.refill, s_next, nw,
                           descs[s_parts[q0].scan], ra);
            else if (!joined)
                walk_parts(tile, tp0.thick, s_parts + q0, q1 - q0, s_slots[g], tp0.refill, s_next, nw);
            if (g + 1 < ngroups)
                first_walks(s_parts + q1, s_group[g + 2] - q1, s_slots[g + 1], nw);
            __syncthreads();
            if constexpr (kCells)
                if (joined) flush_joined(tile, s_parts + q0, q1 - q0, descs);
            for (int q = q0; q < q1 && !joined; ++q) {
                const TilePart &j = s_parts[q];
                const ScanDesc &d = descs[j.scan];
                const TilePlan &tp = d.tp;
                const TileBox b = tile_box(tp, j.tile);
                flush_tile<kRows>(tile + j.offset, b.dx, b.dy, b.dz, j.group >> 1, tp.thick,
                                  (j.group & 1) == 0 ? d.N : d.M, tp.nx, tp.ny, b.x0, b.y0, b.z0);
            }
        }
        __syncthreads();
    }
    if (kRows) {
        if (threadIdx.x == 0) descs[0].pairs.fb_count[blockIdx.x] = s_next[1];
    } else {
        walk_fallback_lists(descs, nscans);
    }
}

static_assert(sizeof(TilePart) <= 64, "the block's lists leave room for the largest tile");
static_assert(kPartList * sizeof(TilePart) >= 4 * 32 * sizeof(unsigned long long), "scan_types");

// Shared memory of a launch whose largest tile has this many words: room for
// up to eight tiles.
static int trace_smem_words(int tile_words)
{
    const int n = kTileSmemBytes / 4 / tile_words;
    return tile_words * (n < 1 ? 1 : (n > 8 ? 8 : n));
}

// Threads of the traversal of Euclidean thick rays: its row loop wants about 100
// registers; 1024 threads leave it 64 (head-sized grid, 2.7e6 histories, 2.5 mm,
// whole scan, in three chunks: 2.00 ms at 1024, 1.84 at 512, 2.23 at 256).
static constexpr int rows_threads(int threads) { return threads > 512 ? 512 : threads; }

template <int kThreads>
int occupancy_of(int smem_words)
{
    // allow the largest tile once, so launches (also inside graph capture)
    // need no attribute change
    if (cudaFuncSetAttribute(trace_tiles_kernel<kThreads, NoRows>,
                             cudaFuncAttributeMaxDynamicSharedMemorySize, kTileSmemBytes) !=
            cudaSuccess ||
        cudaFuncSetAttribute(trace_tiles_kernel<kThreads, Cells<kByBucket>>,
                             cudaFuncAttributeMaxDynamicSharedMemorySize, kTileSmemBytes) !=
            cudaSuccess ||
        cudaFuncSetAttribute(trace_tiles_kernel<kThreads, Cells<kByCell>>,
                             cudaFuncAttributeMaxDynamicSharedMemorySize, kTileSmemBytes) !=
            cudaSuccess ||
        cudaFuncSetAttribute(trace_tiles_kernel<kThreads, Cells<kByCells>>,
                             cudaFuncAttributeMaxDynamicSharedMemorySize, kTileSmemBytes) !=
            cudaSuccess ||
        cudaFuncSetAttribute(trace_tiles_kernel<rows_threads(kThreads), RowsArgs>,
                             cudaFuncAttributeMaxDynamicSharedMemorySize, kTileSmemBytes) !=
            cudaSuccess) {
        cudaGetLastError();
        return 0;
    }
    int nb = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, trace_tiles_kernel<kThreads, NoRows>,
                                                      kThreads, static_cast<size_t>(smem_words) * 4) !=
        cudaSuccess) {
        cudaGetLastError();
        return 0;
    }
    return nb;
}

int trace_tiles_occupancy(int tile_words, int threads)
{
    const int smem_words = trace_smem_words(tile_words);
    switch (threads) {
    case 256: return occupancy_of<256>(smem_words);
    case 512: return occupancy_of<512>(smem_words);
    case 768: return occupancy_of<768>(smem_words);
    case 1024: return occupancy_of<1024>(smem_words);
    default: return 0;
    }
}

template <class RowsT>
static cudaError_t launch_trace(const ScanDesc *descs, int nscans, int tile_words, int threads,
                                int grid, const RowsT &ra, cudaStream_t s)
{
    if (nscans < 1 || nscans > kMaxBatch || tile_words * 4 > kTileSmemBytes)
        return cudaErrorInvalidValue;
    const int smem_words = trace_smem_words(tile_words);
    const size_t smem = static_cast<size_t>(smem_words) * 4;
    switch (threads) {
    case 256:
        return launch_chained(trace_tiles_kernel<256, RowsT>, grid, 256, smem, s, descs, nscans,
                              smem_words, ra);
    case 512:
        return launch_chained(trace_tiles_kernel<512, RowsT>, grid, 512, smem, s, descs, nscans,
                              smem_words, ra);
    case 768:
        return launch_chained(trace_tiles_kernel<768, RowsT>, grid, 768, smem, s, descs, nscans,
                              smem_words, ra);
    case 1024:
        return launch_chained(trace_tiles_kernel<1024, RowsT>, grid, 1024, smem, s, descs, nscans,
                              smem_words, ra);
    default: return cudaErrorInvalidValue;
    }
}

cudaError_t launch_trace_tiles(const ScanDesc *descs, int nscans, int tile_words, int threads,
                               int grid, int buckets, int cells, cudaStream_t s)
{
    if (4 * cells >= 3 * grid) {
        if (buckets <= threads)
            return launch_trace(descs, nscans, tile_words, threads, grid, Cells<kByBucket>{}, s);
        if (buckets / 4 <= threads)
            return launch_trace(descs, nscans, tile_words, threads, grid, Cells<kByCell>{}, s);
        return launch_trace(descs, nscans, tile_words, threads, grid, Cells<kByCells>{}, s);
    }
    return launch_trace(descs, nscans, tile_words, threads, grid, NoRows{}, s);
}

cudaError_t launch_trace_rows(const ScanDesc *desc, int tile_words, int threads, int grid,
                              const RowsArgs &ra, cudaStream_t s)
{
    return launch_trace(desc, 1, tile_words, rows_threads(threads), grid, ra, s);
}

}  // namespace hd
