// Internal definitions shared by the CUDA translation units of libhulld.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "../../include/hulld.h"

namespace hd {

constexpr int64_t kQ16 = 65536;
constexpr int kMaxN = 4096;
constexpr int kMaxTiles = 2048;       // tiles per group for the shared-memory path
constexpr int kGroups = 8;            // groups of records: class + 2 * walk type (hd_geom.cuh)
constexpr int kTileSmemBytes = 224 * 1024;  // shared memory per block for a private tile

// Gantry-rotation constants: theta[i] = round(atan(2^-i) * 180/pi * 2^30)
// (degrees, 30 fractional bits) and K = round(2^30 prod (1 + 2^-2i)^-1/2).
struct Cordic {
    long long theta[32];
    long long K;
};

// One axis of the map from world to grid coordinates: the voxel size s and the
// extent n s (mm * 2^16), floor(2^69 / s) + 1 in two words, and a multiple of s
// that makes every numerator positive, with its quotient.
struct GridDiv {
    int32_t ns;
    uint32_t mlo, mhi;
    uint32_t bias;
    long long off;
};

// Geometry in the fixed-point units the kernels use.
struct GeomQ {
    int32_t nx, ny, nz;
    int32_t pad;
    long long sx, sy, sz;  // voxel sizes, mm * 2^16
    long long T;           // tracker half-separation, mm * 2^16
    GridDiv dx, dy, dz;    // world to grid coordinates (to_grid in hd_geom.cuh)
};

// Device-side counters of one scan.  The block from n_global to the end is
// cleared before every chunk of histories.
struct Ctrl {
    unsigned long long n_in, n_miss, n_hit, n_none, n_reject;
    unsigned long long steps_miss, steps_hit;
    unsigned long long pairs_general;  // pairs sent to the fallback list (cumulative)
    unsigned long long runs;           // runs walked by the tiled pass (cumulative)
    unsigned int n_global;    // records listed for the global path (Records::glist)
    unsigned int n_pair_fallback;  // entries of the pair fallback list
    unsigned int fb_next;          // next fallback entry to hand out
};

// Traversal records of one chunk, one slot per history (slot = the
// history's index in the chunk): grid Q16 entry and exit points, int32 each
// (|G| < 2^30), and a status word (record_status in hd_geom.cuh: path 0 for
// a history without a record, 1 tiled, 2 global; its class; its slices).
// Structure of arrays; each array starts on a 16-byte boundary when the
// chunk's slot count is padded to a multiple of four (records_stride).
struct Records {
    int32_t *g[6];  // x0, y0, z0, x1, y1, z1
    int32_t *status;
    int32_t *glist;  // slots of the global-path records, Ctrl::n_global of them
                     // (null: that path finds them by their status words)
    int64_t cap;     // slots (the chunk's histories)
};

inline int64_t records_stride(int64_t n) { return (n + 3) & ~int64_t(3); }

// How a chunk of n histories is split among the ingest blocks; the scatter
// uses the same split, so that each of its blocks finds the pairs of the
// records one ingest block wrote.  Block b takes histories
// [b per_block, min((b + 1) per_block, n)); per_block is a multiple of 4.
constexpr int kIngestThreads = 256;
constexpr int kIngestBlocksPerSm = 8;
constexpr int kScatterBlocksPerSm = 2;  // resident
struct ChunkSplit {
    int blocks;
    int64_t per_block;
};
inline ChunkSplit chunk_split(int64_t n, int sm_count, int ntiles = 0)
{
    const int64_t units = (n + 3) / 4;  // groups of four histories
    // a block begins and ends with work per bucket: at least 1024 histories, and
    // one for every two buckets; beyond one wave of the scatter in whole waves
    int64_t least = kGroups * static_cast<int64_t>(ntiles) / 8;
    if (least < 256) least = 256;
    int64_t blocks = (units + least - 1) / least;
    const int64_t sms = sm_count > 0 ? sm_count : 1;
    const int64_t wave = sms * kScatterBlocksPerSm;
    if (blocks > wave) blocks -= blocks % wave;
    // but a small chunk is latency, and takes up to a wave of 256 histories each
    // (60 chunks of 5064 histories: 2577 us in blocks of 1024, 2144 of 512, 1817
    // of 256; fewer still exceed their pair budgets one by one)
    int64_t fine = (units + 63) / 64;
    if (fine > wave) fine = wave;
    if (blocks < fine) blocks = fine;
    const int64_t cap = sms * kIngestBlocksPerSm;
    if (blocks > cap) blocks = cap;
    if (blocks < 1) blocks = 1;
    ChunkSplit c;
    c.per_block = 4 * ((units + blocks - 1) / blocks);
    c.blocks = static_cast<int>((n + c.per_block - 1) / c.per_block);
    if (c.blocks < 1) c.blocks = 1;
    return c;
}

// Tiling of the grid into boxes whose counters fit in shared memory.
struct TilePlan {
    int nx, ny, nz;
    int tx, ty, tz;     // tile size in voxels
    int ntx, nty, ntz;  // tiles per axis
    int ntiles;         // tiles per group (0: tiled path off)
    int max_tiles;      // records touching more tiles take the global path
    int pairs_per_record;  // pair budget per history (pair_cap = this * slots)
    int job_size;       // most walks in a tile between two flushes
    long long pair_cap;
    int tile_words;     // 32-bit words of shared memory per block
    int refill;         // idle lanes that trigger a warp refill
    int threads;        // threads per block of the traversal (256, 512, 768, 1024)
    int thick;          // in-plane dilation of the walks, voxels (0: thin paths)
    unsigned mtx, mty, mtz;  // floor(2^32 / t) + 1 (0 when t = 1): division by a tile size
};

// (record, tile) pairs sorted by group and tile: the packed event walk of the
// record clipped to the tile, 32 bytes per pair (two uint4: one 32-byte
// sector; group and tile come from the part).  A pair whose walk has no lean form
// (a tie, a pending start, or a z crossing inside the tile) holds instead
// its tile-local endpoints, tile and class, marked empty for the lean pass,
// and its position goes to the fallback list; traversal blocks that run out
// of parts walk those with the general run walk in global memory.
struct Pairs {
    uint4 *v;   // 2 per pair
    uint2 *fb;  // fallback list: (pair position, 0), pair_cap entries
    // Each ingest block's pairs in the order its budget assigned them, from
    // the block's share (block * per_block * pairs_per_record) on: the
    // record's slot less the block's first slot, times kMaxRecordTiles,
    // plus the pair's tile index within the record.
    uint32_t *stage;
    // Euclidean thick rays use the same buffer with kSliceWords words per pair
    // in v, and fb as the lists of what their closed form leaves open, one per
    // traversal block: fb_count entries in each (the pair, the row in it), room
    // for fb_cap.
    uint32_t fb_cap;
    uint32_t *fb_count;
};
constexpr int kOpenLists = 2048;  // most blocks of that traversal

constexpr int kSliceWords = 12;

// Tiles a record may touch on the tiled path (its box of tiles; more take
// the global path), and the bits of a tile index within a record.
constexpr int kMaxRecordTiles = 32;
constexpr int kRecordTileBits = 5;
static_assert(kMaxRecordTiles == 1 << kRecordTileBits, "tile index bits");

// The buckets of a chunk: its pairs by group and tile (bucket group * ntiles +
// tile), kGroups ntiles of each.
struct Buckets {
    uint32_t *count;             // pairs
    uint32_t *first;             // the bucket's first pair
    unsigned long long *events;  // events of their walks (hd_geom.cuh)
};

// Everything the traversal kernel needs about one scan; a batch passes a
// table of these.
struct ScanDesc {
    TilePlan tp;
    Pairs pairs;
    Buckets buckets;
    Ctrl *ctrl;  // the scan's counters (added to) and fallback list (read)
    uint32_t *N, *M;
    // of a batch's entries: the item's records and the grid they are walked in
    Records rec;
    int32_t nx, ny, nz;
};

constexpr int kMaxBatch = 64;  // scans per batched traversal launch

// What the exact search of a row of Euclidean thick rays needs: the geometry,
// R = 2 q16(d_0), and the chunk's records (world endpoints, mm * 2^16).
struct RowsArgs {
    static constexpr bool kRows = true, kCells = false;
    GeomQ g;
    long long R;
    Records rec;
};

struct Inputs {
    const float *angle, *u_in, *v_in, *u_out, *v_out, *wepl;
};

// Kernels the calling thread has launched on the paths of scans and batches, which
// count theirs by the difference over a call (launch_chained counts itself).
inline int64_t &kernels_launched()
{
    static thread_local int64_t n = 0;
    return n;
}
inline void count_kernels(int n) { kernels_launched() += n; }

// Launch of a kernel that begins with after_previous(): its blocks may come onto
// the SMs, and do what needs none of the previous kernel's results, while that
// one ends (the chain of a small chunk is mostly launches, ends and starts).  Its
// parameters are not declared unaliased where the previous kernel may write what
// they point to: such a load could be moved above the wait.
template <class... P, class... A>
inline cudaError_t launch_chained(void (*kernel)(P...), dim3 grid, dim3 block, size_t smem,
                                  cudaStream_t s, const A &...args)
{
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t c{};
    c.gridDim = grid;
    c.blockDim = block;
    c.dynamicSmemBytes = smem;
    c.stream = s;
    c.attrs = &at;
    c.numAttrs = 1;
    count_kernels(1);
    return cudaLaunchKernelEx(&c, kernel, static_cast<P>(args)...);
}

#ifdef __CUDACC__
// Waits until the previous kernel of the stream has ended and its writes are
// visible; the next one may then be set up.  Every thread of a chained kernel
// calls it before it reads or writes memory.
__device__ __forceinline__ void after_previous()
{
    cudaGridDependencySynchronize();
    cudaTriggerProgrammaticLaunchCompletion();
}
#endif

// ---- launchers (stream-ordered; return the launch's cudaError_t) ----

// Begins a chunk: clears the scan's lists (Ctrl from n_global on) and the
// buckets' counts and events.
cudaError_t launch_chunk_begin(Ctrl *ctrl, const Buckets &buckets, int ntiles, cudaStream_t s);

// Classification, records and pair counts of a chunk.  Block b of the chunk
// split adds its pairs to bucket_count (cleared before) and receives in
// block_base[b kGroups ntiles + t] (null when tp.ntiles is 0) its first place in
// bucket t, where it has pairs there; block_pairs[b] is its pairs in all, listed
// in stage (Pairs::stage).  Each block keeps to a pair budget of
// tp.pairs_per_record per history; its records beyond it take the global
// path.  on_host: the inputs are page-locked host memory read in place.
cudaError_t launch_ingest(const Inputs &in, int64_t n, const GeomQ &g, const Cordic &cordic,
                          float tau_l, float tau_h, int use_miss, int use_hit, const TilePlan &tp,
                          const Records &rec, Ctrl *ctrl, uint32_t *bucket_count,
                          uint32_t *block_base, uint32_t *block_pairs, uint32_t *stage,
                          int on_host, int sm_count, cudaStream_t s);

// Counting sort of the (record, tile) pairs by bucket, with the walk set-up of
// each pair; block b of the chunk split takes the block_pairs[b] pairs that
// ingest block b listed and writes them from its places in the buckets on (the
// buckets' first pairs, an exclusive scan of their counts, are written here),
// adding their events.
cudaError_t launch_scatter(const TilePlan &tp, const Records &rec, int64_t n, Ctrl *ctrl,
                           const Buckets &buckets, const uint32_t *block_base,
                           const uint32_t *block_pairs, const Pairs &pairs, int sm_count,
                           cudaStream_t s);

// Traversal of the pairs of nscans scans (descs on the device) by `grid`
// resident blocks.  tile_words is the largest tile of the scans; threads is
// 256, 512, 768 or 1024; buckets: kGroups ntiles of all scans together; cells: a
// tile's buckets of one class, those of the classes that are counted and that may be
// joined (0: dilated walks, which never are, and chunks of too many histories).
cudaError_t launch_trace_tiles(const ScanDesc *descs, int nscans, int tile_words, int threads,
                               int grid, int buckets, int cells, cudaStream_t s);

// The same over the pairs of Euclidean thick rays of one scan (hd_euclid.cu).
cudaError_t launch_trace_rows(const ScanDesc *desc, int tile_words, int threads, int grid,
                              const RowsArgs &ra, cudaStream_t s);

// Global-memory traversal of the records whose path is 2; upper is the chunk's
// slot count.
cudaError_t launch_trace_global(const Records &rec, Ctrl *ctrl, int64_t upper, const GeomQ &g,
                                uint32_t *N, uint32_t *M, int sm_count, cudaStream_t s);

// The same for the chunks of nscans scans in one launch: most of them have no
// such record, and a launch each, on forked streams, cost a server's thread more
// than the work.  upper: the largest chunk's slots.
cudaError_t launch_trace_global_batch(const ScanDesc *descs, int nscans, int64_t upper,
                                      int sm_count, cudaStream_t s);

// Once per device, before the first launch there: the shared memory ingest and
// scatter may use for the most tiles a plan can have.
cudaError_t init_ingest();
cudaError_t init_scatter();

cudaError_t launch_classify(const float *wepl, int64_t n, float tau_l, float tau_h,
                            uint8_t *cls, cudaStream_t s);

// Blocks per SM the tiled traversal can keep resident with tiles of this many
// words and this many threads (0 when the launch is impossible).
int trace_tiles_occupancy(int tile_words, int threads);

struct DecideArgs {
    int32_t nx, ny, nz;
    int32_t methods;
    int32_t nt, nbhd, sm_ge, sm_per_slice;
    const uint32_t *N;       // null when neither SC nor MSC is on
    const uint32_t *M;       // null when SM is off
    unsigned long long *slice_key;  // nz entries (SM)
    uint32_t *mt, *slope;    // nz entries (SM)
    long long *index;        // nz entries (SM)
    uint8_t *H1, *H2, *H3;
};

// Whether a volume goes to the caller's memory on the device by a chained kernel
// (a copy of the copy engine's kind takes about 4 us more: the five of a small
// scan 78 -> 65 us of the whole, those of a batch of 12 scans 2379 -> 2261).  Up
// to 64 MB where the kernel can move 16 bytes at a time (at 20 to 80 MB a volume
// no difference), to 8 MB where it moves single ones (58 MB: 142 us, 25 by the
// engine).
inline bool copy_by_kernel(const void *dst, const void *src, size_t bytes)
{
    const uintptr_t a = reinterpret_cast<uintptr_t>(dst) | reinterpret_cast<uintptr_t>(src);
    return bytes <= (size_t((a & 15u) == 0 ? 64 : 8) << 20);
}

// A volume of an object of `device` to the caller's memory.
cudaError_t copy_out(void *dst, const void *src, size_t bytes, int32_t dst_on_device, int device,
                     int sm_count, cudaStream_t s);

// A new scan: N and M (V words each, either null) and the counters cleared.
cudaError_t launch_reset(uint32_t *N, uint32_t *M, int64_t V, Ctrl *ctrl, int sm_count, cudaStream_t s);

cudaError_t launch_finalize(const DecideArgs &a, int sm_count, cudaStream_t s);

// sum_v N(v) and sum_v M(v) (each 0 when its volume is null) into out[0],
// out[1]: by Eq. 3.4 and 3.9 these are the sums of |A_i| over the missed and
// the hit histories, the voxel memberships the statistics report.
cudaError_t launch_volume_sums(const uint32_t *N, const uint32_t *M, int64_t V,
                               unsigned long long *out, int sm_count, cudaStream_t s);

cudaError_t launch_pack_bits(const uint8_t *mask, int64_t V, uint32_t *bits, cudaStream_t s);

// Compaction: writes ascending indices of mask != 0 to out (if count fits
// capacity) and the total to *d_count.  `block_counts` holds
// ceil(V / 1024) + 1 uint32 of scratch.
cudaError_t launch_compact(const uint8_t *mask, int64_t V, int32_t *out, int64_t capacity,
                           uint32_t *block_counts, unsigned long long *d_count, cudaStream_t s);

// Shared host helpers of the C ABI (defined with the scan objects).
bool make_cordic_table(Cordic &c);
void note_cuda_error(cudaError_t e, const char *where);
hd_status check_geometry(const hd_geometry *g);

}  // namespace hd
