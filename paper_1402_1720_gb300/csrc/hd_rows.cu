// Rows of the hull-restricted system matrix: for each history, the voxels of
// its path A_i that lie inside a hull, in the order the path meets them.  The
// hull exists to shrink the unknowns of the reconstruction to these voxels
// (Sec. 1); the rows are what an iterative solver reads.
//
// Per chunk of histories one kernel sets every path's walk up (path_lean in
// hd_geom.cuh, 64 bytes each); the count pass and the emit pass (CSR offsets
// from an exclusive scan) walk from there, a lane per path, lanes refilled from
// the warp's share of consecutive histories.  Bound: integer issue of the run
// steps and the hull test.  Head-sized grid, 1.8e6 histories inside the MSC
// hull: 3.29 -> 1.64 ms, of it set-up 0.09, count 0.58, emit 0.88 (before, each
// pass set every path up again and walked it with the general run step, a warp
// waiting for its longest path).
#include "hd_geom.cuh"
#include "hd_rows.cuh"

namespace hd {

namespace {

// One block per SM, the hull in its shared memory.  The emit pass holds more of
// a path: at 1024 threads (64 registers) it spilled, and more rows open at a time
// left more sectors half written (1.39 ms; 768 threads 0.88, 512 threads 1.06).
constexpr int kRowsThreads = 1024;
constexpr int kEmitThreads = 768;
constexpr int kSetupThreads = 256;
constexpr int kRowsRefill = 8;      // idle lanes that take new paths
constexpr int kRunsPerStep = 4;     // runs between refill checks
constexpr int kRowsGrab = 64;       // paths a warp takes at a time
constexpr int kScanThreads = 1024;
constexpr int kScanPerThread = 4;
constexpr int kScanTile = kScanThreads * kScanPerThread;

// Grid endpoints of history i (false when rejected), with the gantry
// cos/sin of the last angle this thread saw kept for reuse.
struct RowsTrig {
    bool valid = false;
    float ang = 0.0f;
    long long c = 0, s = 0;
};

__device__ __forceinline__ bool row_endpoints(const Inputs &in, int64_t i, const GeomQ &g,
                                              const Cordic &cd, RowsTrig &tc, int32_t r[6])
{
    const float ang = in.angle[i];
    if (!(fabsf(ang) < 1048576.0f)) return false;
    if (!tc.valid || ang != tc.ang) {
        cordic_cs(q16_of(ang), cd, tc.c, tc.s);
        tc.ang = ang;
        tc.valid = true;
    }
    return endpoints_cs(g, tc.c, tc.s, in.u_in[i], in.v_in[i], in.u_out[i], in.v_out[i], r);
}

// The voxels of one run of a path inside the hull.  The hull is a bitmap (voxel
// v at bit v & 31 of word v >> 5, one word of padding), in shared memory when it
// fits there.  A run along x covers consecutive bits, counted by a population
// count and listed from the set bits of its words; a run along y has stride nx.
struct HullRuns {
    const uint32_t *bits;
    int nx;

    // up to 32 bits from voxel v on, the first `len` of them
    __device__ __forceinline__ uint32_t window(uint32_t v, int len) const
    {
        const uint32_t w = v >> 5;
        const uint32_t x = __funnelshift_r(bits[w], bits[w + 1], v & 31u);
        return len < 32 ? x & ((1u << len) - 1u) : x;
    }
    __device__ __forceinline__ bool test(uint32_t v) const { return (bits[v >> 5] >> (v & 31u)) & 1u; }

    __device__ __forceinline__ int count(bool ymaj, uint32_t vb, int a, int b) const
    {
        const int lo = min(a, b);
        int len = max(a, b) - lo + 1, c = 0;
        if (!ymaj) {
            uint32_t v = vb + static_cast<uint32_t>(lo);
            for (; len > 32; len -= 32, v += 32u) c += __popc(window(v, 32));
            return c + __popc(window(v, len));
        }
        uint32_t v = vb + static_cast<uint32_t>(nx) * static_cast<uint32_t>(lo);
        for (; len > 0; --len, v += static_cast<uint32_t>(nx)) c += test(v) ? 1 : 0;
        return c;
    }

    // writes the run's hull voxels to out in path order
    __device__ __forceinline__ int32_t *emit(bool ymaj, uint32_t vb, int a, int b, int32_t *out) const
    {
        const bool up = a <= b;
        int len = (up ? b - a : a - b) + 1;
        if (!ymaj) {
            if (up) {
                for (uint32_t v = vb + static_cast<uint32_t>(a); len > 0; len -= 32, v += 32u)
                    for (uint32_t x = window(v, min(len, 32)); x != 0; x &= x - 1u)
                        *out++ = static_cast<int32_t>(v + static_cast<uint32_t>(__ffs(x) - 1));
            } else {
                // windows from the high end down
                uint32_t end = vb + static_cast<uint32_t>(a) + 1u;
                for (; len > 0; len -= 32, end -= 32u) {
                    const int k = min(len, 32);
                    const uint32_t v = end - static_cast<uint32_t>(k);
                    for (uint32_t x = window(v, k); x != 0;) {
                        const int j = 31 - __clz(x);
                        *out++ = static_cast<int32_t>(v + static_cast<uint32_t>(j));
                        x ^= 1u << j;
                    }
                }
            }
            return out;
        }
        const uint32_t st = static_cast<uint32_t>(nx), step = up ? st : 0u - st;
        for (uint32_t v = vb + st * static_cast<uint32_t>(a); len > 0; --len, v += step)
            if (test(v)) *out++ = static_cast<int32_t>(v);
        return out;
    }
};

// What word 11 of a packed path holds above its flags: whether it is a path walk
// or, in words 0 .. 5, the endpoints of a path for the general run walk (else
// the history has no voxel).
constexpr uint32_t kPathLean = 16u, kPathGeneral = 32u;

__global__ void __launch_bounds__(kSetupThreads) rows_setup_kernel(Inputs in, int64_t n, GeomQ g,
                                                                   Cordic cd, uint4 *walks)
{
    RowsTrig tc;
    const int64_t stride = static_cast<int64_t>(gridDim.x) * blockDim.x;
    for (int64_t i = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x; i < n;
         i += stride) {
        int32_t r[6];
        uint32_t o[kPathWords];
#pragma unroll
        for (int k = 0; k < kPathWords; ++k) o[k] = 0u;
        if (row_endpoints(in, i, g, cd, tc, r)) {
            PathWalk L;
            const int k = path_lean(r, r + 3, g.nx, g.ny, g.nz, L);
            if (k > 0) {
                path_pack(L, o);
                o[11] |= kPathLean;
            } else if (k < 0) {
#pragma unroll
                for (int a = 0; a < 6; ++a) o[a] = static_cast<uint32_t>(r[a]);
                o[11] = kPathGeneral;
            }
        }
#pragma unroll
        for (int q = 0; q < kPathWords / 4; ++q)
            walks[(kPathWords / 4) * i + q] = make_uint4(o[4 * q], o[4 * q + 1], o[4 * q + 2], o[4 * q + 3]);
    }
}

// A path without the closed form, whole: its hull voxels counted, or written to
// out (when not null) in path order.
__device__ __noinline__ int general_row(const uint32_t *bits, const uint4 *path, int nx, int ny, int nz,
                                        int32_t *out)
{
    const HullRuns h{bits, nx};
    const uint4 p = path[0], q = path[1];
    const int32_t r[6] = {static_cast<int32_t>(p.x), static_cast<int32_t>(p.y),
                          static_cast<int32_t>(p.z), static_cast<int32_t>(p.w),
                          static_cast<int32_t>(q.x), static_cast<int32_t>(q.y)};
    RunWalk w;
    if (!run_begin(w, r, r + 3, nx, ny, nz)) return 0;
    const bool ymaj = (w.flags >> 5) & 1, up = w.flags & 1;
    int row, lo, hi, c = 0;
    while (run_next(w, row, lo, hi)) {
        const int z = ymaj ? row / nx : 0;
        const uint32_t vb = ymaj ? static_cast<uint32_t>(row - z * nx) +
                                       static_cast<uint32_t>(nx) * static_cast<uint32_t>(ny) *
                                           static_cast<uint32_t>(z)
                                 : static_cast<uint32_t>(nx) * static_cast<uint32_t>(row);
        const int a = up ? lo : hi, b = up ? hi : lo;
        if (out) out = h.emit(ymaj, vb, a, b, out);
        else c += h.count(ymaj, vb, a, b);
    }
    return c;
}

// Copies the packed hull into shared memory.
__device__ __forceinline__ void stage_hull(uint32_t *s_bits, const uint32_t *bits, int64_t words)
{
    for (int64_t w = threadIdx.x; w < words; w += blockDim.x) s_bits[w] = __ldg(bits + w);
    if (threadIdx.x == 0) s_bits[words] = 0u;
    __syncthreads();
}

// A warp's queue of paths: kRowsGrab consecutive ones at a time (their walks are
// alike) from a counter all warps share (walks of other angles take up to three
// times as long: with fixed shares half of the warps waited for the rest).
struct PathQueue {
    unsigned *counter;
    int n, next, end;
    // the path of each idle lane, in order (n: none left); the whole warp calls
    __device__ __forceinline__ int take(unsigned idle, bool mine)
    {
        const unsigned lane = threadIdx.x & 31u;
        if (next >= end) {
            unsigned b = 0;
            if (lane == 0) b = atomicAdd(counter, static_cast<unsigned>(kRowsGrab));
            b = __shfl_sync(0xffffffffu, b, 0);
            next = b < static_cast<unsigned>(n) ? static_cast<int>(b) : n;
            end = min(next + kRowsGrab, n);
        }
        const int i = next + __popc(idle & ((1u << lane) - 1u));
        next += __popc(idle);
        return mine && i < end ? i : n;
    }
    __device__ __forceinline__ bool empty() const { return next >= n; }
};

__device__ __forceinline__ void load_path(const uint4 *walks, int i, uint32_t o[kPathWords])
{
#pragma unroll
    for (int q = 0; q < kPathWords / 4; ++q) {
        const uint4 v = __ldg(walks + (kPathWords / 4) * static_cast<int64_t>(i) + q);
        o[4 * q] = v.x;
        o[4 * q + 1] = v.y;
        o[4 * q + 2] = v.z;
        o[4 * q + 3] = v.w;
    }
}

// path_z_first of the path at `path`, kc and kz of its crossings left: the order
// terms are read again, it is seldom asked.
__device__ __noinline__ bool z_first(const uint4 *path, int kc, int kz)
{
    const uint4 v[4] = {path[0], path[1], path[2], path[3]};
    const uint32_t o[kPathWords] = {v[0].x, v[0].y, v[0].z, v[0].w, v[1].x, v[1].y, v[1].z, v[1].w,
                                    v[2].x, v[2].y, v[2].z, v[2].w, v[3].x, v[3].y, v[3].z, v[3].w};
    PathWalk L;
    path_unpack(o, L);
    L.kc = kc;
    L.kz = kz;
    return path_z_first(L);
}

// The row lengths of a chunk, to row_ptr[i + 1]: a lane per path, run by run.
template <bool kShared>
__global__ void __launch_bounds__(kRowsThreads) rows_count_kernel(const uint4 *__restrict__ walks,
                                                                  int n, int nx, int ny, int nz,
                                                                  const uint32_t *hull_bits,
                                                                  int64_t words, unsigned *counter,
                                                                  int64_t *row_ptr)
{
    extern __shared__ uint32_t s_bits[];
    if (kShared) stage_hull(s_bits, hull_bits, words);
    const HullRuns h{kShared ? s_bits : hull_bits, nx};
    const int plane = nx * ny;
    PathQueue queue{counter, n, 0, 0};
    PathWalk L;
    bool active = false;
    int i = 0, c = 0;
    for (;;) {
        const unsigned idle = __ballot_sync(0xffffffffu, !active);
        if (queue.empty()) {
            if (idle == 0xffffffffu) break;
        } else if (__popc(idle) >= kRowsRefill) {
            const int k = queue.take(idle, !active);
            if (k < n) {
                i = k;
                uint32_t o[kPathWords];
                load_path(walks, i, o);
                c = 0;
                if (o[11] & kPathLean) {
                    path_unpack(o, L);
                    active = true;
                } else {
                    if (o[11] & kPathGeneral)
                        c = general_row(h.bits, walks + (kPathWords / 4) * static_cast<int64_t>(i), nx,
                                        ny, nz, nullptr);
                    row_ptr[i + 1] = c;
                }
            }
            continue;
        }
#pragma unroll 1
        for (int u = 0; u < kRunsPerStep; ++u) {
            if (active) {
                uint32_t vb;
                int a, b;
                active = path_run(L, nx, plane, vb, a, b);
                c += h.count((L.fl & 8) != 0, vb, a, b);
                if (!active) row_ptr[i + 1] = c;
            }
        }
    }
}

// The rows of a chunk, to cols from row_ptr[i] on: a lane per path, voxel by
// voxel (a run's hull voxels differ in number from lane to lane, a step of one
// voxel does not).  A lane's indices gather in its ring of shared memory and
// leave as whole 32-byte sectors: written one by one they reached DRAM 2.7 times
// over, as sectors evicted half full.
constexpr int kRing = 16;  // indices per lane: up to 7 waiting and 8 new ones

template <bool kShared>
__global__ void __launch_bounds__(kEmitThreads) rows_emit_kernel(const uint4 *__restrict__ walks,
                                                                 int n, int nx, int ny, int nz,
                                                                 const uint32_t *hull_bits,
                                                                 int64_t words, unsigned *counter,
                                                                 const int64_t *row_ptr, int32_t *cols)
{
    extern __shared__ uint32_t s_mem[];
    // the rings first (their size depends on the block alone), then the hull
    int32_t *const ring = reinterpret_cast<int32_t *>(s_mem) + threadIdx.x;  // stride blockDim.x
    const int rs = static_cast<int>(blockDim.x);
    uint32_t *const s_bits = s_mem + kRing * blockDim.x;
    if (kShared) stage_hull(s_bits, hull_bits, words);
    const HullRuns h{kShared ? s_bits : hull_bits, nx};
    PathQueue queue{counter, n, 0, 0};
    PathWalk L;
    bool active = false;
    uint32_t v = 0;
    uint32_t mst = 0, cst = 0, zst = 0;
    int jmin = 0;
    const uint4 *path = nullptr;
    // the 32-byte boundary at or before the row, and from there the next index
    // to find a place and the next to be written
    int32_t *out = nullptr;
    int at = 0, done = 0;
    for (;;) {
        const unsigned idle = __ballot_sync(0xffffffffu, !active);
        if (queue.empty()) {
            if (idle == 0xffffffffu) break;
        } else if (__popc(idle) >= kRowsRefill) {
            const int i = queue.take(idle, !active);
            if (i < n) {
                uint32_t o[kPathWords];
                load_path(walks, i, o);
                path = walks + (kPathWords / 4) * static_cast<int64_t>(i);
                out = cols + row_ptr[i];
                at = done = static_cast<int>((reinterpret_cast<uintptr_t>(out) >> 2) & 7u);
                if (o[11] & kPathLean) {
                    path_unpack(o, L);
                    active = true;
                    out -= done;
                    mst = (L.fl & 8) ? static_cast<uint32_t>(nx) : 1u;
                    v = L.vb + mst * static_cast<uint32_t>(L.im0);
                    cst = (L.fl & 8) ? 1u : static_cast<uint32_t>(nx);
                    zst = static_cast<uint32_t>(nx) * static_cast<uint32_t>(ny);
                    if (!(L.fl & 1)) mst = 0u - mst;
                    if (!(L.fl & 2)) cst = 0u - cst;
                    if (!(L.fl & 4)) zst = 0u - zst;
                    jmin = min(L.jn, L.jz);
                } else if (o[11] & kPathGeneral) {
                    general_row(h.bits, path, nx, ny, nz, out);
                }
            }
            continue;
        }
#pragma unroll 4
        for (int u = 0; u < 8; ++u) {
            if (active) {
                if (h.test(v)) {
                    ring[(at & (kRing - 1)) * rs] = static_cast<int32_t>(v);
                    ++at;
                }
                if (L.s != jmin) {
                    // the major axis crosses, or the walk ends
                    active = L.s != L.km;
                    ++L.s;
                    v += mst;
                } else if (L.jz > L.jn || (L.jz == L.jn && !z_first(path, L.kc, L.kz))) {
                    active = L.kc != 0;
                    --L.kc;
                    v += cst;
                    L.rem += L.Ru;
                    L.jn += L.Qu;
                    if (L.rem >= L.ad) {
                        L.rem -= L.ad;
                        ++L.jn;
                    }
                    jmin = min(L.jn, L.jz);
                } else {
                    active = L.kz != 0;
                    --L.kz;
                    v += zst;
                    L.remz += L.Ruz;
                    L.jz += L.Quz;
                    if (L.remz >= L.adz) {
                        L.remz -= L.adz;
                        ++L.jz;
                    }
                    jmin = min(L.jn, L.jz);
                }
            }
        }
        // whole sectors, and what is left of a finished row
        if ((at >> 3) > (done >> 3) || (!active && at > done)) {
            if ((done & 7) == 0 && at - done >= 8) {
                int32_t w[8];
#pragma unroll
                for (int k = 0; k < 8; ++k)
                    w[k] = ring[((done + k) & (kRing - 1)) * rs];
                int4 *const p = reinterpret_cast<int4 *>(out + done);
                p[0] = make_int4(w[0], w[1], w[2], w[3]);
                p[1] = make_int4(w[4], w[5], w[6], w[7]);
                done += 8;
            }
            const int to = active ? (at & ~7) : at;
            for (; done < to; ++done) out[done] = ring[(done & (kRing - 1)) * rs];
        }
    }
}

// Clears a chunk's two path counters; the first chunk also begins row_ptr.
__global__ void rows_first_kernel(unsigned *counters, int64_t *row_ptr)
{
    counters[0] = counters[1] = 0u;
    if (row_ptr != nullptr) row_ptr[0] = 0;
}

// Inclusive block scan of int64 values: `v` is this thread's value; returns
// its inclusive prefix, *total the block's sum.
__device__ __forceinline__ long long block_incl_scan64(long long v, long long *s_warp,
                                                       long long &total)
{
    const unsigned lane = threadIdx.x & 31u, warp = threadIdx.x >> 5;
    long long x = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const long long t = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= static_cast<unsigned>(o)) x += t;
    }
    if (lane == 31) s_warp[warp] = x;
    __syncthreads();
    if (warp == 0) {
        const int nw = blockDim.x >> 5;
        long long y = lane < static_cast<unsigned>(nw) ? s_warp[lane] : 0;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const long long t = __shfl_up_sync(0xffffffffu, y, o);
            if (lane >= static_cast<unsigned>(o)) y += t;
        }
        if (lane < static_cast<unsigned>(nw)) s_warp[lane] = y;
    }
    __syncthreads();
    total = s_warp[(blockDim.x >> 5) - 1];
    const long long before = warp > 0 ? s_warp[warp - 1] : 0;
    __syncthreads();
    return before + x;
}

// Tile b of kScanTile values: inclusive scan in place, its sum to sums[b].
__global__ void __launch_bounds__(kScanThreads) scan_tiles_kernel(int64_t *a, int64_t n,
                                                                  int64_t *sums)
{
    __shared__ long long s_warp[32];
    const int64_t base = static_cast<int64_t>(blockIdx.x) * kScanTile +
                         static_cast<int64_t>(threadIdx.x) * kScanPerThread;
    long long v[kScanPerThread];
    long long acc = 0;
#pragma unroll
    for (int k = 0; k < kScanPerThread; ++k) {
        v[k] = base + k < n ? a[base + k] : 0;
        acc += v[k];
        v[k] = acc;
    }
    long long total;
    const long long before = block_incl_scan64(acc, s_warp, total) - acc;
#pragma unroll
    for (int k = 0; k < kScanPerThread; ++k)
        if (base + k < n) a[base + k] = before + v[k];
    if (threadIdx.x == 0) sums[blockIdx.x] = total;
}

// One block: exclusive scan of the tile sums, kScanThreads at a time.
__global__ void __launch_bounds__(kScanThreads) scan_sums_kernel(int64_t *sums, int64_t nb)
{
    __shared__ long long s_warp[32];
    long long carry = 0;
    for (int64_t base = 0; base < nb; base += kScanThreads) {
        const int64_t i = base + threadIdx.x;
        const long long v = i < nb ? sums[i] : 0;
        long long total;
        const long long incl = block_incl_scan64(v, s_warp, total);
        if (i < nb) sums[i] = carry + incl - v;
        carry += total;
    }
}

__global__ void __launch_bounds__(kScanThreads) scan_add_kernel(int64_t *a, int64_t n,
                                                                const int64_t *offsets)
{
    const long long off = offsets[blockIdx.x];
    const int64_t base = static_cast<int64_t>(blockIdx.x) * kScanTile;
    for (int k = threadIdx.x; k < kScanTile; k += blockDim.x) {
        const int64_t i = base + k;
        if (i < n) a[i] += off;
    }
}

constexpr int kMaxSmem = 227 * 1024;
constexpr int64_t kMaxHullWords = 48 * 1024;  // 192 KB of shared memory

template <class K>
cudaError_t allow_smem(K kernel)
{
    return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kMaxSmem);
}

}  // namespace

int64_t rows_scan_scratch(int64_t n) { return (n + kScanTile - 1) / kScanTile; }

int64_t rows_hull_words(int64_t V) { return (V + 31) / 32; }

cudaError_t launch_rows_setup(const Inputs &in, int64_t n, const GeomQ &g, const Cordic &cd,
                              uint32_t *walks, int sm_count, cudaStream_t s)
{
    int64_t blocks = (n + kSetupThreads - 1) / kSetupThreads;
    const int64_t cap = static_cast<int64_t>(sm_count > 0 ? sm_count : 1) * 16;
    if (blocks > cap) blocks = cap;
    count_kernels(1);
    rows_setup_kernel<<<static_cast<unsigned>(blocks), kSetupThreads, 0, s>>>(
        in, n, g, cd, reinterpret_cast<uint4 *>(walks));
    return cudaGetLastError();
}

cudaError_t launch_rows_count(const uint32_t *walks, int64_t n, const GeomQ &g,
                              const uint32_t *hull_bits, unsigned *counters, int64_t *row_ptr,
                              bool first, int sm_count, cudaStream_t s)
{
    count_kernels(2);
    rows_first_kernel<<<1, 1, 0, s>>>(counters, first ? row_ptr : nullptr);
    const int64_t words = rows_hull_words(int64_t(g.nx) * g.ny * g.nz);
    const int sms = sm_count > 0 ? sm_count : 1;
    const uint4 *w = reinterpret_cast<const uint4 *>(walks);
    if (words < kMaxHullWords) {
        const cudaError_t e = allow_smem(rows_count_kernel<true>);
        if (e != cudaSuccess) return e;
        rows_count_kernel<true><<<sms, kRowsThreads, 4 * static_cast<size_t>(words + 1), s>>>(
            w, static_cast<int>(n), g.nx, g.ny, g.nz, hull_bits, words, counters, row_ptr);
    } else {
        rows_count_kernel<false><<<sms, kRowsThreads, 0, s>>>(
            w, static_cast<int>(n), g.nx, g.ny, g.nz, hull_bits, words, counters, row_ptr);
    }
    return cudaGetLastError();
}

cudaError_t launch_rows_scan(int64_t *a, int64_t n, int64_t *scratch, cudaStream_t s)
{
    if (n <= 0) return cudaSuccess;
    const int64_t nb = rows_scan_scratch(n);
    count_kernels(3);
    scan_tiles_kernel<<<static_cast<unsigned>(nb), kScanThreads, 0, s>>>(a, n, scratch);
    scan_sums_kernel<<<1, kScanThreads, 0, s>>>(scratch, nb);
    scan_add_kernel<<<static_cast<unsigned>(nb), kScanThreads, 0, s>>>(a, n, scratch);
    return cudaGetLastError();
}

cudaError_t launch_rows_emit(const uint32_t *walks, int64_t n, const GeomQ &g,
                             const uint32_t *hull_bits, unsigned *counters, const int64_t *row_ptr,
                             int32_t *cols, int sm_count, cudaStream_t s)
{
    const int64_t words = rows_hull_words(int64_t(g.nx) * g.ny * g.nz);
    const int sms = sm_count > 0 ? sm_count : 1;
    const uint4 *w = reinterpret_cast<const uint4 *>(walks);
    count_kernels(1);
    auto ring = [](int threads) { return sizeof(int32_t) * kRing * static_cast<size_t>(threads); };
    const size_t bits = 4 * static_cast<size_t>(words + 1);
    if (words < kMaxHullWords) {
        // fewer threads when the hull leaves no room for all their rings
        const int threads = bits + ring(kEmitThreads) <= kMaxSmem ? kEmitThreads : kEmitThreads / 2;
        const cudaError_t e = allow_smem(rows_emit_kernel<true>);
        if (e != cudaSuccess) return e;
        rows_emit_kernel<true><<<sms, threads, bits + ring(threads), s>>>(
            w, static_cast<int>(n), g.nx, g.ny, g.nz, hull_bits, words, counters + 1, row_ptr, cols);
    } else {
        const cudaError_t e = allow_smem(rows_emit_kernel<false>);
        if (e != cudaSuccess) return e;
        rows_emit_kernel<false><<<sms, kEmitThreads, ring(kEmitThreads), s>>>(
            w, static_cast<int>(n), g.nx, g.ny, g.nz, hull_bits, words, counters + 1, row_ptr, cols);
    }
    return cudaGetLastError();
}

}  // namespace hd
