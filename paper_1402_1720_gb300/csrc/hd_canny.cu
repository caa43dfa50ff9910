// SM threshold by edge detection: a documented form of the "modified Canny"
// picker the paper used for M_t (Sec. 4, which names the method but not its
// modification).  Per slice of M: binomial smoothing, Sobel derivatives, L1
// magnitude, non-maximum suppression (ties kept on the side of larger M),
// hysteresis at 1/2 and 1/5 of the slice's largest suppressed magnitude
// (8-connected), M_t = a quantile of M over the edge voxels, H_3 = [M >= M_t].
// All integer arithmetic.
//
//   canny_edges_kernel   block per tile of 32 x 32 voxels of a slice, from M to
//                        the suppressed magnitudes in shared memory (S = [1 2 1]^T
//                        [1 2 1] * M, its Sobel derivatives, the local maximum
//                        test), with the tile's largest
//   canny_slice_kernel   block per slice: the slice maximum, hysteresis on bitmaps in shared
//                        memory, the edge voxels' M listed in shared memory,
//                        the quantile by a radix select of four 8-bit steps
//   canny_hull_kernel    thread per voxel: the hull
//
// Latency-bound on volumes of tens of slices.  Head-sized volume: 255 -> 78 us
// (before, three passes over 64-bit volumes, and in the slice's block a step of
// the select per bit, a barrier per row of the hysteresis and the hull).
#include <cuda_runtime.h>

#include "hd_grow.cuh"
#include "hd_internal.cuh"

namespace {

constexpr int kVoxThreads = 256;
constexpr int kSliceThreads = 1024;
constexpr int kMaxWords = 24 * 1024;  // two slice bitmaps of 96 KB
constexpr int kListCap = 4096;        // edge values listed in shared memory

constexpr int kTile = 32;

struct CannyWs {
    long long *sup;   // suppressed magnitude of each voxel (0: not a local maximum)
    long long *tmax;  // the tiles' largest
};

__device__ __forceinline__ int clampi(int v, int lo, int hi) { return v < lo ? lo : (v > hi ? hi : v); }

__global__ void __launch_bounds__(kVoxThreads) canny_edges_kernel(const uint32_t *M, int nx, int ny,
                                                                  long long *sup, long long *tmax)
{
    // rings of 3, 2 and 1 voxels around the tile; outside the grid S and M are
    // read at the nearest voxel, and the magnitude is 0
    __shared__ uint32_t s_m[kTile + 6][kTile + 6];
    __shared__ long long s_s[kTile + 4][kTile + 4];
    __shared__ long long s_g[kTile + 2][kTile + 2];
    __shared__ uint8_t s_dir[kTile + 2][kTile + 2];
    __shared__ long long s_red[kVoxThreads / 32];
    const int x0 = blockIdx.x * kTile, y0 = blockIdx.y * kTile, z = blockIdx.z;
    const int64_t plane = static_cast<int64_t>(nx) * ny;
    const uint32_t *m = M + z * plane;
    for (int i = threadIdx.x; i < (kTile + 6) * (kTile + 6); i += kVoxThreads) {
        const int b = i / (kTile + 6), a = i - b * (kTile + 6);
        const int X = clampi(x0 + a - 3, 0, nx - 1), Y = clampi(y0 + b - 3, 0, ny - 1);
        s_m[b][a] = m[X + static_cast<int64_t>(nx) * Y];
    }
    __syncthreads();
    const int w[3] = {1, 2, 1};
    for (int i = threadIdx.x; i < (kTile + 4) * (kTile + 4); i += kVoxThreads) {
        const int b = i / (kTile + 4), a = i - b * (kTile + 4);
        long long acc = 0;
#pragma unroll
        for (int dy = 0; dy < 3; ++dy)
#pragma unroll
            for (int dx = 0; dx < 3; ++dx)
                acc += static_cast<long long>(w[dx] * w[dy]) * s_m[b + dy][a + dx];
        s_s[b][a] = acc;
    }
    __syncthreads();
    for (int i = threadIdx.x; i < (kTile + 2) * (kTile + 2); i += kVoxThreads) {
        const int b = i / (kTile + 2), a = i - b * (kTile + 2);
        const int x = x0 + a - 1, y = y0 + b - 1;
        long long g = 0;
        int dir = 0;
        if (x >= 0 && x < nx && y >= 0 && y < ny) {
            // S at the neighbours (clamped to the grid), in the array's indices
            const int xm = clampi(x - 1, 0, nx - 1) - x0 + 2, xp = clampi(x + 1, 0, nx - 1) - x0 + 2;
            const int ym = clampi(y - 1, 0, ny - 1) - y0 + 2, yp = clampi(y + 1, 0, ny - 1) - y0 + 2;
            long long gx = 0, gy = 0;
#pragma unroll
            for (int k = -1; k <= 1; ++k) {
                const int Yk = clampi(y + k, 0, ny - 1) - y0 + 2, Xk = clampi(x + k, 0, nx - 1) - x0 + 2;
                gx += w[k + 1] * (s_s[Yk][xp] - s_s[Yk][xm]);
                gy += w[k + 1] * (s_s[yp][Xk] - s_s[ym][Xk]);
            }
            const long long ax = gx < 0 ? -gx : gx, ay = gy < 0 ? -gy : gy;
            const int sx = gx > 0 ? 1 : -1, sy = gy > 0 ? 1 : -1;
            const int dx = 5 * ax < 2 * ay && !(5 * ay < 2 * ax) ? 0 : sx;
            const int dy = 5 * ay < 2 * ax ? 0 : sy;
            g = ax + ay;
            dir = (dx + 1) | ((dy + 1) << 2);
        }
        s_g[b][a] = g;
        s_dir[b][a] = static_cast<uint8_t>(dir);
    }
    __syncthreads();
    long long most = 0;
    for (int i = threadIdx.x; i < kTile * kTile; i += kVoxThreads) {
        const int b = i / kTile, a = i - b * kTile;
        const int x = x0 + a, y = y0 + b;
        if (x >= nx || y >= ny) continue;
        const int d = s_dir[b + 1][a + 1];
        const int dx = (d & 3) - 1, dy = (d >> 2) - 1;
        // along and against the gradient
        const long long fwd = s_g[b + 1 + dy][a + 1 + dx], bwd = s_g[b + 1 - dy][a + 1 - dx];
        const long long g = s_g[b + 1][a + 1];
        const long long v = g > 0 && g >= bwd && g > fwd ? g : 0;
        sup[z * plane + x + static_cast<int64_t>(nx) * y] = v;
        most = max(most, v);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) most = max(most, __shfl_xor_sync(0xffffffffu, most, o));
    if ((threadIdx.x & 31u) == 0) s_red[threadIdx.x >> 5] = most;
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int k = 1; k < kVoxThreads / 32; ++k) most = max(most, s_red[k]);
        tmax[blockIdx.x + gridDim.x * (blockIdx.y + static_cast<int64_t>(gridDim.y) * z)] = most;
    }
}

__device__ __forceinline__ long long block_max(long long v, long long *s_red)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = max(v, __shfl_xor_sync(0xffffffffu, v, o));
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (lane == 0) s_red[warp] = v;
    __syncthreads();
    long long t = 0;
    for (int k = 0; k < static_cast<int>(blockDim.x >> 5); ++k) t = max(t, s_red[k]);
    __syncthreads();
    return t;  // in every thread
}

__global__ void __launch_bounds__(kSliceThreads) canny_slice_kernel(
    const uint32_t *M, const long long *sup, const long long *tmax, int tiles, int nx, int ny, int rw,
    int q_pct, uint32_t *mt, uint8_t *has_edge)
{
    extern __shared__ uint32_t s_bits[];
    __shared__ long long s_red[32];
    uint32_t *W = s_bits;           // weak voxels
    uint32_t *E = s_bits + ny * rw;  // edge voxels found so far
    const int z = blockIdx.x;
    const int64_t plane = static_cast<int64_t>(nx) * ny;
    const uint32_t *m = M + z * plane;
    const long long *mg = sup + z * plane;
    // the slice's largest suppressed magnitude
    long long mloc = 0;
    for (int j = threadIdx.x; j < tiles; j += blockDim.x)
        mloc = max(mloc, tmax[static_cast<int64_t>(z) * tiles + j]);
    const long long mmax = block_max(mloc, s_red);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
    const int words = ny * rw;
    const hd::WordRows row_of(rw);
    for (int k0 = warp; k0 < words; k0 += 8 * nwarps) {  // a ballot per word, eight loads in flight
        long long a[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const int k = k0 + i * nwarps, y = row_of(k), x = (k - y * rw) * 32 + lane;
            a[i] = k < words && x < nx ? mg[static_cast<int64_t>(y) * nx + x] : 0;
        }
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const int k = k0 + i * nwarps;
            const uint32_t wb = __ballot_sync(0xffffffffu, a[i] > 0 && 5 * a[i] >= mmax);
            const uint32_t sb = __ballot_sync(0xffffffffu, a[i] > 0 && 2 * a[i] >= mmax);
            if (lane == 0 && k < words) {
                W[k] = wb;
                E[k] = sb;
            }
        }
    }
    __syncthreads();
    // hysteresis: the weak voxels joined to the strong ones, 8-connected
    hd::grow_region<true>(W, E, rw, ny, plane);
    // the edge voxels' M values, listed in shared memory when they fit
    __shared__ int s_n;
    uint32_t *L = s_bits + 2 * words;
    if (threadIdx.x == 0) s_n = 0;
    __syncthreads();
    for (int k = threadIdx.x; k < words; k += blockDim.x) {
        const int y = row_of(k), x0 = (k - y * rw) * 32;
        for (uint32_t bits = E[k]; bits != 0; bits &= bits - 1u) {
            const int slot = atomicAdd(&s_n, 1);
            if (slot < kListCap) L[slot] = m[static_cast<int64_t>(y) * nx + x0 + __ffs(bits) - 1];
        }
    }
    __syncthreads();
    const long long kedge = s_n;
    if (kedge == 0) {
        if (threadIdx.x == 0) {
            mt[z] = 0;
            has_edge[z] = 0;
        }
        return;
    }
    // the element of rank t among the edge voxels' M: radix select, the highest
    // byte first (over the list, or over the edge bitmap when it overflowed)
    const bool listed = kedge <= kListCap;
    long long t = (static_cast<long long>(q_pct) * (kedge - 1)) / 100;
    __shared__ int s_hist[256];
    __shared__ int s_digit, s_before;
    uint32_t prefix = 0;
    for (int b = 24; b >= 0; b -= 8) {
        const uint32_t above = b == 24 ? 0u : ~((1u << (b + 8)) - 1u);  // the bytes settled
        for (int i = threadIdx.x; i < 256; i += blockDim.x) s_hist[i] = 0;
        __syncthreads();
        if (listed) {
            // one update per value among a warp's: the high bytes are mostly alike
            for (int i0 = 32 * warp; i0 < kedge; i0 += 32 * nwarps) {
                const bool in = i0 + lane < kedge && (L[i0 + lane] & above) == prefix;
                const int d = in ? static_cast<int>((L[i0 + lane] >> b) & 255u) : 256;
                const unsigned same = __match_any_sync(0xffffffffu, d);
                if (in && lane == __ffs(same) - 1) atomicAdd(&s_hist[d], __popc(same));
            }
        } else {
            for (int k = threadIdx.x; k < words; k += blockDim.x) {
                const int y = row_of(k), x0 = (k - y * rw) * 32;
                for (uint32_t bits = E[k]; bits != 0; bits &= bits - 1u) {
                    const uint32_t v = m[static_cast<int64_t>(y) * nx + x0 + __ffs(bits) - 1];
                    if ((v & above) == prefix) atomicAdd(&s_hist[(v >> b) & 255u], 1);
                }
            }
        }
        __syncthreads();
        if (warp == 0) {  // the digit whose values hold rank t
            int c[8], sum = 0;
#pragma unroll
            for (int i = 0; i < 8; ++i) sum += c[i] = s_hist[8 * lane + i];
            int before = sum;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int u = __shfl_up_sync(0xffffffffu, before, o);
                if (lane >= o) before += u;
            }
            before -= sum;
            if (t >= before && t < before + sum) {  // one lane
                int i = 0;
                while (t >= before + c[i]) before += c[i++];
                s_digit = 8 * lane + i;
                s_before = before;
            }
        }
        __syncthreads();
        t -= s_before;
        prefix |= static_cast<uint32_t>(s_digit) << b;
    }
    if (threadIdx.x == 0) {
        mt[z] = prefix;
        has_edge[z] = 1;
    }
}

__global__ void __launch_bounds__(kVoxThreads) canny_hull_kernel(const uint32_t *M, int64_t plane,
                                                                 const uint32_t *mt,
                                                                 const uint8_t *has_edge,
                                                                 uint8_t *H3)
{
    const int z = blockIdx.y;
    const uint32_t t = mt[z];
    const bool edge = has_edge[z] != 0;
    const int64_t j0 = static_cast<int64_t>(blockIdx.x) * (4 * kVoxThreads) + threadIdx.x;
    const uint32_t *m = M + z * plane;
    uint8_t *h = H3 + z * plane;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const int64_t j = j0 + k * kVoxThreads;
        if (j < plane) h[j] = edge && m[j] >= t ? 1 : 0;
    }
}

size_t align256(size_t b) { return (b + 255) & ~size_t(255); }

// Two 64-bit words and two bytes per voxel, of which the suppressed magnitudes
// and the tiles' maxima (at most one per voxel) take the first and the second.
bool layout(int32_t nx, int32_t ny, int32_t nz, void *base, CannyWs *ws, size_t *bytes)
{
    const size_t V = static_cast<size_t>(nx) * ny * nz;
    const size_t a = align256(8 * V);
    if (bytes) *bytes = 2 * a + 2 * align256(V);
    if (ws && base) {
        char *p = static_cast<char *>(base);
        ws->sup = reinterpret_cast<long long *>(p);
        ws->tmax = reinterpret_cast<long long *>(p + a);
    }
    return true;
}

hd_status check_dims(int32_t nx, int32_t ny, int32_t nz)
{
    if (nx < 1 || ny < 1 || nz < 1) return HD_ERR_ARG;
    if (static_cast<int64_t>(nx) * ny * nz > (int64_t(1) << 31)) return HD_ERR_RANGE;
    if (static_cast<int64_t>((nx + 31) / 32) * ny > kMaxWords) return HD_ERR_RANGE;
    return HD_OK;
}

}  // namespace

extern "C" {

hd_status hd_sm_canny_workspace(int32_t nx, int32_t ny, int32_t nz, size_t *bytes)
{
    if (!bytes) return HD_ERR_ARG;
    const hd_status s = check_dims(nx, ny, nz);
    if (s != HD_OK) return s;
    layout(nx, ny, nz, nullptr, nullptr, bytes);
    return HD_OK;
}

hd_status hd_sm_canny(const uint32_t *M, int32_t nx, int32_t ny, int32_t nz, int32_t q_pct,
                      void *workspace, size_t workspace_bytes, uint32_t *mt, uint8_t *has_edge,
                      uint8_t *H3, void *stream)
{
    if (!M || !workspace || !mt || !has_edge || !H3) return HD_ERR_ARG;
    if (q_pct < 0 || q_pct > 100) return HD_ERR_ARG;
    const hd_status s = check_dims(nx, ny, nz);
    if (s != HD_OK) return s;
    size_t need = 0;
    CannyWs ws{};
    layout(nx, ny, nz, workspace, &ws, &need);
    if (workspace_bytes < need) return HD_ERR_ARG;
    if ((reinterpret_cast<uintptr_t>(workspace) & 255) != 0) return HD_ERR_ARG;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    const int rw = (nx + 31) / 32;
    const int64_t plane = static_cast<int64_t>(nx) * ny;
    cudaError_t e =
        cudaFuncSetAttribute(canny_slice_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             static_cast<int>(sizeof(uint32_t) * (2 * kMaxWords + kListCap)));
    const unsigned tx = static_cast<unsigned>((nx + kTile - 1) / kTile),
                   ty = static_cast<unsigned>((ny + kTile - 1) / kTile);
    // slices beyond a launch's third and second dimension in turns
    for (int z0 = 0; z0 < nz && e == cudaSuccess; z0 += 65535) {
        const unsigned zs = static_cast<unsigned>(nz - z0 < 65535 ? nz - z0 : 65535);
        const uint32_t *m = M + z0 * plane;
        long long *sup = ws.sup + z0 * plane;
        long long *tmax = ws.tmax + static_cast<int64_t>(z0) * tx * ty;
        canny_edges_kernel<<<dim3(tx, ty, zs), kVoxThreads, 0, st>>>(m, nx, ny, sup, tmax);
        canny_slice_kernel<<<zs, kSliceThreads, sizeof(uint32_t) * (2 * rw * ny + kListCap), st>>>(
            m, sup, tmax, static_cast<int>(tx * ty), nx, ny, rw, q_pct, mt + z0, has_edge + z0);
        canny_hull_kernel<<<dim3(static_cast<unsigned>((plane + 4 * kVoxThreads - 1) / (4 * kVoxThreads)), zs),
                            kVoxThreads, 0, st>>>(m, plane, mt + z0, has_edge + z0,
                                                  H3 + z0 * plane);
        e = cudaGetLastError();
    }
    if (e != cudaSuccess) {
        hd::note_cuda_error(e, "hd_sm_canny");
        return HD_ERR_CUDA;
    }
    return HD_OK;
}

}  // extern "C"
