// Hull diagnostics: extra and missing voxels of a hull against the true
// object, per slice (the counts of Tables 1-2, Sec. 4), and the part of a
// mask that it encloses within each slice (applied to the literal MSC hull
// H_2 of Eq. 3.6, whose excluded voxels form a shell around the object, it
// keeps the region the shell encloses).
//
//   compare_kernel  blocks over pieces of a slice: sums of the two counts
//   fill_kernel     one block per slice: the mask and the exterior (mask
//                   voxels joined to the slice border) as bitmaps in shared
//                   memory, one row of words per voxel row; the exterior grows
//                   tile by tile (hd_grow.cuh)
#include <cuda_runtime.h>

#include "hd_grow.cuh"
#include "hd_internal.cuh"

namespace {

constexpr int kDiagThreads = 1024;
constexpr int kFillMaxWords = 24 * 1024;  // two bitmaps of 96 KB

constexpr int kCompareThreads = 256;
constexpr int kComparePiece = 16 * kCompareThreads;  // voxels of a block

// Nonzero bytes of h where o is zero, over four bytes.
__device__ __forceinline__ unsigned only(unsigned h, unsigned o)
{
    return static_cast<unsigned>(__popc(__vcmpne4(h, 0u) & __vcmpeq4(o, 0u))) >> 3;
}

// A block per piece of a slice, 16 voxels a thread (one 16-byte load of each
// volume where both slices allow it).  Latency-bound: a block per slice took 16 us
// on the head-sized volume, in 40 steps of one voxel.
__global__ void __launch_bounds__(kCompareThreads) compare_kernel(const uint8_t *hull,
                                                                  const uint8_t *object,
                                                                  int64_t plane, int nz,
                                                                  unsigned long long *counts)
{
    const int z = blockIdx.y;
    const uint8_t *h = hull + static_cast<int64_t>(z) * plane;
    const uint8_t *o = object + static_cast<int64_t>(z) * plane;
    const int64_t j0 = static_cast<int64_t>(blockIdx.x) * kComparePiece;
    unsigned extra = 0, missing = 0;
    const int64_t j = j0 + 16 * static_cast<int>(threadIdx.x);
    if (((reinterpret_cast<uintptr_t>(h) | reinterpret_cast<uintptr_t>(o)) & 15u) == 0 &&
        j0 + kComparePiece <= plane) {
        const uint4 a = *reinterpret_cast<const uint4 *>(h + j);
        const uint4 b = *reinterpret_cast<const uint4 *>(o + j);
        extra = only(a.x, b.x) + only(a.y, b.y) + only(a.z, b.z) + only(a.w, b.w);
        missing = only(b.x, a.x) + only(b.y, a.y) + only(b.z, a.z) + only(b.w, a.w);
    } else {
#pragma unroll
        for (int k = 0; k < 16; ++k) {
            const int64_t q = j0 + k * kCompareThreads + static_cast<int>(threadIdx.x);
            const bool hv = q < plane && h[q] != 0, ov = q < plane && o[q] != 0;
            extra += hv && !ov ? 1u : 0u;
            missing += ov && !hv ? 1u : 0u;
        }
    }
    extra = __reduce_add_sync(0xffffffffu, extra);
    missing = __reduce_add_sync(0xffffffffu, missing);
    __shared__ unsigned s_sum[2];
    if (threadIdx.x < 2) s_sum[threadIdx.x] = 0u;
    __syncthreads();
    if ((threadIdx.x & 31u) == 0) {
        atomicAdd(&s_sum[0], extra);
        atomicAdd(&s_sum[1], missing);
    }
    __syncthreads();
    if (threadIdx.x < 2 && s_sum[threadIdx.x] != 0u) {
        const unsigned long long c = s_sum[threadIdx.x];
        atomicAdd(counts + static_cast<int64_t>(threadIdx.x) * nz + z, c);
        atomicAdd(counts + 2 * static_cast<int64_t>(nz) + threadIdx.x, c);
    }
}

// Bitmaps: word (y, w) = y * rw + w holds voxels x = 32 w .. 32 w + 31 of
// row y (bit x & 31); bits past nx are 0 in the mask, so nothing grows there.
__global__ void __launch_bounds__(kDiagThreads) fill_kernel(const uint8_t *mask, int nx, int ny,
                                                            int rw, uint8_t *out)
{
    extern __shared__ uint32_t s_bits[];
    uint32_t *M = s_bits;
    uint32_t *E = s_bits + ny * rw;
    const int z = blockIdx.x;
    const int64_t plane = static_cast<int64_t>(nx) * ny;
    const uint8_t *m = mask + static_cast<int64_t>(z) * plane;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
    const int words = ny * rw;
    const hd::WordRows row_of(rw);
    // mask bits, a warp per word (coalesced bytes, one ballot)
    for (int k0 = warp; k0 < words; k0 += 8 * nwarps) {  // eight loads in flight
        uint8_t v[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const int k = k0 + i * nwarps, y = row_of(k), x = (k - y * rw) * 32 + lane;
            v[i] = k < words && x < nx ? m[static_cast<int64_t>(y) * nx + x] : 0;
        }
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const int k = k0 + i * nwarps;
            const uint32_t word = __ballot_sync(0xffffffffu, v[i] != 0);
            if (lane == 0 && k < words) M[k] = word;
        }
    }
    __syncthreads();
    // seeds: the mask voxels on the slice border
    for (int k = threadIdx.x; k < words; k += blockDim.x) {
        const int y = row_of(k), w = k - y * rw;
        uint32_t seed = 0;
        if (y == 0 || y == ny - 1) {
            seed = 0xffffffffu;
        } else {
            if (w == 0) seed |= 1u;
            if (w == (nx - 1) >> 5) seed |= 1u << ((nx - 1) & 31);
        }
        E[k] = seed & M[k];
    }
    __syncthreads();
    hd::grow_region<false>(M, E, rw, ny, plane);
    // enclosed = mask, not exterior
    uint8_t *o = out + static_cast<int64_t>(z) * plane;
    for (int k = warp; k < words; k += nwarps) {
        const int y = row_of(k), x = (k - y * rw) * 32 + lane;
        if (x < nx)
            o[static_cast<int64_t>(y) * nx + x] =
                static_cast<uint8_t>(((M[k] & ~E[k]) >> lane) & 1u);
    }
}

}  // namespace

extern "C" {

hd_status hd_hull_compare(const uint8_t *hull, const uint8_t *object, int32_t nx, int32_t ny,
                          int32_t nz, int64_t *counts, void *stream)
{
    if (!hull || !object || !counts || nx < 1 || ny < 1 || nz < 1) return HD_ERR_ARG;
    if (nz > 65535) return HD_ERR_RANGE;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    const int64_t plane = static_cast<int64_t>(nx) * ny;
    const int64_t pieces = (plane + kComparePiece - 1) / kComparePiece;
    if (pieces > 0x7fffffff) return HD_ERR_RANGE;
    cudaError_t e = cudaMemsetAsync(counts, 0, (2 * static_cast<size_t>(nz) + 2) * sizeof(int64_t), st);
    if (e == cudaSuccess) {
        compare_kernel<<<dim3(static_cast<unsigned>(pieces), static_cast<unsigned>(nz)), kCompareThreads,
                         0, st>>>(hull, object, plane, nz,
                                  reinterpret_cast<unsigned long long *>(counts));
        e = cudaGetLastError();
    }
    if (e != cudaSuccess) {
        hd::note_cuda_error(e, "hd_hull_compare");
        return HD_ERR_CUDA;
    }
    return HD_OK;
}

hd_status hd_fill_enclosed(const uint8_t *mask, int32_t nx, int32_t ny, int32_t nz, uint8_t *out,
                           void *stream)
{
    if (!mask || !out || nx < 1 || ny < 1 || nz < 1) return HD_ERR_ARG;
    if (nz > 65535) return HD_ERR_RANGE;
    const int rw = (nx + 31) / 32;
    const int64_t words = static_cast<int64_t>(rw) * ny;
    if (words > kFillMaxWords) return HD_ERR_RANGE;
    const size_t smem = 2 * sizeof(uint32_t) * static_cast<size_t>(words);
    cudaError_t e = cudaFuncSetAttribute(fill_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         static_cast<int>(2 * sizeof(uint32_t) * kFillMaxWords));
    if (e == cudaSuccess) {
        fill_kernel<<<nz, kDiagThreads, smem, static_cast<cudaStream_t>(stream)>>>(mask, nx, ny,
                                                                                   rw, out);
        e = cudaGetLastError();
    }
    if (e != cudaSuccess) {
        hd::note_cuda_error(e, "hd_fill_enclosed");
        return HD_ERR_CUDA;
    }
    return HD_OK;
}

}  // extern "C"
