// Binned SC: SC as the paper ran it (Sec. 2.2 data cuts; Sec. 3.2, its
// implementation paragraphs).  Histories are binned by gantry angle and by
// the mid-point displacement of their path; per bin, 3 sigma cuts on WEPL
// and both slopes; a bin whose kept histories average below the WEPL cutoff
// is missed and its line is carved in every slice it covers; the carved
// image is averaged over a window in each slice and thresholded.
//
// Stream-ordered kernels, all integer arithmetic.  Two passes over the
// histories, each in one of two forms:
//   binned_stats_tiles_kernel, binned_cut_tiles_kernel  a block per SM takes
//                        consecutive histories and keeps the bins of one gantry
//                        angle in shared memory (histories arrive angle by
//                        angle); the finished table goes out with one atomic per
//                        bin and word.  Sums of n, S and Q of 3 values; then the
//                        3 sigma test against bounds taken once per bin
//   binned_stats_kernel, binned_cut_kernel  one thread per history, 7 and 2
//                        64-bit atomics into its bin's row of the table: few
//                        histories, or an angle's bins beyond shared memory
// and the image:
//   binned_carve_kernel  one block per (angle bin, vertical bin): the lines of
//                        the block's missed bins walked run by run into a bitmap
//                        in shared memory, merged into the volume bitmap of each
//                        slice of the bin with one atomicAnd per changed word
//   binned_filter_kernel one thread per voxel: the window count of uncarved
//                        voxels, the hull byte and the carved byte
#include <cmath>
#include <new>

#include "hd_geom.cuh"

namespace hd {

struct BinQ {
    int n_ang, n_u, n_v, k;
    long long ang_q, u_q, v_q, u_lo_q, v_lo_q;  // Q16 degrees and mm
    long long miss_q8;                          // 1/256 mm
    float r_ang, r_u, r_v;                      // rcp_int of twice the bin sizes
    int w, min_count;
};

// Slices z0 .. z1 - 1 share the lines of vertical bin iv; count: the bin's
// statistics are counted with this group (the first of its bin).
struct SliceGroup {
    int iv, z0, z1, count;
};

namespace {

constexpr int kBinThreads = 256;
constexpr int kPassBlocksPerSm = 6;  // resident blocks of the per-history passes (40 registers)
constexpr int kCarveThreads = 192;
constexpr int kAccWords = 9;
constexpr int kCtrWords = 8;
constexpr int kMaxSmemWords = 48 * 1024;  // slice bitmaps up to 192 KB in shared memory
constexpr long long kFull = 360LL * 65536;

__device__ __forceinline__ int q8_of(float x) { return __float2int_rn(x * 256.0f); }

// floor(a / b) for |a| < 2^30, 0 < b < 2^30 and |a / b| < 2^18, rb = rcp_int(b):
// the float quotient is within one of it.
__device__ __forceinline__ int bin_div(int a, int b, float rb)
{
    int q = __float2int_rd(static_cast<float>(a) * rb);
    const int r = a - q * b;
    if (r < 0) --q;
    if (r >= b) ++q;
    return q;
}

struct BinAt {
    int ia, iu, iv;
    int x[3];  // WEPL (|.| <= 2^18), lateral and vertical slope (< 2^18) in 1/256 mm
};

// Angle bin of an angle with |ang| < 2^20.
__device__ __forceinline__ int angle_bin(const BinQ &b, float ang)
{
    int a;
    if (ang >= 0.0f && ang < 360.0f) {
        a = __float2int_rn(ang * 65536.0f);
        if (a == static_cast<int>(kFull)) a = 0;
    } else {
        const long long t = q16_of(ang);  // |t| < 2^36: a small quotient
        a = static_cast<int>(t - floordiv_small(t, kFull) * kFull);
    }
    const int q = static_cast<int>(b.ang_q);
    const int ia = bin_div(2 * a + q, 2 * q, b.r_ang);  // nearest centre
    return ia == b.n_ang ? 0 : ia;
}

// Bin of one history; false when it is not binned.  All in 32 bits: u and v in
// Q16 stay below 2^28, twice a bin size and twice a lower edge below 2^29.
__device__ __forceinline__ bool bin_of(const BinQ &b, float ang, float ui, float vi, float uo,
                                       float vo, float wepl, BinAt &o)
{
    if (!(fabsf(ang) < 1048576.0f) || !(fabsf(wepl) < 1024.0f)) return false;
    if (!(fabsf(ui) < 4096.0f) || !(fabsf(vi) < 4096.0f) || !(fabsf(uo) < 4096.0f) ||
        !(fabsf(vo) < 4096.0f))
        return false;
    o.x[0] = q8_of(wepl);
    o.x[1] = q8_of(uo) - q8_of(ui);
    o.x[2] = q8_of(vo) - q8_of(vi);
    if (abs(o.x[1]) >= 1024 * 256 || abs(o.x[2]) >= 1024 * 256) return false;
    o.ia = angle_bin(b, ang);
    const int u2 = q16_small(ui) + q16_small(uo) - 2 * static_cast<int>(b.u_lo_q);
    const int v2 = q16_small(vi) + q16_small(vo) - 2 * static_cast<int>(b.v_lo_q);
    o.iu = bin_div(u2, 2 * static_cast<int>(b.u_q), b.r_u);
    o.iv = bin_div(v2, 2 * static_cast<int>(b.v_q), b.r_v);
    return o.iu >= 0 && o.iu < b.n_u && o.iv >= 0 && o.iv < b.n_v;
}

__device__ __forceinline__ long long row_of(const BinQ &b, const BinAt &o)
{
    return o.ia + static_cast<long long>(b.n_ang) * (o.iu + static_cast<long long>(b.n_u) * o.iv);
}

// x within k population standard deviations of a bin holding n values of
// sum S and sum of squares Q: (n x - S)^2 <= k^2 (n Q - S^2).
__device__ __forceinline__ bool within(long long n, long long S, long long Q, long long x, int k)
{
    const __int128 d = static_cast<__int128>(n) * x - S;
    const __int128 var_n2 = static_cast<__int128>(n) * Q - static_cast<__int128>(S) * S;
    return d * d <= static_cast<__int128>(k * k) * var_n2;
}

__device__ __forceinline__ bool bin_missed(const unsigned long long *a, long long miss_q8)
{
    const long long kn = static_cast<long long>(a[7]);
    const long long ks = static_cast<long long>(a[8]);
    return kn > 0 && ks < miss_q8 * kn;
}

__device__ __forceinline__ void warp_add(unsigned long long v, unsigned long long *dst)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if ((threadIdx.x & 31) == 0 && v != 0) atomicAdd(dst, v);
}

__device__ __forceinline__ unsigned long long u64_of(int x)
{
    return static_cast<unsigned long long>(static_cast<long long>(x));
}

// The six sums of one history into its bin's row.
__device__ __forceinline__ void add_sums(unsigned long long *a, const int x[3])
{
#pragma unroll
    for (int q = 0; q < 3; ++q) {
        atomicAdd(a + 1 + q, u64_of(x[q]));
        atomicAdd(a + 4 + q, static_cast<unsigned long long>(static_cast<long long>(x[q]) * x[q]));
    }
}

// The 3 sigma test of one history against its bin's finished statistics
// (words 0-6, while other threads add to words 7 and 8).
__device__ __forceinline__ bool keep_of(const BinQ &b, const unsigned long long *a, const int x[3])
{
    const long long cnt = static_cast<long long>(a[0]);
    bool keep = true;
#pragma unroll
    for (int q = 0; q < 3; ++q)
        keep = keep && within(cnt, static_cast<long long>(a[1 + q]),
                              static_cast<long long>(a[4 + q]), x[q], b.k);
    return keep;
}

// Clears 64-bit words: the bin table (16 bytes a thread and step: cudaMalloc's
// alignment) and the counters.
__global__ void __launch_bounds__(512) binned_clear_kernel(unsigned long long *acc, int64_t words,
                                                           unsigned long long *ctr)
{
    after_previous();
    const int64_t i0 = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
    const int64_t stride = static_cast<int64_t>(gridDim.x) * blockDim.x;
    for (int64_t i = i0; i < words / 2; i += stride)
        reinterpret_cast<uint4 *>(acc)[i] = make_uint4(0u, 0u, 0u, 0u);
    if (i0 == 0 && (words & 1)) acc[words - 1] = 0ull;
    if (i0 < kCtrWords) ctr[i0] = 0ull;
}

// Begins the image: nothing carved, its four counters cleared.
__global__ void __launch_bounds__(512) binned_image_kernel(uint32_t *bits, int64_t words,
                                                           unsigned long long *ctr)
{
    after_previous();
    const int64_t i0 = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
    for (int64_t i = i0; i < words; i += static_cast<int64_t>(gridDim.x) * blockDim.x)
        bits[i] = 0xffffffffu;
    if (i0 < 4) ctr[2 + i0] = 0ull;
}

// Histories i, i + stride, .. below end without a table, those of vertical bins
// v0 .. v1 - 1: seven and two atomics each.  kAtOnce of them are in flight.  (Plain
// loads here and below: these kernels come right behind the caller's work, which
// may still write the histories while they start.)
template <int kAtOnce>
__device__ __forceinline__ void load_histories(const Inputs &in, int64_t i, int64_t end,
                                               int64_t stride, float h[kAtOnce][6])
{
#pragma unroll
    for (int k = 0; k < kAtOnce; ++k) {
        const int64_t j = i + k * stride;
        h[k][0] = 2097152.0f;  // not binned
        if (j < end) {
            h[k][0] = in.angle[j];
            h[k][1] = in.u_in[j];
            h[k][2] = in.v_in[j];
            h[k][3] = in.u_out[j];
            h[k][4] = in.v_out[j];
            h[k][5] = in.wepl[j];
        }
    }
}

template <int kAtOnce>
__device__ __forceinline__ unsigned stats_direct(const Inputs &in, int64_t i, int64_t end,
                                                 int64_t stride, const BinQ &b, int v0, int v1,
                                                 unsigned long long *acc)
{
    unsigned binned = 0;
    for (; i < end; i += kAtOnce * stride) {
        float h[kAtOnce][6];
        load_histories<kAtOnce>(in, i, end, stride, h);
#pragma unroll
        for (int k = 0; k < kAtOnce; ++k) {
            BinAt o;
            if (!bin_of(b, h[k][0], h[k][1], h[k][2], h[k][3], h[k][4], h[k][5], o)) continue;
            if (o.iv < v0 || o.iv >= v1) continue;
            unsigned long long *a = acc + kAccWords * row_of(b, o);
            atomicAdd(a, 1ull);
            add_sums(a, o.x);
            ++binned;
        }
    }
    return binned;
}

template <int kAtOnce>
__device__ __forceinline__ unsigned cut_direct(const Inputs &in, int64_t i, int64_t end,
                                               int64_t stride, const BinQ &b, int v0, int v1,
                                               unsigned long long *acc)
{
    unsigned cut = 0;
    for (; i < end; i += kAtOnce * stride) {
        float h[kAtOnce][6];
        load_histories<kAtOnce>(in, i, end, stride, h);
        unsigned long long *a[kAtOnce];
        unsigned long long w[kAtOnce][7];
        int x[kAtOnce][3];
#pragma unroll
        for (int k = 0; k < kAtOnce; ++k) {
            BinAt o;
            a[k] = nullptr;
            if (!bin_of(b, h[k][0], h[k][1], h[k][2], h[k][3], h[k][4], h[k][5], o)) continue;
            if (o.iv < v0 || o.iv >= v1) continue;
            a[k] = acc + kAccWords * row_of(b, o);
#pragma unroll
            for (int f = 0; f < 7; ++f) w[k][f] = a[k][f];
#pragma unroll
            for (int q = 0; q < 3; ++q) x[k][q] = o.x[q];
        }
#pragma unroll
        for (int k = 0; k < kAtOnce; ++k) {
            if (a[k] == nullptr) continue;
            if (!keep_of(b, w[k], x[k])) {
                ++cut;
                continue;
            }
            atomicAdd(a[k] + 7, 1ull);
            atomicAdd(a[k] + 8, u64_of(x[k][0]));
        }
    }
    return cut;
}

__global__ void __launch_bounds__(kBinThreads, kPassBlocksPerSm) binned_stats_kernel(
    Inputs in, int64_t n, BinQ b, unsigned long long *acc, unsigned long long *ctr)
{
    after_previous();
    const int64_t i = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
    warp_add(stats_direct<1>(in, i, n, static_cast<int64_t>(gridDim.x) * blockDim.x, b, 0, b.n_v, acc),
             ctr + 0);
}

__global__ void __launch_bounds__(kBinThreads, kPassBlocksPerSm) binned_cut_kernel(
    Inputs in, int64_t n, BinQ b, unsigned long long *acc, unsigned long long *ctr)
{
    after_previous();
    const int64_t i = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
    warp_add(cut_direct<1>(in, i, n, static_cast<int64_t>(gridDim.x) * blockDim.x, b, 0, b.n_v, acc),
             ctr + 1);
}

// ---- the passes with an angle's bins in shared memory ----
//
// Bound: shared-memory atomics (ten per history, random banks) and integer issue.
// Head grid, 9e6 histories: statistics 365 -> 97 us, cuts 250 -> 112 us (7 and 2
// 64-bit atomics per history in L2 before, and 128-bit tests for each).

constexpr int kTileThreads = 768;   // one block per SM
constexpr int kTileUnroll = 2;      // histories per thread and chunk, the next chunk's in flight
constexpr int kTileChunk = kTileThreads * kTileUnroll;
constexpr int kStatsWords = 10;     // n, S x 3, Q low 18 bits x 3, Q high x 3
constexpr int kCutWords = 8;        // bounds x 6, kept n, kept sum
constexpr int kTileBytes = 224000;  // of the 227 KB a block can have
// Sums of one flush's histories per bin: beyond this many in a bin the rest of
// its values go straight to the table.  2^18 times it stays below 2^31.
constexpr unsigned kTileCount = 8191;
constexpr int kMaxWindows = 4;
// Histories per bin of an angle and block that pay for a table (head grid, 4544
// bins an angle: at 1.1 million histories in all 245 us with it, 228 without; at
// 1.8 million 265 and 279).
constexpr int kTileFill = 2;

// The window of vertical bins a block keeps (n_v split into n_win windows of
// rows bins each, a block per window and segment of histories).
struct BinTiles {
    int n_win, rows;
};

// Chunks of kTileThreads * kTileUnroll consecutive histories; the table holds
// the angle bin of a chunk's first history, and a chunk that begins with another
// angle changes it.  Where angles come in no order a table buys nothing: chunks
// whose first, middle and last history lie in three angles change nothing, and a
// block that meets many of them hands its histories to the direct loop.
struct TileAngle {
    int cur = -1, stray = 0, chunks = 0;
    // next: the angle to change to; s: the three histories' angles
    __device__ __forceinline__ bool due(const BinQ &b, const float s[3], int &next)
    {
        ++chunks;
        next = fabsf(s[0]) < 1048576.0f ? angle_bin(b, s[0]) : cur;
        if (next == cur) return false;
        if (s[0] != s[1] && s[1] != s[2]) {
            ++stray;
            return false;
        }
        return true;
    }
    __device__ __forceinline__ bool lost() const { return stray > 2 + chunks / 4; }
};

// Columns of this thread's histories of the chunk at c0; past i1 an angle that is
// not binned.
__device__ __forceinline__ void load_chunk(const Inputs &in, int64_t c0, int64_t i1,
                                           float h[kTileUnroll][6], float s[3])
{
    if (c0 >= i1) return;
    s[0] = in.angle[c0];
    s[1] = in.angle[min(c0 + kTileChunk / 2, i1 - 1)];
    s[2] = in.angle[min(c0 + kTileChunk, i1) - 1];
    load_histories<kTileUnroll>(in, c0 + threadIdx.x, i1, kTileThreads, h);
}

__global__ void __launch_bounds__(kTileThreads) binned_stats_tiles_kernel(Inputs in, int64_t n,
                                                                          BinQ b, BinTiles t,
                                                                          unsigned long long *acc,
                                                                          unsigned long long *ctr)
{
    extern __shared__ uint32_t s_tab[];  // word f of bin e at f * E + e
    const int win = blockIdx.x % t.n_win, seg = blockIdx.x / t.n_win, n_seg = gridDim.x / t.n_win;
    const int64_t i0 = n * seg / n_seg, i1 = n * (seg + 1) / n_seg;
    const int v0 = win * t.rows, v1 = min(b.n_v, v0 + t.rows);
    const int E = b.n_u * (v1 - v0);
    for (int e = threadIdx.x; e < kStatsWords * E; e += kTileThreads) s_tab[e] = 0u;
    after_previous();
    unsigned long long binned = 0;
    TileAngle ang;
    auto flush = [&]() {
        __syncthreads();
        if (ang.cur >= 0) {
            for (int e = threadIdx.x; e < E; e += kTileThreads) {
                const uint32_t c = s_tab[e];
                if (c == 0u) continue;
                unsigned long long *a =
                    acc + kAccWords * (ang.cur + static_cast<long long>(b.n_ang) *
                                                     (e + static_cast<long long>(b.n_u) * v0));
                atomicAdd(a, static_cast<unsigned long long>(c));
                s_tab[e] = 0u;
#pragma unroll
                for (int q = 0; q < 3; ++q) {
                    uint32_t *const S = s_tab + (1 + q) * E + e, *const L = S + 3 * E,
                                   *const H = S + 6 * E;
                    atomicAdd(a + 1 + q, u64_of(static_cast<int>(*S)));
                    atomicAdd(a + 4 + q, (static_cast<unsigned long long>(*H) << 18) + *L);
                    *S = *L = *H = 0u;
                }
            }
        }
        __syncthreads();
    };
    float ahead[kTileUnroll][6] = {}, sample[3] = {};
    load_chunk(in, i0, i1, ahead, sample);
    int64_t c0 = i0;
    for (; c0 < i1 && !ang.lost(); c0 += kTileChunk) {
        int next;
        if (ang.due(b, sample, next)) {
            flush();
            ang.cur = next;
        }
        float h[kTileUnroll][6];
#pragma unroll
        for (int k = 0; k < kTileUnroll; ++k)
#pragma unroll
            for (int f = 0; f < 6; ++f) h[k][f] = ahead[k][f];
        load_chunk(in, c0 + kTileChunk, i1, ahead, sample);
#pragma unroll
        for (int k = 0; k < kTileUnroll; ++k) {
            BinAt o;
            if (!bin_of(b, h[k][0], h[k][1], h[k][2], h[k][3], h[k][4], h[k][5], o)) continue;
            if (o.iv < v0 || o.iv >= v1) continue;
            ++binned;
            if (o.ia != ang.cur) {
                unsigned long long *a = acc + kAccWords * row_of(b, o);
                atomicAdd(a, 1ull);
                add_sums(a, o.x);
                continue;
            }
            const int e = o.iu + b.n_u * (o.iv - v0);
            if (atomicAdd(s_tab + e, 1u) >= kTileCount) {
                add_sums(acc + kAccWords * row_of(b, o), o.x);
                continue;
            }
#pragma unroll
            for (int q = 0; q < 3; ++q) {
                uint32_t *const S = s_tab + (1 + q) * E + e;
                atomicAdd(S, static_cast<uint32_t>(o.x[q]));
                const unsigned long long x2 =
                    static_cast<unsigned long long>(static_cast<long long>(o.x[q]) * o.x[q]);
                atomicAdd(S + 3 * E, static_cast<uint32_t>(x2) & 0x3ffffu);
                const uint32_t hi = static_cast<uint32_t>(x2 >> 18);
                if (hi != 0u) atomicAdd(S + 6 * E, hi);
            }
        }
    }
    flush();
    binned += stats_direct<2>(in, c0 + threadIdx.x, i1, kTileThreads, b, v0, v1, acc);
    warp_add(binned, ctr + 0);
}

// The test of within() as |x - m| <= r with m = S / n and r = k sqrt(n Q - S^2) / n
// in float: m is off by less than 3 2^-24 of 2^18 and the difference by half a
// unit of 2^19, together less than kCutSlack, and r by less than kCutEps of itself.  A
// value inside by both margins is kept, one outside by both is cut, the rest
// take the test in integers.  Empty bins keep everything (r infinite); a variance
// that wrapped below zero leaves all to the integers (r a NaN).  (Integer bounds
// per bin needed exact roots and divisions: 29 of the pass's 82 million warp
// instructions.)
constexpr float kCutSlack = 0.25f, kCutEps = 3.814697265625e-6f;  // 2^-18

__device__ __forceinline__ float2 cut_limits(int k, const unsigned long long *a, int q)
{
    const unsigned long long n = a[0];
    const long long S = static_cast<long long>(a[1 + q]), Q = static_cast<long long>(a[4 + q]);
    if (n == 0) return make_float2(0.0f, INFINITY);
    float var;
    if (n < 8192) {  // n Q and S^2 below 2^62
        var = __ll2float_rn(static_cast<long long>(n) * Q - S * S);
    } else {
        const __int128 v = static_cast<__int128>(n) * Q - static_cast<__int128>(S) * S;
        var = __ll2float_rn(static_cast<long long>(v >> 62)) * 4611686018427387904.0f +
              __ll2float_rn(static_cast<long long>(v & ((static_cast<__int128>(1) << 62) - 1)));
    }
    const float fn = __ull2float_rn(n);
    return make_float2(__fdiv_rn(__ll2float_rn(S), fn),
                       __fdiv_rn(static_cast<float>(k) * __fsqrt_rn(var), fn));
}

__global__ void __launch_bounds__(kTileThreads) binned_cut_tiles_kernel(Inputs in, int64_t n, BinQ b,
                                                                        BinTiles t,
                                                                        unsigned long long *acc,
                                                                        unsigned long long *ctr)
{
    extern __shared__ uint32_t s_tab[];  // limits of the 3 values, kept n, kept sum
    float2 *const s_lim = reinterpret_cast<float2 *>(s_tab);
    const int win = blockIdx.x % t.n_win, seg = blockIdx.x / t.n_win, n_seg = gridDim.x / t.n_win;
    const int64_t i0 = n * seg / n_seg, i1 = n * (seg + 1) / n_seg;
    const int v0 = win * t.rows, v1 = min(b.n_v, v0 + t.rows);
    const int E = b.n_u * (v1 - v0);
    after_previous();
    unsigned long long cut = 0;
    TileAngle ang;
    auto row_at = [&](int e) {
        return acc + kAccWords * (ang.cur + static_cast<long long>(b.n_ang) *
                                                (e + static_cast<long long>(b.n_u) * v0));
    };
    auto flush = [&]() {
        __syncthreads();
        if (ang.cur >= 0) {
            for (int e = threadIdx.x; e < E; e += kTileThreads) {
                const uint32_t c = s_tab[6 * E + e];
                if (c == 0u) continue;
                unsigned long long *a = row_at(e);
                atomicAdd(a + 7, static_cast<unsigned long long>(c));
                atomicAdd(a + 8, u64_of(static_cast<int>(s_tab[7 * E + e])));
            }
        }
    };
    float ahead[kTileUnroll][6] = {}, sample[3] = {};
    load_chunk(in, i0, i1, ahead, sample);
    int64_t c0 = i0;
    for (; c0 < i1 && !ang.lost(); c0 += kTileChunk) {
        int next;
        if (ang.due(b, sample, next)) {
            flush();
            ang.cur = next;
            for (int e = threadIdx.x; e < E; e += kTileThreads) {
                const unsigned long long *a = row_at(e);
#pragma unroll
                for (int q = 0; q < 3; ++q) s_lim[q * E + e] = cut_limits(b.k, a, q);
                s_tab[6 * E + e] = s_tab[7 * E + e] = 0u;
            }
            __syncthreads();
        }
        float h[kTileUnroll][6];
#pragma unroll
        for (int k = 0; k < kTileUnroll; ++k)
#pragma unroll
            for (int f = 0; f < 6; ++f) h[k][f] = ahead[k][f];
        load_chunk(in, c0 + kTileChunk, i1, ahead, sample);
#pragma unroll
        for (int k = 0; k < kTileUnroll; ++k) {
            BinAt o;
            if (!bin_of(b, h[k][0], h[k][1], h[k][2], h[k][3], h[k][4], h[k][5], o)) continue;
            if (o.iv < v0 || o.iv >= v1) continue;
            if (o.ia != ang.cur) {
                unsigned long long *a = acc + kAccWords * row_of(b, o);
                if (!keep_of(b, a, o.x)) {
                    ++cut;
                    continue;
                }
                atomicAdd(a + 7, 1ull);
                atomicAdd(a + 8, u64_of(o.x[0]));
                continue;
            }
            const int e = o.iu + b.n_u * (o.iv - v0);
            bool keep = true, out = false;
#pragma unroll
            for (int q = 0; q < 3; ++q) {
                const float2 lim = s_lim[q * E + e];
                const float d = fabsf(static_cast<float>(o.x[q]) - lim.x);
                keep = keep && d <= lim.y * (1.0f - kCutEps) - kCutSlack;
                out = out || d > lim.y * (1.0f + kCutEps) + kCutSlack;
            }
            if (!keep && !out) keep = keep_of(b, row_at(e), o.x);
            if (!keep) {
                ++cut;
                continue;
            }
            if (atomicAdd(s_tab + 6 * E + e, 1u) >= kTileCount)
                atomicAdd(row_at(e) + 8, u64_of(o.x[0]));
            else
                atomicAdd(s_tab + 7 * E + e, static_cast<uint32_t>(o.x[0]));
        }
    }
    flush();
    cut += cut_direct<2>(in, c0 + threadIdx.x, i1, kTileThreads, b, v0, v1, acc);
    warp_add(cut, ctr + 1);
}

// Bins used and missed, where the carving blocks do not count them.
__global__ void __launch_bounds__(kBinThreads) binned_bins_kernel(const unsigned long long *acc,
                                                                  int64_t nb, long long miss_q8,
                                                                  unsigned long long *ctr)
{
    after_previous();
    unsigned long long used = 0, missed = 0;
    const int64_t stride = static_cast<int64_t>(gridDim.x) * blockDim.x;
    for (int64_t i = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x; i < nb;
         i += stride) {
        const unsigned long long *a = acc + kAccWords * i;
        used += a[0] != 0 ? 1 : 0;
        missed += bin_missed(a, miss_q8) ? 1 : 0;
    }
    warp_add(used, ctr + 2);
    warp_add(missed, ctr + 3);
}

// Clears the bits of one run of a line in a slice bitmap (bit x + nx y,
// 1 = not carved).  An x-major run is a row segment, contiguous bits cleared
// a word at a time; a y-major run (row = x) is a column segment, one bit per
// voxel.  Runs come from a walk clipped to the slice, so they lie inside it;
// the checks only guard the bitmap.
__device__ __forceinline__ void clear_run(uint32_t *img, bool ymaj, int row, int lo, int hi,
                                          int nx, uint32_t plane)
{
    if (!ymaj) {
        const uint32_t l0 = static_cast<uint32_t>(row * nx + lo);
        const uint32_t l1 = static_cast<uint32_t>(row * nx + hi);
        if (l1 >= plane || l0 > l1) return;
        const uint32_t w0 = l0 >> 5, w1 = l1 >> 5;
        for (uint32_t w = w0; w <= w1; ++w) {
            const uint32_t a = w == w0 ? (l0 & 31u) : 0u;
            const uint32_t b = w == w1 ? (l1 & 31u) : 31u;
            const uint32_t m = b - a == 31u ? 0xffffffffu : ((1u << (b - a + 1u)) - 1u) << a;
            atomicAnd(img + w, ~m);
        }
    } else {
        for (int y = lo; y <= hi; ++y) {
            const uint32_t l = static_cast<uint32_t>(row + nx * y);
            if (l < plane) atomicAnd(img + (l >> 5), ~(1u << (l & 31u)));
        }
    }
}

// Host-computed line tables: centre angle of each angle bin, lateral centre
// of each u bin, centre height of each slice, and the groups of slices.
struct LineTables {
    const float *ang_c, *u_c, *zc;
    const SliceGroup *groups;
};

constexpr int kMaxLinesPerBlock = 1024;  // lateral bins a block lists at once

// One block per (angle bin, group of slices): the block's missed bins are
// listed in shared memory, then each thread walks lines from the list.  A line
// lies at a slice's centre height, so its walk is clipped to the slice (a box one
// voxel deep) and is lean unless a crossing ties with another: the runs then
// come from the closed-form cursor, otherwise from the general run walk.  The
// lines of one vertical bin differ between its slices in their height alone, and a
// height inside the slice crosses nothing: one walk serves every slice of a group
// (slices of 2.5 mm in bins of 5 mm: 154 -> 108 us on the head grid).
template <bool kShared>
__global__ void __launch_bounds__(kCarveThreads) binned_carve_kernel(
    const unsigned long long *acc, BinQ b, GeomQ g, Cordic cd, LineTables t, uint32_t *bits,
    int wps, unsigned long long *ctr)
{
    extern __shared__ uint32_t sm[];
    __shared__ int s_list[kMaxLinesPerBlock];
    __shared__ int s_warp[kCarveThreads / 32];
    __shared__ long long s_cs[2];
    const int ia = blockIdx.x;
    const SliceGroup grp = t.groups[blockIdx.y];
    const int iv = grp.iv, z = grp.z0;
    const bool empty = grp.z1 == grp.z0;  // no slice: the bin is only counted
    uint32_t *gimg = bits + static_cast<size_t>(z) * wps;
    uint32_t *img = kShared ? sm : gimg;
    if (kShared)
        for (int w = threadIdx.x; w < wps; w += blockDim.x) sm[w] = 0xffffffffu;
    const uint32_t plane = static_cast<uint32_t>(g.nx) * static_cast<uint32_t>(g.ny);
    const float zc = empty ? 0.0f : t.zc[z];
    if (threadIdx.x == 0) {  // the block's gantry cos and sin, once
        long long c, sn;
        cordic_cs(q16_of(t.ang_c[ia]), cd, c, sn);
        s_cs[0] = c;
        s_cs[1] = sn;
    }
    after_previous();
    const unsigned lane = threadIdx.x & 31u, warp = threadIdx.x >> 5;
    unsigned long long lines = 0, outside = 0, used = 0, missed = 0;
    for (int base = 0; base < b.n_u; base += kMaxLinesPerBlock) {
        // the chunk's missed bins, listed in lateral order (neighbouring
        // lanes then walk neighbouring, similar lines)
        const int end = min(b.n_u, base + kMaxLinesPerBlock);
        int nl = 0;
        for (int c0 = base; c0 < end; c0 += blockDim.x) {
            const int iu = c0 + static_cast<int>(threadIdx.x);
            bool miss = false;
            if (iu < end) {
                const long long bi = ia + static_cast<long long>(b.n_ang) *
                                              (iu + static_cast<long long>(b.n_u) * iv);
                const unsigned long long *a = acc + kAccWords * bi;
                miss = bin_missed(a, b.miss_q8);
                if (grp.count) {
                    used += a[0] != 0 ? 1 : 0;
                    missed += miss ? 1 : 0;
                }
                miss = miss && !empty;
            }
            const unsigned bal = __ballot_sync(0xffffffffu, miss);
            if (lane == 0) s_warp[warp] = __popc(bal);
            __syncthreads();
            int off = nl, tot = 0;
            for (int k = 0; k < static_cast<int>(blockDim.x >> 5); ++k) {
                off += k < static_cast<int>(warp) ? s_warp[k] : 0;
                tot += s_warp[k];
            }
            if (miss) s_list[off + __popc(bal & ((1u << lane) - 1u))] = iu;
            nl += tot;
            __syncthreads();
        }
        const long long cs = s_cs[0], sn = s_cs[1];
        for (int j = threadIdx.x; j < nl; j += blockDim.x) {
            ++lines;
            const float lu = t.u_c[s_list[j]];
            int32_t r[6];
            if (!endpoints_cs(g, cs, sn, lu, zc, lu, zc, r)) {
                ++outside;
                continue;
            }
            const int32_t gi[3] = {r[0], r[1], r[2] - (z << 16)};
            const int32_t go[3] = {r[3], r[4], r[5] - (z << 16)};
            RunWalk w;
            if (!run_begin(w, gi, go, g.nx, g.ny, 1)) continue;
            const bool ymaj = (w.flags >> 5) & 1;
            LeanWalk L;
            int row, lo, hi;
            if (lean_of(w, L)) {
                uint32_t o[kLeanWords];
                lean_pack(L, o);
                LeanCursor c;
                if (!lean_start(o, 1, c)) continue;  // rows counted one by one
                unsigned ends = 0;
                bool more;
                do {
                    more = lean_run(c, row, lo, hi, ends);
                    clear_run(img, ymaj, row, lo, hi, g.nx, plane);
                } while (more);
            } else {
                while (run_next(w, row, lo, hi)) clear_run(img, ymaj, row, lo, hi, g.nx, plane);
            }
        }
        __syncthreads();  // the list is rebuilt next round
    }
    if (kShared) {
        for (int w = threadIdx.x; w < wps; w += blockDim.x) {
            const uint32_t m = sm[w];
            if (m != 0xffffffffu)
                for (int k = 0; k < grp.z1 - grp.z0; ++k)
                    atomicAnd(gimg + static_cast<size_t>(k) * wps + w, m);
        }
    }
    const unsigned long long slices = static_cast<unsigned long long>(grp.z1 - grp.z0);
    warp_add(used, ctr + 2);
    warp_add(missed, ctr + 3);
    warp_add(lines * slices, ctr + 4);
    warp_add(outside * slices, ctr + 5);
}

// Window count of uncarved voxels in each slice (outside the grid counts as
// carved); hull = count >= min_count.
__global__ void __launch_bounds__(256) binned_filter_kernel(const uint32_t *bits, int wps, int nx,
                                                            int ny, int r, int min_count,
                                                            uint8_t *mask, uint8_t *carved)
{
    after_previous();
    const int x = blockIdx.x * blockDim.x + threadIdx.x;
    const int y = blockIdx.y * blockDim.y + threadIdx.y;
    const int z = blockIdx.z;
    if (x >= nx || y >= ny) return;
    const uint32_t *img = bits + static_cast<size_t>(z) * wps;
    // a row of the window is at most 15 consecutive bits, in one word or two
    const int xl = max(x - r, 0), width = min(x + r, nx - 1) - xl + 1;
    const uint32_t wmask = (1u << width) - 1u;
    int c = 0;
    uint32_t own = 0u;
    for (int Y = max(y - r, 0); Y <= min(y + r, ny - 1); ++Y) {
        const uint32_t l = static_cast<uint32_t>(xl) + static_cast<uint32_t>(nx) * Y;
        const int w = static_cast<int>(l >> 5);
        const uint32_t row = __funnelshift_r(img[w], img[min(w + 1, wps - 1)],
                                             l & 31u) & wmask;
        c += __popc(row);
        if (Y == y) own = row >> (x - xl);
    }
    const size_t v = static_cast<size_t>(x) + static_cast<size_t>(nx) * (y + static_cast<size_t>(ny) * z);
    mask[v] = c >= min_count ? 1 : 0;
    carved[v] = static_cast<uint8_t>(own & 1u);
}

int grid_for(int64_t n, int sm_count, int per_sm = 8)
{
    int64_t blocks = (n + kBinThreads - 1) / kBinThreads;
    const int64_t cap = static_cast<int64_t>(sm_count > 0 ? sm_count : 1) * per_sm;
    if (blocks > cap) blocks = cap;
    return static_cast<int>(blocks < 1 ? 1 : blocks);
}

}  // namespace
}  // namespace hd

// ------------------------------------------------------------------ C ABI

struct hd_binned {
    int device = 0;
    int sm_count = 0;
    hd_geometry geom{};
    hd_binned_params params{};
    hd::GeomQ gq{};
    hd::Cordic cordic{};
    hd::BinQ bq{};
    int64_t V = 0;
    int64_t nb = 0;
    int wps = 0;  // bitmap words per slice
    unsigned long long *acc = nullptr;  // nb x 9
    unsigned long long *ctr = nullptr;  // 8 counters
    uint32_t *bits = nullptr;           // nz x wps carved bitmap (1 = not carved)
    uint8_t *mask = nullptr, *carved = nullptr;
    float *tables = nullptr;  // n_ang angle centres, n_u lateral centres, nz heights
    hd::SliceGroup *groups = nullptr;
    int n_groups = 0;
    bool count_apart = false;  // the bins are counted by binned_bins_kernel
    int phase = 0;  // 0 statistics, 1 cuts, 2 finalised
};

namespace {

#define HB_CUDA(call)                              \
    do {                                           \
        cudaError_t e_ = (call);                   \
        if (e_ != cudaSuccess) {                   \
            hd::note_cuda_error(e_, #call);        \
            return HD_ERR_CUDA;                    \
        }                                          \
    } while (0)

struct BinDevice {
    int prev = -1;
    bool ok = true;
    explicit BinDevice(int dev)
    {
        if (cudaGetDevice(&prev) != cudaSuccess) {
            ok = false;
            return;
        }
        if (prev != dev && cudaSetDevice(dev) != cudaSuccess) ok = false;
    }
    ~BinDevice()
    {
        int cur = -1;
        if (prev >= 0 && cudaGetDevice(&cur) == cudaSuccess && cur != prev) cudaSetDevice(prev);
    }
};

long long fixed_of(float v, double scale) { return llrint(static_cast<double>(v) * scale); }

hd_status make_binq(const hd_binned_params *p, hd::BinQ &b)
{
    auto finite = [](float v) { return std::isfinite(v); };
    if (!finite(p->angle_bin_deg) || !finite(p->u_bin_mm) || !finite(p->v_bin_mm) ||
        !finite(p->u_lo_mm) || !finite(p->v_lo_mm) || !finite(p->miss_wepl_mm))
        return HD_ERR_ARG;
    if (!(p->angle_bin_deg >= 1.0f / 16.0f && p->angle_bin_deg <= 360.0f)) return HD_ERR_RANGE;
    if (!(p->u_bin_mm >= 1.0f / 16.0f && p->u_bin_mm <= 4096.0f)) return HD_ERR_RANGE;
    if (!(p->v_bin_mm >= 1.0f / 16.0f && p->v_bin_mm <= 4096.0f)) return HD_ERR_RANGE;
    if (std::fabs(p->u_lo_mm) > 4096.0f || std::fabs(p->v_lo_mm) > 4096.0f) return HD_ERR_RANGE;
    if (std::fabs(p->miss_wepl_mm) >= 1024.0f) return HD_ERR_RANGE;
    if (p->n_u < 1 || p->n_v < 1 || p->k_sigma < 1 || p->k_sigma > 64) return HD_ERR_RANGE;
    if (p->window < 1 || p->window > 15 || p->window % 2 == 0) return HD_ERR_RANGE;
    if (p->min_count < 0 || p->min_count > p->window * p->window) return HD_ERR_RANGE;
    b.ang_q = fixed_of(p->angle_bin_deg, 65536.0);
    if (hd::kFull % b.ang_q != 0) return HD_ERR_RANGE;
    b.n_ang = static_cast<int>(hd::kFull / b.ang_q);
    b.n_u = p->n_u;
    b.n_v = p->n_v;
    if (static_cast<int64_t>(b.n_ang) * b.n_u * b.n_v > (int64_t(1) << 24)) return HD_ERR_RANGE;
    b.u_q = fixed_of(p->u_bin_mm, 65536.0);
    b.v_q = fixed_of(p->v_bin_mm, 65536.0);
    b.u_lo_q = fixed_of(p->u_lo_mm, 65536.0);
    b.v_lo_q = fixed_of(p->v_lo_mm, 65536.0);
    b.r_ang = hd::rcp_int(static_cast<int>(2 * b.ang_q));
    b.r_u = hd::rcp_int(static_cast<int>(2 * b.u_q));
    b.r_v = hd::rcp_int(static_cast<int>(2 * b.v_q));
    b.k = p->k_sigma;
    b.miss_q8 = fixed_of(p->miss_wepl_mm, 256.0);
    b.w = p->window;
    b.min_count = p->min_count;
    return HD_OK;
}

long long floordiv_host(long long a, long long b)  // b > 0
{
    long long q = a / b;
    if (a % b != 0 && a < 0) --q;
    return q;
}

void free_binned(hd_binned *b)
{
    if (!b) return;
    if (b->acc) cudaFree(b->acc);
    if (b->ctr) cudaFree(b->ctr);
    if (b->bits) cudaFree(b->bits);
    if (b->mask) cudaFree(b->mask);
    if (b->carved) cudaFree(b->carved);
    if (b->tables) cudaFree(b->tables);
    if (b->groups) cudaFree(b->groups);
    delete b;
}

// Every input pointer must be readable by the device; host: some input lies in
// host memory.
hd_status check_inputs(const float *const *p, int k, bool &host)
{
    host = false;
    for (int i = 0; i < k; ++i) {
        if (!p[i]) return HD_ERR_ARG;
        cudaPointerAttributes at{};
        if (cudaPointerGetAttributes(&at, p[i]) != cudaSuccess) {
            cudaGetLastError();
            return HD_ERR_ARG;
        }
        if (at.type == cudaMemoryTypeUnregistered) return HD_ERR_ARG;
        if (at.type != cudaMemoryTypeDevice) host = true;
    }
    return HD_OK;
}

// Blocks of 512 threads for `items` of them, at most four per SM.
unsigned blocks_of(const hd_binned *b, int64_t items)
{
    int64_t n = (items + 511) / 512;
    const int64_t cap = 4 * int64_t(b->sm_count > 0 ? b->sm_count : 1);
    if (n > cap) n = cap;
    return static_cast<unsigned>(n < 1 ? 1 : n);
}

// How a pass of n histories keeps an angle's bins in shared memory (words 32-bit
// words each); n_win 0 when it does not: more than four windows (each reads every
// history again), too few histories to fill and empty a block's table, or host
// inputs: the host link bounds those, and the one block per SM of a table keeps
// fewer reads of it in flight (4e6 histories 1205 us, 1038 without a table).
hd::BinTiles tiles_of(const hd_binned *b, int64_t n, int words, bool host)
{
    if (host) return {0, 0};
    const int64_t bins = hd::kTileBytes / (4 * words);
    const int64_t rows = bins / b->bq.n_u;
    if (rows < 1) return {0, 0};
    const int64_t n_win = (b->bq.n_v + rows - 1) / rows;
    if (n_win > hd::kMaxWindows || n_win > b->sm_count) return {0, 0};
    const int64_t per_angle = int64_t(b->bq.n_u) * b->bq.n_v;
    if (n < per_angle * b->sm_count * hd::kTileFill) return {0, 0};
    return {static_cast<int>(n_win), static_cast<int>((b->bq.n_v + n_win - 1) / n_win)};
}

hd_status pass(hd_binned *b, const float *angle_deg, const float *u_in, const float *v_in,
               const float *u_out, const float *v_out, const float *wepl, int64_t n, bool cut,
               cudaStream_t st)
{
    if (n < 0) return HD_ERR_ARG;
    if (n == 0) return HD_OK;
    const float *p[6] = {angle_deg, u_in, v_in, u_out, v_out, wepl};
    bool host;
    const hd_status v = check_inputs(p, 6, host);
    if (v != HD_OK) return v;
    const hd::Inputs in{angle_deg, u_in, v_in, u_out, v_out, wepl};
    const int words = cut ? hd::kCutWords : hd::kStatsWords;
    const hd::BinTiles t = tiles_of(b, n, words, host);
    const int grid = hd::grid_for(n, b->sm_count, hd::kPassBlocksPerSm);  // one wave
    if (t.n_win > 0) {
        const unsigned blocks = static_cast<unsigned>(b->sm_count / t.n_win * t.n_win);
        const size_t smem = sizeof(uint32_t) * words * size_t(b->bq.n_u) * t.rows;
        HB_CUDA(hd::launch_chained(cut ? hd::binned_cut_tiles_kernel : hd::binned_stats_tiles_kernel,
                                   blocks, hd::kTileThreads, smem, st, in, n, b->bq, t, b->acc,
                                   b->ctr));
    } else {
        HB_CUDA(hd::launch_chained(cut ? hd::binned_cut_kernel : hd::binned_stats_kernel,
                                   static_cast<unsigned>(grid), hd::kBinThreads, 0, st, in, n, b->bq,
                                   b->acc, b->ctr));
    }
    return HD_OK;
}

}  // namespace

extern "C" {

hd_status hd_binned_params_default(const hd_geometry *geom, hd_binned_params *out)
{
    if (!geom || !out) return HD_ERR_ARG;
    const hd_status gs = hd::check_geometry(geom);
    if (gs != HD_OK) return gs;
    out->angle_bin_deg = 4.0f;
    out->u_bin_mm = 1.0f;
    out->v_bin_mm = 5.0f;
    const double wx = static_cast<double>(geom->nx) * geom->sx;
    const double wy = static_cast<double>(geom->ny) * geom->sy;
    const double half_u = std::ceil(std::hypot(wx, wy) / 2.0 / out->u_bin_mm) * out->u_bin_mm;
    const double half_v =
        std::ceil(static_cast<double>(geom->nz) * geom->sz / 2.0 / out->v_bin_mm) * out->v_bin_mm;
    out->u_lo_mm = static_cast<float>(-half_u);
    out->v_lo_mm = static_cast<float>(-half_v);
    out->n_u = static_cast<int32_t>(std::lround(2.0 * half_u / out->u_bin_mm));
    out->n_v = static_cast<int32_t>(std::lround(2.0 * half_v / out->v_bin_mm));
    out->k_sigma = 3;
    out->miss_wepl_mm = 1.0f;
    out->window = 5;
    out->min_count = 11;
    return HD_OK;
}

hd_status hd_binned_create(const hd_geometry *geom, const hd_binned_params *params,
                           hd_binned **out)
{
    if (!out || !geom || !params) return HD_ERR_ARG;
    *out = nullptr;
    const hd_status gs = hd::check_geometry(geom);
    if (gs != HD_OK) return gs;
    hd::BinQ bq{};
    const hd_status ps = make_binq(params, bq);
    if (ps != HD_OK) return ps;
    hd_binned *b = new (std::nothrow) hd_binned();
    if (!b) return HD_ERR_NOMEM;
    b->geom = *geom;
    b->params = *params;
    b->bq = bq;
    if (!hd::make_cordic_table(b->cordic)) {
        delete b;
        return HD_ERR_RANGE;
    }
    cudaError_t e = cudaGetDevice(&b->device);
    if (e == cudaSuccess)
        e = cudaDeviceGetAttribute(&b->sm_count, cudaDevAttrMultiProcessorCount, b->device);
    if (e != cudaSuccess) {
        hd::note_cuda_error(e, "hd_binned_create: device query");
        delete b;
        return HD_ERR_CUDA;
    }
    b->gq = hd::make_geomq(geom->nx, geom->ny, geom->nz, geom->sx, geom->sy, geom->sz,
                           geom->tracker_half_sep_mm);
    b->V = int64_t(geom->nx) * geom->ny * geom->nz;
    b->nb = int64_t(bq.n_ang) * bq.n_u * bq.n_v;
    const int64_t plane = int64_t(geom->nx) * geom->ny;
    b->wps = static_cast<int>((plane + 31) / 32);
    // line tables, computed as the method states them: centre angle ia
    // times the bin size, lateral centre lo + (iu + 1/2) size, slice centre
    // height from the Q16 slice thickness and its vertical bin
    const int nz = geom->nz;
    const size_t nt = static_cast<size_t>(bq.n_ang) + bq.n_u + nz;
    float *tab = new (std::nothrow) float[nt];
    b->count_apart = bq.n_v > 2 * nz + 64;
    hd::SliceGroup *grp = new (std::nothrow)
        hd::SliceGroup[size_t(nz) + (b->count_apart ? 0 : size_t(bq.n_v))];
    if (!tab || !grp) {
        delete[] tab;
        delete[] grp;
        delete b;
        return HD_ERR_NOMEM;
    }
    for (int ia = 0; ia < bq.n_ang; ++ia)
        tab[ia] = static_cast<float>(static_cast<double>(ia * bq.ang_q) / 65536.0);
    for (int iu = 0; iu < bq.n_u; ++iu)
        tab[bq.n_ang + iu] = static_cast<float>(
            static_cast<double>(2 * bq.u_lo_q + (2LL * iu + 1) * bq.u_q) / (2.0 * 65536.0));
    // groups: a bin's slices (heights rise with z) together while the heights lie
    // inside their slices and a bitmap in shared memory collects the lines; bins
    // without slices have an empty group, unless they are so many that counting
    // them takes a kernel of its own
    int ng = 0, next_iv = 0;
    bool open = false;
    for (int z = 0; z < nz; ++z) {
        const long long c2 = (2LL * z + 1 - nz) * b->gq.sz;
        const float zc = static_cast<float>(static_cast<double>(c2) / (2.0 * 65536.0));
        tab[bq.n_ang + bq.n_u + z] = zc;
        const long long iv = floordiv_host(c2 - 2 * bq.v_lo_q, 2 * bq.v_q);
        if (iv < 0 || iv >= bq.n_v) continue;
        const long long at = std::fabs(zc) < 4096.0f
                                 ? hd::to_grid(hd::q16_small(zc), b->gq.dz) - (int64_t(z) << 16) : 0;
        const bool inside = at > 0 && at < 65536 && b->wps <= hd::kMaxSmemWords;
        if (inside && open && grp[ng - 1].iv == iv) {
            grp[ng - 1].z1 = z + 1;
            continue;
        }
        if (next_iv <= iv) {
            while (!b->count_apart && next_iv < iv) grp[ng++] = {next_iv++, 0, 0, 1};
            grp[ng++] = {static_cast<int>(iv), z, z + 1, b->count_apart ? 0 : 1};
            next_iv = static_cast<int>(iv) + 1;
        } else {
            grp[ng++] = {static_cast<int>(iv), z, z + 1, 0};
        }
        open = inside;
    }
    while (!b->count_apart && next_iv < bq.n_v) grp[ng++] = {next_iv++, 0, 0, 1};
    b->n_groups = ng;
    bool ok = true;
    auto alloc = [&](void **p, size_t bytes) {
        if (!ok) return;
        if (cudaMalloc(p, bytes) != cudaSuccess) {
            cudaGetLastError();
            *p = nullptr;
            ok = false;
        }
    };
    alloc(reinterpret_cast<void **>(&b->acc), sizeof(unsigned long long) * hd::kAccWords * b->nb);
    alloc(reinterpret_cast<void **>(&b->ctr), sizeof(unsigned long long) * hd::kCtrWords);
    alloc(reinterpret_cast<void **>(&b->bits), sizeof(uint32_t) * size_t(b->wps) * nz);
    alloc(reinterpret_cast<void **>(&b->mask), size_t(b->V));
    alloc(reinterpret_cast<void **>(&b->carved), size_t(b->V));
    alloc(reinterpret_cast<void **>(&b->tables), sizeof(float) * nt);
    alloc(reinterpret_cast<void **>(&b->groups), sizeof(hd::SliceGroup) * (ng > 0 ? ng : 1));
    if (ok) {
        cudaError_t c = cudaMemcpy(b->tables, tab, sizeof(float) * nt, cudaMemcpyHostToDevice);
        if (c == cudaSuccess)
            c = cudaMemcpy(b->groups, grp, sizeof(hd::SliceGroup) * ng, cudaMemcpyHostToDevice);
        if (c == cudaSuccess)
            c = cudaMemset(b->acc, 0, sizeof(unsigned long long) * hd::kAccWords * b->nb);
        if (c == cudaSuccess) c = cudaMemset(b->ctr, 0, sizeof(unsigned long long) * hd::kCtrWords);
        if (c == cudaSuccess) c = cudaDeviceSynchronize();
        if (c != cudaSuccess) {
            hd::note_cuda_error(c, "hd_binned_create: initialise");
            delete[] tab;
            delete[] grp;
            free_binned(b);
            return HD_ERR_CUDA;
        }
    }
    delete[] tab;
    delete[] grp;
    if (!ok) {
        free_binned(b);
        return HD_ERR_NOMEM;
    }
    // the largest slice bitmap any object uses, so objects of different
    // sizes never lower one another's limit
    if (cudaFuncSetAttribute(hd::binned_carve_kernel<true>,
                             cudaFuncAttributeMaxDynamicSharedMemorySize,
                             static_cast<int>(sizeof(uint32_t) * hd::kMaxSmemWords)) !=
            cudaSuccess ||
        cudaFuncSetAttribute(hd::binned_stats_tiles_kernel,
                             cudaFuncAttributeMaxDynamicSharedMemorySize, hd::kTileBytes) !=
            cudaSuccess ||
        cudaFuncSetAttribute(hd::binned_cut_tiles_kernel,
                             cudaFuncAttributeMaxDynamicSharedMemorySize, hd::kTileBytes) !=
            cudaSuccess) {
        cudaGetLastError();
        free_binned(b);
        return HD_ERR_CUDA;
    }
    *out = b;
    return HD_OK;
}

hd_status hd_binned_destroy(hd_binned *b)
{
    if (!b) return HD_ERR_ARG;
    BinDevice g(b->device);
    cudaDeviceSynchronize();
    free_binned(b);
    return HD_OK;
}

hd_status hd_binned_reset(hd_binned *b, void *stream)
{
    if (!b) return HD_ERR_ARG;
    BinDevice g(b->device);
    if (!g.ok) return HD_ERR_CUDA;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    const int64_t words = hd::kAccWords * b->nb;
    HB_CUDA(hd::launch_chained(hd::binned_clear_kernel, blocks_of(b, words / 2), 512, 0, st, b->acc,
                               words, b->ctr));
    b->phase = 0;
    return HD_OK;
}

hd_status hd_binned_add_histories(hd_binned *b, const float *angle_deg, const float *u_in,
                                  const float *v_in, const float *u_out, const float *v_out,
                                  const float *wepl, int64_t n, void *stream)
{
    if (!b) return HD_ERR_ARG;
    if (b->phase != 0) return HD_ERR_STATE;
    BinDevice g(b->device);
    if (!g.ok) return HD_ERR_CUDA;
    return pass(b, angle_deg, u_in, v_in, u_out, v_out, wepl, n, false,
                static_cast<cudaStream_t>(stream));
}

hd_status hd_binned_cut_histories(hd_binned *b, const float *angle_deg, const float *u_in,
                                  const float *v_in, const float *u_out, const float *v_out,
                                  const float *wepl, int64_t n, void *stream)
{
    if (!b) return HD_ERR_ARG;
    if (b->phase == 2) return HD_ERR_STATE;
    BinDevice g(b->device);
    if (!g.ok) return HD_ERR_CUDA;
    const hd_status s = pass(b, angle_deg, u_in, v_in, u_out, v_out, wepl, n, true,
                             static_cast<cudaStream_t>(stream));
    if (s == HD_OK) b->phase = 1;
    return s;
}

hd_status hd_binned_finalize(hd_binned *b, void *stream)
{
    if (!b) return HD_ERR_ARG;
    if (b->phase == 0) return HD_ERR_STATE;
    BinDevice g(b->device);
    if (!g.ok) return HD_ERR_CUDA;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    const int nz = b->geom.nz;
    const int64_t words = int64_t(b->wps) * nz;
    HB_CUDA(hd::launch_chained(hd::binned_image_kernel, blocks_of(b, words), 512, 0, st, b->bits, words,
                               b->ctr));
    if (b->count_apart)
        HB_CUDA(hd::launch_chained(hd::binned_bins_kernel,
                                   static_cast<unsigned>(hd::grid_for(b->nb, b->sm_count)),
                                   hd::kBinThreads, 0, st, b->acc, b->nb, b->bq.miss_q8, b->ctr));
    const hd::LineTables t{b->tables, b->tables + b->bq.n_ang, b->tables + b->bq.n_ang + b->bq.n_u,
                           b->groups};
    const dim3 cg(static_cast<unsigned>(b->bq.n_ang), static_cast<unsigned>(b->n_groups));
    if (b->n_groups > 0) {
        const bool shared = b->wps <= hd::kMaxSmemWords;
        HB_CUDA(hd::launch_chained(shared ? hd::binned_carve_kernel<true> : hd::binned_carve_kernel<false>,
                                   cg, hd::kCarveThreads, shared ? sizeof(uint32_t) * b->wps : 0, st,
                                   b->acc, b->bq, b->gq, b->cordic, t, b->bits, b->wps, b->ctr));
    }
    const dim3 fb(32, 8);
    const dim3 fg(static_cast<unsigned>((b->geom.nx + 31) / 32),
                  static_cast<unsigned>((b->geom.ny + 7) / 8), static_cast<unsigned>(nz));
    HB_CUDA(hd::launch_chained(hd::binned_filter_kernel, fg, fb, 0, st, b->bits, b->wps, b->geom.nx,
                               b->geom.ny, b->bq.w / 2, b->bq.min_count, b->mask, b->carved));
    b->phase = 2;
    return HD_OK;
}

hd_status hd_binned_run(hd_binned *b, const float *angle_deg, const float *u_in,
                        const float *v_in, const float *u_out, const float *v_out,
                        const float *wepl, int64_t n, void *stream)
{
    hd_status s = hd_binned_reset(b, stream);
    if (s == HD_OK) s = hd_binned_add_histories(b, angle_deg, u_in, v_in, u_out, v_out, wepl, n, stream);
    if (s == HD_OK) s = hd_binned_cut_histories(b, angle_deg, u_in, v_in, u_out, v_out, wepl, n, stream);
    if (s == HD_OK && b->phase == 0) b->phase = 1;  // n == 0: nothing to cut
    if (s == HD_OK) s = hd_binned_finalize(b, stream);
    return s;
}

hd_status hd_binned_get_image(hd_binned *b, int32_t which, uint8_t *dst, int64_t n,
                              int32_t dst_on_device, void *stream)
{
    if (!b || !dst || (which != HD_BINNED_HULL && which != HD_BINNED_CARVED)) return HD_ERR_ARG;
    if (n < b->V) return HD_ERR_ARG;
    if (b->phase != 2) return HD_ERR_STATE;
    BinDevice g(b->device);
    if (!g.ok) return HD_ERR_CUDA;
    HB_CUDA(hd::copy_out(dst, which == HD_BINNED_HULL ? b->mask : b->carved, size_t(b->V), dst_on_device,
                         b->device, b->sm_count, static_cast<cudaStream_t>(stream)));
    return HD_OK;
}

hd_status hd_binned_get_bins(hd_binned *b, int64_t *dst, int64_t n_bins, int32_t dst_on_device,
                             void *stream)
{
    if (!b || !dst || n_bins < b->nb) return HD_ERR_ARG;
    BinDevice g(b->device);
    if (!g.ok) return HD_ERR_CUDA;
    HB_CUDA(hd::copy_out(dst, b->acc, sizeof(int64_t) * hd::kAccWords * b->nb, dst_on_device, b->device,
                         b->sm_count, static_cast<cudaStream_t>(stream)));
    return HD_OK;
}

hd_status hd_binned_get_stats(hd_binned *b, hd_binned_stats *out, void *stream)
{
    if (!b || !out) return HD_ERR_ARG;
    BinDevice g(b->device);
    if (!g.ok) return HD_ERR_CUDA;
    unsigned long long c[hd::kCtrWords];
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    HB_CUDA(cudaMemcpyAsync(c, b->ctr, sizeof(c), cudaMemcpyDeviceToHost, st));
    HB_CUDA(cudaStreamSynchronize(st));
    out->histories_binned = static_cast<int64_t>(c[0]);
    out->histories_cut = static_cast<int64_t>(c[1]);
    out->bins = b->nb;
    out->bins_used = static_cast<int64_t>(c[2]);
    out->bins_missed = static_cast<int64_t>(c[3]);
    out->lines = static_cast<int64_t>(c[4]);
    out->lines_outside = static_cast<int64_t>(c[5]);
    return HD_OK;
}

}  // extern "C"
