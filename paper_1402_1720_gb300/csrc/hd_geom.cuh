// Fixed-point geometry and the exact voxel traversal (host and device).
//
// Geometry (Sec. 2.1-2.2): the path L_i is the closed segment from the entry
// point -T b + u_in e_u + v_in e_v to the exit point +T b + u_out e_u +
// v_out e_v, b = (cos phi, sin phi, 0), e_u = (-sin phi, cos phi, 0).  Each
// float32 input is rounded once to 16 fractional bits (ties to even); cos
// and sin come from an integer CORDIC with 30 fractional bits; world and
// grid coordinates follow by integer floor division.  After that every step
// is exact.
//
// Voxel set (Eq. 3.2 with d_0 = 0 against half-open voxel cubes): the voxels
// floor(P(t) / 2^16), t in [0, 1], of P(t) = G_in + t D inside the box.  The
// walk orders plane crossings with the three cross-multiplied terms
// E_ab = num_a |D_b| - num_b |D_a| (num_a / |D_a| is the parameter of axis
// a's next crossing) and updates them with additions only.  At equal
// parameters an axis moving + enters its next voxel at the crossing itself
// and an axis moving - leaves its voxel just after it, so a mixed tie visits
// the corner voxel between the two.  The walk starts at the exact rational
// parameter where the segment enters the box.
//
// Magnitudes: |G| < 2^30 + 2^28 (grid coordinates, possibly shifted to a
// tile origin), |D| < 2^31, so every product below stays under 2^62.
#pragma once

#include <cmath>
#include <cstdint>

#include "hd_internal.cuh"

#define HD_HD __host__ __device__ __forceinline__

namespace hd {

HD_HD unsigned long long umulhi64(unsigned long long a, unsigned long long b)
{
#ifdef __CUDA_ARCH__
    return __umul64hi(a, b);
#else
    return static_cast<unsigned long long>((static_cast<unsigned __int128>(a) * b) >> 64);
#endif
}

HD_HD unsigned umulhi32(unsigned a, unsigned b)
{
#ifdef __CUDA_ARCH__
    return __umulhi(a, b);
#else
    return static_cast<unsigned>((static_cast<unsigned long long>(a) * b) >> 32);
#endif
}

// Q16 of a value known to satisfy |x| < 4096: the 32-bit conversion rounds
// exactly as the 64-bit one does.
HD_HD int q16_small(float x)
{
#ifdef __CUDA_ARCH__
    return __float2int_rn(x * 65536.0f);
#else
    return static_cast<int>(lrintf(x * 65536.0f));
#endif
}

HD_HD long long q16_of(float x)
{
    // x * 2^16 is exact in float32 for |x| < 2^20 * ..., so the conversion
    // is the only rounding (to nearest, ties to even).
#ifdef __CUDA_ARCH__
    return __float2ll_rn(x * 65536.0f);
#else
    return llrintf(x * 65536.0f);
#endif
}

HD_HD long long floordiv_pos(long long a, long long b)
{
    long long q = a / b;
    if (a - q * b != 0 && a < 0) --q;
    return q;
}

// Float value of a 64-bit integer (relative error below 2^-22) built from
// two 32-bit conversions.
HD_HD float float_of(long long a)
{
    return static_cast<float>(static_cast<int>(a >> 32)) * 4294967296.0f +
           static_cast<float>(static_cast<unsigned>(a & 0xffffffffLL));
}

// floor(a / b), b > 0, for quotients known to be small (|a / b| < 2^20 and
// |a| < 2^62): a float estimate corrected with exact integer arithmetic, so
// no 64-bit division is needed.
HD_HD long long floordiv_small(long long a, long long b)
{
    // an approximate float quotient: the integer steps below make it exact
#ifdef __CUDA_ARCH__
    long long q = static_cast<long long>(static_cast<int>(floorf(__fdividef(float_of(a), float_of(b)))));
#else
    long long q = static_cast<long long>(static_cast<int>(floorf(float_of(a) / float_of(b))));
#endif
    long long r = a - q * b;
    while (r < 0) {
        --q;
        r += b;
    }
    while (r >= b) {
        ++q;
        r -= b;
    }
    return q;
}

// floor(a / b) for b > 0 and |a / b| < 2^20: a correctly rounded float
// quotient estimate (relative error below 2^-21) is within one of the
// floor, so one correction step each way settles it.  The 64-bit form of fdiv32,
// which the kernels use; the host tests compare it with the floor.
HD_HD long long fdiv_small(long long a, long long b)
{
#ifdef __CUDA_ARCH__
    long long q = static_cast<long long>(
        static_cast<int>(floorf(__fdividef(__ll2float_rn(a), __ll2float_rn(b)))));
#else
    long long q = static_cast<long long>(
        static_cast<int>(std::floor(static_cast<float>(a) / static_cast<float>(b))));
#endif
    long long r = a - q * b;
    if (r < 0) {
        --q;
        r += b;
    }
    if (r >= b) ++q;
    return q;
}
// Approximate reciprocal of b > 0 (within two units of the last place).
HD_HD float rcp_int(int b)
{
#ifdef __CUDA_ARCH__
    return __fdividef(1.0f, static_cast<float>(b));
#else
    return 1.0f / static_cast<float>(b);
#endif
}

// floor(a / b) and its remainder for 0 < b < 2^31, |a / b| < 2^20, rb =
// rcp_int(b): the estimate is within one of the floor (relative error below
// 2^-21), so one step each way settles it; the remainder is one 32 x 32
// product, and a divisor used twice has its reciprocal taken once.
HD_HD int fdiv32(long long a, int b, float rb, long long &rem)
{
#ifdef __CUDA_ARCH__
    int q = __float2int_rd(__ll2float_rn(a) * rb);
#else
    int q = static_cast<int>(std::floor(static_cast<float>(a) * rb));
#endif
    rem = a - static_cast<long long>(q) * static_cast<long long>(b);
    if (rem < 0) {
        --q;
        rem += b;
    }
    if (rem >= b) {
        ++q;
        rem -= b;
    }
    return q;
}

// Rotation-mode CORDIC of an angle in degrees * 2^16: cos and sin * 2^30.
HD_HD void cordic_cs(long long a_q16, const Cordic &cd, long long &c, long long &s)
{
    const long long full = 360LL * kQ16, quarter = 90LL * kQ16;
    long long a = a_q16 % full;
    if (a < 0) a += full;
    const int k = static_cast<int>(a / quarter);
    const long long r = a - k * quarter;
    long long z = r << 14;
    // |x|, |y| stay below 2^31 (unit vector scaled by 2^30)
    int x = static_cast<int>(cd.K), y = 0;
#pragma unroll
    for (int i = 0; i < 32; ++i) {
        const int xs = x >> i, ys = y >> i;
        const long long th = cd.theta[i];
        if (z >= 0) {
            x -= ys;
            y += xs;
            z -= th;
        } else {
            x += ys;
            y -= xs;
            z += th;
        }
    }
    switch (k) {
    case 0: c = x; s = y; break;
    case 1: c = -y; s = x; break;
    case 2: c = -x; s = -y; break;
    default: c = y; s = -x; break;
    }
}

// Grid coordinate (voxel units, Q16) of a world coordinate w (mm, Q16):
// floor((2 w + n s) 2^16 / (2 s)) = floor((2 w + n s) 2^15 / s).  The numerator
// N = 2 w + n s lies within 1.61e9 in magnitude (|w| < 2^29, n s <= 2^29), so N
// plus the bias is an unsigned 32-bit n', and floor(n' M / 2^54) with M =
// floor(2^69 / s) + 1 is the quotient exactly: its error n' / 2^54 stays below
// 1 / s (n' < 2^32, s <= 2^22).  Two 32 x 32 products, where a 64-bit
// multiply-high division took about four times the instructions.
HD_HD long long to_grid(int w, const GridDiv &d)
{
    const uint32_t n = static_cast<uint32_t>(2 * w + d.ns) + d.bias;
    const unsigned long long lo = static_cast<unsigned long long>(n) * d.mlo;
    const unsigned long long hi = static_cast<unsigned long long>(n) * d.mhi + (lo >> 32);
    return static_cast<long long>(hi >> 22) - d.off;
}

// Host-side construction of the fixed-point geometry.
inline GeomQ make_geomq(int nx, int ny, int nz, float sx, float sy, float sz, float T)
{
    GeomQ g{};
    g.nx = nx;
    g.ny = ny;
    g.nz = nz;
    g.sx = llrint(static_cast<double>(sx) * 65536.0);
    g.sy = llrint(static_cast<double>(sy) * 65536.0);
    g.sz = llrint(static_cast<double>(sz) * 65536.0);
    g.T = llrint(static_cast<double>(T) * 65536.0);
    auto axis = [](int n, long long s) {
        GridDiv d;
        const unsigned long long m = static_cast<unsigned long long>(
                                         (static_cast<unsigned __int128>(1) << 69) /
                                         static_cast<unsigned long long>(s)) + 1;
        d.mlo = static_cast<uint32_t>(m);
        d.mhi = static_cast<uint32_t>(m >> 32);
        d.ns = static_cast<int32_t>(n * s);
        const long long k = (1620000000LL + s - 1) / s;  // >= the largest |N|
        d.bias = static_cast<uint32_t>(k * s);
        d.off = k << 15;
        return d;
    };
    g.dx = axis(nx, g.sx);
    g.dy = axis(ny, g.sy);
    g.dz = axis(nz, g.sz);
    return g;
}

// World entry and exit points (mm, Q16) of one history from its gantry
// cos/sin: W = (x_in, y_in, z_in, x_out, y_out, z_out).  The inputs must
// satisfy |u|, |v| < 4096 mm (endpoints_cs checks it).
HD_HD void world_cs(const GeomQ &g, long long c, long long s, float ui, float vi, float uo,
                    float vo, long long W[6])
{
    // every factor fits 32 bits (T < 2^28 since the tracker distance is below
    // 4096 mm, |c|, |s| <= 2^30, |u| Q16 < 2^28): exact 32 x 32 -> 64 products
    const int T = static_cast<int>(g.T);
    const int ci = static_cast<int>(c), si = static_cast<int>(s);
    const int qui = q16_small(ui), quo = q16_small(uo);
    auto mul = [](int a, int b) { return static_cast<long long>(a) * static_cast<long long>(b); };
    W[0] = (-mul(T, ci) - mul(qui, si)) >> 30;
    W[1] = (-mul(T, si) + mul(qui, ci)) >> 30;
    W[2] = q16_small(vi);
    W[3] = (mul(T, ci) - mul(quo, si)) >> 30;
    W[4] = (mul(T, si) + mul(quo, ci)) >> 30;
    W[5] = q16_small(vo);
}

// Grid Q16 endpoints of one history from its gantry cos/sin; false when the
// history is rejected.
HD_HD bool endpoints_cs(const GeomQ &g, long long c, long long s, float ui, float vi, float uo,
                        float vo, int32_t out[6])
{
    if (!(fabsf(ui) < 4096.0f) || !(fabsf(vi) < 4096.0f) || !(fabsf(uo) < 4096.0f) ||
        !(fabsf(vo) < 4096.0f))
        return false;
    long long W[6];
    world_cs(g, c, s, ui, vi, uo, vo, W);
    const GridDiv *const d[3] = {&g.dx, &g.dy, &g.dz};
    bool ok = true;
#pragma unroll
    for (int a = 0; a < 6; ++a) {
        const long long G = to_grid(static_cast<int>(W[a]), *d[a % 3]);
        // |G| < 2^30
        ok = ok && static_cast<unsigned long long>(G + ((1LL << 30) - 1)) < (1ULL << 31) - 1;
        out[a] = static_cast<int32_t>(G);
    }
    return ok;
}

// Grid Q16 endpoints of one history; false when the history is rejected.
HD_HD bool endpoints(const GeomQ &g, const Cordic &cd, float ang, float ui, float vi, float uo,
                     float vo, int32_t out[6])
{
    if (!(fabsf(ang) < 1048576.0f)) return false;
    long long c, s;
    cordic_cs(q16_of(ang), cd, c, s);
    return endpoints_cs(g, c, s, ui, vi, uo, vo, out);
}

// The slices the part of a segment inside the grid's x-y extent can touch: a
// superset of the slices that hold voxels of the segment (z is monotone along
// it); false when the segment misses the grid (it then has no voxel at all,
// though a segment that barely misses it may get slices).  In float, the extent
// widened by 16 eps (eps = 2^-24) of the numbers that enter a parameter, whose
// roundings are below 8 eps of them, and z by 8 eps of its own (exact rationals
// took three times the instructions and gave the same slices but for one in a
// thousand).
HD_HD bool grid_z_range(const TilePlan &tp, const int32_t r[6], int &zlo, int &zhi)
{
    const float eps = 5.9604644775390625e-8f;
    float t0 = 0.0f, t1 = 1.0f;
#pragma unroll
    for (int a = 0; a < 2; ++a) {
        const float H = static_cast<float>((a == 0 ? tp.nx : tp.ny) << 16);
        const float p = static_cast<float>(r[a]);
        const int di = r[a + 3] - r[a];
        const float d = static_cast<float>(di);
        const float m = fmaf(16.0f * eps, fabsf(p) + fabsf(d) + H, 1.0f);
        if (di == 0) {
            if (p < -m || p > H + m) return false;
        } else {
#ifdef __CUDA_ARCH__
            const float i = __frcp_rn(d);
#else
            const float i = 1.0f / d;
#endif
            const float ta = (-m - p) * i, tb = (H + m - p) * i;
            t0 = fmaxf(t0, fminf(ta, tb));
            t1 = fminf(t1, fmaxf(ta, tb));
        }
    }
    if (t0 > t1) return false;
    const float z = static_cast<float>(r[2]), dz = static_cast<float>(r[5] - r[2]);
    const float za = fmaf(t0, dz, z), zb = fmaf(t1, dz, z);
    const float m = fmaf(8.0f * eps, fabsf(z) + fabsf(dz), 1.0f);
    const int z0 = static_cast<int>(floorf((fminf(za, zb) - m) * (1.0f / 65536.0f)));
    const int z1 = static_cast<int>(floorf((fmaxf(za, zb) + m) * (1.0f / 65536.0f)));
    if (z1 < 0 || z0 >= tp.nz) return false;
    zlo = z0 < 0 ? 0 : z0;
    zhi = z1 >= tp.nz ? tp.nz - 1 : z1;
    return true;
}

// Tiles a record can touch, given its slices zlo..zhi (grid_z_range): in x
// and y the bounding box of its segment clamped to the grid, in z those
// slices, in tile units.  Returns the number of tiles (0 when the box
// misses the grid).
HD_HD int tile_range_z(const TilePlan &tp, const int32_t r[6], int zlo, int zhi, int lo[3],
                       int hi[3])
{
    const int n[3] = {tp.nx, tp.ny, tp.nz};
    const unsigned m[3] = {tp.mtx, tp.mty, tp.mtz};
    int cnt = 1;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        const int a0 = r[a] >> 16, a1 = r[a + 3] >> 16;
        int mn = a0 < a1 ? a0 : a1, mx = a0 < a1 ? a1 : a0;
        if (a == 2) {
            mn = zlo;
            mx = zhi;
        }
        if (mx < 0 || mn >= n[a]) return 0;
        mn = mn < 0 ? 0 : mn;
        mx = mx >= n[a] ? n[a] - 1 : mx;
        // floor(v / t) = umulhi(v, floor(2^32 / t) + 1) for v, t <= 4096;
        // m = 0 stands for t = 1
        lo[a] = m[a] ? static_cast<int>(umulhi32(static_cast<unsigned>(mn), m[a])) : mn;
        hi[a] = m[a] ? static_cast<int>(umulhi32(static_cast<unsigned>(mx), m[a])) : mx;
        cnt *= hi[a] - lo[a] + 1;
    }
    return cnt;
}

// tile_range_z with the slices of grid_z_range; 0 when the segment misses
// the grid (it then has no voxel at all).
HD_HD int tile_range(const TilePlan &tp, const int32_t r[6], int lo[3], int hi[3])
{
    int zlo, zhi;
    if (!grid_z_range(tp, r, zlo, zhi)) return 0;
    return tile_range_z(tp, r, zlo, zhi, lo, hi);
}

// Orients a segment so that its major in-plane axis (the one with the larger
// |D|, x when equal) moves + (A_i is a set of points, so swapping the ends
// does not change it) and returns the type of its walks: bit 1 the major axis
// is y, bit 0 the other in-plane axis moves -.
HD_HD int orient_record(int32_t r[6])
{
    const int dx = r[3] - r[0], dy = r[4] - r[1];  // |G| < 2^30: no overflow
    const int ax = dx < 0 ? -dx : dx, ay = dy < 0 ? -dy : dy;
    const bool ymaj = ay > ax;
    const bool flip = (ymaj ? dy : dx) < 0;
    const int dm = ymaj ? dx : dy;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        const int32_t t = r[a];
        r[a] = flip ? r[a + 3] : t;
        r[a + 3] = flip ? t : r[a + 3];
    }
    return (ymaj ? 2 : 0) | ((flip ? dm > 0 : dm < 0) ? 1 : 0);
}

// A record's status word: bits 0-1 the path (0 no record, 1 tiled, 2
// global), bits 2-4 its group (class + 2 type: the class, 0 missed or 1
// hit, in bit 2, the walk type of orient_record in bits 3-4), bits 8-19 and 20-31 its first and last slice (grid_z_range, computed once).
HD_HD int32_t record_status(int path, int cls, int type, int zlo, int zhi)
{
    return static_cast<int32_t>(static_cast<uint32_t>(path) | (static_cast<uint32_t>(cls) << 2) |
                                (static_cast<uint32_t>(type) << 3) |
                                (static_cast<uint32_t>(zlo) << 8) |
                                (static_cast<uint32_t>(zhi) << 20));
}
HD_HD int status_path(int32_t s) { return s & 3; }
HD_HD int status_cls(int32_t s) { return (s >> 2) & 1; }
HD_HD int status_group(int32_t s) { return (s >> 2) & 7; }  // class + 2 type
HD_HD int status_zlo(int32_t s) { return (static_cast<uint32_t>(s) >> 8) & 0xfff; }
HD_HD int status_zhi(int32_t s) { return static_cast<uint32_t>(s) >> 20; }

// ------------------------------------------------------------------ walk

// Resumable traversal state of one segment inside a box of nx*ny*nz voxels.
struct Walk {
    long long exy, exz, eyz;     // crossing-order terms
    long long ax16, ay16, az16;  // |D_a| * 2^16
    int idx;                     // linear index (x fastest) of the current voxel
    int kx, ky, kz;              // remaining valid crossings per axis
    int stx, sty, stz;           // signed index strides
    int flags;                   // bits 0-2: axis moves +; bits 4-6: pending - group
};

HD_HD void walk_apply(Walk &w, int mask)
{
    if (mask & 1) { --w.kx; w.idx += w.stx; w.exy += w.ay16; w.exz += w.az16; }
    if (mask & 2) { --w.ky; w.idx += w.sty; w.exy -= w.ax16; w.eyz += w.az16; }
    if (mask & 4) { --w.kz; w.idx += w.stz; w.exz -= w.ax16; w.eyz -= w.ay16; }
}

HD_HD bool walk_exhausted(const Walk &w, int mask)
{
    return ((mask & 1) && w.kx == 0) || ((mask & 2) && w.ky == 0) || ((mask & 4) && w.kz == 0);
}

// Advance to the next voxel of the set; false when the set is exhausted.
HD_HD bool walk_next(Walk &w)
{
    const int pend = (w.flags >> 4) & 7;
    if (pend) {
        // the - half of a tie: those axes leave their voxels just after the
        // crossing, before any later event
        w.flags &= 7;
        if (walk_exhausted(w, pend)) return false;
        walk_apply(w, pend);
        return true;
    }
    if (w.exy != 0 && w.exz != 0 && w.eyz != 0) {
        // one axis crosses strictly first (the common case, branch-free)
        const bool cxy = w.exy < 0, cxz = w.exz < 0, cyz = w.eyz < 0;
        const bool sx = cxy && cxz;
        const bool sy = !cxy && cyz;
        const int k = sx ? w.kx : (sy ? w.ky : w.kz);
        if (k == 0) return false;
        w.kx -= sx;
        w.ky -= sy;
        w.kz -= (!sx && !sy);
        w.idx += sx ? w.stx : (sy ? w.sty : w.stz);
        w.exy += sx ? w.ay16 : (sy ? -w.ax16 : 0);
        w.exz += sx ? w.az16 : (sy ? 0 : -w.ax16);
        w.eyz += sx ? 0 : (sy ? w.az16 : -w.ay16);
        return true;
    }
    // several axes cross at the same parameter
    const int in = ((w.ax16 != 0 && w.exy <= 0 && w.exz <= 0) ? 1 : 0) |
                   ((w.ay16 != 0 && w.exy >= 0 && w.eyz <= 0) ? 2 : 0) |
                   ((w.az16 != 0 && w.exz >= 0 && w.eyz >= 0) ? 4 : 0);
    const int plus = in & w.flags & 7, minus = in & ~w.flags & 7;
    if (plus) {
        if (walk_exhausted(w, plus)) return false;
        walk_apply(w, plus);
        w.flags |= minus << 4;
        return true;
    }
    if (walk_exhausted(w, minus)) return false;
    walk_apply(w, minus);
    return true;
}

// Set up the walk of segment gi -> go (grid Q16, relative to the box
// origin) through the box [0, nx) x [0, ny) x [0, nz).  Returns false when
// the segment has no voxel in the box; otherwise w.idx is its first voxel.
HD_HD bool walk_begin(Walk &w, const int32_t gi[3], const int32_t go[3], int nx, int ny, int nz,
                      int *ijk = nullptr)
{
    const long long hx = static_cast<long long>(nx) << 16, hy = static_cast<long long>(ny) << 16,
                    hz = static_cast<long long>(nz) << 16;
    const long long x0 = gi[0], y0 = gi[1], z0 = gi[2];
    const long long dx = static_cast<long long>(go[0]) - x0;
    const long long dy = static_cast<long long>(go[1]) - y0;
    const long long dz = static_cast<long long>(go[2]) - z0;

    // t_enter = tN / tQ: the largest per-axis entry parameter
    long long tN = 0, tQ = 1;
    bool ok = true;
    auto entry = [&](long long p0, long long d, long long hi) {
        long long cN = -1, cQ = 1;
        if (d > 0) {
            if (p0 >= hi) ok = false;
            else if (p0 < 0) { cN = -p0; cQ = d; }
        } else if (d < 0) {
            if (p0 < 0) ok = false;
            else if (p0 >= hi) { cN = p0 - hi; cQ = -d; }
        } else if (p0 < 0 || p0 >= hi) {
            ok = false;
        }
        if (cN >= 0 && cN * tQ > tN * cQ) { tN = cN; tQ = cQ; }
    };
    entry(x0, dx, hx);
    entry(y0, dy, hy);
    entry(z0, dz, hz);
    if (!ok || tN > tQ) return false;

    int ix, iy, iz;
    if (tN == 0) {
        ix = static_cast<int>(x0 >> 16);
        iy = static_cast<int>(y0 >> 16);
        iz = static_cast<int>(z0 >> 16);
    } else {
        const long long den = tQ << 16;
        // voxel indices at the entry parameter: quotients below 2^15
        ix = static_cast<int>(floordiv_small(x0 * tQ + tN * dx, den));
        iy = static_cast<int>(floordiv_small(y0 * tQ + tN * dy, den));
        iz = static_cast<int>(floordiv_small(z0 * tQ + tN * dz, den));
    }
    if ((dx > 0 && ix >= nx) || (dx < 0 && ix < 0)) return false;
    if ((dy > 0 && iy >= ny) || (dy < 0 && iy < 0)) return false;
    if ((dz > 0 && iz >= nz) || (dz < 0 && iz < 0)) return false;

    long long ax, ay, az, nmx, nmy, nmz;
    {
        const int fx = go[0] >> 16, fy = go[1] >> 16, fz = go[2] >> 16;
        if (dx > 0) { ax = dx; nmx = ((static_cast<long long>(ix) + 1) << 16) - x0; w.kx = (fx < nx - 1 ? fx : nx - 1) - ix; }
        else if (dx < 0) { ax = -dx; nmx = x0 - (static_cast<long long>(ix) << 16); w.kx = ix - (fx > 0 ? fx : 0); }
        else { ax = 0; nmx = 1; w.kx = 0; }
        if (dy > 0) { ay = dy; nmy = ((static_cast<long long>(iy) + 1) << 16) - y0; w.ky = (fy < ny - 1 ? fy : ny - 1) - iy; }
        else if (dy < 0) { ay = -dy; nmy = y0 - (static_cast<long long>(iy) << 16); w.ky = iy - (fy > 0 ? fy : 0); }
        else { ay = 0; nmy = 1; w.ky = 0; }
        if (dz > 0) { az = dz; nmz = ((static_cast<long long>(iz) + 1) << 16) - z0; w.kz = (fz < nz - 1 ? fz : nz - 1) - iz; }
        else if (dz < 0) { az = -dz; nmz = z0 - (static_cast<long long>(iz) << 16); w.kz = iz - (fz > 0 ? fz : 0); }
        else { az = 0; nmz = 1; w.kz = 0; }
    }
    w.exy = nmx * ay - nmy * ax;
    w.exz = nmx * az - nmz * ax;
    w.eyz = nmy * az - nmz * ay;
    // two axes that never move never cross: give their term a fixed sign so
    // it is never read as a tie
    if (ax == 0 && ay == 0) w.exy = 1;
    if (ax == 0 && az == 0) w.exz = 1;
    if (ay == 0 && az == 0) w.eyz = 1;
    w.ax16 = ax << 16;
    w.ay16 = ay << 16;
    w.az16 = az << 16;
    w.stx = dx > 0 ? 1 : -1;
    w.sty = dy > 0 ? nx : -nx;
    w.stz = dz > 0 ? nx * ny : -(nx * ny);
    w.flags = (dx > 0 ? 1 : 0) | (dy > 0 ? 2 : 0) | (dz > 0 ? 4 : 0);
    w.idx = ix + nx * (iy + ny * iz);
    // an axis moving - that enters through the box's upper face starts one
    // voxel outside; its first crossing brings it in
    int out = (ix >= nx ? 1 : 0) | (iy >= ny ? 2 : 0) | (iz >= nz ? 4 : 0);
    const int k0x = w.kx, k0y = w.ky, k0z = w.kz;
    while (out) {
        if (!walk_next(w)) return false;
        if ((out & 1) && w.kx < k0x) out &= ~1;
        if ((out & 2) && w.ky < k0y) out &= ~2;
        if ((out & 4) && w.kz < k0z) out &= ~4;
    }
    if (ijk) {
        ijk[0] = ix + (dx > 0 ? 1 : -1) * (k0x - w.kx);
        ijk[1] = iy + (dy > 0 ? 1 : -1) * (k0y - w.ky);
        ijk[2] = iz + (dz > 0 ? 1 : -1) * (k0z - w.kz);
    }
    return true;
}

// ------------------------------------------------------------- run walk
//
// The same voxel set, produced as runs along the major in-plane axis m (x
// or y, the one with the larger |D|): only crossings of the two minor axes
// (the other in-plane axis and z) are explicit events.  For a minor axis c,
// D_c = num_c |D_m| - num_m |D_c| orders m's pending crossings against c's:
// m crosses ceil(D_c / S_c) times strictly before c does (S_c = |D_c| 2^16),
// and exactly when c does if D_c is a multiple of S_c.  D_c is kept as
// q S_c + rh 2^16 + rl: every update adds a multiple of 2^16, so rl (the low
// 16 bits) never changes and q, rh are 32-bit, updated Bresenham-style with
// no division after the set-up.  A quotient of 2^29 or more stands for
// "after the major axis has run out" (a box has at most 4096 crossings per
// axis), so q saturates there.  Events are processed in exactly the order
// and with exactly the tie rules of walk_next; crossings of m alone are
// batched.
constexpr int kQBig = 1 << 29;

struct RunWalk {
    long long e12;       // crossing order of the two minors (num_0 |D_1| - num_1 |D_0|)
    int q[2];            // D_c = q S_c + rh 2^16 + rl (q saturated at kQBig)
    unsigned rh[2];      // 0 <= rh < ad
    unsigned ad[2];      // |D_c|, so S_c = ad 2^16
    int Qu[2];           // |D_m| = Qu |D_c| + Ru (Qu saturated at kQBig)
    unsigned Ru[2];
    int km, kc[2];       // remaining valid crossings
    int im, run_start;   // major index now and where the current run began
    int row;             // row of the current run in the major axis' layout
    int rstride[2];      // signed row change when minor c crosses
    int nmaj;            // box size along the major axis
    int flags;           // bit 0: major moves +, bits 1-2: minor moves +, bits 3-4: minor
                         // moves at all, bit 5: major is y, bits 6-8: pending part,
                         // bit 9: done, bits 10-11: rl of minor c is nonzero
};

HD_HD int sat_add(int q, int d)
{
    const int v = q + d;  // both <= kQBig, so no overflow
    return v > kQBig ? kQBig : v;
}

HD_HD bool run_rpos(const RunWalk &w, int c)  // r > 0 for minor c
{
    return w.rh[c] != 0 || ((w.flags >> (10 + c)) & 1);
}

// Minor c crosses: D_c grows by |D_m| 2^16.
HD_HD void run_minor_step(RunWalk &w, int c)
{
    unsigned rh = w.rh[c] + w.Ru[c];
    int q = sat_add(w.q[c], w.Qu[c]);
    if (rh >= w.ad[c]) {
        rh -= w.ad[c];
        q = sat_add(q, 1);
    }
    w.rh[c] = rh;
    w.q[c] = q;
    --w.kc[c];
    w.row += w.rstride[c];
    if (c == 0) w.e12 += static_cast<long long>(w.ad[1]) << 16;
    else w.e12 -= static_cast<long long>(w.ad[0]) << 16;
}

// Apply one part (a set of axes crossing together) of an event: bit 0 the
// major axis, bits 1-2 the minors.  Returns 1 and the finished run when a
// minor crossed (a new row begins), 0 when only the major moved, and -1 with
// the last run when an axis in the part has no valid crossing left (end).
HD_HD int run_apply(RunWalk &w, int part, int &row, int &lo, int &hi)
{
    if (((part & 1) && w.km == 0) || ((part & 2) && w.kc[0] == 0) ||
        ((part & 4) && w.kc[1] == 0)) {
        row = w.row;
        lo = w.run_start < w.im ? w.run_start : w.im;
        hi = w.run_start < w.im ? w.im : w.run_start;
        w.flags |= 1 << 9;
        return -1;
    }
    const int im_before = w.im;
    if (part & 1) {
        w.im += (w.flags & 1) ? 1 : -1;
        --w.km;
        w.q[0] -= (w.q[0] < kQBig) ? 1 : 0;
        w.q[1] -= (w.q[1] < kQBig) ? 1 : 0;
    }
    if (!(part & 6)) return 0;
    row = w.row;
    lo = w.run_start < im_before ? w.run_start : im_before;
    hi = w.run_start < im_before ? im_before : w.run_start;
    if (part & 2) run_minor_step(w, 0);
    if (part & 4) run_minor_step(w, 1);
    w.run_start = w.im;
    return 1;
}

// General step of the run walk (every case, including ties and the end).
HD_HD bool run_next_general(RunWalk &w, int &row, int &lo, int &hi)
{
    if (w.flags & (1 << 9)) return false;
    for (;;) {
        const int pend = (w.flags >> 6) & 7;
        if (pend) {
            w.flags &= ~(7 << 6);
            const int res = run_apply(w, pend, row, lo, hi);
            if (res != 0) return true;
            continue;
        }
        const bool act0 = (w.flags >> 3) & 1, act1 = (w.flags >> 4) & 1;
        int g;  // minors in the event (bits 1-2 of a part)
        if (act0 && act1) g = w.e12 < 0 ? 2 : (w.e12 > 0 ? 4 : 6);
        else g = act0 ? 2 : (act1 ? 4 : 0);
        const bool c0 = (g & 2) != 0;  // minor 0 takes part (else minor 1)
        int j;
        if (g == 0) {
            j = kQBig;
        } else {
            const int qc = c0 ? w.q[0] : w.q[1];
            const bool rp = c0 ? run_rpos(w, 0) : run_rpos(w, 1);
            j = (qc > 0 || (qc == 0 && rp)) ? qc + (rp ? 1 : 0) : 0;
        }
        if (j > w.km) {
            // the major axis runs out before any minor crossing: last run
            w.im += (w.flags & 1) ? w.km : -w.km;
            w.km = 0;
            row = w.row;
            lo = w.run_start < w.im ? w.run_start : w.im;
            hi = w.run_start < w.im ? w.im : w.run_start;
            w.flags |= 1 << 9;
            return true;
        }
        if (j > 0) {
            w.im += (w.flags & 1) ? j : -j;
            w.km -= j;
            w.q[0] -= (w.q[0] < kQBig) ? j : 0;
            w.q[1] -= (w.q[1] < kQBig) ? j : 0;
        }
        if (g != 0 && (c0 ? (w.q[0] == 0 && !run_rpos(w, 0)) : (w.q[1] == 0 && !run_rpos(w, 1))))
            g |= 1;  // the major crosses at the same parameter
        const int posmask = w.flags & 7;
        const int plus = g & posmask, minus = g & ~posmask & 7;
        if (plus) {
            const int res = run_apply(w, plus, row, lo, hi);
            if (res < 0) return true;
            if (minus) w.flags |= minus << 6;
            if (res > 0) return true;
            continue;
        }
        const int res = run_apply(w, minus, row, lo, hi);
        if (res != 0) return true;
    }
}

// Next run of the set: returns false when there is none.  row indexes the
// run's line in the major axis' layout (x-major: y + ny z, y-major:
// x + nx z); lo..hi is the inclusive range of major indices.  The common
// case (one minor axis crossing alone after j major crossings, or the end
// of the walk) is done inline without branching on which minor crossed;
// ties and the parts they leave go to run_next_general.
HD_HD bool run_next(RunWalk &w, int &row, int &lo, int &hi)
{
    const int fl = w.flags;
    if (fl & (1 << 9)) return false;
    const bool act0 = (fl >> 3) & 1, act1 = (fl >> 4) & 1;
    if ((fl & (7 << 6)) == 0 && !(act0 && act1 && w.e12 == 0)) {
        const bool cz = !(act0 && (!act1 || w.e12 < 0));  // minor 1 crosses first
        const int qc = cz ? w.q[1] : w.q[0];
        const bool rp = cz ? run_rpos(w, 1) : run_rpos(w, 0);
        const int kcc = cz ? w.kc[1] : w.kc[0];
        const bool any = act0 || act1;
        const int j = !any ? kQBig : ((qc > 0 || (qc == 0 && rp)) ? qc + (rp ? 1 : 0) : 0);
        const bool runs_out = j > w.km;
        const bool major_tie = any && !rp && qc >= 0;
        if (runs_out || !major_tie) {
            const int ji = runs_out ? w.km : j;
            const int end = w.im + ((fl & 1) ? ji : -ji);
            row = w.row;
            lo = w.run_start < end ? w.run_start : end;
            hi = w.run_start < end ? end : w.run_start;
            if (runs_out || kcc == 0) {
                w.flags = fl | (1 << 9);
                return true;
            }
            w.km -= ji;
            w.q[0] -= (w.q[0] < kQBig) ? ji : 0;
            w.q[1] -= (w.q[1] < kQBig) ? ji : 0;
            // minor cz crosses alone
            const unsigned adc = cz ? w.ad[1] : w.ad[0];
            unsigned rh = (cz ? w.rh[1] : w.rh[0]) + (cz ? w.Ru[1] : w.Ru[0]);
            int qn = sat_add(cz ? w.q[1] : w.q[0], cz ? w.Qu[1] : w.Qu[0]);
            if (rh >= adc) {
                rh -= adc;
                qn = sat_add(qn, 1);
            }
            w.q[1] = cz ? qn : w.q[1];
            w.rh[1] = cz ? rh : w.rh[1];
            w.q[0] = cz ? w.q[0] : qn;
            w.rh[0] = cz ? w.rh[0] : rh;
            w.kc[1] -= cz ? 1 : 0;
            w.kc[0] -= cz ? 0 : 1;
            w.row += cz ? w.rstride[1] : w.rstride[0];
            w.e12 += cz ? -(static_cast<long long>(w.ad[0]) << 16)
                        : (static_cast<long long>(w.ad[1]) << 16);
            w.im = end;
            w.run_start = end;
            return true;
        }
    }
    return run_next_general(w, row, lo, hi);
}

// Set up the run walk of segment gi -> go in the box (see walk_begin).
HD_HD bool run_begin(RunWalk &rw, const int32_t gi[3], const int32_t go[3], int nx, int ny,
                     int nz)
{
    Walk w;
    int ijk[3];
    if (!walk_begin(w, gi, go, nx, ny, nz, ijk)) return false;
    const bool ymaj = w.ay16 > w.ax16;
    // axes: major m, minor 0 (the other in-plane axis), minor 1 (z)
    const unsigned am = static_cast<unsigned>((ymaj ? w.ay16 : w.ax16) >> 16);
    const unsigned a0 = static_cast<unsigned>((ymaj ? w.ax16 : w.ay16) >> 16);
    const unsigned a1 = static_cast<unsigned>(w.az16 >> 16);
    // D_c = -E_mc
    const long long d0 = ymaj ? w.exy : -w.exy;
    const long long d1 = ymaj ? -w.eyz : -w.exz;
    rw.e12 = ymaj ? w.exz : w.eyz;
    const int fl = w.flags;
    const int pm = ymaj ? ((fl >> 1) & 1) : (fl & 1);
    const int p0 = ymaj ? (fl & 1) : ((fl >> 1) & 1);
    const int p1 = (fl >> 2) & 1;
    int flags = pm | (p0 << 1) | (p1 << 2) | ((a0 != 0) << 3) | ((a1 != 0) << 4) | (ymaj << 5);
    const int pend = (fl >> 4) & 7;  // pending - part of walk_begin, in x,y,z bits
    if (pend) {
        const int bm = ymaj ? ((pend >> 1) & 1) : (pend & 1);
        const int b0 = ymaj ? (pend & 1) : ((pend >> 1) & 1);
        const int b1 = (pend >> 2) & 1;
        flags |= (bm | (b0 << 1) | (b1 << 2)) << 6;
    }
    rw.km = ymaj ? w.ky : w.kx;
    rw.kc[0] = ymaj ? w.kx : w.ky;
    rw.kc[1] = w.kz;
    const unsigned A[2] = {a0, a1};
    const long long Dc[2] = {d0, d1};
#pragma unroll
    for (int c = 0; c < 2; ++c) {
        if (A[c] != 0) {
            rw.ad[c] = A[c];
            const unsigned qu = am / A[c];
            rw.Qu[c] = qu >= (1u << 20) ? kQBig : static_cast<int>(qu);
            rw.Ru[c] = am - qu * A[c];
            // D = Dh 2^16 + Dl with 0 <= Dl < 2^16, q = floor(Dh / ad)
            const long long dh = Dc[c] >> 16;
            const unsigned dl = static_cast<unsigned>(Dc[c] & 0xffff);
            if (float_of(dh) >= 1048576.0f * static_cast<float>(A[c])) {
                rw.q[c] = kQBig;
                rw.rh[c] = 1;  // any remainder > 0: never a tie
            } else {
                const long long q = floordiv_small(dh, static_cast<long long>(A[c]));
                rw.q[c] = static_cast<int>(q);
                rw.rh[c] = static_cast<unsigned>(dh - q * static_cast<long long>(A[c]));
            }
            if (dl != 0) flags |= 1 << (10 + c);
        } else {
            rw.ad[c] = 1;
            rw.Qu[c] = kQBig;
            rw.Ru[c] = 0;
            rw.q[c] = kQBig;
            rw.rh[c] = 0;
            flags |= 1 << (10 + c);
        }
    }
    rw.flags = flags;
    if (!ymaj) {
        rw.im = ijk[0];
        rw.row = ijk[1] + ny * ijk[2];
        rw.rstride[0] = (fl & 2) ? 1 : -1;
        rw.rstride[1] = (fl & 4) ? ny : -ny;
        rw.nmaj = nx;
    } else {
        rw.im = ijk[1];
        rw.row = ijk[0] + nx * ijk[2];
        rw.rstride[0] = (fl & 1) ? 1 : -1;
        rw.rstride[1] = (fl & 4) ? nx : -nx;
        rw.nmaj = ny;
    }
    rw.run_start = rw.im;
    return true;
}

// -------------------------------------------------------------- path walk
//
// The whole-grid walk of one path as runs in path order, for segments with no
// tie (nearly all): both minors cross between two major crossings, never at
// the same parameter as one, and never together.  Counting major crossings
// from the start, minor 0's next crossing comes after jn of them and z's after
// jz (Bresenham steps of 32-bit integers, as in the lean walks below); when
// both fall between the same two, the sign of e12 (advanced from the crossings
// so far, only then) tells which comes first.  These are exactly the runs
// run_next produces; a run costs about 20 instructions where the general step,
// with its 64-bit order term and its saturated quotients, took about 90.
struct PathWalk {
    unsigned ad, Ru, rem;     // |D_0|, |D_m| mod |D_0|, Bresenham remainder
    unsigned adz, Ruz, remz;  // the same for z
    int jn, Qu, jz, Quz;      // next crossings, and |D_m| div |D_c| (capped)
    int km, kc, kz;           // valid crossings left: major in all, minor 0, z
    int im0;                  // major index of the first voxel
    uint32_t vb;              // voxel of major index 0 in the current row
    int fl;                   // bit 0 major +, 1 minor 0 +, 2 z +, 3 major is y
    long long e12;            // order of minor 0 against z at the start (< 0: minor 0 first)
    int c0, z0;               // kc and kz at the start
    int s;                    // major crossings before the current run
};
constexpr int kPathWords = 16;  // packed size (64 bytes)

// The path walk of gi -> go (grid Q16) over the grid: 1, 0 (no voxel), or -1
// (a tie, or no in-plane motion: the general run walk).  The set-up is
// slab_lean's with z an axis like the others.
HD_HD int path_lean(const int32_t gi[3], const int32_t go[3], int nx, int ny, int nz, PathWalk &L)
{
    const int P[3] = {gi[0], gi[1], gi[2]};
    const int D[3] = {go[0] - gi[0], go[1] - gi[1], go[2] - gi[2]};
    const int n[3] = {nx, ny, nz};
    if (D[0] == 0 && D[1] == 0) return -1;
    unsigned tN = 0, tQ = 1;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        const int H = n[a] << 16;
        unsigned cN = 0, cQ = 1;
        bool cand = false;
        if (D[a] > 0) {
            if (P[a] >= H) return 0;
            if (P[a] < 0) { cN = static_cast<unsigned>(-P[a]); cQ = static_cast<unsigned>(D[a]); cand = true; }
        } else if (D[a] < 0) {
            if (P[a] < 0) return 0;
            if (P[a] >= H) { cN = static_cast<unsigned>(P[a] - H); cQ = static_cast<unsigned>(-D[a]); cand = true; }
        } else if (P[a] < 0 || P[a] >= H) {
            return 0;
        }
        if (cand && static_cast<unsigned long long>(cN) * tQ > static_cast<unsigned long long>(tN) * cQ) {
            tN = cN;
            tQ = cQ;
        }
    }
    if (tN > tQ) return 0;
    int idx[3];
    bool onp[3];
    const float rQ = rcp_int(static_cast<int>(tQ));
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        const long long num = static_cast<long long>(P[a]) * tQ + static_cast<long long>(tN) * D[a];
        long long rem;
        idx[a] = fdiv32(num >> 16, static_cast<int>(tQ), rQ, rem);
        onp[a] = rem == 0 && (num & 0xffff) == 0;
    }
#pragma unroll
    for (int a = 0; a < 3; ++a)
        if ((D[a] > 0 && idx[a] >= n[a]) || (D[a] < 0 && idx[a] < 0)) return 0;
    // an axis moving - that enters through its upper face (see slab_lean)
    int out = -1;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        if (idx[a] >= n[a]) {
            if (out >= 0) return -1;
            out = a;
        }
    }
    if (out >= 0) {
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            if (a != out && D[a] < 0 && onp[a]) return -1;
            if (a == out) idx[a] -= 1;
        }
    }
    int nm[3], k[3];
    unsigned A[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        const int f = go[a] >> 16;
        const bool pos = D[a] > 0, neg = D[a] < 0;
        A[a] = pos ? static_cast<unsigned>(D[a]) : (neg ? static_cast<unsigned>(-D[a]) : 0u);
        nm[a] = pos ? ((idx[a] + 1) << 16) - P[a] : (neg ? P[a] - (idx[a] << 16) : 1);
        k[a] = pos ? (f < n[a] - 1 ? f : n[a] - 1) - idx[a] : (neg ? idx[a] - (f > 0 ? f : 0) : 0);
    }
    if (k[0] < 0 || k[1] < 0 || k[2] < 0) return 0;  // the walk ends where it enters
    const bool ymaj = A[1] > A[0];
    const unsigned am = ymaj ? A[1] : A[0], a0 = ymaj ? A[0] : A[1], a1 = A[2];
    const long long nmm = ymaj ? nm[1] : nm[0], nmc = ymaj ? nm[0] : nm[1], nmz = nm[2];
    // minor against the major axis: the quotient and remainder of its first
    // crossing, and of the step to the next
    auto minor = [&](unsigned a, long long d, int &j, unsigned &rem, int &Qu, unsigned &Ru) {
        j = kQBig;
        rem = 0;
        Qu = kQBig;
        Ru = 0;
        if (a == 0) return true;
        if ((d & 0xffff) == 0) return false;  // may tie with the major axis
        const unsigned qu = am / a;
        Qu = qu >= (1u << 20) ? kQBig : static_cast<int>(qu);
        Ru = am - qu * a;
        const long long dh = d >> 16;
        if (float_of(dh) < 1048576.0f * static_cast<float>(a)) {
            long long rm;
            const int q = fdiv32(dh, static_cast<int>(a), rcp_int(static_cast<int>(a)), rm);
            if (q < -1) return false;
            j = q + 1;
            rem = static_cast<unsigned>(rm);
        }
        return true;
    };
    if (!minor(a0, nmc * am - nmm * a0, L.jn, L.rem, L.Qu, L.Ru)) return -1;
    if (!minor(a1, nmz * am - nmm * a1, L.jz, L.remz, L.Quz, L.Ruz)) return -1;
    L.e12 = a0 == 0 ? 1 : (a1 == 0 ? -1 : nmc * a1 - nmz * a0);
    if (a0 != 0 && a1 != 0 && (L.e12 & 0xffff) == 0) return -1;  // the minors may tie
    constexpr int kCap = 16383, kQuCap = 8192;  // beyond any box: never reached
    L.jn = L.jn < kCap ? L.jn : kCap;
    L.jz = L.jz < kCap ? L.jz : kCap;
    L.Qu = L.Qu < kQuCap ? L.Qu : kQuCap;
    L.Quz = L.Quz < kQuCap ? L.Quz : kQuCap;
    L.ad = a0 != 0 ? a0 : 1u;
    L.adz = a1 != 0 ? a1 : 1u;
    L.km = ymaj ? k[1] : k[0];
    L.kc = L.c0 = ymaj ? k[0] : k[1];
    L.kz = L.z0 = k[2];
    L.im0 = ymaj ? idx[1] : idx[0];
    L.vb = static_cast<uint32_t>(ymaj ? idx[0] : nx * idx[1]) +
           static_cast<uint32_t>(nx) * static_cast<uint32_t>(ny) * static_cast<uint32_t>(idx[2]);
    L.fl = ((ymaj ? D[1] : D[0]) > 0 ? 1 : 0) | ((ymaj ? D[0] : D[1]) > 0 ? 2 : 0) |
           (D[2] > 0 ? 4 : 0) | (ymaj ? 8 : 0);
    L.s = 0;
    return 1;
}

HD_HD void path_pack(const PathWalk &L, uint32_t o[kPathWords])
{
    o[0] = L.ad;
    o[1] = L.Ru;
    o[2] = L.rem;
    o[3] = L.adz;
    o[4] = L.Ruz;
    o[5] = L.remz;
    o[6] = static_cast<uint32_t>(L.jn) | (static_cast<uint32_t>(L.Qu) << 16);
    o[7] = static_cast<uint32_t>(L.jz) | (static_cast<uint32_t>(L.Quz) << 16);
    o[8] = static_cast<uint32_t>(L.km) | (static_cast<uint32_t>(L.kc) << 16);
    o[9] = static_cast<uint32_t>(L.kz) | (static_cast<uint32_t>(L.im0) << 16);
    o[10] = L.vb;
    o[11] = static_cast<uint32_t>(L.fl);
    o[12] = static_cast<uint32_t>(static_cast<unsigned long long>(L.e12) & 0xffffffffull);
    o[13] = static_cast<uint32_t>(static_cast<unsigned long long>(L.e12) >> 32);
    o[14] = o[15] = 0;
}

HD_HD void path_unpack(const uint32_t o[kPathWords], PathWalk &L)
{
    L.ad = o[0];
    L.Ru = o[1];
    L.rem = o[2];
    L.adz = o[3];
    L.Ruz = o[4];
    L.remz = o[5];
    L.jn = static_cast<int>(o[6] & 0xffffu);
    L.Qu = static_cast<int>(o[6] >> 16);
    L.jz = static_cast<int>(o[7] & 0xffffu);
    L.Quz = static_cast<int>(o[7] >> 16);
    L.km = static_cast<int>(o[8] & 0xffffu);
    L.kc = L.c0 = static_cast<int>(o[8] >> 16);
    L.kz = L.z0 = static_cast<int>(o[9] & 0xffffu);
    L.im0 = static_cast<int>(o[9] >> 16);
    L.vb = o[10];
    L.fl = static_cast<int>(o[11]);
    L.e12 = static_cast<long long>((static_cast<unsigned long long>(o[13]) << 32) | o[12]);
    L.s = 0;
}

// When minor 0 and z both cross between the same two major crossings: whether z
// does first.
HD_HD bool path_z_first(const PathWalk &L)
{
    return L.e12 + ((static_cast<long long>(L.c0 - L.kc) * L.adz) << 16) -
               ((static_cast<long long>(L.z0 - L.kz) * L.ad) << 16) >
           0;
}

// The current run: vb the voxel of major index 0 in its row, a .. b its major
// indices in path order (a > b when the major axis moves -).  Returns whether
// more runs follow.
HD_HD bool path_run(PathWalk &L, int nx, int plane, uint32_t &vb, int &a, int &b)
{
    const int j = L.jn < L.jz ? L.jn : L.jz;
    const bool out = j > L.km;
    const int e = out ? L.km : j;
    vb = L.vb;
    a = (L.fl & 1) ? L.im0 + L.s : L.im0 - L.s;
    b = (L.fl & 1) ? L.im0 + e : L.im0 - e;
    if (out) return false;
    bool zc = L.jz < L.jn;
    if (L.jz == L.jn) zc = path_z_first(L);
    L.s = e;
    if (!zc) {
        if (L.kc == 0) return false;
        --L.kc;
        const int st = (L.fl & 8) ? 1 : nx;
        L.vb += static_cast<uint32_t>((L.fl & 2) ? st : -st);
        L.rem += L.Ru;
        const bool carry = L.rem >= L.ad;
        L.rem = carry ? L.rem - L.ad : L.rem;
        L.jn += L.Qu + (carry ? 1 : 0);
    } else {
        if (L.kz == 0) return false;
        --L.kz;
        L.vb += static_cast<uint32_t>((L.fl & 4) ? plane : -plane);
        L.remz += L.Ruz;
        const bool carry = L.remz >= L.adz;
        L.remz = carry ? L.remz - L.adz : L.remz;
        L.jz += L.Quz + (carry ? 1 : 0);
    }
    return true;
}

// ---------------------------------------------------------- lean run walk
//
// Most walks inside a one-voxel-deep tile are "lean": the in-plane minor
// axis (minor 0) never crosses at the same parameter as the major axis
// (rl_0 != 0: D_0 is never a multiple of S_0), z never ties with the major
// axis (rl_1 != 0) nor with minor 0 (e12 is never a multiple of 2^16, and
// every update adds one), no tie is pending at the start, and z has no valid
// crossing inside the box, so its first crossing (if any) ends the walk.
// Then every event is a lone crossing and the runs have a closed form.
// Counting major crossings from the start, minor 0's k-th crossing (k >= 1)
// comes after J_k = q_0 + 1 + (k - 1) Qu_0 + floor((rh_0 + (k - 1) Ru_0) / ad_0)
// of them (so J_1 = q_0 + 1, and J_{k+1} = J_k + Qu_0 + carry, Bresenham
// style); z crosses after j_z = q_1 + 1; the major axis runs out after km.
// Crossing k of minor 0 happens iff k <= K = min(kc_0, K_z), K_z being the
// number of minor-0 crossings before z's (from the sign of
// e12 + k ad_1 2^16), and J_k <= km.  Run k (k = 0, 1, ...) covers major
// counts J_k .. J_{k+1} (J_0 = 0) in row row_0 + k s_0 (s_0 the signed
// minor-0 row stride), the last ending at min(J_{k+1}, km, j_z) instead.
// These are exactly the runs run_next produces.  With kmz = min(km, j_z),
// run k is the last iff k = K or J_{k+1} > kmz (a crossing k + 1 <= K_z comes
// no later than z's), and it ends at min(J_{k+1}, kmz).
struct LeanWalk {
    unsigned ad, Ru, rem;  // |D_0|, |D_m| mod |D_0|, (rh_0 + k Ru_0) mod ad_0
    int jn;                // J_{k+1} (capped: any value above kmz acts alike)
    int Qu;                // floor(|D_m| / |D_0|), capped at kLeanQuCap
    int kmz;               // min(km, j_z)
    int kleft, K;          // crossings of minor 0 left, and in all
    int s;                 // J_k: where the current run starts
    int im0;               // major index of the first voxel
    int row;               // row of the current run (major axis' layout)
    int fl;                // bit 0 major +, bit 1 minor 0 +, bit 2 major is y, bit 3 empty
};
constexpr int kLeanWords = 8;   // packed size (32 bytes)
constexpr int kLeanQuCap = 8192;  // > any box extent (4096): one step beyond the box suffices
constexpr int kLeanJCap = 16383;

// The lean form of a freshly begun walk, when it has one.
HD_HD bool lean_of(const RunWalk &w, LeanWalk &L)
{
    const int fl = w.flags;
    if (fl & ((7 << 6) | (1 << 9))) return false;  // a tie pending, or empty
    const bool act0 = (fl >> 3) & 1, act1 = (fl >> 4) & 1;
    if (w.kc[1] != 0) return false;                            // z crosses inside the box
    if (!((fl >> 10) & 1) || !((fl >> 11) & 1)) return false;  // a tie with the major axis
    if (w.q[0] < -1 || w.q[1] < -1) return false;
    int kz;  // minor-0 crossings before z's
    if (!act0) {
        kz = 0;
    } else if (!act1) {
        kz = w.kc[0];
    } else {
        if ((w.e12 & 0xffff) == 0) return false;  // minor 0 and z may tie
        if (w.e12 > 0) {
            kz = 0;
        } else {
            // ceil(-e12 / step) = floor((-e12 - 1) / step) + 1 (e12 < 0), needed
            // only up to kc_0 <= 4096: a float estimate settles larger ones
            const long long step = static_cast<long long>(w.ad[1]) << 16;
            const long long num = -w.e12 - 1;
            if (float_of(num) >= (static_cast<float>(w.kc[0]) + 2.0f) * float_of(step)) {
                kz = w.kc[0];
            } else {
                const long long n = floordiv_small(num, step) + 1;
                kz = n < w.kc[0] ? static_cast<int>(n) : w.kc[0];
            }
        }
    }
    L.K = act0 ? (kz < w.kc[0] ? kz : w.kc[0]) : 0;
    L.kleft = L.K;
    const int jz = act1 ? w.q[1] + 1 : kQBig;
    L.kmz = w.km < jz ? w.km : jz;
    const int j1 = act0 ? w.q[0] + 1 : kQBig;
    L.jn = j1 < kLeanJCap ? j1 : kLeanJCap;
    L.Qu = w.Qu[0] < kLeanQuCap ? w.Qu[0] : kLeanQuCap;
    L.ad = w.ad[0];
    L.Ru = w.Ru[0];
    L.rem = w.rh[0];
    L.s = 0;
    L.im0 = w.im;
    L.row = w.row;
    L.fl = (fl & 3) | (((fl >> 5) & 1) << 2);
    return true;
}

HD_HD void lean_pack(const LeanWalk &L, uint32_t o[kLeanWords])
{
    o[0] = L.ad;
    o[1] = L.Ru;
    o[2] = L.rem;
    o[3] = static_cast<uint32_t>(L.jn) | (static_cast<uint32_t>(L.Qu) << 16);
    o[4] = static_cast<uint32_t>(L.kmz) | (static_cast<uint32_t>(L.K) << 16);
    o[5] = static_cast<uint32_t>(L.im0) | (static_cast<uint32_t>(L.fl) << 16);
    o[6] = static_cast<uint32_t>(L.row);
    o[7] = 0;
}

// The lean walk of the segment gi -> go (grid Q16, relative to the box
// origin) in a one-slice box [0, nx) x [0, ny) x [0, 1), computed directly:
// the same LeanWalk as lean_of(run_begin(...)) gives, without the general
// set-up's machinery.  In a one-slice box z never crosses inside (its only
// crossing ends the walk), the z index at the entry point is 0 or 1 (one
// comparison), the axis that sets the entry parameter needs no division,
// and z's crossing matters only through j_z, so its major-step quotient is
// not needed.  An axis moving - that enters through its upper face starts
// one voxel outside and takes that crossing first (as walk_begin does);
// when another axis moving - is exactly on a plane at the entry (a tie) or
// two axes enter that way, and for walks without in-plane motion, it
// returns -1 and the caller takes the general set-up.  Returns 1 (lean, L
// filled), 0 (no voxel in the box) or -1 (use run_begin and lean_of).
HD_HD int slab_lean(const int32_t gi[3], const int32_t go[3], int nx, int ny, LeanWalk &L)
{
    // 32-bit storage throughout (|P| < 2^30, |D| < 2^31, plane distances
    // below 2^31); only products are 64-bit
    const int P[3] = {gi[0], gi[1], gi[2]};
    const int D[3] = {go[0] - gi[0], go[1] - gi[1], go[2] - gi[2]};
    const int n[3] = {nx, ny, 1};
    const int H[3] = {nx << 16, ny << 16, 1 << 16};
    if (D[0] == 0 && D[1] == 0) return -1;
    // entry parameter tN / tQ (the largest per-axis entry) and its axis
    unsigned tN = 0, tQ = 1;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        unsigned cN = 0, cQ = 1;
        bool cand = false;
        if (D[a] > 0) {
            if (P[a] >= H[a]) return 0;
            if (P[a] < 0) { cN = static_cast<unsigned>(-P[a]); cQ = static_cast<unsigned>(D[a]); cand = true; }
        } else if (D[a] < 0) {
            if (P[a] < 0) return 0;
            if (P[a] >= H[a]) { cN = static_cast<unsigned>(P[a] - H[a]); cQ = static_cast<unsigned>(-D[a]); cand = true; }
        } else if (P[a] < 0 || P[a] >= H[a]) {
            return 0;
        }
        if (cand && static_cast<unsigned long long>(cN) * tQ > static_cast<unsigned long long>(tN) * cQ) {
            tN = cN;
            tQ = cQ;
        }
    }
    if (tN > tQ) return 0;
    // voxel indices at the entry point, and whether that point lies on a
    // plane of each axis (remainder 0)
    int idx[3];
    bool onp[3];
    const long long den = static_cast<long long>(tQ) << 16;
    const float rQ = rcp_int(static_cast<int>(tQ));
    // the entry point's coordinate along each axis, P tQ + tN D over den
    // (also right for the entry axis and when the segment starts inside)
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        const long long num = static_cast<long long>(P[a]) * tQ + static_cast<long long>(tN) * D[a];
        if (a == 2) {
            idx[2] = num < 0 ? -1 : (num >= den ? 1 : 0);
            onp[2] = num == 0 || num == den;
        } else {
            long long rem;
            idx[a] = fdiv32(num >> 16, static_cast<int>(tQ), rQ, rem);
            onp[a] = rem == 0 && (num & 0xffff) == 0;
        }
    }
#pragma unroll
    for (int a = 0; a < 3; ++a)
        if ((D[a] > 0 && idx[a] >= n[a]) || (D[a] < 0 && idx[a] < 0)) return 0;
    // an axis moving - that enters through its upper face starts one voxel
    // outside; its crossing at the entry parameter comes first unless another
    // axis moving - is on a plane there too (a tie: general set-up)
    int out = -1;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        if (idx[a] >= n[a]) {
            if (out >= 0) return -1;
            out = a;
        }
    }
    if (out >= 0) {
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            if (a != out && D[a] < 0 && onp[a]) return -1;
            if (a == out) idx[a] -= 1;
        }
    }
    // distances from the segment's start to each axis' next plane, and the
    // crossings left inside the box
    int nm[3], k[3];
    unsigned A[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        const int f = go[a] >> 16;
        const bool pos = D[a] > 0, neg = D[a] < 0;
        A[a] = pos ? static_cast<unsigned>(D[a]) : (neg ? static_cast<unsigned>(-D[a]) : 0u);
        nm[a] = pos ? ((idx[a] + 1) << 16) - P[a] : (neg ? P[a] - (idx[a] << 16) : 1);
        k[a] = pos ? (f < n[a] - 1 ? f : n[a] - 1) - idx[a] : (neg ? idx[a] - (f > 0 ? f : 0) : 0);
    }
    if (k[0] < 0 || k[1] < 0 || k[2] < 0) return 0;  // the walk ends where it enters
    if (k[2] != 0) return -1;
    // axes: major m, minor 0 (the other in-plane axis), minor 1 (z); every
    // array is read at constant indices (a runtime index would put it in
    // local memory)
    const bool ymaj = A[1] > A[0];
    const unsigned am = ymaj ? A[1] : A[0];
    const unsigned a0 = ymaj ? A[0] : A[1];
    const unsigned a1 = A[2];
    const long long nmm = ymaj ? nm[1] : nm[0], nmc = ymaj ? nm[0] : nm[1];
    const long long nmz = nm[2];
    // crossing-order terms against the major axis (D_c of run_begin), and
    // between the minors (e12); two axes that never move never cross
    const long long d0 = a0 == 0 ? -1 : nmc * am - nmm * a0;
    const long long d1 = a1 == 0 ? -1 : nmz * am - nmm * a1;
    const long long e12 = (a0 == 0 && a1 == 0) ? 1 : nmc * a1 - nmz * a0;
    const bool act0 = a0 != 0, act1 = a1 != 0;
    int q0 = kQBig, q1 = kQBig;
    unsigned rh0 = 0, Ru0 = 0;
    int Qu0 = kQBig;
    if (act0) {
        if ((d0 & 0xffff) == 0) return -1;  // minor 0 may tie with the major axis
        const unsigned qu = am / a0;
        Qu0 = qu >= (1u << 20) ? kQBig : static_cast<int>(qu);
        Ru0 = am - qu * a0;
        const long long dh = d0 >> 16;
        if (float_of(dh) >= 1048576.0f * static_cast<float>(a0)) {
            q0 = kQBig;
            rh0 = 1;
        } else {
            long long rem;
            q0 = fdiv32(dh, static_cast<int>(a0), rcp_int(static_cast<int>(a0)), rem);
            rh0 = static_cast<unsigned>(rem);
        }
    }
    const float r1 = act1 ? rcp_int(static_cast<int>(a1)) : 0.0f;
    if (act1) {
        if ((d1 & 0xffff) == 0) return -1;  // z may tie with the major axis
        const long long dh = d1 >> 16;
        if (float_of(dh) >= 1048576.0f * static_cast<float>(a1)) {
            q1 = kQBig;
        } else {
            long long rem;
            q1 = fdiv32(dh, static_cast<int>(a1), r1, rem);
        }
    }
    if (q0 < -1 || q1 < -1) return -1;
    const int km = ymaj ? k[1] : k[0], kc0 = ymaj ? k[0] : k[1];
    int kz;  // minor-0 crossings before z's
    if (!act0) {
        kz = 0;
    } else if (!act1) {
        kz = kc0;
    } else {
        if ((e12 & 0xffff) == 0) return -1;  // minor 0 and z may tie
        if (e12 > 0) {
            kz = 0;
        } else {
            const long long step = static_cast<long long>(a1) << 16;
            const long long num = -e12 - 1;
            if (float_of(num) >= (static_cast<float>(kc0) + 2.0f) * float_of(step)) {
                kz = kc0;
            } else {
                // floor(num / (a1 2^16)) = floor(floor(num / 2^16) / a1)
                long long rem;
                const int q = fdiv32(num >> 16, static_cast<int>(a1), r1, rem) + 1;
                kz = q < kc0 ? q : kc0;
            }
        }
    }
    L.K = act0 ? (kz < kc0 ? kz : kc0) : 0;
    L.kleft = L.K;
    const int jz = act1 ? q1 + 1 : kQBig;
    L.kmz = km < jz ? km : jz;
    const int j1 = act0 ? q0 + 1 : kQBig;
    L.jn = j1 < kLeanJCap ? j1 : kLeanJCap;
    L.Qu = Qu0 < kLeanQuCap ? Qu0 : kLeanQuCap;
    L.ad = act0 ? a0 : 1u;
    L.Ru = Ru0;
    L.rem = rh0;
    L.s = 0;
    L.im0 = ymaj ? idx[1] : idx[0];
    L.row = ymaj ? idx[0] : idx[1];
    const bool pm = (ymaj ? D[1] : D[0]) > 0, pc = (ymaj ? D[0] : D[1]) > 0;
    L.fl = (pm ? 1 : 0) | ((pc ? 1 : 0) << 1) | ((ymaj ? 1 : 0) << 2);
    return 1;
}

HD_HD void lean_unpack(const uint32_t o[kLeanWords], LeanWalk &L)
{
    L.ad = o[0];
    L.Ru = o[1];
    L.rem = o[2];
    L.jn = static_cast<int>(o[3] & 0xffffu);
    L.Qu = static_cast<int>(o[3] >> 16);
    L.kmz = static_cast<int>(o[4] & 0xffffu);
    L.K = static_cast<int>(o[4] >> 16);
    L.kleft = L.K;
    L.im0 = static_cast<int>(o[5] & 0xffffu);
    L.fl = static_cast<int>(o[5] >> 16);
    L.row = static_cast<int>(o[6]);
    L.s = 0;
}

HD_HD bool lean_empty(const LeanWalk &L) { return (L.fl >> 3) & 1; }

// The traversal kernel's form of a lean walk: the same runs, with the row
// offset (row * nmaj), the run's start and the direction kept as signed
// increments so that a run costs a few integer operations.
struct LeanCursor {
    unsigned ad, Ru, rem;  // as in LeanWalk
    int jn, Qu, kmz, kleft;
    int im0, sg;  // major index of the first voxel, major direction (+1 or -1)
    int ms;       // major index where the current run starts
    int rb;       // row * nmaj of the current run
    int rstep;    // change of rb per minor-0 crossing (+nmaj or -nmaj)
};

// A packed lean walk as a cursor over rows of nmaj voxels (nmaj: the box's
// extent along the walk's major axis).  Returns false for an empty walk.
HD_HD bool lean_start(const uint32_t o[kLeanWords], int nmaj, LeanCursor &c)
{
    const int fl = static_cast<int>(o[5] >> 16);
    c.ad = o[0];
    c.Ru = o[1];
    c.rem = o[2];
    c.jn = static_cast<int>(o[3] & 0xffffu);
    c.Qu = static_cast<int>(o[3] >> 16);
    c.kmz = static_cast<int>(o[4] & 0xffffu);
    c.kleft = static_cast<int>(o[4] >> 16);
    c.im0 = static_cast<int>(o[5] & 0xffffu);
    c.sg = (fl & 1) ? 1 : -1;
    c.ms = c.im0;
    c.rb = static_cast<int>(o[6]) * nmaj;
    c.rstep = (fl & 2) ? nmaj : -nmaj;
    return !((fl >> 3) & 1);
}

// The current run: *rb its row offset, lo..hi its major range (inclusive).
// Returns whether more runs follow.  With the last run it adds e (the major
// count where the walk ends) to `ends`: the walk's voxel count is e plus its
// number of runs (see lean_step), so a caller that counts the runs gets the
// voxels as runs + ends.  Branch-free: the cursor also advances past the
// last run, where it is not used again.
HD_HD bool lean_run(LeanCursor &c, int &rb, int &lo, int &hi, unsigned &ends)
{
    const int jn = c.jn;
    const int e = jn < c.kmz ? jn : c.kmz;
    const int b = c.im0 + c.sg * e;
    lo = c.ms < b ? c.ms : b;
    hi = c.ms < b ? b : c.ms;
    rb = c.rb;
    const bool last = c.kleft == 0 || jn > c.kmz;
    ends += last ? static_cast<unsigned>(e) : 0u;
    c.ms = b;  // before the last run e = jn: the next run starts where this one ends
    const unsigned rem = c.rem + c.Ru;
    const bool carry = rem >= c.ad;
    c.rem = carry ? rem - c.ad : rem;
    c.jn = jn + c.Qu + (carry ? 1 : 0);
    --c.kleft;
    c.rb += c.rstep;
    return !last;
}

// The current run of a non-empty lean walk: row, and the inclusive range
// lo..hi of major indices.  Returns whether more runs follow; with the last
// run it adds the walk's voxel count (e + K + 1: the major cells covered
// plus one per row change) to `steps`.
HD_HD bool lean_step(LeanWalk &L, int &row, int &lo, int &hi, unsigned &steps)
{
    const int jn = L.jn;
    const int e = jn < L.kmz ? jn : L.kmz;
    const int a = (L.fl & 1) ? L.im0 + L.s : L.im0 - L.s;
    const int b = (L.fl & 1) ? L.im0 + e : L.im0 - e;
    lo = a < b ? a : b;
    hi = a < b ? b : a;
    row = L.row;
    if (L.kleft == 0 || jn > L.kmz) {
        steps += static_cast<unsigned>(e + (L.K - L.kleft) + 1);
        return false;
    }
    L.s = jn;
    const unsigned rem = L.rem + L.Ru;
    const bool carry = rem >= L.ad;
    L.rem = carry ? rem - L.ad : rem;
    L.jn = jn + L.Qu + (carry ? 1 : 0);
    --L.kleft;
    L.row += (L.fl & 2) ? 1 : -1;
    return true;
}

// The updates of a joined tile (below) stated run by run, as the host tests check
// them; the traversal itself takes them from event walks (JoinedCursor).  The
// same runs as lean_run, as byte offsets into a tile box of dx x dy x dz voxels stored one 32-bit
// word per voxel, x fastest, with one padding column and one padding row:
// word(x, y, z) = x + Wx (y + Hy z), Wx = dx + 1, Hy = dy + 1.  A run adds
// inc (1 for runs along x, 65536 for runs along y: the two halves of a
// word) at its first voxel and subtracts it just past its last one, which
// for a run ending at the box's edge lies in the padding.  Consecutive runs
// share a major index (the walk changes row there), so a run is fixed by
// the major positions b_prev (where it starts in walk order) and b (where
// it ends): with the major axis moving +, inc goes at b_prev and -inc just
// past b; moving -, inc goes at b and -inc just past b_prev.  The cursor
// keeps the row base and the positions as byte offsets (plus a base the
// caller chooses, such as the tile's shared-memory address) and the two
// per-walk offsets and values that this choice implies, so a run costs a
// few integer steps and no comparison of its ends.
struct TileCursor {
    unsigned ad, Ru, rem;  // Bresenham state of minor 0 (as in LeanWalk)
    int jn, Qu, kmz, kleft;
    int m0b;    // byte offset of the first voxel's major index within its row
    int sgm;    // signed bytes per major step
    int bprev;  // byte offset of the current run's start (walk order) in its row
    int rowb;   // base + byte offset of the current row's major index 0
    int rstep;  // change of rowb per minor-0 crossing
    int oprev, ocur;     // byte offsets added to the run's ends: 0 or one major step
    uint32_t vprev, vcur;  // values added there: inc and -inc, in walk order
};

// Start a packed lean walk (lean_pack's form) in a box of dx x dy x dz
// voxels whose word 0 is at byte address `base`; false for an empty walk.
HD_HD bool tile_cursor_start(const uint32_t o[kLeanWords], int dx, int dy, int dz, int base,
                             TileCursor &c)
{
    const int fl = static_cast<int>(o[5] >> 16);
    const bool ymaj = (fl >> 2) & 1;
    const bool plus = fl & 1;
    const int Wx = dx + 1, Hy = dy + 1;
    c.ad = o[0];
    c.Ru = o[1];
    c.rem = o[2];
    c.jn = static_cast<int>(o[3] & 0xffffu);
    c.Qu = static_cast<int>(o[3] >> 16);
    c.kmz = static_cast<int>(o[4] & 0xffffu);
    c.kleft = static_cast<int>(o[4] >> 16);
    const int im0 = static_cast<int>(o[5] & 0xffffu);
    // the row in the major axis' layout of the box: x-major y + dy z,
    // y-major x + dx z; a lean walk never changes z
    const int row = static_cast<int>(o[6]);
    const int nminor = ymaj ? dx : dy;
    const int z = dz == 1 ? 0 : row / nminor;
    const int a = row - z * nminor;  // the minor-0 index (y for x-major, x for y-major)
    const int mstep = ymaj ? 4 * Wx : 4;
    c.sgm = plus ? mstep : -mstep;
    c.m0b = im0 * mstep;
    c.bprev = c.m0b;
    c.rowb = base + (ymaj ? 4 * (a + Wx * Hy * z) : 4 * Wx * (a + Hy * z));
    const int rs = ymaj ? 4 : 4 * Wx;
    c.rstep = (fl & 2) ? rs : -rs;
    const uint32_t inc = ymaj ? 65536u : 1u;
    c.oprev = plus ? 0 : mstep;
    c.ocur = plus ? mstep : 0;
    c.vprev = plus ? inc : 0u - inc;
    c.vcur = plus ? 0u - inc : inc;
    return !((fl >> 3) & 1);
}

// The current run: vprev is added at byte address `at_prev` and vcur at
// `at_cur`.  Returns whether more runs follow.  Past its last run the
// cursor holds kleft = (crossings left at the start) - (runs walked).
HD_HD bool tile_cursor_run(TileCursor &c, int &at_prev, int &at_cur)
{
    const int jn = c.jn;
    const int e = jn < c.kmz ? jn : c.kmz;
    const int b = c.m0b + c.sgm * e;
    at_prev = c.rowb + c.bprev + c.oprev;
    at_cur = c.rowb + b + c.ocur;
    const bool last = c.kleft == 0 || jn > c.kmz;
    c.bprev = b;  // the next run starts where this one ends (in the next row)
    const unsigned rem = c.rem + c.Ru;
    const bool carry = rem >= c.ad;
    c.rem = carry ? rem - c.ad : rem;
    c.jn = jn + c.Qu + (carry ? 1 : 0);
    --c.kleft;
    c.rowb += c.rstep;
    return !last;
}

// ------------------------------------------------------------- event walk
//
// The tiled traversal's form of a lean walk whose major axis moves + (every
// record is stored oriented that way).  Consecutive runs of such a walk share
// a major index: run k ends at major index b in its row and run k + 1 begins at
// b one row on (always in the same direction).  So instead of adding +1 where
// each run begins and -1 past its end, the walk adds 1 to an event count E at
// (row, b) for each change of row, and marks only its own first and last voxel
// in P: one update per run where the two ends took two.  With the walks of a
// tile sorted by type (major axis, row direction s), E and P decode together:
//   count(m, row) = SP(m, row) + SE(m, row - s) - SE(m - 1, row)
// SE and SP the prefix sums of E and P along the major axis (P is +1 at the
// walk's first voxel, -1 just past its last).  A row of a walk holds at most
// one event, so SE and SP stay within the pairs of a part (32767).
//
// Rays dilated by t voxels in-plane decode from the same events: the
// dilated set's interval in a row runs from where the run t rows earlier began,
// less t, to where the run t rows later ends, plus t, so
//   count(m, row) = sum_{|j| <= t} SP(m, row + j)
//                   + SE(m + t, row - (t + 1) s) - SE(m - t - 1, row + t s)
// with P marked t before the first voxel and t past the last (clamped to the
// row), SE read as 0 left of the row and as the row's total right of it.
//
// Layout: one word per voxel, E in the low and P in the high half (added as 1
// and +-65536, so a row's prefix sum of words is SE + 65536 SP mod 2^32), the
// major axis fastest, rows of W words (at least one past the voxels, for the
// end marks), row = minor index + nminor * slice.

// Words per row: one more than the voxels, rounded up to an odd number when
// the box still fits in the (nx + 1)(ny + 1) words a tile is planned with, so
// that the lanes of a warp that are in different rows at one major index hit
// different banks.
HD_HD int tile_row_words(int nmaj, int nminor)
{
    const int w = nmaj + 1;
    return (w & 1) == 0 && nminor <= nmaj + 1 ? w + 1 : w;
}

// Packed event walk (kLeanWords words): |D_0|, |D_m| mod |D_0|, the Bresenham
// remainder; then byte offsets from the tile's first word: of one event to the
// next without the carry, of the first event, of the last place the end mark
// can have, of the first mark; and the number of events (bit 31: no walk).
HD_HD void event_pack(const LeanWalk &L, int nmaj, int nminor, int thick, uint32_t o[kLeanWords])
{
    const int W = tile_row_words(nmaj, nminor);
    // events: the K' = min(K, ceil(X / |D_m|)) crossings k of minor 0 with
    // J_k <= kmz, J_k = J_1 + floor(((k - 1) |D_m| + rem) / |D_0|) and
    // X = (kmz - J_1 + 1) |D_0| - rem
    int n = 0;
    if (L.K > 0 && L.jn <= L.kmz) {
        const long long X =
            static_cast<long long>(L.kmz - L.jn + 1) * L.ad - static_cast<long long>(L.rem);
        const long long am = static_cast<long long>(L.Qu) * L.ad + L.Ru;
        long long rem;  // X >= 1: L.rem < |D_0|
        const int k = fdiv32(X - 1, static_cast<int>(am), rcp_int(static_cast<int>(am)), rem) + 1;
        n = k < L.K ? k : L.K;
    }
    const int s = (L.fl & 2) ? 1 : -1;
    const int row0 = L.row * W;
    const int m0 = L.im0 - thick > 0 ? L.im0 - thick : 0;
    const int j1 = L.jn < L.kmz ? L.jn : L.kmz;
    const int rowk = row0 + s * n * W;
    const int last = L.im0 + L.kmz + thick + 1;
    o[0] = L.ad;
    o[1] = L.Ru;
    o[2] = L.rem;
    o[3] = static_cast<uint32_t>(4 * (L.Qu + s * W));
    o[4] = static_cast<uint32_t>(4 * (row0 + L.im0 + j1));
    o[5] = static_cast<uint32_t>(4 * (rowk + (last < nmaj ? last : nmaj)));
    o[6] = static_cast<uint32_t>(4 * (row0 + m0));
    o[7] = static_cast<uint32_t>(n);
}

// A packed event walk with no voxel.
HD_HD void event_pack_empty(uint32_t o[kLeanWords])
{
    for (int i = 0; i < kLeanWords; ++i) o[i] = 0;
    o[7] = 0x80000000u;
}

// An event walk in progress; addresses are byte offsets from a base the
// caller chooses (such as the tile's shared-memory address).
struct EventCursor {
    unsigned ad, Ru, rem;
    int addr;  // of the next event
    int step;  // to the one after it, without the carry
    int left;  // events left
    int endl;  // the last address the end mark can have
};

// Starts a packed walk; *first receives the address of its first mark.
// False when there is no walk (no events left then either).
HD_HD bool event_start(const uint32_t o[kLeanWords], int base, EventCursor &c, int &first)
{
    c.ad = o[0];
    c.Ru = o[1];
    c.rem = o[2];
    c.step = static_cast<int>(o[3]);
    c.addr = base + static_cast<int>(o[4]);
    c.endl = base + static_cast<int>(o[5]);
    first = base + static_cast<int>(o[6]);
    const bool walk = static_cast<int>(o[7]) >= 0;
    c.left = walk ? static_cast<int>(o[7]) : 0;
    return walk;
}

// Moves past one event.
HD_HD void event_next(EventCursor &c)
{
    c.rem += c.Ru;
    const bool carry = c.rem >= c.ad;
    c.addr += c.step;
    if (carry) {
        c.rem -= c.ad;
        c.addr += 4;
    }
    --c.left;
}

// Address of the end mark once no event is left (the cursor then stands at
// the event that would follow, in the last row); thick4 = 4 (t + 1).
HD_HD int event_end(const EventCursor &c, int thick4)
{
    const int e = c.addr + thick4;
    return e < c.endl ? e : c.endl;
}

// ------------------------------------------------------------ joined tiles
//
// Event walks of all four types in one tile: for tiles whose walks of a type
// are too few to pay for a flush of their own.  One layout, x fastest in rows of
// nx + 1 words and ny + 1 rows to a slice; the low half of a word holds the
// difference counts of x-major runs along x, the high half those of y-major
// runs along y, so that
//   count(x, y) = sum_{x' <= x} low(x', y) + sum_{y' <= y} high(x, y').
// An event then takes two updates: it ends its row's run past its major index
// and begins the next row's there.  A walk adds at most one to a half of a word
// and to a prefix sum of it, so both stay within the pairs of a part (32767).

// How walks of one type lie in a joined tile (bytes from one index to the next,
// the minor one's in the direction the walks go), and in their own layout.
struct JoinedBox {
    float rW;  // 1 / W
    int major, minor, slice;
    int16_t W, nminor;  // words per row and rows per slice of the own layout
};

HD_HD JoinedBox joined_box(int type, int dx, int dy)
{
    const bool ymaj = (type & 2) != 0;
    JoinedBox b;
    b.nminor = static_cast<int16_t>(ymaj ? dx : dy);
    b.W = static_cast<int16_t>(tile_row_words(ymaj ? dy : dx, b.nminor));
    b.rW = 1.0f / static_cast<float>(b.W);
    const int row = 4 * (dx + 1);
    b.major = ymaj ? row : 4;
    b.minor = ymaj ? 4 : row;
    if (type & 1) b.minor = -b.minor;
    b.slice = row * (dy + 1);
    return b;
}

// A walk in progress in a joined tile: an event at `addr` adds -v at addr + major
// and v at addr + minor.
struct JoinedCursor {
    unsigned ad, Ru, rem;
    int addr, step, left, endl;
    int major, minor;
    uint32_t v;
};

// Starts a packed event walk there; *first receives the address of its first
// mark (v).  False when there is no walk.  The row of a word is a division by W
// of a number below 2^16: (q + 1/2) / W is at least 1 / (2 W) from a whole
// number, W <= 4098, its float error at most 2^-22 of it.
HD_HD bool joined_start(const uint32_t o[kLeanWords], const JoinedBox &b, int base, JoinedCursor &c,
                        int &first)
{
    c.ad = o[0];
    c.Ru = o[1];
    c.rem = o[2];
    const bool walk = static_cast<int>(o[7]) >= 0;
    c.left = walk ? static_cast<int>(o[7]) : 0;
    const int f = static_cast<int>(o[6]) >> 2;
    const int row = static_cast<int>((static_cast<float>(f) + 0.5f) * b.rW);
    const int z = row < b.nminor ? 0 : row / b.nminor;
    const int sgn = b.minor < 0 ? -1 : 1;  // rows per event
    const int at = base + z * b.slice + (row - z * b.nminor) * sgn * b.minor;  // the first row's start
    const int own = row * b.W;
    first = at + (f - own) * b.major;
    c.addr = at + ((static_cast<int>(o[4]) >> 2) - own) * b.major;
    const int n = c.left * sgn;  // rows to the last one
    c.endl = at + c.left * b.minor + ((static_cast<int>(o[5]) >> 2) - own - n * b.W) * b.major;
    c.step = ((static_cast<int>(o[3]) >> 2) - sgn * b.W) * b.major + b.minor;
    c.major = b.major;
    c.minor = b.minor;
    c.v = b.major == 4 ? 1u : 65536u;  // (a row has at least two words)
    return walk;
}

// Moves past one event.
HD_HD void joined_next(JoinedCursor &c)
{
    c.rem += c.Ru;
    const bool carry = c.rem >= c.ad;
    c.addr += c.step;
    if (carry) {
        c.rem -= c.ad;
        c.addr += c.major;
    }
    --c.left;
}

// Address of the end mark (-v) once no event is left.
HD_HD int joined_end(const JoinedCursor &c)
{
    const int e = c.addr + c.major;
    return e < c.endl ? e : c.endl;
}

// The high half of a word, its low half being a signed count.
HD_HD uint32_t joined_high(uint32_t w) { return (w + 0x8000u) >> 16; }

// Packed run-walk state: 16 32-bit words, so a walk prepared by one kernel
// can be resumed by another.  The row strides and the major size follow
// from the box (nx, ny) and the flags.
constexpr int kPackedWords = 16;

HD_HD void run_pack(const RunWalk &w, uint32_t o[kPackedWords])
{
    o[0] = static_cast<uint32_t>(static_cast<unsigned long long>(w.e12) & 0xffffffffull);
    o[1] = static_cast<uint32_t>(static_cast<unsigned long long>(w.e12) >> 32);
    o[2] = static_cast<uint32_t>(w.q[0]);
    o[3] = static_cast<uint32_t>(w.q[1]);
    o[4] = w.rh[0];
    o[5] = w.rh[1];
    o[6] = w.ad[0];
    o[7] = w.ad[1];
    o[8] = static_cast<uint32_t>(w.Qu[0]);
    o[9] = static_cast<uint32_t>(w.Qu[1]);
    o[10] = w.Ru[0];
    o[11] = w.Ru[1];
    o[12] = static_cast<uint32_t>(w.row);
    o[13] = (static_cast<uint32_t>(w.im) & 0xffffu) | (static_cast<uint32_t>(w.km) << 16);
    o[14] = (static_cast<uint32_t>(w.kc[0]) & 0xffffu) | (static_cast<uint32_t>(w.kc[1]) << 16);
    o[15] = static_cast<uint32_t>(w.flags);
}

// A packed state that yields no run.
HD_HD void run_pack_empty(uint32_t o[kPackedWords])
{
    for (int i = 0; i < kPackedWords; ++i) o[i] = 0;
    o[15] = 1u << 9;
}

HD_HD void run_unpack(const uint32_t o[kPackedWords], int nx, int ny, RunWalk &w)
{
    w.e12 = static_cast<long long>((static_cast<unsigned long long>(o[1]) << 32) | o[0]);
    w.q[0] = static_cast<int>(o[2]);
    w.q[1] = static_cast<int>(o[3]);
    w.rh[0] = o[4];
    w.rh[1] = o[5];
    w.ad[0] = o[6];
    w.ad[1] = o[7];
    w.Qu[0] = static_cast<int>(o[8]);
    w.Qu[1] = static_cast<int>(o[9]);
    w.Ru[0] = o[10];
    w.Ru[1] = o[11];
    w.row = static_cast<int>(o[12]);
    w.im = static_cast<int>(o[13] & 0xffffu);
    w.km = static_cast<int>(o[13] >> 16);
    w.kc[0] = static_cast<int>(o[14] & 0xffffu);
    w.kc[1] = static_cast<int>(o[14] >> 16);
    w.flags = static_cast<int>(o[15]);
    const bool ymaj = (w.flags >> 5) & 1;
    w.run_start = w.im;
    w.rstride[0] = (w.flags & 2) ? 1 : -1;
    w.rstride[1] = (w.flags & 4) ? (ymaj ? nx : ny) : -(ymaj ? nx : ny);
    w.nmaj = ymaj ? ny : nx;
}

// Call visit(v) for every voxel of the set in traversal order; returns |A_i|.
template <class VisitT>
HD_HD unsigned walk_all(const int32_t gi[3], const int32_t go[3], int nx, int ny, int nz,
                        const VisitT &visit)
{
    Walk w;
    if (!walk_begin(w, gi, go, nx, ny, nz)) return 0;
    unsigned c = 0;
    do {
        visit(static_cast<uint32_t>(w.idx));
        ++c;
    } while (walk_next(w));
    return c;
}

}  // namespace hd
