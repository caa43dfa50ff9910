// Host build of the closed form of Euclidean rows (hd_euclid.cuh) for
// tests/test_host_slice_rows.py.
#include "../../paper_1402_1720_gb300/csrc/hd_euclid.cuh"

// Every row of every slice of one history (world endpoints W, mm * 2^16)
// against the exact search: the rows the closed form calls certain, cut to the
// strip [m0, m0 + len) of the major axis, and the rows it leaves out.
// Returns the number of certain rows, or -1 a certain row that differs, -2 a
// row with voxels outside the slices or rows handed out, -3 such a row when
// euclid_range finds none.  *open: rows left to the exact search; *closed.
extern "C" long long hx_slice_rows(const long long *W, int nx, int ny, int nz, float sx, float sy,
                                   float sz, float T, float d0, int m0, int len, long long *open,
                                   int *closed)
{
    const hd::GeomQ g = hd::make_geomq(nx, ny, nz, sx, sy, sz, T);
    const long long R = 2 * hd::q16_of(d0);
    long long A[3], B[3];
    bool ymaj;
    int blo[3], bhi[3];
    float S;
    *open = 0;
    *closed = 0;
    const bool box = hd::capsule_frame(g, W, R, A, B, ymaj, blo, bhi, S);
    hd::CapX cx;
    hd::capx_of(g, A, B, ymaj, R, cx);
    const hd::CapF cf = hd::capf_of(cx, S, R);
    int klo, khi, ylo, yhi;
    bool cl = false;
    const bool any = hd::euclid_range(g, W, R, klo, khi, ylo, yhi, cl);
    *closed = cl;
    int32_t w[6];
    for (int q = 0; q < 6; ++q) w[q] = static_cast<int32_t>(W[q]);
    const int n1 = ymaj ? nx : ny, n0 = ymaj ? ny : nx;
    if (m0 + len > n0) len = n0 - m0;
    long long certain = 0;
    for (int k = 0; k < nz; ++k) {
        hd::SliceRows r{};
        const bool rows = any && cl && k >= klo && k <= khi &&
                          hd::slice_rows(g, w, R, k, 0, n1, m0, len, r);
        for (int a = 0; a < n1; ++a) {
            int lo = 1, hi = 0;
            if (!box || !hd::row_interval(cf, cx, a, k, lo, hi)) lo = 1, hi = 0;
            const bool have = lo <= hi;
            if (have && !any) return -3;
            if (have && (k < klo || k > khi)) return -2;
            if (have && (ymaj ? (hi < ylo || lo > yhi || lo < ylo || hi > yhi) : (a < ylo || a > yhi)))
                return -2;
            if (!any || !cl) continue;
            int tl = lo - m0, th = hi - m0;  // the tile's part
            if (tl < 0) tl = 0;
            if (th > len - 1) th = len - 1;
            const bool part = have && tl <= th;
            if (!rows || a < r.row || a >= r.row + r.n) {
                if (part) return -2;
                continue;
            }
            float x0, x1, y0, y1;
            const float q = hd::slice_row(r, static_cast<float>(a - r.row), x0, x1, y0, y1);
            if (!(q > 4.0f * r.dq) && !(q < -r.dq)) {
                ++*open;
                continue;
            }
            ++certain;
            if (q < 0.0f) {
                if (part) return -1;
                continue;
            }
            if (x0 != x1 || y0 != y1) ++*open;
            // x1 .. y0 inside, below x0 and above y1 outside (tile indices)
            for (int m = 0; m < len; ++m) {
                const float f = hd::kWhole + static_cast<float>(m);
                const bool in = have && m >= lo - m0 && m <= hi - m0;
                if (f >= x1 && f <= y0 && !in) return -1;
                if ((f < x0 || f > y1) && in) return -1;
            }
        }
    }
    return certain;
}
