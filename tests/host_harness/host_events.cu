// Host build of the event walks (hd_geom.cuh) for tests/test_host_events.py.
#include <vector>

#include "../../paper_1402_1720_gb300/csrc/hd_geom.cuh"

// to_grid against floor((2 w + n s) 2^16 / (2 s)) in 128 bits; mismatches.
extern "C" long long hx_to_grid(int n, float s, const int32_t *w, long long count)
{
    const hd::GeomQ g = hd::make_geomq(n, n, n, s, s, s, 1.0f);
    long long bad = 0;
    for (long long i = 0; i < count; ++i) {
        const __int128 num = (2 * (__int128)w[i] + (__int128)n * g.sx) * 65536, den = 2 * g.sx;
        __int128 q = num / den;
        if (num % den != 0 && num < 0) --q;
        if ((__int128)hd::to_grid(w[i], g.dx) != q) ++bad;
    }
    return bad;
}

// The path walk (through pack and unpack) against the general run walk, run by
// run: returns its runs, 0 when neither has a voxel, -1 when it declines, -2
// when only one of them has a voxel, -3 when a run differs.
extern "C" int hx_path(const int32_t *gi, const int32_t *go, int nx, int ny, int nz)
{
    hd::PathWalk P;
    hd::RunWalk w;
    const int r = hd::path_lean(gi, go, nx, ny, nz, P);
    const bool have = hd::run_begin(w, gi, go, nx, ny, nz);
    if (r < 0) return -1;
    if (r == 0) return have ? -2 : 0;
    if (!have) return -2;
    uint32_t o[hd::kPathWords];
    hd::path_pack(P, o);
    hd::path_unpack(o, P);
    const bool ymaj = (w.flags >> 5) & 1, plus = w.flags & 1;
    int row, lo, hi, n = 0;
    bool more = true;
    while (hd::run_next(w, row, lo, hi)) {
        if (!more) return -3;
        uint32_t vb;
        int a, b;
        more = hd::path_run(P, nx, nx * ny, vb, a, b);
        const uint32_t base = ymaj ? row % nx + nx * ny * (row / nx) : nx * row;
        if (vb != base || a != (plus ? lo : hi) || b != (plus ? hi : lo)) return -3;
        ++n;
    }
    return more ? -3 : n;
}

// The event walk of the oriented segment in a box of dx x dy x dz voxels,
// dilated by `thick`: its updates applied to plain counters in the tile's
// layout, decoded by the definition (prefix sums along the major axis), the
// voxels with a nonzero count returned box-linear (x fastest).  direct: the
// one-slice set-up the scatter uses (dz = 1), else the general one.  Returns
// -1 when the walk has no event form, -2 an update outside the box's words or
// in another row than its walk's, -3 a voxel counted other than once.
extern "C" int hx_events(const int32_t *seg, int dx, int dy, int dz, int thick, int direct,
                         int32_t *out, int *nruns)
{
    int32_t r[6];
    for (int a = 0; a < 6; ++a) r[a] = seg[a];
    const int type = hd::orient_record(r);
    const int32_t gi[3] = {r[0], r[1], r[2]}, go[3] = {r[3], r[4], r[5]};
    const bool ymaj = (type & 2) != 0;
    const int s = (type & 1) ? -1 : 1;
    const int nmaj = ymaj ? dy : dx, nmin = ymaj ? dx : dy;
    const int W = hd::tile_row_words(nmaj, nmin);
    if (nmin * W * dz > (dx + 1) * (dy + 1) * dz) return -2;
    *nruns = 0;
    hd::LeanWalk L;
    if (direct) {
        const int rl = hd::slab_lean(gi, go, dx, dy, L);
        if (rl == 0) return 0;
        if (rl < 0) return -1;
    } else {
        hd::RunWalk w;
        if (!hd::run_begin(w, gi, go, dx, dy, dz)) return 0;
        if (!hd::lean_of(w, L)) return -1;
    }
    const bool moves = gi[0] != go[0] || gi[1] != go[1];
    if (((L.fl >> 2) & 1) != (ymaj ? 1 : 0) || (moves && !(L.fl & 1))) return -4;
    uint32_t o[hd::kLeanWords];
    hd::event_pack(L, nmaj, nmin, thick, o);
    const int words = nmin * W * dz;
    std::vector<int> E(words, 0), P(words, 0);
    hd::EventCursor c;
    int first;
    if (!hd::event_start(o, 0, c, first)) return -2;
    auto ok = [&](int at) { return at >= 0 && at / 4 < words && (at & 3) == 0; };
    if (!ok(first)) return -2;
    P[first / 4] += 1;
    int row = first / 4 / W;
    *nruns = c.left + 1;
    while (c.left) {
        if (!ok(c.addr) || c.addr / 4 / W != row || c.addr / 4 % W >= nmaj) return -2;
        E[c.addr / 4] += 1;
        hd::event_next(c);
        row += s;
    }
    const int end = hd::event_end(c, 4 * (thick + 1));
    if (!ok(end) || end / 4 / W != row) return -2;
    P[end / 4] -= 1;
    std::vector<int> SE(words), SP(words);
    for (int q = 0; q < nmin * dz; ++q) {
        int e = 0, p = 0;
        for (int m = 0; m < W; ++m) {
            SE[q * W + m] = e += E[q * W + m];
            SP[q * W + m] = p += P[q * W + m];
        }
    }
    int n = 0;
    for (int z = 0; z < dz; ++z)
        for (int y = 0; y < dy; ++y)
            for (int x = 0; x < dx; ++x) {
                const int i = ymaj ? x : y, m = ymaj ? y : x;
                int v = 0;
                for (int j = -thick; j <= thick; ++j)
                    if (i + j >= 0 && i + j < nmin) v += SP[(i + j + nmin * z) * W + m];
                const int ia = i - (thick + 1) * s, ib = i + thick * s;
                if (ia >= 0 && ia < nmin)
                    v += SE[(ia + nmin * z) * W + (m + thick < nmaj ? m + thick : nmaj)];
                if (ib >= 0 && ib < nmin && m - thick - 1 >= 0)
                    v -= SE[(ib + nmin * z) * W + m - thick - 1];
                if (v != 0 && v != 1) return -3;
                if (v) out[n++] = x + dx * (y + dy * z);
            }
    return n;
}

// The chunk split for a plan of ntiles tiles.
extern "C" void hx_chunk_split(long long n, int sm_count, int ntiles, int *blocks, long long *per_block)
{
    const hd::ChunkSplit c = hd::chunk_split(n, sm_count, ntiles);
    *blocks = c.blocks;
    *per_block = c.per_block;
}
