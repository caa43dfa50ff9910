// Host build of event walks in joined tiles (hd_geom.cuh) for tests/test_host_joined.py.
#include <vector>

#include "../../paper_1402_1720_gb300/csrc/hd_geom.cuh"

// The event walks of n oriented segments in a box of dx x dy x dz voxels, added to
// the words of one joined tile as the traversal does, and decoded as its flush
// does: counts receives each voxel's.  Returns the walks added (segments without
// an event walk are marked in skipped), or -2 for an update outside the tile.
extern "C" int hx_joined(const int32_t *segs, int n, int dx, int dy, int dz, int direct,
                         int32_t *counts, uint8_t *skipped)
{
    const int P = dx + 1, words = P * (dy + 1) * dz;
    std::vector<uint32_t> tile(words, 0u);
    auto add = [&](int at, uint32_t v) {
        if (at < 0 || at / 4 >= words || (at & 3) != 0) return false;
        tile[at / 4] += v;
        return true;
    };
    int walks = 0;
    for (int i = 0; i < n; ++i) {
        int32_t r[6];
        for (int a = 0; a < 6; ++a) r[a] = segs[6 * i + a];
        const int type = hd::orient_record(r);
        const int32_t gi[3] = {r[0], r[1], r[2]}, go[3] = {r[3], r[4], r[5]};
        const bool ymaj = (type & 2) != 0;
        hd::LeanWalk L;
        uint32_t o[hd::kLeanWords];
        skipped[i] = 0;
        bool have;
        if (direct) {
            const int rl = hd::slab_lean(gi, go, dx, dy, L);
            have = rl == 1;
            skipped[i] = rl < 0;
        } else {
            hd::RunWalk w;
            have = hd::run_begin(w, gi, go, dx, dy, dz);
            if (have && !hd::lean_of(w, L)) {
                have = false;
                skipped[i] = 1;
            }
        }
        if (have) hd::event_pack(L, ymaj ? dy : dx, ymaj ? dx : dy, 0, o);
        else hd::event_pack_empty(o);
        const hd::JoinedBox b = hd::joined_box(type, dx, dy);
        hd::JoinedCursor c;
        int first;
        const bool walk = hd::joined_start(o, b, 0, c, first);
        if (walk != have) return -3;
        if (!walk) continue;
        ++walks;
        bool ok = add(first, c.v);
        while (c.left) {
            ok = ok && add(c.addr + c.major, 0u - c.v) && add(c.addr + c.minor, c.v);
            hd::joined_next(c);
        }
        if (!ok || !add(hd::joined_end(c), 0u - c.v)) return -2;
    }
    for (int z = 0; z < dz; ++z)
        for (int x = 0; x < dx; ++x) {
            uint32_t sum = 0;
            for (int y = 0; y < dy; ++y) {
                uint32_t &w = tile[x + P * (y + (dy + 1) * z)];
                sum += hd::joined_high(w);
                w = (w & 0xffffu) | (sum << 16);
            }
        }
    for (int z = 0; z < dz; ++z)
        for (int y = 0; y < dy; ++y) {
            uint32_t sum = 0;
            for (int x = 0; x < dx; ++x) {
                const uint32_t w = tile[x + P * (y + (dy + 1) * z)];
                sum += w;
                counts[x + dx * (y + dy * z)] = static_cast<int32_t>((sum & 0xffffu) + (w >> 16));
            }
        }
    return walks;
}
