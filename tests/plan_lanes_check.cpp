// plan_lanes_check.cpp -- builds a tensor-core plan's host part on the CPU and
// checks what the kernel takes from it without looking again: the lanes of every
// tile, their sign patterns, and the units of every x chunk length.
// Usage: plan_lanes_check ng box_len n_k1 n_mu ntri_file edges_file
// stdout: "tiles mixed_tiles violations" (violations described on stderr)
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <map>
#include <vector>

#include "plan.hpp"

using namespace bisp;

static int bad = 0;
static void expect(bool ok, const char *what, size_t tile)
{
    if (ok) return;
    ++bad;
    std::fprintf(stderr, "tile %zu: %s\n", tile, what);
}

int main(int argc, char **argv)
{
    if (argc != 7) return 2;
    const int ng = std::atoi(argv[1]), nk1 = std::atoi(argv[3]), nmu = std::atoi(argv[4]);
    HostPlan P;
    P.desc.n_g = ng;
    P.desc.n_k1 = nk1;
    P.desc.n_mu = P.desc.n_t = nmu;
    P.desc.l_max = 6;
    P.desc.max_batch = 1;
    P.desc.precision = BISP_PREC_MIXED_TC;
    P.kf = 2.0 * M_PI / std::atof(argv[2]);
    P.k1_edges.resize(size_t(nk1) + 1);
    FILE *f = std::fopen(argv[6], "rb");
    if (!f || std::fread(P.k1_edges.data(), sizeof(double), P.k1_edges.size(), f) != P.k1_edges.size()) return 4;
    std::fclose(f);
    P.desc.k1_edges = P.k1_edges.data();
    if (!build_rings(ng, P.rings)) return 3;
    const int nr = P.rings.nr;
    P.ntri.resize(size_t(nr) * nr * nr);
    f = std::fopen(argv[5], "rb");
    if (!f || std::fread(P.ntri.data(), sizeof(int64_t), P.ntri.size(), f) != P.ntri.size()) return 4;
    std::fclose(f);
    P.celem = 8;
    P.max_cls = 4;
    P.tensor = true;
    size_t mixed = 0, ntile = 0;
    for (int64_t chunk : {int64_t(16384), int64_t(512)}) {
        const std::string err = enumerate(P, chunk);
        if (!err.empty()) {
            std::fprintf(stderr, "enumerate: %s\n", err.c_str());
            return 5;
        }
        ntile = P.tc_tiles.size();
        mixed = 0;
        expect(P.tc_lanes.size() == ntile * kTcRows, "lanes of every tile", 0);
        for (size_t t = 0; t < ntile; ++t) {
            const TcTile &T = P.tc_tiles[t];
            std::vector<int> seen(size_t(T.nrow), 0);
            int patterns[9] = {};
            for (int l = 0; l < kTcRows; ++l) {
                const TcLane &L = P.tc_lanes[t * kTcRows + l];
                if (L.row == kTcNoRow) {
                    expect(L.s1 < T.nslot && L.s2 < T.nslot, "a lane without a row reads staged slots", t);
                    continue;
                }
                if (L.row >= T.nrow) {
                    expect(false, "a lane's row is one of the tile's", t);
                    continue;
                }
                ++seen[L.row];
                const TcRow &R = P.tc_rows[size_t(T.row0) + L.row];
                expect(L.s1 == R.s1 && L.s2 == R.s2, "the lane's slots are its row's", t);
                expect(R.s1 < T.nslot && R.s2 < T.nslot, "slots in range", t);
                expect(R.flags == T.qflags[l / 32], "a warp's rows have its sign pattern", t);
                expect((R.flags & 1) == 0, "n1 >= 0", t);
                patterns[R.flags & 7] = 1;
            }
            for (int s : seen) expect(s == 1, "every row on one lane", t);
            int n = 0, one = 0;
            for (int k = 0; k < 8; ++k)
                if (patterns[k]) {
                    ++n;
                    one = k;
                }
            expect(n == 1 ? T.flags == one : T.flags == kTcMixed, "the tile's sign pattern", t);
            mixed += n > 1;
            // the fields a row reads are those of its groups' planes and rings
            for (int s = 0; s < T.nslot; ++s) {
                const int32_t v = P.tc_slots[size_t(T.slot0) + s];
                expect((v & 255) <= nr && (v >> 8) <= P.rings.nz, "slot names a field or none", t);
            }
        }
        std::map<std::pair<int, int>, int> units;
        for (const TcUnit &U : P.tc_units) ++units[{U.tile, U.chunk}];
        size_t want = 0;
        for (size_t t = 0; t < ntile; ++t) {
            const int64_t m2 = int64_t(P.tc_tiles[t].M) * P.tc_tiles[t].M;
            for (int64_t c = 0; c * chunk < m2; ++c) {
                ++want;
                const auto it = units.find({int(t), int(c)});
                expect(it != units.end() && it->second == 1, "every x chunk of a tile is one unit", t);
            }
        }
        expect(units.size() == want && P.tc_units.size() == want, "no other units", 0);
    }
    std::printf("%zu %zu %d\n", ntile, mixed, bad);
    return 0;
}
