// plan_chunk_check.cpp -- a tensor-core plan's host part on the CPU: one enumerated for
// long x chunks and given another length (set_x_chunk) is the one enumerated for that.
// Usage: plan_chunk_check ng box_len n_k1 ntri_file edges_file
// stdout: "units differences"
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <vector>

#include "plan.hpp"

using namespace bisp;

template <typename T> static int differ(const std::vector<T> &a, const std::vector<T> &b)
{
    return a.size() != b.size() || (!a.empty() && std::memcmp(a.data(), b.data(), a.size() * sizeof(T)) != 0);
}

int main(int argc, char **argv)
{
    if (argc != 6) return 2;
    const int ng = std::atoi(argv[1]), nk1 = std::atoi(argv[3]);
    HostPlan P[2];
    size_t units = 0;
    int bad = 0;
    for (int64_t chunk : {int64_t(8192), int64_t(512), int64_t(16384)}) {
        for (int k = 0; k < 2; ++k) {
            HostPlan &p = P[k];
            p = HostPlan{};
            p.desc.n_g = ng;
            p.desc.n_k1 = nk1;
            p.desc.n_mu = p.desc.n_t = 5;
            p.desc.l_max = 6;
            p.desc.max_batch = 1;
            p.desc.precision = BISP_PREC_MIXED_TC;
            p.kf = 2.0 * M_PI / std::atof(argv[2]);
            p.k1_edges.resize(size_t(nk1) + 1);
            FILE *f = std::fopen(argv[5], "rb");
            if (!f || std::fread(p.k1_edges.data(), sizeof(double), p.k1_edges.size(), f) != p.k1_edges.size()) return 4;
            std::fclose(f);
            p.desc.k1_edges = p.k1_edges.data();
            if (!build_rings(ng, p.rings)) return 3;
            p.ntri.resize(size_t(p.rings.nr) * p.rings.nr * p.rings.nr);
            f = std::fopen(argv[4], "rb");
            if (!f || std::fread(p.ntri.data(), sizeof(int64_t), p.ntri.size(), f) != p.ntri.size()) return 4;
            std::fclose(f);
            p.celem = 8;
            p.tensor = true;
            if (!enumerate(p, k == 0 ? 16384 : chunk).empty()) return 5;
        }
        set_x_chunk(P[0], chunk);
        const HostPlan &a = P[0], &b = P[1];
        bad += differ(a.groups, b.groups) + differ(a.tc_tiles, b.tc_tiles) + differ(a.tc_rows, b.tc_rows) +
               differ(a.tc_units, b.tc_units) + differ(a.tc_slots, b.tc_slots) + differ(a.tc_lanes, b.tc_lanes) +
               differ(a.doff, b.doff) + (a.n_partials != b.n_partials) +
               (std::memcmp(a.tc_class_begin, b.tc_class_begin, sizeof(a.tc_class_begin)) != 0);
        units += b.tc_units.size();
    }
    std::printf("%zu %d\n", units, bad);
    return 0;
}
