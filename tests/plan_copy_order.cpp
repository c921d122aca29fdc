// The split schedule lets the slicer of a step write that step's operand back to the front, ahead of the
// step's GEMM (SplitStep::fuse_copy).  A plan's own schedule does so; a GEMM whose result is made to meet
// the copy's destination must not.  Prints one line per case; exits non-zero on a wrong decision.
#include <algorithm>
#include <cstdio>
#include <string>
#include <vector>

#include "plan.hpp"
#include "split_gemm.cuh"

namespace ndsi {
void set_last_error(const std::string&) {}
}  // namespace ndsi
using namespace ndsi;

int main() {
    // a box of 5 x 4 x 4 atoms, 3 orbitals each, all 26 neighbours
    const int nx = 5, ny = 4, nz = 4, o = 3, na = nx * ny * nz, n = na * o;
    std::vector<int64_t> rowptr(1, 0);
    std::vector<int32_t> col;
    for (int i = 0; i < n; ++i) {
        const int a = i / o, x = a % nx, y = a / nx % ny, z = a / (nx * ny);
        std::vector<int> cs;
        for (int b = 0; b < na; ++b) {
            const int dx = b % nx - x, dy = b / nx % ny - y, dz = b / (nx * ny) - z;
            if (std::max({dx, -dx, dy, -dy, dz, -dz}) <= 1)
                for (int q = 0; q < o; ++q) cs.push_back(b * o + q);
        }
        for (int c : cs) col.push_back(c);
        rowptr.push_back(static_cast<int64_t>(col.size()));
    }
    std::vector<double> centers(3 * na);
    for (int a = 0; a < na; ++a) {
        centers[3 * a] = a % nx;
        centers[3 * a + 1] = a / nx % ny;
        centers[3 * a + 2] = a / (nx * ny);
    }
    std::vector<int32_t> aob(n);
    for (int i = 0; i < n; ++i) aob[i] = i / o;
    ndsi_pattern pat{n, rowptr.data(), col.data()};
    ndsi_options opt{};
    opt.leaf_atoms = 6;
    opt.block = 16;
    opt.outer_block = 128;
    opt.m0_radius = 1e7;
    opt.precision = NDSI_PREC_SPLIT;
    opt.split_slices = 6;
    Plan P;
    std::string err;
    if (analyze(&pat, na, centers.data(), aob.data(), opt, P, err)) {
        std::printf("analyze failed: %s\n", err.c_str());
        return 2;
    }
    const std::vector<int8_t> bands(P.launches.size(), 0);
    auto fused = [&](int tag) {  // per launch of this tag: 1 when its copy is done by the slicer
        std::vector<SplitItem> items;
        std::vector<SplitStep> steps;
        std::vector<GemmTile> tiles;
        std::vector<SliceBlock> blocks;
        build_split_schedule(P, 6, bands, items, steps, tiles, blocks);
        std::vector<std::pair<size_t, int>> out;
        size_t k = 0;
        for (size_t li = 0; li < P.launches.size(); ++li) {
            if (!split_eligible(P.launches[li])) continue;
            if (P.launches[li].tag == tag) out.emplace_back(li, steps[k].fuse_copy);
            ++k;
        }
        return out;
    };
    int bad = 0, planted = 0;
    for (const int tag : {static_cast<int>(T_SCHUR), static_cast<int>(T_SEL_D)}) {
        const auto clean = fused(tag);
        int on = 0;
        for (const auto& c : clean) on += c.second;
        std::printf("tag %d: %d of %zu steps copy ahead\n", tag, on, clean.size());
        if (on == 0) ++bad;
        for (const auto& c : clean) {
            if (!c.second) continue;
            const Launch& l = P.launches[c.first];
            const CopyItem& y = P.copy_items[P.launches[c.first + 1].first];
            GemmItem& g = P.gemm_items[l.first];
            const int64_t keep = g.c_off;
            const int32_t ld = g.ldc;
            g.c_off = y.dst_off;  // the result over the copy's destination
            g.ldc = y.ldd;
            for (const auto& d : fused(tag))
                if (d.first == c.first && d.second) ++bad, std::printf("tag %d launch %zu: copies over the result\n", tag, c.first);
            g.c_off = keep;
            g.ldc = ld;
            ++planted;
        }
        if (fused(tag) != clean) ++bad;
    }
    std::printf("planted %d\n", planted);
    return bad || !planted ? 1 : 0;
}
