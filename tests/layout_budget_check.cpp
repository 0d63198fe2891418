// Host-side check of the work items that mm_layout.cpp packs with the values the
// library gives it (SMs, the items' fixed cost, a supplied order), built and run
// by tests/test_layout_budget.py.
//
// Checks for every item that its sweep bundles' compartments lie side by side
// over the whole item, each holding exactly its own paths (the FP64 kernel
// divides bundle by bundle), and for giants that their scratch ranges do; prints
// the classes, the number of items solved by clusters, the largest item of
// several neurons, the largest shared-memory need, and the giants' sizes.
//
// Usage: layout_budget_check <network file> <group_comps> <sms> <fp64: 0 | 1>
// Network file: int32 N | int64 C | int64 comp_offset[N+1] | int32 parent[C] | int32 cost given | float cost[N].
#include <algorithm>
#include <cstdio>
#include <cstdlib>
#include <string>
#include <vector>

#include "mm_layout.h"

using namespace mmk;

template <class N, class P>
static int bundles_bad(const GroupRec &G, const unsigned char *b)
{
    const N *nr = (const N *)b;
    const P *paths = (const P *)(b + G.path_off);
    int bad = 0, comp = 0;
    for (int k = 0; k < G.nbundle; ++k) {
        if (nr[k].comp0 != comp || nr[k].ncomp < 1) ++bad;
        comp += nr[k].ncomp;
        int covered = 0;
        for (int p = nr[k].path0; p < nr[k].path0 + nr[k].npath; ++p) {
            if (paths[p].head < nr[k].comp0 || paths[p].end > comp) ++bad;
            covered += paths[p].end - paths[p].head;
        }
        if (covered != nr[k].ncomp) ++bad;
    }
    return bad + (comp != G.ncomp);
}

int main(int argc, char **argv)
{
    if (argc != 5) return 2;
    FILE *f = std::fopen(argv[1], "rb");
    if (!f) return 2;
    int32_t N, given;
    int64_t C;
    if (std::fread(&N, 4, 1, f) != 1 || std::fread(&C, 8, 1, f) != 1) return 2;
    std::vector<int64_t> off((size_t)N + 1);
    std::vector<int32_t> par((size_t)C);
    std::vector<float> cost((size_t)N);
    if (std::fread(off.data(), 8, off.size(), f) != off.size() || std::fread(par.data(), 4, par.size(), f) != par.size() ||
        std::fread(&given, 4, 1, f) != 1 || std::fread(cost.data(), 4, cost.size(), f) != cost.size())
        return 2;
    std::fclose(f);
    const bool fp64 = std::atoi(argv[4]) != 0;
    std::vector<double> L((size_t)C, 10.0), D((size_t)C, 1.0);
    mmh::LayoutInput in{};
    in.N = N;
    in.comp_offset = off.data();
    in.parent = par.data();
    in.length_um = L.data();
    in.diam_um = D.data();
    in.cost = given ? cost.data() : nullptr;
    in.dt = 0.025;
    in.group_comps = std::atoi(argv[2]);
    in.sms = std::atoi(argv[3]);
    in.item_cost = fp64 ? 300 : 700;
    in.max_group_comps = fp64 ? 8192 : 1 << 30;
    in.smem_per_comp = fp64 ? 16 : 24;
    in.smem_per_path = fp64 ? 0 : 8;
    in.giant_smem_limit = fp64 ? 0 : 110 * 1024;
    in.big_smem_limit = fp64 ? 0 : 224 * 1024;
    mmh::Layout lay;
    bool invalid = false;
    const std::string err = mmh::build_layout(in, lay, &invalid);
    if (!err.empty()) {
        std::printf("layout error: %s\n", err.c_str());
        return 1;
    }
    int bad = 0, several = 0;
    int64_t comps = 0, paths = 0, covered = 0;
    const int nitems = (int)lay.groups.size();
    for (int g = 0; g < nitems; ++g) {
        const GroupRec &G = lay.groups[(size_t)g];
        const unsigned char *b = lay.meta.data() + G.meta_off;
        const bool wide = g >= lay.n_small + lay.n_big;
        bad += wide ? bundles_bad<NrnG, PathG>(G, b) : bundles_bad<NrnQ, PathQ>(G, b);
        if (wide) {
            bad += G.scratch0 != comps || G.pscratch0 != paths;
            comps += G.ncomp;
            paths += G.npath;
        }
        covered += G.ncomp;
        if (G.nneuron > 1) several = std::max(several, (int)G.ncomp);
    }
    bad += covered != C || comps != lay.giant_comps || paths != lay.giant_paths;
    std::printf("items=%d small=%d large=%d giant=%d huge=%d several=%d smem=%lld bad=%d giants=", nitems, lay.n_small,
                lay.n_big, nitems - lay.n_small - lay.n_big, lay.n_huge, several, (long long)lay.max_smem, bad);
    for (int g = lay.n_small + lay.n_big; g < nitems; ++g) std::printf("%d,", lay.groups[(size_t)g].ncomp);
    std::printf("\n");
    return bad ? 1 : 0;
}
