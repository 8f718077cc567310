// The columns that the busiest warp of the grid-resident engine walks (see
// test_grid_walk_host.py).
#include <cstdio>
#include <vector>

#include "snp_internal.h"

using namespace snp;

static std::vector<int32_t> starts(const std::vector<int32_t>& cols) {
    std::vector<int32_t> p(1, 0);
    for (int32_t c : cols) p.push_back(p.back() + c);
    return p;
}

int main() {
    int bad = 0;
    // one group per CTA: the longest list, shared by the group's warps
    bad += grid_longest_walk(starts({5, 9, 7}), 3, 4, 1) != 9;
    bad += grid_longest_walk(starts({5, 9, 7}), 3, 4, 4) != 3;
    bad += grid_longest_walk(starts({5, 9, 7}), 3, 8, 2) != 5;
    // groups 0, 2, 4, 6 on the first of two CTAs, one warp each or in turn
    const std::vector<int32_t> p = starts({1, 10, 2, 20, 4, 40, 8, 80});
    bad += grid_longest_walk(p, 2, 4, 1) != 80;
    bad += grid_longest_walk(p, 2, 2, 1) != 20 + 80;
    bad += grid_longest_walk(p, 2, 1, 1) != 10 + 20 + 40 + 80;
    // the widths come from the in-degrees: 300 neurons, one of 77 in-edges in the second group
    HostPack hp;
    hp.q = 300;
    for (int32_t i = 0; i < hp.q; ++i) {
        hp.perm.push_back(i);
        hp.indeg.push_back(i == 130 ? 77 : i % 3);
    }
    std::vector<int32_t> ptr;
    quad_list_starts(hp, 1, &ptr);
    bad += ptr != std::vector<int32_t>({0, 2, 79, 81});
    quad_list_starts(hp, 2, &ptr);
    bad += ptr != std::vector<int32_t>({0, 1, 40, 41});
    // more columns than 32 bits count: 5,000 groups with a list of 600,000 each
    hp.q = 5000 * kGroup;
    hp.perm.resize((size_t)hp.q);
    hp.indeg.assign((size_t)hp.q, 0);
    for (int32_t i = 0; i < hp.q; ++i) hp.perm[(size_t)i] = i;
    for (int32_t g = 0; g < 5000; ++g) hp.indeg[(size_t)g * kGroup + 5] = 600'000;
    bad += quad_list_starts(hp, 1, &ptr);
    bad += !quad_list_starts(hp, 2, &ptr) || ptr.back() != 5000 * 300'000;
    std::printf("bad=%d\n", bad);
    return bad;
}
