// Packs the tiled layout of 60,000 neurons with uniform in-degrees and with one
// neuron of 20,000 in-edges; prints both times (see test_pack_skew_time_host.py).
#include <algorithm>
#include <chrono>
#include <cstdio>
#include <random>
#include <vector>

#include "snp_internal.h"

using namespace snp;

static double pack_ms(int32_t hub) {
    const int32_t q = 60000;
    std::mt19937 rng(5);
    std::vector<std::vector<int32_t>> out((size_t)q);
    for (int32_t t = 0; t < q; ++t)
        for (int32_t u = 0; u < (t == 777 ? hub : 10); ++u) {
            const int32_t s = (int32_t)(rng() % (unsigned)q);
            if (s != t) out[(size_t)s].push_back(t);
        }
    std::vector<int64_t> ro((size_t)q + 1), so((size_t)q + 1, 0);
    std::vector<int32_t> one((size_t)q, 1), zero((size_t)q, 0), tg;
    for (int32_t i = 0; i < q; ++i) {
        std::vector<int32_t>& o = out[(size_t)i];
        std::sort(o.begin(), o.end());
        o.erase(std::unique(o.begin(), o.end()), o.end());
        tg.insert(tg.end(), o.begin(), o.end());
        ro[(size_t)i + 1] = i + 1;
        so[(size_t)i + 1] = (int64_t)tg.size();
    }
    snp_desc d{};
    d.q = q;
    d.init_spikes = one.data();
    d.rule_offsets = ro.data();
    d.rule_k = d.rule_c = d.rule_p = one.data();
    d.rule_j = d.rule_d = zero.data();
    d.num_syn = (int64_t)tg.size();
    d.syn_offsets = so.data();
    d.syn_targets = tg.data();
    int clusters[17] = {0};
    for (int p = 1; p <= 8; ++p) clusters[p] = 152 / p;
    double best = 1e30;
    for (int rep = 0; rep < 2; ++rep) {
        HostPack hp;
        TiledPack tp;
        if (pack_system(&d, false, false, 0, &hp)) return -1.0;
        const auto t = std::chrono::steady_clock::now();
        if (pack_tiled(&d, hp, 152, 225 * 1024, &tp, clusters)) return -1.0;
        best = std::min(best, std::chrono::duration<double, std::milli>(std::chrono::steady_clock::now() - t).count());
    }
    return best;
}

int main() {
    const double even = pack_ms(10), skewed = pack_ms(20000);
    std::printf("%.3f %.3f\n", even, skewed);
    return even > 0.0 && skewed > 0.0 ? 0 : 1;
}
