// Packs 128 neurons with the same long in-list, once with sources that all
// share a bank of shared memory and once with mixed ones; prints both times
// (see test_pack_time_host.py).
#include <algorithm>
#include <chrono>
#include <cstdio>
#include <vector>

#include "snp_internal.h"

using namespace snp;

static double pack_ms(bool one_bank) {
    const int32_t q = 65408;
    std::vector<int64_t> ro((size_t)q + 1), so((size_t)q + 1, 0);
    std::vector<int32_t> one((size_t)q, 1), zero((size_t)q, 0), tg;
    for (int32_t i = 0; i < q; ++i) {
        ro[(size_t)i + 1] = i + 1;
        // slots keep the caller's order here, so neuron i's emission lies in bank i / 4 mod 32
        const bool source = i >= kGroup && (one_bank ? (i / 4) % 32 == 0 : i % 32 == i / 128 * 4 % 32);
        for (int32_t t = 0; source && t < kGroup; ++t) tg.push_back(t);
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
    double best = 1e30;
    for (int rep = 0; rep < 3; ++rep) {
        HostPack hp;
        if (pack_system(&d, false, false, 8192, &hp, true)) return -1.0;
        const auto t = std::chrono::steady_clock::now();
        pack_in_quads(&d, &hp);
        best = std::min(best, std::chrono::duration<double, std::milli>(std::chrono::steady_clock::now() - t).count());
    }
    return best;
}

int main() {
    const double mixed = pack_ms(false), shared = pack_ms(true);
    std::printf("%.3f %.3f\n", mixed, shared);
    return mixed > 0.0 && shared > 0.0 ? 0 : 1;
}
