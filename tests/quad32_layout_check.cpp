// Packs a random system in quad order with 32-bit lists over packed emissions and
// decodes them back into in-edges (see test_quad32_layout_host.py).
#include <algorithm>
#include <cstdio>
#include <cstdlib>
#include <random>
#include <set>
#include <vector>

#include "snp_internal.h"

using namespace snp;

int main(int argc, char** argv) {
    if (argc != 5) return 2;
    const int32_t q = std::atoi(argv[1]), deg = std::atoi(argv[2]);
    std::mt19937 rng((unsigned)std::atoi(argv[3]));
    std::vector<int64_t> ro((size_t)q + 1), so((size_t)q + 1, 0);
    std::vector<int32_t> C0((size_t)q, 1), k((size_t)q, 1), j((size_t)q, 0), p((size_t)q, 1), dl((size_t)q, 0), tg;
    std::vector<std::vector<int32_t>> in((size_t)q);
    for (int32_t i = 0; i < q; ++i) {
        ro[(size_t)i + 1] = i + 1;
        std::set<int32_t> t;
        // a few hubs: targets are squared towards 0
        for (int n = q > 1 ? (int)(rng() % (unsigned)(deg + 1)) : 0; n > 0; --n) {
            const double u = (double)rng() / 4294967296.0;
            const int32_t x = (int32_t)(u * u * q);
            if (x != i) t.insert(x);
        }
        for (int32_t x : t) {
            tg.push_back(x);
            in[(size_t)x].push_back(i);
        }
        so[(size_t)i + 1] = (int64_t)tg.size();
    }
    snp_desc d{};
    d.q = q;
    d.init_spikes = C0.data();
    d.rule_offsets = ro.data();
    d.rule_k = k.data();
    d.rule_j = j.data();
    d.rule_c = k.data();
    d.rule_p = p.data();
    d.rule_d = dl.data();
    d.num_syn = (int64_t)tg.size();
    d.syn_offsets = so.data();
    d.syn_targets = tg.data();
    const int eb = std::atoi(argv[4]);  // bits per emission
    HostPack hp;
    if (pack_system(&d, false, false, 8192, &hp, true) || !hp.quads) return 3;
    pack_in_quads32(&d, &hp, eb);

    const int32_t ng = (q + kGroup - 1) / kGroup;
    std::vector<int32_t> neuron((size_t)(ng + 1) * kGroup, -1);  // place -> neuron
    for (int32_t g = 0; g < ng; ++g)
        for (int32_t l = 0; l < 32; ++l)
            for (int32_t u = 0; u < 4; ++u) {
                const int32_t s = quad_slot(g, l, u, q);
                if (s >= 0) neuron[(size_t)(g * kGroup + 4 * l + u)] = hp.perm[(size_t)s];
            }
    // the place an entry names: byte address of its word, first bit in the word
    long long bad = 0, edges = 0;
    const long long bytes = ((long long)ng * kGroup * eb / 8 + 31) / 16 * 16;  // of a packed vector
    auto place = [&](uint32_t e) -> int32_t {
        const long long word = e >> 8, bit = e & 255u;
        if (word % 4 != 0 || word + 4 > bytes || bit > 31 || (word * 8 + bit) % eb != 0) {
            ++bad;
            return ng * kGroup;
        }
        const long long x = (word * 8 + bit) / eb;
        if (x > (long long)ng * kGroup) {
            ++bad;
            return ng * kGroup;
        }
        return (int32_t)x;
    };
    const size_t cols = (size_t)hp.quad_ptr32[(size_t)ng];
    bad += hp.in_quads32.size() != (cols + kQuadSlack) * 128;
    for (int32_t g = 0; g < ng; ++g)
        for (int32_t l = 0; l < 32; ++l)
            for (int32_t u = 0; u < 4; ++u) {
                std::vector<int32_t> got;
                for (int32_t c = hp.quad_ptr32[(size_t)g]; c < hp.quad_ptr32[(size_t)g + 1]; ++c) {
                    const int32_t x = place(hp.in_quads32[((size_t)c * 32 + l) * 4 + u]);
                    if (x == ng * kGroup) continue;
                    if (neuron[(size_t)x] < 0)
                        ++bad;
                    else
                        got.push_back(neuron[(size_t)x]);
                }
                std::sort(got.begin(), got.end());
                const int32_t i = neuron[(size_t)(g * kGroup + 4 * l + u)];
                if (i < 0 ? !got.empty() : got != in[(size_t)i]) ++bad;
                edges += (long long)got.size();
            }
    for (size_t x = cols * 128; x < hp.in_quads32.size(); ++x) bad += place(hp.in_quads32[x]) != ng * kGroup;
    std::printf("bad=%lld edges=%lld num_syn=%lld\n", bad, edges, (long long)d.num_syn);
    return bad || edges != d.num_syn;
}
