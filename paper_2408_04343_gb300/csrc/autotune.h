// Online autotuner of a batch's resident launches.  Host code only, checked on
// the CPU.
#pragma once

#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <map>
#include <tuple>

namespace snp {

// A candidate is how many groups of 128 neurons one CTA may hold: a system of
// more takes a cluster of 2, 4 or 8 CTAs (kernels_cluster.cu), so a small bound
// shortens the largest systems and a large one spends fewer CTAs and barriers.
//
// Rounds are compared with their like only: by bits per emission, log2 of the
// largest system and log2 of the round's work (a small round says nothing about
// a large one: systems join piecemeal at first and leave one by one).  For each
// such level every candidate is tried on one real round (the work is not
// wasted: results do not depend on the candidate), then the fastest by measured
// synaptic updates per second is used.  A level met for the first time takes
// the choice of the nearest level that has tried them all, so a load that rises
// or falls through many levels does not start over at each of them.
//
// With SNP_AUTOTUNE_CACHE naming a file, measurements are read at batch creation
// and written back at destroy, a line each: bits, log2 of the size + 64 x level,
// kFirst + candidate (smaller numbers belonged to an earlier set), work,
// seconds.  Lines without a level serve any level as its nearest.
class Autotune {
public:
    static constexpr int kN = 3;
    static constexpr int kFirst = 6;
    static int groups_of(int c) { return 16 << c; }

    // The candidate for a round of `work` synaptic updates.
    int pick(int e_bits, int log_q, double work) const {
        const int level = level_of(work);
        const auto it = stats_.find({e_bits, log_q, level});
        if (it != stats_.end() && it->second.tried() > 0) {
            for (int c = 0; c < kN; ++c)
                if (it->second.secs[c] == 0.0) return c;
            return it->second.best();
        }
        int choice = 0, apart = 1 << 30;
        for (const auto& kv : stats_) {
            if (std::get<0>(kv.first) != e_bits || std::get<1>(kv.first) != log_q || kv.second.tried() < kN) continue;
            const int away = std::abs(std::get<2>(kv.first) - level);
            if (away < apart) {
                apart = away;
                choice = kv.second.best();
            }
        }
        return choice;
    }
    void record(int e_bits, int log_q, int c, double work, double secs) { add(e_bits, log_q, level_of(work), c, work, secs); }

    void load(const char* path) {
        FILE* f = path ? std::fopen(path, "r") : nullptr;
        if (!f) return;
        int eb, lq, c;
        double w, t;
        while (std::fscanf(f, "%d %d %d %lf %lf", &eb, &lq, &c, &w, &t) == 5)
            if (c >= kFirst && c < kFirst + kN && lq >= 0) add(eb, lq % 64, lq / 64, c - kFirst, w, t);
        std::fclose(f);
    }
    void save(const char* path) const {
        FILE* f = path ? std::fopen(path, "w") : nullptr;
        if (!f) return;
        for (const auto& kv : stats_)
            for (int c = 0; c < kN; ++c)
                if (kv.second.secs[c] > 0.0)
                    std::fprintf(f, "%d %d %d %.6g %.6g\n", std::get<0>(kv.first),
                                 std::get<1>(kv.first) + 64 * std::get<2>(kv.first), c + kFirst, kv.second.work[c],
                                 kv.second.secs[c]);
        std::fclose(f);
    }

private:
    struct Stat {
        double work[kN] = {0, 0, 0};
        double secs[kN] = {0, 0, 0};
        int tried() const {
            int n = 0;
            for (int c = 0; c < kN; ++c) n += secs[c] > 0.0 ? 1 : 0;
            return n;
        }
        int best() const {
            int b = 0;
            for (int c = 1; c < kN; ++c)
                if (work[c] / secs[c] > work[b] / secs[b]) b = c;
            return b;
        }
    };
    // 1, 2, ...: work up to 3, from 4, from 8, ...
    static int level_of(double work) { return work < 4.0 ? 1 : std::ilogb(work); }
    void add(int e_bits, int log_q, int level, int c, double work, double secs) {
        Stat& st = stats_[{e_bits, log_q, level}];
        st.work[c] += work;
        st.secs[c] += secs > 1e-9 ? secs : 1e-9;
    }
    std::map<std::tuple<int, int, int>, Stat> stats_;  // by bits, log2 of the size, level (0: none given)
};

}  // namespace snp
