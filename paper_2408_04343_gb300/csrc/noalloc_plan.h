// The one-launch form of snp_step_noalloc: how many neurons a CTA owns.  Host
// arithmetic only, checked on the CPU over made-up devices.
#pragma once

#include <algorithm>
#include <cstdint>

#include "snp_internal.h"

namespace snp {

struct NaPlan {
    int N, G, smem;  // neurons per CTA, CTAs (0: a launch per step instead), dynamic shared memory
};

// Shared memory that N neurons' state takes: spikes, status words, first and
// end rules, list starts and ends, the rules chosen at two steps.
SNP_HD inline long long na_state_bytes(long long n) { return (n * 28 + 15) / 16 * 16; }

// 128 neurons per CTA at least (fewer CTAs meet sooner), one CTA per SM at
// most, since the CTAs wait for one another.  Beside the state, what 1 KB per
// neuron holds of its rules and in-neighbours.  152 SMs of 227 KB hold the
// state of the largest system in 49 KB a CTA; below 32 such SMs it does not fit.
inline NaPlan na_plan(int32_t q, int32_t sms, int32_t cap) {
    NaPlan p{0, 0, 0};
    if (sms < 1) return p;
    const long long N = std::max<long long>(128, ((long long)q + sms - 1) / sms);
    if (na_state_bytes(N) > (long long)cap - 1024) return p;
    p.N = (int)N;
    p.G = (int)((q + N - 1) / N);
    p.smem = (int)std::min<long long>((long long)cap - 1024, N * 1024);
    return p;
}

}  // namespace snp

// snp_step_noalloc as on a device of sms SMs (0: no cooperative launches) with
// cap bytes of shared memory per CTA.
extern "C" int snp_noalloc_on(const snp_device_system* sys, int32_t select, uint64_t seed, uint64_t step, int64_t n,
                              void* stream, int64_t* steps_done, int32_t sms, int32_t cap);
