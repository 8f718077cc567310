// na_plan over made-up devices: what a CTA keeps in shared memory fits, and
// every neuron has a CTA (see test_noalloc_plan_host.py).
#include <cstdio>

#include "noalloc_plan.h"

using namespace snp;

int main() {
    long long bad = 0, one = 0, steps = 0;
    for (int cap : {48 * 1024, 100 * 1024, 164 * 1024, 228 * 1024 - 1024})
        for (int sms = 0; sms <= 200; ++sms)
            for (int q : {1, 127, 128, 129, 4096, 20000, 65537, 149000, 200001, SNP_NOALLOC_MAX_Q}) {
                const NaPlan p = na_plan(q, sms, cap);
                if (p.G == 0) {
                    ++steps;
                    // only where even an equal share of the neurons does not fit
                    const long long share = sms > 0 ? ((long long)q + sms - 1) / sms : 0;
                    bad += sms > 0 && 28 * (share < 128 ? 128 : share) + 15 <= cap - 1024;
                    continue;
                }
                ++one;
                bad += p.G < 1 || p.G > sms || (long long)p.G * p.N < q || (long long)(p.G - 1) * p.N >= q;
                bad += p.smem > cap - 1024 || 28ll * p.N > p.smem;
            }
    // the devices of the limit: 152 SMs hold every size, 18 SMs no longer the largest
    bad += na_plan(SNP_NOALLOC_MAX_Q, 152, 227 * 1024).G == 0 || na_plan(SNP_NOALLOC_MAX_Q, 18, 227 * 1024).G != 0;
    std::printf("bad=%lld one=%lld steps=%lld\n", bad, one, steps);
    return bad || !one || !steps;
}
