// snp_step_noalloc: the pull step for callers that must not allocate.
//
// Some callers cannot call cudaMalloc: code running inside a host framework
// that owns every byte of device memory (a plugin or custom operator whose
// framework hands out memory only through its own pool), or latency-critical
// loops where an allocation may synchronize the device at an unpredictable
// moment.  This entry point takes the system and its state in the caller's
// device arrays and keeps its own working buffers (the two emission vectors
// and a few flag words) in one file-scope device array of fixed size, so it
// allocates nothing.
//
// One cooperative launch runs all steps of a call (k_na_run): every CTA owns a
// contiguous range of neurons whose state, in-neighbour list and rules it
// keeps in shared memory as far as they fit; emissions go through L2, and the
// CTAs meet at a counter after every step.  A launch per step spent most of
// its time on starting and on two dependent trips to L2 per in-edge and per
// rule field (65,537 neurons of 10 in-edges: 16.4 us per step); it remains for
// devices that cannot hold the one launch (k_na_step).  Every index
// read from the caller's arrays is bounds-checked, and so are the fields of
// every rule a step fires (the ranges snp_create enforces on the host:
// k, j, c >= 0, p and d in [0, 65535], no delay on a forgetting rule) and the
// number of rules of a neuron; a bad one sets an error flag and the call
// returns SNP_ERR_INVALID instead of silently packing an out-of-range value.
#include <cuda_runtime.h>

#include <algorithm>
#include <mutex>
#include <string>

#include "device_common.cuh"
#include "noalloc_plan.h"
#include "quad.cuh"
#include "snp_internal.h"

namespace snp {

// ---- the static scratch ----------------------------------------------------
// Layout (32-bit words): [0, 16) flag words (words 8 to 11 are the two 64-bit
// barrier counters), [16, 24) step counters (four 64-bit values), then two
// emission vectors of SNP_NOALLOC_MAX_Q + 1 words (the spikes sent; k_na_step
// adds the selected rule).
constexpr int kNaFlagWords = 16;
constexpr int kNaStepWords = 8;
constexpr long long kNaEWords = (long long)SNP_NOALLOC_MAX_Q + 1;
constexpr long long kNaWords = kNaFlagWords + kNaStepWords + 2 * kNaEWords;
enum : int { kNaAct0 = 0, kNaHalted = 3, kNaOverflow = 4, kNaInvalid = 5, kNaTimeout = 6, kNaCounters = 8 };
enum : int { kNaBase = 0, kNaStart = 1, kNaExec = 2, kNaHalt = 3 };

static __device__ __align__(256) uint32_t g_noalloc_scratch[kNaWords];

struct NaSys {
    int32_t q;
    long long m;
    const int32_t* rule_off;
    const int32_t* rk;
    const int32_t* rj;
    const int32_t* rc;
    const int32_t* rp;
    const int32_t* rd;
    const int32_t* in_off;
    const int32_t* in_src;
    long long nin;
    int32_t* C;
    int32_t* D;
    int32_t* P;
    int32_t* S;
    uint32_t* scratch;  // device address of g_noalloc_scratch
    uint64_t seed;
};

__device__ __forceinline__ uint32_t* na_flags(const NaSys& s) { return s.scratch; }
__device__ __forceinline__ unsigned long long* na_steps(const NaSys& s) {
    return reinterpret_cast<unsigned long long*>(s.scratch + kNaFlagWords);
}
__device__ __forceinline__ uint32_t* na_e(const NaSys& s, unsigned long long k) {
    return s.scratch + kNaFlagWords + kNaStepWords + (k & 1ull) * kNaEWords;
}

__device__ __forceinline__ RuleF na_rule(const NaSys& s, int32_t r) {
    RuleF f;
    f.k = s.rk[r];
    f.j = s.rj[r];
    f.c = s.rc[r];
    f.p = s.rp[r];
    f.d = s.rd[r];
    return f;
}

// The field ranges snp_create's validation enforces on the host; the status
// word and the emission words below hold p and d in 16 bits.
__device__ __forceinline__ bool na_rule_ok(const RuleF& f) {
    return f.k >= 0 && f.j >= 0 && f.c >= 0 && f.p >= 0 && f.p <= kMaxP && f.d >= 0 && f.d <= kMaxDelay &&
           (f.p != 0 || f.d == 0);
}

// A rule staged in shared memory: its test without a division (the constants
// of build_test_records, for any j) and its outcome.  Rules with a field out
// of range are left to the caller's arrays.
struct NaRule {
    uint32_t k, c, j, M;  // M = 0: the remainder is x & mask
    uint32_t pd;          // p | d << 16
    uint32_t how;         // sh | kNaMaskJ | kNaOdd
};
constexpr uint32_t kNaMaskJ = 64u;  // j is a power of two: mask j - 1, else no mask
constexpr uint32_t kNaOdd = 128u;   // a field out of range

__device__ __forceinline__ NaRule na_stage(const RuleF& f) {
    NaRule r;
    r.k = (uint32_t)f.k;
    r.c = (uint32_t)f.c;
    r.j = (uint32_t)f.j;
    r.M = 0u;
    r.pd = 0u;
    r.how = kNaOdd;
    if (!na_rule_ok(f)) return r;
    r.pd = (uint32_t)f.p | ((uint32_t)f.d << 16);
    r.how = 0u;
    if (f.j > 0 && (r.j & (r.j - 1u)) == 0u) {
        r.how = kNaMaskJ;
    } else if (f.j > 0) {
        const uint32_t l = 32u - (uint32_t)__clz((int)(r.j - 1u));  // ceil(log2 j), j >= 3
        r.M = (uint32_t)(((1ull << (31u + l)) + r.j - 1ull) / r.j);
        r.how = l - 1u;
    }
    return r;
}
__device__ __forceinline__ bool na_applies(uint32_t n, const NaRule& f) {
    const uint32_t x = n - f.k;
    const uint32_t r = (f.how & kNaMaskJ) ? (x & (f.j - 1u)) : x - (__umulhi(x, f.M) >> (f.how & 31u)) * f.j;
    return n >= f.k && n >= f.c && r == 0u;
}

// A CTA's rules: the staged ones [lo, hi), the rest in the caller's arrays.
struct NaRules {
    const NaRule* staged;
    int32_t lo, hi;
};
__device__ __forceinline__ bool na_rule_applies(const NaSys& s, const NaRules& rs, int32_t r, int32_t n) {
    if (r >= rs.lo && r < rs.hi && !(rs.staged[r - rs.lo].how & kNaOdd)) return na_applies((uint32_t)n, rs.staged[r - rs.lo]);
    return rule_applies(n, na_rule(s, r));
}
// c, p and d of rule r; false when a field is out of range.
__device__ __forceinline__ bool na_outcome(const NaSys& s, const NaRules& rs, int32_t r, int32_t* c, int32_t* p, int32_t* d) {
    if (r >= rs.lo && r < rs.hi && !(rs.staged[r - rs.lo].how & kNaOdd)) {
        const NaRule& f = rs.staged[r - rs.lo];
        *c = (int32_t)f.c;
        *p = (int32_t)(f.pd & 0xffffu);
        *d = (int32_t)(f.pd >> 16);
        return true;
    }
    const RuleF f = na_rule(s, r);
    *c = f.c;
    *p = f.p;
    *d = f.d;
    return na_rule_ok(f);
}

// Select phase of neuron j at step k on the caller's state; same rules as
// select_neuron in device_common.cuh, over rule fields held as separate arrays.
// *bad is set when a rule the step fires has a field out of range (the step
// then treats the neuron as idle).
template <int SEL>
__device__ __forceinline__ SelOut na_select(const NaSys& s, const NaRules& rs, int32_t j, int32_t r0, int32_t r1,
                                            int32_t n, uint32_t st, unsigned long long k, bool* bad) {
    SelOut o;
    o.c_after = n;
    o.emit = 0;
    o.s = -1;
    int32_t c, p, d;
    const uint32_t pend = st >> kPendShift;
    if (pend != 0u) {
        o.active = true;
        if ((st & kDMask) == 0u) {
            if (!na_outcome(s, rs, r0 + (int32_t)pend - 1, &c, &p, &d)) {
                *bad = true;
                o.active = false;
            } else {
                o.emit = p;
            }
            o.st = 0u;
        } else {
            o.st = st - 1u;
        }
        return o;
    }
    o.st = 0u;
    o.active = false;
    int32_t pick = -1;
    if (SEL == SNP_SELECT_FIRST) {
        for (int32_t r = r0; r < r1 && pick < 0; ++r)
            if (na_rule_applies(s, rs, r, n)) pick = r;
    } else if (r1 - r0 <= 32) {  // one pass: bit i = rule r0 + i applies
        uint32_t m = 0u;
        for (int32_t r = r0; r < r1; ++r) m |= (na_rule_applies(s, rs, r, n) ? 1u : 0u) << (r - r0);
        uint32_t idx = 0u;
        if ((m & (m - 1u)) != 0u) idx = __umulhi(philox_draw(k, (uint32_t)j, s.seed), (uint32_t)__popc(m));
        for (; idx > 0u; --idx) m &= m - 1u;
        if (m != 0u) pick = r0 + __ffs(m) - 1;
    } else {
        int32_t cnt = 0;
        for (int32_t r = r0; r < r1; ++r) cnt += na_rule_applies(s, rs, r, n) ? 1 : 0;
        if (cnt > 0) {
            int32_t idx = cnt > 1 ? (int32_t)__umulhi(philox_draw(k, (uint32_t)j, s.seed), (uint32_t)cnt) : 0;
            for (int32_t r = r0; r < r1 && pick < 0; ++r)
                if (na_rule_applies(s, rs, r, n) && idx-- == 0) pick = r;
        }
    }
    if (pick >= 0) {
        if (!na_outcome(s, rs, pick, &c, &p, &d)) {
            *bad = true;
            return o;
        }
        o.active = true;
        o.s = pick - r0;
        o.c_after = n - c;
        if (d == 0)
            o.emit = p;
        else
            o.st = ((uint32_t)(o.s + 1) << kPendShift) | (uint32_t)(d - 1);
    }
    return o;
}

constexpr int kNaThreads = 512;

// Runs up to n steps from the base step.  Shared memory (smem bytes), for the
// CTA's N neurons: spikes, status words, first rules, list starts, the rules
// chosen at two steps; then as many of the CTA's in-neighbours and rules as fit
// (all or none of each).  more: a further launch of the same call.
template <int SEL>
__global__ void __launch_bounds__(kNaThreads, 1) k_na_run(const __grid_constant__ NaSys s, long long n, int N, int smem,
                                                         int more) {
    extern __shared__ __align__(16) unsigned char sm[];
    __shared__ int s_go;
    uint32_t* fl = na_flags(s);
    unsigned long long* steps = na_steps(s);
    if (more && __ldcg(fl + kNaHalted) != 0u) return;
    const int32_t lo = (int32_t)blockIdx.x * N, own = min(N, s.q - lo);
    int32_t* Csm = reinterpret_cast<int32_t*>(sm);
    uint32_t* Ssm = reinterpret_cast<uint32_t*>(Csm + N);
    int32_t* rsm = reinterpret_cast<int32_t*>(Ssm + N);  // first rule; second half: past the last
    int32_t* osm = rsm + 2 * N;                          // list start; second half: end
    int16_t* chosen = reinterpret_cast<int16_t*>(osm + 2 * N);  // of step k at (k & 1) * N
    const int used = (int)na_state_bytes(N);
    const unsigned long long base = steps[kNaBase];
    // what the CTA's first and last offsets span, when it is in range and fits
    int left = smem - used;
    NaRules rs{reinterpret_cast<const NaRule*>(sm + used), 0, 0};
    {
        const int32_t a = s.rule_off[lo], b = s.rule_off[lo + own];
        if (a >= 0 && a <= b && (long long)b <= s.m && (long long)(b - a) * (long long)sizeof(NaRule) <= left) {
            rs.lo = a;
            rs.hi = b;
        }
        // counted from 0: a rule id near INT32_MAX plus a stride would wrap
        for (int32_t i = threadIdx.x; i < rs.hi - rs.lo; i += blockDim.x)
            const_cast<NaRule*>(rs.staged)[i] = na_stage(na_rule(s, rs.lo + i));
    }
    const int rbytes = (int)((rs.hi - rs.lo) * (int)sizeof(NaRule));
    left -= rbytes;
    int32_t* const esm = reinterpret_cast<int32_t*>(sm + used + rbytes);
    int32_t e_lo = 0, e_hi = 0;  // staged in-neighbours
    {
        const int32_t a = s.in_off[lo], b = s.in_off[lo + own];
        if (a >= 0 && a <= b && (long long)b <= s.nin && (long long)(b - a) * 4 <= left) {
            e_lo = a;
            e_hi = b;
        }
        for (int32_t i = threadIdx.x; i < e_hi - e_lo; i += blockDim.x) esm[i] = s.in_src[e_lo + i];
    }
    for (int i = threadIdx.x; i < own; i += blockDim.x) {
        const int32_t j = lo + i;
        int32_t r0 = s.rule_off[j], r1 = s.rule_off[j + 1];
        const int32_t c = s.C[j], P = s.P[j], D = s.D[j];
        bool ok = r0 >= 0 && r0 <= r1 && (long long)r1 <= s.m && r1 - r0 <= kMaxRulesPerNeuron && c >= 0;
        uint32_t st = 0u;
        if (P != -1) {
            ok = ok && P >= r0 && P < r1 && D >= 0 && D <= (int32_t)kDMask;
            st = ((uint32_t)(P - r0 + 1) << kPendShift) | ((uint32_t)D & kDMask);
        } else {
            ok = ok && D == 0;  // a neuron can only be closed by a pending rule
        }
        if (!ok) {  // idle for the rest of the call
            atomicOr(fl + kNaInvalid, 1u);
            r0 = r1 = 0;
            st = 0u;
        }
        Csm[i] = c;
        Ssm[i] = st;
        rsm[i] = r0;
        rsm[N + i] = r1;
        osm[i] = s.in_off[j];
        osm[N + i] = s.in_off[j + 1];
    }
    __syncthreads();
    // select of step `base`; a thread keeps to its own neurons from here on
    bool act = false, invalid = false;
    for (int i = threadIdx.x; i < own; i += blockDim.x) {
        const SelOut o = na_select<SEL>(s, rs, lo + i, rsm[i], rsm[N + i], Csm[i], Ssm[i], base, &invalid);
        Csm[i] = o.c_after;
        Ssm[i] = o.st;
        chosen[(int)(base & 1ull) * N + i] = (int16_t)o.s;
        na_e(s, base)[lo + i] = (uint32_t)o.emit;
        act |= o.active;
    }
    uint32_t seen[2] = {0u, 0u};  // thread 0: active arrivals so far, by counter
    long long exec = 0;
    bool halted = false;
    for (long long t = 0; t < n; ++t) {
        // every CTA's emissions of step base + t are written: meet
        const bool any = __syncthreads_or(act);
        if (threadIdx.x == 0) {
            const int go = grid_meet(reinterpret_cast<unsigned long long*>(fl + kNaCounters), t, any, seen);
            if (go < 0) atomicOr(fl + kNaTimeout, 1u);
            s_go = go;
        }
        __syncthreads();
        if (s_go <= 0) {
            halted = s_go == 0;  // the same in every CTA
            break;
        }
        const unsigned long long kg = base + (unsigned long long)t, ks = kg + 1ull;
        const uint32_t* const Ek = na_e(s, kg);
        act = false;
        for (int i = threadIdx.x; i < own; i += blockDim.x) {
            const int32_t j = lo + i, a = osm[i], b = osm[N + i];
            long long sum = 0;
            if (a < 0 || a > b || (long long)b > s.nin) {
                invalid = true;
            } else {
                // eight emissions in flight: an index out of range gives none.
                // What is left is counted down: a list may end at INT32_MAX.
                auto gather = [&](const int32_t* p) {
                    for (int32_t left = b - a; left > 0; left -= 8, p += 8) {
                        uint32_t v[8];
#pragma unroll
                        for (int u = 0; u < 8; ++u) {
                            const bool there = u < left;
                            const int32_t x = there ? p[u] : 0;
                            const bool in = x >= 0 && x < s.q;
                            invalid |= !in;
                            v[u] = there && in ? __ldcg(Ek + x) : 0u;
                        }
#pragma unroll
                        for (int u = 0; u < 8; ++u) sum += (long long)v[u];
                    }
                };
                if (a >= e_lo && b <= e_hi)
                    gather(esm + (a - e_lo));
                else
                    gather(s.in_src + a);
            }
            int32_t c = Csm[i];
            const uint32_t st = Ssm[i];
            if ((st >> kPendShift) == 0u) {
                long long nc = (long long)c + sum;
                if (nc > 2147483647ll) {
                    atomicOr(fl + kNaOverflow, 1u);
                    nc = 2147483647ll;
                }
                c = (int32_t)nc;
            }
            if (t + 1 < n) {
                const SelOut o = na_select<SEL>(s, rs, j, rsm[i], rsm[N + i], c, st, ks, &invalid);
                c = o.c_after;
                Ssm[i] = o.st;
                chosen[(int)(ks & 1ull) * N + i] = (int16_t)o.s;
                na_e(s, ks)[j] = (uint32_t)o.emit;
                act |= o.active;
            }
            Csm[i] = c;
        }
        ++exec;
    }
    if (invalid) atomicOr(fl + kNaInvalid, 1u);
    const int last = (int)((base + (unsigned long long)exec + 1ull) & 1ull) * N;  // the last executed step's choices
    for (int i = threadIdx.x; i < own; i += blockDim.x) {
        const int32_t j = lo + i, r0 = rsm[i];
        const uint32_t st = Ssm[i], pend = st >> kPendShift;
        s.C[j] = Csm[i];
        s.D[j] = pend ? (int32_t)(st & kDMask) : 0;
        s.P[j] = pend ? r0 + (int32_t)pend - 1 : -1;
        if (exec > 0) s.S[j] = chosen[last + i] >= 0 ? r0 + chosen[last + i] : -1;
    }
    // every CTA has read the base step and the halt flag: it was at a barrier since
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        steps[kNaBase] = base + (unsigned long long)exec;
        steps[kNaExec] = base + (unsigned long long)exec - steps[kNaStart];
        fl[kNaHalted] = halted ? 1u : 0u;
    }
}

// One step with the state in the caller's arrays, a launch of its own: for
// devices, partitions and contexts that cannot hold k_na_run's grid with the
// neurons' state in shared memory (na_plan).  An emission word holds the spikes
// sent (low 16 bits) and 1 + the local index of the selected rule.
template <bool GATHER, bool SELECT, int SEL>
__global__ void __launch_bounds__(256) k_na_step(NaSys s, int32_t t) {
    uint32_t* fl = na_flags(s);
    unsigned long long* steps = na_steps(s);
    const unsigned long long kg = steps[kNaBase] + (unsigned long long)t;
    const unsigned long long ks = GATHER ? kg + 1ull : kg;
    if (GATHER) {
        if (ld_volatile(fl + kNaHalted)) return;
        if (ld_volatile(fl + kNaAct0 + (int)(kg % 3ull)) == 0u) {
            if (threadIdx.x == 0) {
                steps[kNaHalt] = kg;
                __threadfence();
                atomicExch(fl + kNaHalted, 1u);
            }
            return;
        }
        if (SELECT && blockIdx.x == 0 && threadIdx.x == 0) fl[kNaAct0 + (int)((kg + 2ull) % 3ull)] = 0u;
    }
    const int32_t j = (int32_t)(blockIdx.x * blockDim.x + threadIdx.x);
    bool active = false;
    if (j < s.q) {
        int32_t r0 = s.rule_off[j], r1 = s.rule_off[j + 1];
        int32_t c = s.C[j];
        bool ok = r0 >= 0 && r0 <= r1 && (long long)r1 <= s.m && r1 - r0 <= kMaxRulesPerNeuron && c >= 0;
        const int32_t P = s.P[j], D = s.D[j];
        uint32_t st = 0u;
        if (P != -1) {
            ok = ok && P >= r0 && P < r1 && D >= 0 && D <= (int32_t)kDMask;
            st = ((uint32_t)(P - r0 + 1) << kPendShift) | ((uint32_t)D & kDMask);
        } else {
            ok = ok && D == 0;  // a neuron can only be closed by a pending rule
        }
        if (!ok) {
            atomicOr(fl + kNaInvalid, 1u);
            r0 = r1 = 0;
            st = 0u;
        }
        if (GATHER) {
            const uint32_t* Ek = na_e(s, kg);
            const int32_t a = s.in_off[j], b = s.in_off[j + 1];
            long long sum = 0;
            if (a < 0 || a > b || (long long)b > s.nin) {
                atomicOr(fl + kNaInvalid, 1u);
            } else {
                for (int32_t e = a; e < b; ++e) {
                    const int32_t src = s.in_src[e];
                    if (src < 0 || src >= s.q) {
                        atomicOr(fl + kNaInvalid, 1u);
                        continue;
                    }
                    sum += (long long)(Ek[src] & 0xffffu);
                }
            }
            if ((st >> kPendShift) == 0u) {
                long long nc = (long long)c + sum;
                if (nc > 2147483647ll) {
                    atomicOr(fl + kNaOverflow, 1u);
                    nc = 2147483647ll;
                }
                c = (int32_t)nc;
            }
            // step kg is executed: publish its spiking vector
            const uint32_t sel = Ek[j] >> 16;
            s.S[j] = sel ? r0 + (int32_t)sel - 1 : -1;
        }
        if (SELECT) {
            const NaRules none{nullptr, 0, 0};
            bool bad = false;
            const SelOut o = na_select<SEL>(s, none, j, r0, r1, c, st, ks, &bad);
            if (bad) atomicOr(fl + kNaInvalid, 1u);
            c = o.c_after;
            active = o.active;
            na_e(s, ks)[j] = ((uint32_t)o.emit & 0xffffu) | ((uint32_t)(o.s + 1) << 16);
            const uint32_t pend = o.st >> kPendShift;
            s.P[j] = pend ? r0 + (int32_t)pend - 1 : -1;
            s.D[j] = pend ? (int32_t)(o.st & kDMask) : 0;
        }
        s.C[j] = c;
    }
    if (SELECT) {
        if (__syncthreads_or(active) && threadIdx.x == 0) {
            uint32_t* a = fl + kNaAct0 + (int)(ks % 3ull);
            if (ld_volatile(a) == 0u) atomicExch(a, 1u);
        }
    }
}

// Clears the flags and sets the base step (first), or clears the barrier
// counters for a further launch of the call.
__global__ void k_na_begin(NaSys s, unsigned long long k0, int first) {
    uint32_t* fl = na_flags(s);
    if (threadIdx.x < kNaFlagWords && (first || threadIdx.x >= kNaCounters)) fl[threadIdx.x] = 0u;
    if (first && threadIdx.x == 0) {
        unsigned long long* st = na_steps(s);
        st[kNaBase] = k0;
        st[kNaStart] = k0;
        st[kNaExec] = 0ull;
        st[kNaHalt] = 0ull;
    }
}

__global__ void k_na_finish(NaSys s, int32_t tail) {
    if (threadIdx.x == 0 && blockIdx.x == 0) {
        unsigned long long* st = na_steps(s);
        if (ld_volatile(na_flags(s) + kNaHalted))
            st[kNaBase] = st[kNaHalt];
        else
            st[kNaBase] += (unsigned long long)tail;
        st[kNaExec] = st[kNaBase] - st[kNaStart];
    }
}

template <bool G, bool S>
static void na_launch(const NaSys& s, int32_t t, int sel, cudaStream_t st) {
    const unsigned grid = (unsigned)((s.q + 255) / 256);
    if (sel == SNP_SELECT_FIRST)
        k_na_step<G, S, SNP_SELECT_FIRST><<<grid, 256, 0, st>>>(s, t);
    else
        k_na_step<G, S, SNP_SELECT_PHILOX><<<grid, 256, 0, st>>>(s, t);
}

// Device address of the scratch array, looked up once per device.  The
// cached address belongs to the device's primary context: cudaDeviceReset
// makes it stale, which the library cannot detect (documented in snp.h).
static std::mutex g_na_mu;
static uint32_t* g_na_ptr[64] = {nullptr};

static int na_scratch(uint32_t** out) {
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) {
        cudaGetLastError();
        return fail(SNP_ERR_CUDA, "no current CUDA device");
    }
    std::lock_guard<std::mutex> lk(g_na_mu);
    if (!g_na_ptr[dev]) {
        void* p = nullptr;
        cudaError_t e = cudaGetSymbolAddress(&p, g_noalloc_scratch);
        if (e != cudaSuccess || !p) {
            cudaGetLastError();
            return fail(SNP_ERR_CUDA, std::string("cudaGetSymbolAddress: ") + cudaGetErrorString(e));
        }
        g_na_ptr[dev] = (uint32_t*)p;
    }
    *out = g_na_ptr[dev];
    return SNP_OK;
}

// All steps by k_na_run.
static cudaError_t na_run(const NaSys& s, const NaPlan& pl, int cap, int select, uint64_t step, int64_t n,
                          cudaStream_t st) {
    auto fn = select == SNP_SELECT_FIRST ? k_na_run<SNP_SELECT_FIRST> : k_na_run<SNP_SELECT_PHILOX>;
    // the same bound for every launch: threads may launch different sizes at once
    cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, cap - 1024);
    for (int64_t done = 0; done < n && e == cudaSuccess; done += kLaunchMaxSteps) {
        k_na_begin<<<1, 32, 0, st>>>(s, (unsigned long long)step, done == 0 ? 1 : 0);
        if ((e = cudaGetLastError()) != cudaSuccess) break;
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3((unsigned)pl.G);
        cfg.blockDim = dim3(kNaThreads);
        cfg.dynamicSmemBytes = (size_t)pl.smem;
        cfg.stream = st;
        cudaLaunchAttribute at[1];
        at[0].id = cudaLaunchAttributeCooperative;
        at[0].val.cooperative = 1;
        cfg.attrs = at;
        cfg.numAttrs = 1;
        e = cudaLaunchKernelEx(&cfg, fn, s, (long long)std::min<int64_t>(n - done, kLaunchMaxSteps), pl.N, pl.smem,
                               done > 0 ? 1 : 0);
    }
    return e;
}

// All steps by a launch of k_na_step each.
static cudaError_t na_run_steps(const NaSys& s, int select, uint64_t step, int64_t n, cudaStream_t st) {
    k_na_begin<<<1, 32, 0, st>>>(s, (unsigned long long)step, 1);
    na_launch<false, true>(s, 0, select, st);
    for (int64_t t = 0; t + 1 < n; ++t) na_launch<true, true>(s, (int32_t)t, select, st);
    na_launch<true, false>(s, (int32_t)(n - 1), select, st);
    k_na_finish<<<1, 32, 0, st>>>(s, (int32_t)n);
    return cudaGetLastError();
}

}  // namespace snp

using namespace snp;

extern "C" int snp_noalloc_on(const snp_device_system* d, int32_t select, uint64_t seed, uint64_t step, int64_t n,
                              void* stream, int64_t* steps_done, int32_t sms, int32_t cap) {
    if (steps_done) *steps_done = 0;
    if (!d) return fail(SNP_ERR_INVALID, "system is NULL");
    if (d->q < 1 || d->q > SNP_NOALLOC_MAX_Q)
        return fail(SNP_ERR_INVALID, "q must be in [1, SNP_NOALLOC_MAX_Q] (262,144) for snp_step_noalloc");
    if (d->m < 0 || d->m > INT32_MAX - 1 || d->num_in < 0 || d->num_in > INT32_MAX)
        return fail(SNP_ERR_INVALID, "m or num_in out of range");
    if (!d->rule_offsets || (d->m > 0 && (!d->rule_k || !d->rule_j || !d->rule_c || !d->rule_p || !d->rule_d)) ||
        !d->in_offsets || (d->num_in > 0 && !d->in_sources) || !d->C || !d->D || !d->P || !d->S)
        return fail(SNP_ERR_INVALID, "NULL array");
    if (select != SNP_SELECT_FIRST && select != SNP_SELECT_PHILOX) return fail(SNP_ERR_INVALID, "bad select");
    if (n < 0 || n > INT32_MAX) return fail(SNP_ERR_INVALID, "n must be in [0, 2^31 - 1]");
    if (n == 0) return SNP_OK;
    uint32_t* scratch = nullptr;
    int rc = na_scratch(&scratch);
    if (rc) return rc;
    NaSys s;
    s.q = d->q;
    s.m = d->m;
    s.rule_off = d->rule_offsets;
    s.rk = d->rule_k;
    s.rj = d->rule_j;
    s.rc = d->rule_c;
    s.rp = d->rule_p;
    s.rd = d->rule_d;
    s.in_off = d->in_offsets;
    s.in_src = d->in_sources;
    s.nin = d->num_in;
    s.C = d->C;
    s.D = d->D;
    s.P = d->P;
    s.S = d->S;
    s.scratch = scratch;
    s.seed = seed;
    cudaStream_t st = (cudaStream_t)stream;
    const NaPlan pl = na_plan(d->q, sms, cap);
    cudaError_t le = pl.G > 0 ? na_run(s, pl, cap, select, step, n, st) : cudaErrorCooperativeLaunchTooLarge;
    if (le == cudaErrorCooperativeLaunchTooLarge) {  // the state, or the grid, does not fit at once
        cudaGetLastError();
        le = na_run_steps(s, select, step, n, st);
    }
    if (le != cudaSuccess) cudaGetLastError();
    if (le != cudaSuccess) return fail(SNP_ERR_CUDA, std::string("snp_step_noalloc launch: ") + cudaGetErrorString(le));
    if (!steps_done) return SNP_OK;
    uint32_t fl[kNaFlagWords];
    unsigned long long sw[4];
    if (cudaMemcpyAsync(fl, scratch, sizeof(fl), cudaMemcpyDeviceToHost, st) != cudaSuccess ||
        cudaMemcpyAsync(sw, scratch + kNaFlagWords, sizeof(sw), cudaMemcpyDeviceToHost, st) != cudaSuccess ||
        cudaStreamSynchronize(st) != cudaSuccess) {
        cudaError_t e = cudaGetLastError();
        return fail(SNP_ERR_CUDA, std::string("snp_step_noalloc: ") + cudaGetErrorString(e));
    }
    *steps_done = (int64_t)sw[kNaExec];
    if (fl[kNaTimeout]) return fail(SNP_ERR_TIMEOUT, "a bounded device wait gave up");
    if (fl[kNaInvalid]) return fail(SNP_ERR_INVALID, "an index or a fired rule's field in the device arrays was out of range");
    if (fl[kNaOverflow]) return fail(SNP_ERR_OVERFLOW, "a spike count left the int32 range");
    return SNP_OK;
}

extern "C" int snp_step_noalloc(const snp_device_system* d, int32_t select, uint64_t seed, uint64_t step, int64_t n,
                                void* stream, int64_t* steps_done) {
    int dev = 0, sms = 0, cap = 0, coop = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&cap, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev) != cudaSuccess) {
        cudaGetLastError();
        sms = cap = coop = 0;  // the arguments are checked before the device
    }
    return snp_noalloc_on(d, select, seed, step, n, stream, steps_done, coop ? sms : 0, cap);
}
