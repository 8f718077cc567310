// The ELL form and the uncompressed ("Sparse") form of the transition matrix.
//
// Both forms keep the paper's per-rule view: the spiking vector has one entry
// per rule (Sec. 2: S_k of length m), and spikes travel as (rule, value)
// pairs.  Em_k[r] = 1 when rule r emits at step k (it fired with d = 0, or
// its delay ran out), stored as bytes, double-buffered by step parity.
//
//  * ELL pull: each target neuron sums Em_k[r] * p over the (rule, p) pairs
//    of its in-ELL column (the transpose of M^s_Pi's +p rows, Sec. 4);
//  * ELL push: each emitting rule walks its column of M^s_Pi and adds p into
//    every open target with warp-aggregated atomics (Alg. 4's direction),
//    the columns dealt to warps in equal runs (push_balanced.cuh);
//  * dense: each neuron walks its column of M_Pi over all m rules and adds
//    Em_k[r] * M[r, j] (Alg. 3's direction); the (row block x neuron tile)
//    partial sums meet in an in-flow vector, and the select launch applies it.
// Consumption (-c) is applied when a rule is selected (the pair in row 0 of
// M^s_Pi is not walked): with delays a rule consumes at t and emits at t+d.
#include <cuda_runtime.h>

#include "device_common.cuh"
#include "kernels.h"
#include "push_balanced.cuh"
#include "quad.cuh"

namespace snp {

// Select for step ks on one slot, writing the per-rule emission bytes.
template <bool COMPACT, int SEL>
__device__ __forceinline__ bool ell_select_slot(const DevSys& s, const EllSys& e, int32_t slot, int32_t& c,
                                                unsigned long long ks) {
    const uint32_t st = s.st[slot];
    const int32_t r0 = rule_lo(s, slot), r1 = rule_hi(s, slot);
    const SelOut o = select_slot<COMPACT, SEL>(s, slot, c, st, ks);
    int32_t emitting = -1;  // local index of the rule that emits at ks
    if ((st >> kPendShift) != 0u && (st & kDMask) == 0u) emitting = (int32_t)(st >> kPendShift) - 1;
    else if (o.s >= 0 && o.emit > 0) emitting = o.s;
    uint8_t* Em = SNP_PICK(e.Em, ks);
    for (int32_t r = r0; r < r1; ++r) Em[r] = (r - r0) == emitting ? 1 : 0;
    c = o.c_after;
    SNP_PICK(s.S, ks)[slot] = o.s;
    s.st[slot] = o.st;
    return o.active;
}

// ELL pull: gather of step kg (+ select of kg+1), like k_step_pull.
template <bool GATHER, bool SELECT, bool COMPACT, int SEL>
__global__ void __launch_bounds__(256) k_ell_pull(DevSys s, EllSys e, int32_t t) {
    uint32_t* fl = s.flags;
    const unsigned long long kg = s.step[kStepBase] + (unsigned long long)t;
    const unsigned long long ks = GATHER ? kg + 1ull : kg;
    if (GATHER) {
        if (step_blocked(fl, s.step, kg)) return;
        if (SELECT && blockIdx.x == 0 && threadIdx.x == 0) fl[kFlagAct0 + (int)((kg + 2ull) % 3ull)] = 0u;
    }
    const int lane = threadIdx.x & 31;
    const int32_t slice = (int32_t)((blockIdx.x * blockDim.x + threadIdx.x) >> 5);
    const int32_t slot = slice * kSlice + lane;
    bool active = false;
    if (slice < s.nslices) {
        const bool valid = slot < s.q;
        int32_t c = valid ? s.C[slot] : 0;
        if (GATHER) {
            const uint8_t* __restrict__ Em = SNP_PICK(e.Em, kg);
            const int32_t b = __ldg(e.in_ptr + slice);
            const int32_t w = __ldg(e.in_ptr + slice + 1) - b;
            const int2* __restrict__ p = e.in_ent + (size_t)b * kSlice + lane;
            long long sum = 0;
            int32_t col = 0;
            for (; col + 4 <= w; col += 4) {
                const int2 a0 = __ldg(p + (col + 0) * kSlice), a1 = __ldg(p + (col + 1) * kSlice);
                const int2 a2 = __ldg(p + (col + 2) * kSlice), a3 = __ldg(p + (col + 3) * kSlice);
                sum += (Em[SNP_IDX(fl, 4, a0.x, e.m + 1)] ? a0.y : 0) + (Em[SNP_IDX(fl, 4, a1.x, e.m + 1)] ? a1.y : 0) +
                       (Em[SNP_IDX(fl, 4, a2.x, e.m + 1)] ? a2.y : 0) + (Em[SNP_IDX(fl, 4, a3.x, e.m + 1)] ? a3.y : 0);
            }
            for (; col < w; ++col) {
                const int2 a = __ldg(p + col * kSlice);
                sum += Em[SNP_IDX(fl, 4, a.x, e.m + 1)] ? a.y : 0;
            }
            if (valid && (s.st[slot] >> kPendShift) == 0u) {
                long long nc = (long long)c + sum;
                if (nc > 2147483647ll) {
                    atomicOr(fl + kFlagOverflow, 1u);
                    nc = 2147483647ll;
                }
                c = (int32_t)nc;
            }
        }
        if (SELECT && valid) active = ell_select_slot<COMPACT, SEL>(s, e, slot, c, ks);
        if (valid) s.C[slot] = c;
    }
    if (SELECT) raise_step_activity(fl, ks, active);
}

// All steps of an ELL pull call in one cooperative launch.  The step of
// k_ell_pull is bound by its random one-byte reads of Em, which L2 serves at
// some 2.6e11 a second.  Here the step's emitting rules are a bit vector (4
// bits per neuron) that every CTA copies into shared memory, a pair is one
// word instead of two, and the CTAs meet at a counter between steps
// (grid_meet) with their slices' state in shared memory.  262,144 neurons,
// 5.2M pairs, 48 steps with import and reads: 1,335 us before (27.8 a step), 583
// so (12.1), 496 of them this kernel.
constexpr int kEllThreads = 1024;

size_t ell_run_smem(const EllSys& e) { return (size_t)e.bit_words * 4 + (size_t)e.own * kSlice * 8; }

template <int SEL>
__global__ void __launch_bounds__(kEllThreads, 1)
    k_ell_run(const __grid_constant__ DevSys s, const __grid_constant__ EllSys e, long long n, int more) {
    extern __shared__ __align__(16) unsigned char sm[];
    __shared__ uint2 s_mod[16];
    __shared__ uint8_t s_pick[64];
    __shared__ int s_go;
    if (more && __ldcg(s.flags + kFlagHalted) != 0u) return;  // a further launch of a call that has halted
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    const int G = (int)gridDim.x, rank = (int)blockIdx.x;
    const int own = (s.nslices - rank + G - 1) / G;  // slices rank, rank + G, ...
    uint32_t* const bits = reinterpret_cast<uint32_t*>(sm);
    int32_t* const Csm = reinterpret_cast<int32_t*>(bits + e.bit_words);
    uint32_t* const Ssm = reinterpret_cast<uint32_t*>(Csm + e.own * kSlice);
    fill_mod_table(s_mod);
    fill_pick_table(s_pick);
    const unsigned long long base = s.step[kStepBase];
    const unsigned long long start = more ? s.step[kStepCallStart] : base;
    // the lane's emitting rule as a bit of its four, eight lanes a word
    auto put = [&](unsigned long long k, int32_t slice, uint32_t mask) {
        uint32_t w = mask << (4 * (lane & 7));
        w |= __shfl_xor_sync(0xffffffffu, w, 1);
        w |= __shfl_xor_sync(0xffffffffu, w, 2);
        w |= __shfl_xor_sync(0xffffffffu, w, 4);
        if ((lane & 7) == 0) SNP_PICK(e.bits, k)[slice * 4 + lane / 8] = w;
    };
    auto emitting = [](uint32_t st, const SelOut& o) {  // st: before the select
        if ((st >> kPendShift) != 0u) return (st & kDMask) == 0u ? 1u << ((st >> kPendShift) - 1u) : 0u;
        return o.s >= 0 && o.emit > 0 ? 1u << o.s : 0u;
    };
    bool act = false;
    for (int i = warp; i < own; i += nw) {
        const int32_t slice = rank + i * G, slot = slice * kSlice + lane;
        uint32_t mask = 0u, nst = 0u;
        int32_t c = 0;
        if (slot < s.q) {
            const uint32_t st = s.st[slot];
            const SelOut o = s.compact ? select_slot<true, SEL>(s, slot, s.C[slot], st, base)
                                       : select_slot<false, SEL>(s, slot, s.C[slot], st, base);
            mask = emitting(st, o);
            SNP_PICK(s.S, base)[slot] = o.s;
            c = o.c_after;
            nst = o.st;
            act |= o.active;
        }
        Csm[i * kSlice + lane] = c;
        Ssm[i * kSlice + lane] = nst;
        put(base, slice, mask);
    }
    uint32_t rk[20];
    {
        uint32_t k0 = (uint32_t)s.seed, k1 = (uint32_t)(s.seed >> 32);
#pragma unroll
        for (int r = 0; r < 10; ++r) {
            rk[2 * r] = k0;
            rk[2 * r + 1] = k1;
            k0 += 0x9E3779B9u;
            k1 += 0xBB67AE85u;
        }
    }
    const uint32_t b0 = cl_smem_u32(bits);
    uint32_t seen[2] = {0u, 0u};
    long long exec = 0;
    bool halted = false;
    for (long long t = 0; t < n; ++t) {
        const bool any = __syncthreads_or(act);
        if (threadIdx.x == 0) {
            const int go = grid_meet(e.ctr, t, any, seen);
            if (go < 0) atomicOr(s.flags + kFlagTimeout, 1u);
            s_go = go;
        }
        __syncthreads();
        if (s_go <= 0) {
            halted = s_go == 0;  // the same in every CTA
            break;
        }
        const unsigned long long ks = base + (unsigned long long)t + 1ull;
        copy_from_l2(reinterpret_cast<uint4*>(bits), reinterpret_cast<const uint4*>(SNP_PICK(e.bits, ks + 1ull)),
                     e.bit_words / 4);
        __syncthreads();
        const bool do_sel = t + 1 < n;
        PhiloxHead ph{};
        if (SEL == SNP_SELECT_PHILOX) ph = philox_head(ks, rk);
        act = false;
        for (int i = warp; i < own; i += nw) {
            const int32_t slice = rank + i * G, slot = slice * kSlice + lane;
            const bool valid = slot < s.q;
            const int32_t a = __ldg(e.bit_ptr + slice), b = __ldg(e.bit_ptr + slice + 1);
            uint4 rec = make_uint4(0u, 0u, 0u, 0u);
            uint32_t nid = 0u;
            if (valid && do_sel) {
                if (e.rec) rec = __ldg(reinterpret_cast<const uint4*>(e.rec) + slot);
                nid = neuron_id(s, slot);
            }
            uint32_t in = 0u;  // one rule of a source emits: at most in-degree x p <= INT32_MAX
            auto pair = [&](uint32_t w) {
                const uint32_t word = sm_load_u32(b0 + (uint32_t)SNP_IDX(s.flags, 4, w >> 16, e.bit_words) * 4u);
                in += (word >> ((w >> 11) & 31u)) & 1u ? w & 2047u : 0u;
            };
            auto four = [&](const uint4& x) {
                pair(x.x);
                pair(x.y);
                pair(x.z);
                pair(x.w);
            };
            const uint4* __restrict__ p = e.bit_ent + (size_t)a * kSlice + lane;
            int32_t u = a;
            for (; u + 4 <= b; u += 4, p += 4 * kSlice) {
                const uint4 x0 = __ldg(p), x1 = __ldg(p + kSlice), x2 = __ldg(p + 2 * kSlice), x3 = __ldg(p + 3 * kSlice);
                four(x0);
                four(x1);
                four(x2);
                four(x3);
            }
            for (; u < b; ++u, p += kSlice) four(__ldg(p));
            int32_t c = Csm[i * kSlice + lane];
            const uint32_t st = Ssm[i * kSlice + lane];
            if ((st >> kPendShift) == 0u) {
                const uint32_t nc = (uint32_t)c + in;
                if (nc > 2147483647u) atomicOr(s.flags + kFlagOverflow, 1u);
                c = (int32_t)min(nc, 2147483647u);
            }
            if (do_sel) {
                SelOut o;
                o.c_after = c;
                o.st = 0u;
                o.emit = 0;
                o.s = -1;
                o.active = false;
                if (e.rec)  // a zero record past the system's end: nothing applies
                    o = select_rec_flat<SEL>(rec, c, st, nid, ph, rk, s_mod, s_pick);
                else if (valid && s.compact)
                    o = select_neuron<true, SEL>(s.rules, rule_lo(s, slot), rule_hi(s, slot), c, st, ks, nid, s.seed);
                else if (valid)
                    o = select_neuron<false, SEL>(s.rules, rule_lo(s, slot), rule_hi(s, slot), c, st, ks, nid, s.seed);
                put(ks, slice, emitting(st, o));
                c = o.c_after;
                act |= o.active;
                if (valid) SNP_PICK(s.S, ks)[slot] = o.s;
                Ssm[i * kSlice + lane] = o.st;
            }
            Csm[i * kSlice + lane] = c;
        }
        ++exec;
    }
    for (int i = warp; i < own; i += nw) {
        const int32_t slot = (rank + i * G) * kSlice + lane;
        if (slot < s.q) {
            s.C[slot] = Csm[i * kSlice + lane];
            s.st[slot] = Ssm[i * kSlice + lane];
        }
    }
    // every CTA has read the step words and the halt flag: it was at a barrier since
    if (rank == 0 && threadIdx.x == 0) {
        s.step[kStepCallStart] = start;
        s.step[kStepBase] = base + (unsigned long long)exec;
        s.step[kStepExec] = base + (unsigned long long)exec - start;
        s.step[kStepHalt] = halted ? base + (unsigned long long)exec : 0ull;
        s.flags[kFlagHalted] = halted ? 1u : 0u;
    }
}

cudaError_t launch_ell_run(const DevSys& s, const EllSys& e, long long n, bool more, int sel, cudaStream_t st) {
    auto fn = sel == SNP_SELECT_FIRST ? k_ell_run<SNP_SELECT_FIRST> : k_ell_run<SNP_SELECT_PHILOX>;
    const size_t smem = ell_run_smem(e);
    // the same bound for every launch: threads may launch different sizes at once
    cudaError_t err = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, resident_max_smem() - 1024);
    if (err == cudaSuccess) err = cudaMemsetAsync(e.ctr, 0, 2 * sizeof(unsigned long long), st);
    if (err != cudaSuccess) return err;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)e.G);
    cfg.blockDim = dim3((unsigned)kEllThreads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeCooperative;
    at[0].val.cooperative = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, fn, s, e, n, more ? 1 : 0);
}

// Select launch of step ks = base + t for the push and dense variants.  With
// INFLOW it first finishes step ks - 1 by adding the in-flow accumulated by
// the dense launch (to open neurons) and clears it; with !SELECT it only
// finishes.
template <bool INFLOW, bool SELECT, bool COMPACT, int SEL>
__global__ void __launch_bounds__(256) k_ell_select(DevSys s, EllSys e, int32_t t) {
    uint32_t* fl = s.flags;
    const unsigned long long ks = s.step[kStepBase] + (unsigned long long)t;
    if (call_halted(fl)) return;
    const int32_t slot = (int32_t)(blockIdx.x * blockDim.x + threadIdx.x);
    bool active = false;
    if (slot < s.q) {
        int32_t c = s.C[slot];
        if (INFLOW) {
            const int32_t in = e.inflow[slot];
            e.inflow[slot] = 0;
            if ((s.st[slot] >> kPendShift) == 0u) {
                long long nc = (long long)c + in;
                if (nc > 2147483647ll) {
                    atomicOr(fl + kFlagOverflow, 1u);
                    nc = 2147483647ll;
                }
                c = (int32_t)nc;
            }
        }
        if (SELECT) active = ell_select_slot<COMPACT, SEL>(s, e, slot, c, ks);
        s.C[slot] = c;
    }
    if (SELECT) raise_step_activity(fl, ks, active);
}

// ELL push of step kg = base + t: per-rule columns of (target, p) pairs in
// slices of 32 consecutive rules; each warp takes an equal run of their
// columns (push_balanced.cuh).
struct PushEllSrc {
    using Ent = int2;
    const uint8_t* Em;
    int64_t m;
    __device__ __forceinline__ Ent pad() const { return make_int2(-1, 0); }
    __device__ __forceinline__ int32_t value(int32_t slice, int lane) const {
        const int64_t r = (int64_t)slice * kSlice + lane;
        return r < m && Em[r] ? 1 : 0;
    }
    __device__ __forceinline__ int32_t target(Ent e) const { return e.x; }
    __device__ __forceinline__ int32_t amount(Ent e, int32_t) const { return e.y; }
};

constexpr int kEllPushBlocksPerSm = 6;

template <bool INFLOW>
__global__ void __launch_bounds__(256, kEllPushBlocksPerSm) k_ell_push(DevSys s, EllSys e, int32_t t) {
    uint32_t* fl = s.flags;
    const unsigned long long kg = s.step[kStepBase] + (unsigned long long)t;
    if (step_blocked(fl, s.step, kg)) return;
    if (blockIdx.x == 0 && threadIdx.x == 0) fl[kFlagAct0 + (int)((kg + 1ull) % 3ull)] = 0u;
    PushEllSrc src;
    src.Em = SNP_PICK(e.Em, kg);
    src.m = e.m;
    const int32_t nrs = (int32_t)((e.m + kSlice - 1) / kSlice);
    push_scatter_balanced<8, INFLOW>(src, e.out_ptr, nrs, e.out_ent, INFLOW ? e.inflow : s.C, s.st, fl, s.q,
                                     s.hubs != 0);
}

// Dense accumulation of step kg = base + t: CTA (bx, by) covers neurons
// [bx*256, bx*256+256) and rules [by*rows, (by+1)*rows); every rule row of
// M_Pi is read whether or not the rule emits, as Alg. 3 walks all m rules.
__global__ void __launch_bounds__(256) k_dense_accum(DevSys s, EllSys e, int32_t t, int32_t rows) {
    uint32_t* fl = s.flags;
    const unsigned long long kg = s.step[kStepBase] + (unsigned long long)t;
    if (step_blocked(fl, s.step, kg)) return;
    if (blockIdx.x == 0 && blockIdx.y == 0 && threadIdx.x == 0) fl[kFlagAct0 + (int)((kg + 2ull) % 3ull)] = 0u;
    const int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int64_t r0 = (int64_t)blockIdx.y * rows;
    const int64_t r1 = r0 + rows < e.m ? r0 + rows : e.m;
    const uint8_t* __restrict__ Em = SNP_PICK(e.Em, kg);
    if (j >= s.q) return;
    long long sum = 0;
    const int32_t* __restrict__ col = e.dense + j;
    for (int64_t r = r0; r < r1; ++r) sum += (long long)Em[r] * __ldg(col + r * (int64_t)s.q);
    if (sum) {
        const int old = atomicAdd(e.inflow + j, (int)sum);
        if ((long long)old + sum > 2147483647ll) atomicOr(fl + kFlagOverflow, 1u);
    }
}

// ---- launchers ----------------------------------------------------------

template <bool G, bool S>
static cudaError_t ell_pull_t(const DevSys& s, const EllSys& e, int32_t t, cudaStream_t st, bool compact, int sel) {
    const dim3 grid((unsigned)((s.nslices + 7) / 8));
    if (compact) {
        if (sel == SNP_SELECT_FIRST) k_ell_pull<G, S, true, SNP_SELECT_FIRST><<<grid, 256, 0, st>>>(s, e, t);
        else k_ell_pull<G, S, true, SNP_SELECT_PHILOX><<<grid, 256, 0, st>>>(s, e, t);
    } else {
        if (sel == SNP_SELECT_FIRST) k_ell_pull<G, S, false, SNP_SELECT_FIRST><<<grid, 256, 0, st>>>(s, e, t);
        else k_ell_pull<G, S, false, SNP_SELECT_PHILOX><<<grid, 256, 0, st>>>(s, e, t);
    }
    return cudaGetLastError();
}

cudaError_t launch_ell_pull(const DevSys& s, const EllSys& e, int kind, int32_t t, cudaStream_t st, bool compact,
                            int sel) {
    switch (kind) {
        case kPullSelectOnly: return ell_pull_t<false, true>(s, e, t, st, compact, sel);
        case kPullFused: return ell_pull_t<true, true>(s, e, t, st, compact, sel);
        case kPullGatherOnly: return ell_pull_t<true, false>(s, e, t, st, compact, sel);
        default: return cudaErrorInvalidValue;
    }
}

template <bool IN, bool S>
static cudaError_t ell_select_t(const DevSys& s, const EllSys& e, int32_t t, cudaStream_t st, bool compact, int sel) {
    const dim3 grid((unsigned)((s.q + 255) / 256));
    if (compact) {
        if (sel == SNP_SELECT_FIRST) k_ell_select<IN, S, true, SNP_SELECT_FIRST><<<grid, 256, 0, st>>>(s, e, t);
        else k_ell_select<IN, S, true, SNP_SELECT_PHILOX><<<grid, 256, 0, st>>>(s, e, t);
    } else {
        if (sel == SNP_SELECT_FIRST) k_ell_select<IN, S, false, SNP_SELECT_FIRST><<<grid, 256, 0, st>>>(s, e, t);
        else k_ell_select<IN, S, false, SNP_SELECT_PHILOX><<<grid, 256, 0, st>>>(s, e, t);
    }
    return cudaGetLastError();
}

cudaError_t launch_ell_select(const DevSys& s, const EllSys& e, bool inflow, bool select, int32_t t, cudaStream_t st,
                              bool compact, int sel) {
    if (inflow) return select ? ell_select_t<true, true>(s, e, t, st, compact, sel)
                              : ell_select_t<true, false>(s, e, t, st, compact, sel);
    return ell_select_t<false, true>(s, e, t, st, compact, sel);
}

cudaError_t launch_ell_push(const DevSys& s, const EllSys& e, int32_t t, cudaStream_t st) {
    const int64_t nrs = (e.m + kSlice - 1) / kSlice;
    if (nrs == 0) {
        k_ell_push<false><<<1, 32, 0, st>>>(s, e, t);  // still settles the halt test
        return cudaGetLastError();
    }
    if (e.inflow)
        k_ell_push<true><<<push_blocks(kEllPushBlocksPerSm, nrs), 256, 0, st>>>(s, e, t);
    else
        k_ell_push<false><<<push_blocks(kEllPushBlocksPerSm, nrs), 256, 0, st>>>(s, e, t);
    return cudaGetLastError();
}

cudaError_t launch_dense_accum(const DevSys& s, const EllSys& e, int32_t t, cudaStream_t st) {
    const int32_t rows = 512;
    const unsigned gy = (unsigned)((e.m + rows - 1) / rows);
    const dim3 grid((unsigned)((s.q + 255) / 256), gy > 0 ? gy : 1u);
    k_dense_accum<<<grid, 256, 0, st>>>(s, e, t, rows);
    return cudaGetLastError();
}

}  // namespace snp
