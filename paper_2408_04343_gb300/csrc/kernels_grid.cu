// Grid-resident engine: one cooperative launch runs all steps of one system,
// every SM holding a part of it.
//
// The tiled engine's launch per step costs a middle-sized system (8,193 to
// some 690,000 neurons) more than its work: the launch, the fixed-point flag,
// the state read and written, entries padded to 1,024 runs.  Here group i of
// 128 slots in quad order (see pack_system) belongs to CTA i mod G for the
// whole call; its spikes, status words and, where they fit (LSM), in-lists and
// records stay in shared memory.  Per step a CTA
//   * copies the packed emission vector E_k (2 to 16 bits per neuron) from L2
//     into shared memory;
//   * gathers and selects its groups, one lane per quad (quad.cuh), and writes
//     its quads' packed E_{k+1} to global memory;
//   * meets the other CTAs at a counter in L2.  The counter's upper half counts
//     the CTAs that saw a pending or selecting neuron, so the barrier carries
//     the fixed-point test.  Two counters alternate: a CTA can run ahead into
//     the next step's, never into the one a slower CTA still reads.
// The launch is cooperative, so all CTAs are resident; the wait is bounded all
// the same.  us per step, a launch per step / so: 9,000 neurons 8.1 / 3.0,
// 32,768 8.2 / 3.3, 100,003 9.1 / 4.0, 200,003 9.9 / 5.7, 450,000 12.8 / 9.4;
// 100,003 neurons of wide rules 17.6 / 6.0.  Systems with long in-lists are left
// to the tiled engine (grid_plan in api.cu says where the line lies).
#include <cuda_runtime.h>

#include <algorithm>

#include "device_common.cuh"
#include "kernels.h"
#include "quad.cuh"

namespace snp {

namespace {

// A quad's emissions, EB bits each, packed in w.
__device__ __forceinline__ void put_emissions(uint8_t* E, int32_t quad, unsigned long long w, int eb) {
    if (eb == 2)
        E[quad] = (uint8_t)w;
    else if (eb == 4)
        reinterpret_cast<uint16_t*>(E)[quad] = (uint16_t)w;
    else if (eb == 8)
        reinterpret_cast<uint32_t*>(E)[quad] = (uint32_t)w;
    else
        reinterpret_cast<unsigned long long*>(E)[quad] = w;
}

__host__ __device__ constexpr bool grid_byte_rules(int mode) { return mode == kClusterRec || mode == kClusterTest8; }

}  // namespace

// Shared memory of one CTA: the packed emissions; for `own` groups spikes,
// status words, (up to 32 rules) the chosen rules of two steps, list pointers
// and quad ids; several warps per group: their partial in-flows; LSM: records
// and in-lists; test records as in cluster_smem_bytes.
size_t grid_smem_bytes(int mode, const GridSys& gs, bool lsm, int lsm_cols, int rules) {
    const size_t own = (size_t)gs.own;
    size_t b = (size_t)gs.e_bytes + own * (1024 + (grid_byte_rules(mode) ? 256 : 0) + 8 + 128);
    b = (b + 15) & ~(size_t)15;
    if (gs.warps_per_group > 1) b += kClusterThreads / 32 * 512;
    if (lsm) b += (mode == kClusterRec ? own * 2048 : 0) + (size_t)lsm_cols * 512;
    if (mode == kClusterTest8) b += own * 516 + 16 + (size_t)rules * 16;
    return b;
}

template <int MODE, int SEL, bool LSM>
__global__ void __launch_bounds__(kClusterThreads, 1)
    k_grid_run(const __grid_constant__ DevSys s, const __grid_constant__ GridSys gs, long long n, int more) {
    constexpr bool REC = MODE == kClusterRec, BYTE = grid_byte_rules(MODE);
    constexpr bool WORDS = SEL == SNP_SELECT_PHILOX && MODE != kClusterGeneral;  // Philox words by quad
    extern __shared__ __align__(16) unsigned char sm[];
    __shared__ uint2 s_mod[16];
    __shared__ uint8_t s_pick[64];
    __shared__ int s_go;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    const int G = (int)gridDim.x, rank = (int)blockIdx.x;
    const int ng = (s.q + kGroup - 1) / kGroup;
    const int own = (ng - rank + G - 1) / G;  // groups rank, rank + G, ...
    const int S = gs.warps_per_group;
    const int eb = gs.e_bits;
    const uint32_t emask = (1u << eb) - 1u;
    if (more && __ldcg(s.flags + kFlagHalted) != 0u) return;  // a further launch of a call that has halted
    int4* Csm = reinterpret_cast<int4*>(sm + gs.e_bytes);
    uint4* Ssm = reinterpret_cast<uint4*>(Csm + gs.own * 32);
    uint32_t* Rsm = reinterpret_cast<uint32_t*>(Ssm + gs.own * 32);
    int2* gptr = reinterpret_cast<int2*>(Rsm + (BYTE ? gs.own * 64 : 0));
    uint32_t* qsm = reinterpret_cast<uint32_t*>(gptr + gs.own);
    uint4* part0 =
        reinterpret_cast<uint4*>(sm + ((gs.e_bytes + gs.own * (1024 + (BYTE ? 256 : 0) + 136) + 15) & ~15));
    uint4* rsm = part0 + (S > 1 ? kClusterThreads : 0);
    uint4* lsm = rsm + (REC ? gs.own * 128 : 0);
    uint4* const part = part0 + threadIdx.x;
    fill_mod_table(s_mod);
    fill_pick_table(s_pick);
    for (int i = warp; i < own; i += nw) {
        const int g = rank + i * G;
        int32_t c[4] = {0, 0, 0, 0};
        uint32_t st[4] = {0u, 0u, 0u, 0u};
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int32_t slot = quad_slot(g, lane, j, s.q);
            uint4 rec = make_uint4(0u, 0u, 0u, 0u);
            if (slot >= 0) {
                c[j] = s.C[slot];
                st[j] = s.st[slot];
                if (REC && LSM) rec = __ldg(reinterpret_cast<const uint4*>(s.rec) + slot);
                if (j == 0) qsm[i * 32 + lane] = neuron_id(s, slot) >> 2;
            } else if (j == 0) {
                qsm[i * 32 + lane] = 0u;
            }
            if (REC && LSM) rsm[(i * 4 + j) * 32 + lane] = rec;
        }
        Csm[i * 32 + lane] = make_int4(c[0], c[1], c[2], c[3]);
        Ssm[i * 32 + lane] = make_uint4(st[0], st[1], st[2], st[3]);
    }
    if (warp == 0)
        warp_group_starts(
            own, lane, [&](int i) { return __ldg(gs.ptr + rank + i * G + 1) - __ldg(gs.ptr + rank + i * G); },
            [&](int i, int32_t at, int32_t w) { gptr[i] = make_int2(LSM ? at : __ldg(gs.ptr + rank + i * G), w); });
    __syncthreads();
    const uint4* __restrict__ listg = gs.lists + lane;
    if (LSM) {
        for (int i = warp; i < own; i += nw) {
            const int2 pw = gptr[i];
            const uint4* __restrict__ p = listg + (size_t)__ldg(gs.ptr + rank + i * G) * 32;
            for (int c = 0; c < pw.y; ++c) lsm[(pw.x + c) * 32 + lane] = __ldg(p + c * 32);
        }
    }
    const int lcols = LSM ? gptr[own - 1].x + gptr[own - 1].y : 0;
    uint4* const tsm = lsm + (size_t)lcols * 32;  // test records
    int32_t* const rstart = reinterpret_cast<int32_t*>(tsm + gs.own * 32);
    uint4* const rrec = tsm + gs.own * 32 + (gs.own + 3) / 4;
    const uint4* const recs = gs.rules > 0 ? rrec : reinterpret_cast<const uint4*>(s.trec);
    if (MODE == kClusterTest8) {
        if (warp == 0)
            warp_group_starts(
                own, lane,
                [&](int i) {
                    const int32_t a = (rank + i * G) * kGroup;
                    return __ldg(s.rule_off + min(s.q, a + kGroup)) - __ldg(s.rule_off + a);
                },
                [&](int i, int32_t at, int32_t) { rstart[i] = at; });
        __syncthreads();
        for (int i = warp; i < own; i += nw)
            stage_tests(s, rank + i * G, lane, tsm + i * 32, rrec, gs.rules > 0, rstart[i]);
    }
    const unsigned long long base = s.step[kStepBase];
    const unsigned long long start = more ? s.step[kStepCallStart] : base;

    // select of step `base`
    bool act = false;
    for (int i = warp; i < own; i += nw) {
        const int g = rank + i * G;
        unsigned long long w = 0ull;
        uint32_t chosen = 0u;
#pragma unroll 1
        for (int j = 0; j < 4; ++j) {
            const int32_t slot = quad_slot(g, lane, j, s.q);
            if (slot < 0) continue;
            int32_t* c = reinterpret_cast<int32_t*>(Csm + i * 32 + lane) + j;
            uint32_t* st = reinterpret_cast<uint32_t*>(Ssm + i * 32 + lane) + j;
            const SelOut o = s.compact ? select_slot<true, SEL>(s, slot, *c, *st, base)
                                       : select_slot<false, SEL>(s, slot, *c, *st, base);
            *c = o.c_after;
            *st = o.st;
            if (BYTE)
                chosen |= (uint32_t)(uint8_t)o.s << (8 * j);
            else
                SNP_PICK(s.S, base)[slot] = o.s;
            w |= (unsigned long long)(uint32_t)o.emit << (eb * j);
            act |= o.active;
        }
        if (BYTE) Rsm[((int)(base & 1ull) * gs.own + i) * 32 + lane] = chosen;
        put_emissions(SNP_PICK(gs.E, base), g * 32 + lane, w, eb);
    }

    const uint32_t e0 = cl_smem_u32(sm);
    const uint32_t mod0 = cl_smem_u32(s_mod), pick0 = cl_smem_u32(s_pick);
    const uint32_t list0 = cl_smem_u32(lsm) + (uint32_t)lane * 16u;
    const int first = S > 1 ? warp / S : warp, helper = S > 1 ? warp % S : 0;
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
    uint32_t seen[2] = {0u, 0u};  // thread 0: active arrivals so far, by counter
    long long exec = 0;
    bool halted = false;
    for (long long t = 0; t < n; ++t) {
        // every CTA's E_{base + t} is written: arrive, wait, learn whether any
        // neuron was active
        const bool any = __syncthreads_or(act);
        if (threadIdx.x == 0) {
            const int go = grid_meet(gs.ctr, t, any, seen);
            if (go < 0) atomicOr(s.flags + kFlagTimeout, 1u);
            s_go = go;
        }
        __syncthreads();
        if (s_go <= 0) {
            halted = s_go == 0;  // the same in every CTA
            break;
        }
        const unsigned long long ks = base + (unsigned long long)t + 1ull;
        copy_from_l2(reinterpret_cast<uint4*>(sm), reinterpret_cast<const uint4*>(SNP_PICK(gs.E, ks + 1ull)), gs.e_bytes / 16);
        __syncthreads();
        const bool do_sel = t + 1 < n;
        uint8_t* const En = SNP_PICK(gs.E, ks);
        PhiloxHead ph{};
        if (WORDS) ph = philox_head(ks, rk);
        act = false;
        for (int i = first; i < own; i += nw) {
            const int g = rank + i * G;
            int2 pw = gptr[i];
            if (S > 1) {
                const int c0 = pw.y * helper / S;
                pw = make_int2(pw.x + c0, pw.y * (helper + 1) / S - c0);
            }
            uint4 rec[4];
            if (REC && helper == 0) {
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    if (LSM) {
                        rec[j] = rsm[(i * 4 + j) * 32 + lane];
                    } else {
                        const int32_t slot = quad_slot(g, lane, j, s.q);
                        rec[j] = slot >= 0 ? __ldg(reinterpret_cast<const uint4*>(s.rec) + slot) : make_uint4(0u, 0u, 0u, 0u);
                    }
                }
            }
            Philox4 px{};
            if (WORDS && helper == 0) px = quad_philox(ph, qsm[i * 32 + lane], s.seed);
            uint32_t in[4] = {0u, 0u, 0u, 0u};  // at most INT32_MAX each (checked when the system is made)
            auto column = [&](const uint4& x) {
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    // byte address of the source's word << 8 | its bit in the word
                    const uint32_t e = (&x.x)[j];
                    const uint32_t w = sm_load_u32(e0 + (uint32_t)SNP_IDX(s.flags, 1, e >> 8, gs.e_bytes - 3));
                    in[j] += __funnelshift_r(w, w, e) & emask;
                }
            };
            if (LSM) {
                uint32_t a = list0 + (uint32_t)pw.x * 512u;
                int c = 0;
                for (; c + 4 <= pw.y; c += 4, a += 2048u) {
                    const uint4 x0 = sm_load_v4(a), x1 = sm_load_v4(a + 512u);
                    const uint4 x2 = sm_load_v4(a + 1024u), x3 = sm_load_v4(a + 1536u);
                    column(x0);
                    column(x1);
                    column(x2);
                    column(x3);
                }
                for (; c < pw.y; ++c, a += 512u) column(sm_load_v4(a));
            } else {
                // four columns in flight while four are added (the loads past
                // the last column read the slack after the lists)
                const uint4* __restrict__ p = listg + (size_t)pw.x * 32;
                uint4 x0 = __ldg(p), x1 = __ldg(p + 32), x2 = __ldg(p + 64), x3 = __ldg(p + 96);
                int c = 0;
                for (; c + 4 <= pw.y; c += 4) {
                    p += 128;
                    const uint4 y0 = __ldg(p), y1 = __ldg(p + 32), y2 = __ldg(p + 64), y3 = __ldg(p + 96);
                    column(x0);
                    column(x1);
                    column(x2);
                    column(x3);
                    x0 = y0;
                    x1 = y1;
                    x2 = y2;
                    x3 = y3;
                }
                if (c < pw.y) column(x0);
                if (c + 1 < pw.y) column(x1);
                if (c + 2 < pw.y) column(x2);
            }
            if (S > 1) {  // the group's warps meet: named barrier i + 1
                if (helper > 0) *part = make_uint4(in[0], in[1], in[2], in[3]);
                asm volatile("bar.sync %0, %1;" ::"r"(i + 1), "r"(S * 32) : "memory");
                if (helper > 0) continue;
                for (int h = 1; h < S; ++h) {
                    const uint4 x = part[h * 32];
                    in[0] += x.x;
                    in[1] += x.y;
                    in[2] += x.z;
                    in[3] += x.w;
                }
            }
            int4 c4 = Csm[i * 32 + lane];
            uint4 st4 = Ssm[i * 32 + lane];
            if (quad_receive<uint32_t>(c4, st4, in)) atomicOr(s.flags + kFlagOverflow, 1u);
            if (do_sel) {
                int32_t slot[4];
                uint32_t emit[4];
#pragma unroll
                for (int j = 0; j < 4; ++j) slot[j] = BYTE ? 0 : quad_slot(g, lane, j, s.q);
                if (BYTE) {
                    uint32_t chosen;
                    if (REC)
                        quad_select_rec<SEL>(rec, c4, st4, px, mod0, pick0, emit, chosen, act);
                    else
                        quad_select_test<SEL>(recs, tsm[i * 32 + lane], c4, st4, px, emit, chosen, act);
                    Rsm[((int)(ks & 1ull) * gs.own + i) * 32 + lane] = chosen;
                } else if (MODE == kClusterTable) {
                    int32_t chosen[4];
                    quad_select_table<SEL>(s, slot, c4, st4, px.v, emit, chosen, act);
#pragma unroll
                    for (int j = 0; j < 4; ++j)
                        if (slot[j] >= 0) SNP_PICK(s.S, ks)[slot[j]] = chosen[j];
                } else {
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        emit[j] = 0u;
                        if (slot[j] < 0) continue;
                        const uint32_t nid = qsm[i * 32 + lane] * 4u + (uint32_t)j;
                        const int32_t r0 = rule_lo(s, slot[j]), r1 = rule_hi(s, slot[j]);
                        const SelOut o =
                            s.compact
                                ? select_neuron<true, SEL>(s.rules, r0, r1, (&c4.x)[j], (&st4.x)[j], ks, nid, s.seed)
                                : select_neuron<false, SEL>(s.rules, r0, r1, (&c4.x)[j], (&st4.x)[j], ks, nid, s.seed);
                        (&c4.x)[j] = o.c_after;
                        (&st4.x)[j] = o.st;
                        act |= o.active;
                        emit[j] = (uint32_t)o.emit;
                        SNP_PICK(s.S, ks)[slot[j]] = o.s;
                    }
                }
                unsigned long long w = emit[0];
#pragma unroll
                for (int j = 1; j < 4; ++j) w |= (unsigned long long)emit[j] << (eb * j);
                put_emissions(En, g * 32 + lane, w, eb);
                Ssm[i * 32 + lane] = st4;
            }
            Csm[i * 32 + lane] = c4;
        }
        ++exec;
    }
    if (S > 1) __syncthreads();  // with one warp per group a lane wrote its own quads only
    int32_t* const Sl = SNP_PICK(s.S, base + (unsigned long long)exec + 1ull);  // of the last executed step
    const int rl = (int)((base + (unsigned long long)exec + 1ull) & 1ull) * gs.own * 32;
    for (int i = warp; i < own; i += nw) {
        const int4 c4 = Csm[i * 32 + lane];
        const uint4 st4 = Ssm[i * 32 + lane];
        const uint32_t chosen = BYTE ? Rsm[rl + i * 32 + lane] : 0u;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int32_t slot = quad_slot(rank + i * G, lane, j, s.q);
            if (slot < 0) continue;
            s.C[slot] = (&c4.x)[j];
            s.st[slot] = (&st4.x)[j];
            if (BYTE && exec > 0) Sl[slot] = (int32_t)(int8_t)(chosen >> (8 * j));
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

template <int MODE, int SEL, bool LSM>
static cudaError_t launch_grid_t(const DevSys& s, const GridSys& gs, long long n, bool more, cudaStream_t st) {
    auto fn = k_grid_run<MODE, SEL, LSM>;
    // the same bound for every launch: threads may launch different sizes at once
    cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, resident_max_smem() - 1024);
    if (e == cudaSuccess) e = cudaMemsetAsync(gs.ctr, 0, 2 * sizeof(unsigned long long), st);
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)gs.G);
    cfg.blockDim = dim3((unsigned)gs.threads);
    cfg.dynamicSmemBytes = (size_t)gs.smem;
    cfg.stream = st;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeCooperative;
    at[0].val.cooperative = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, fn, s, gs, n, more ? 1 : 0);
}

template <int MODE, int SEL>
static cudaError_t launch_grid_l(const DevSys& s, const GridSys& gs, long long n, bool more, cudaStream_t st) {
    return gs.lsm ? launch_grid_t<MODE, SEL, true>(s, gs, n, more, st)
                  : launch_grid_t<MODE, SEL, false>(s, gs, n, more, st);
}

cudaError_t launch_grid(const DevSys& s, const GridSys& gs, long long n, bool more, int sel, cudaStream_t st) {
    const bool first = sel == SNP_SELECT_FIRST;
    switch (gs.mode) {
        case kClusterRec:
            return first ? launch_grid_l<kClusterRec, SNP_SELECT_FIRST>(s, gs, n, more, st)
                         : launch_grid_l<kClusterRec, SNP_SELECT_PHILOX>(s, gs, n, more, st);
        case kClusterTest8:
            return first ? launch_grid_l<kClusterTest8, SNP_SELECT_FIRST>(s, gs, n, more, st)
                         : launch_grid_l<kClusterTest8, SNP_SELECT_PHILOX>(s, gs, n, more, st);
        case kClusterTable:
            return first ? launch_grid_l<kClusterTable, SNP_SELECT_FIRST>(s, gs, n, more, st)
                         : launch_grid_l<kClusterTable, SNP_SELECT_PHILOX>(s, gs, n, more, st);
        case kClusterGeneral:
            return first ? launch_grid_l<kClusterGeneral, SNP_SELECT_FIRST>(s, gs, n, more, st)
                         : launch_grid_l<kClusterGeneral, SNP_SELECT_PHILOX>(s, gs, n, more, st);
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace snp
