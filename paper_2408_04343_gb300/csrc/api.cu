// C-ABI of libsnp: system life cycle, stepping, state access.
#include <cuda.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdio>
#include <atomic>
#include <cstring>
#include <mutex>
#include <new>
#include <string>
#include <vector>

#include "kernels.h"
#include "snp_internal.h"
#include "pointer_kind.h"
#include "system.h"

namespace snp {

const char* last_error();

// ---- device memory -----------------------------------------------------

void* sys_alloc(snp_system* s, size_t bytes) {
    if (bytes == 0) bytes = 16;
    bytes = (bytes + 255) & ~(size_t)255;
    void* p = nullptr;
    if (s->alloc.alloc) {
        p = s->alloc.alloc(s->alloc.ctx, bytes, (void*)s->stream);
    } else if (cudaMalloc(&p, bytes) != cudaSuccess) {
        cudaGetLastError();
        p = nullptr;
    }
    if (p) {
        s->allocs.push_back({p, bytes});
        s->device_bytes += bytes;
    }
    return p;
}

static void sys_free_all(snp_system* s) {
    for (auto& a : s->allocs) {
        if (s->alloc.release)
            s->alloc.release(s->alloc.ctx, a.first, a.second, (void*)s->stream);
        else
            cudaFree(a.first);
    }
    s->allocs.clear();
    s->device_bytes = 0;
}

// Short-lived device buffers of one call (staging of host arrays): from the
// caller's allocator when the system has one, else stream-ordered cudaMalloc.
static void* stage_alloc(snp_system* s, size_t bytes) {
    bytes = (bytes + 255) & ~(size_t)255;
    if (s->alloc.alloc) return s->alloc.alloc(s->alloc.ctx, bytes, (void*)s->stream);
    void* p = nullptr;
    if (cudaMallocAsync(&p, bytes, s->stream) != cudaSuccess) {
        cudaGetLastError();
        return nullptr;
    }
    return p;
}

static void stage_free(snp_system* s, void* p, size_t bytes) {
    if (!p) return;
    bytes = (bytes + 255) & ~(size_t)255;
    if (s->alloc.release)
        s->alloc.release(s->alloc.ctx, p, bytes, (void*)s->stream);
    else
        cudaFreeAsync(p, s->stream);
}

static int cuda_fail(const char* what) {
    cudaError_t e = cudaGetLastError();
    return fail(SNP_ERR_CUDA, std::string(what) + ": " + cudaGetErrorString(e));
}

// ---- one allocation per system ---------------------------------------------
// Every device buffer of a system is carved from one allocation: the host
// image is turned into a list of pieces (destination pointer field, source or
// fill byte, size), the sizes are summed at 256-byte alignment, one block is
// allocated, and each piece is copied or filled into its place.

size_t plan_bytes(const std::vector<Piece>& plan) {
    size_t t = 0;
    for (const Piece& p : plan) t += (p.bytes + 255) & ~(size_t)255;
    return t;
}

void build_plan(snp_system* s, std::vector<Piece>& plan) {
    HostImage& im = *s->img;
    HostPack& hp = im.hp;
    DevSys& d = s->dev;
    const size_t q = (size_t)hp.q;
    const int32_t nslices = (hp.q + kSlice - 1) / kSlice;
    auto vec = [&](void* field, const auto& v) {
        plan.push_back({reinterpret_cast<void**>(field), v.data(), v.size() * sizeof(v[0]), -1});
    };
    auto fill = [&](void* field, size_t bytes, int byte) {
        plan.push_back({reinterpret_cast<void**>(field), nullptr, bytes, byte});
    };
    d.q = hp.q;
    d.nslices = nslices;
    vec(&d.slice_ptr, hp.slice_ptr);
    if (s->has_in_lists) vec(&d.in_idx, hp.in_idx);
    d.in_quads = nullptr;
    if (s->quad_lists) {
        vec(&d.quad_ptr, hp.quad_ptr);
        vec(&d.in_quads, hp.in_quads);
    }
    if (s->has_grid) {
        vec(&s->grid.ptr, hp.quad_ptr32);
        vec(&s->grid.lists, hp.in_quads32);
        for (int b = 0; b < 2; ++b) fill(&s->grid.E[b], (size_t)s->grid.e_bytes, 0);
        fill(&s->grid.ctr, 2 * sizeof(unsigned long long), 0);
    }
    d.tab_off = nullptr;
    if (s->tables) {
        vec(&d.tab_off, hp.tab_off);
        vec(&d.tab, hp.tab);
        vec(&d.tab_app, hp.tab_app);
        vec(&d.tab_p, hp.tab_p);
    }
    d.trec = nullptr;
    if (s->test_recs) vec(&d.trec, hp.trec);
    // a push's in-flow fits 32 bits (else the targets' counts are added to directly)
    const bool inflow = s->opt.prop == SNP_PROP_PUSH && (int64_t)hp.max_in * (int64_t)hp.max_p <= (int64_t)INT32_MAX;
    d.inflow = nullptr;
    if (s->opt.form == SNP_FORM_OPT && s->opt.prop == SNP_PROP_PUSH) {
        vec(&d.out_ptr, hp.out_ptr);
        vec(&d.out_idx, hp.out_idx);
        if (inflow) fill(&d.inflow, q * 4, 0);
    }
    vec(&d.rule_off, hp.rule_off);
    vec(&d.rules, hp.rules);
    d.rec = nullptr;
    if ((s->opt.form == SNP_FORM_OPT || s->unions) && !hp.rec.empty()) vec(&d.rec, hp.rec);
    vec(&d.orig, hp.perm);
    vec(&s->d_rule_base, hp.rule_base);
    vec(&d.C, hp.C0);
    fill(&d.st, q * 4, 0);
    for (int b = 0; b < 2; ++b) {
        if (s->opt.form == SNP_FORM_OPT) fill(&d.E[b], (q + 1) * 4, 0);
        fill(&d.S[b], q * 4, 0xff);  // -1: no rule selected yet
    }
    fill(&d.flags, kStatusBytes, 0);  // and the step counters
    fill(&s->scratch, q * 4, 0);
    fill(&s->d_nsteps, 8, 0);
    fill(&s->d_work, 4, 0);
    fill(&s->d_self, sizeof(DevSys), 0);
    if (s->opt.form != SNP_FORM_OPT) {
        EllSys& e = s->ell;
        e.m = hp.m;
        e.bit_ent = nullptr;
        e.rec = nullptr;
        if (!im.ep.bit_ent.empty()) {
            vec(&e.bit_ptr, im.ep.bit_ptr);
            vec(&e.bit_ent, im.ep.bit_ent);
            for (int b = 0; b < 2; ++b) fill(&e.bits[b], (size_t)e.bit_words * 4, 0);
            fill(&e.ctr, 2 * sizeof(unsigned long long), 0);
            if (!hp.rec.empty()) vec(&e.rec, hp.rec);
        } else if (!im.ep.in_ptr.empty()) {
            vec(&e.in_ptr, im.ep.in_ptr);
            vec(&e.in_ent, im.ep.in_ent);
        }
        if (!im.ep.out_ptr.empty()) {
            vec(&e.out_ptr, im.ep.out_ptr);
            vec(&e.out_ent, im.ep.out_ent);
        }
        if (s->opt.form == SNP_FORM_DENSE) {
            vec(&e.dense, im.dense);
        }
        e.inflow = nullptr;
        if (s->opt.form == SNP_FORM_DENSE || inflow) fill(&e.inflow, q * 4, 0);
        e.Em[0] = e.Em[1] = nullptr;  // one-word pairs step on bits instead
        for (int b = 0; b < 2 && im.ep.bit_ent.empty(); ++b) fill(&e.Em[b], (size_t)hp.m + 1, 0);
    }
    if (s->has_tiled) {
        TiledSys& tl = s->tiled;
        const TiledPack& tp = im.tp;
        tl.P = tp.P;
        tl.part_words = tp.part_words;
        tl.e_bits = tp.e_bits;
        tl.G = tp.G;
        tl.acc_words = tp.acc_words;
        tl.rin_words = tp.rin_words;
        tl.acc8 = tp.acc8;
        tl.rin_esm = tp.rin_esm;
        tl.src_bits = tp.src_bits;
        tl.pairs = tp.pairs;
        tl.rle = tp.rle;
        tl.tstart = nullptr;
        if (tp.rle) vec(&tl.tstart, tp.tstart);
        tl.ent_words = (int64_t)tp.ent.size();
        vec(&tl.sub, tp.sub);
        vec(&tl.ent, tp.ent);
        vec(&tl.cta_lo, tp.cta_lo);
        tl.inflow = nullptr;  // the fused step sums the partitions' in-flows in distributed shared memory
        if (tp.P > kTiledMaxCluster) fill(&tl.inflow, (size_t)tp.P * nslices * kSlice * 4, 0);
        for (int b = 0; b < 2; ++b) fill(&tl.Eg[b], (size_t)tp.P * tp.part_words * 4, 0);
    }
}

// Id of the current context, unique for the life of the process (0: unknown):
// after cudaDeviceReset the same device has another one.
static unsigned long long context_id() {
    using Fn = CUresult (*)(CUcontext, unsigned long long*);
    static const Fn fn = [] {
        void* p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuCtxGetId", &p, 12000, cudaEnableDefault, &q) != cudaSuccess ||
            q != cudaDriverEntryPointSuccess) {
            cudaGetLastError();
            p = nullptr;
        }
        return reinterpret_cast<Fn>(p);
    }();
    unsigned long long id = 0;
    return fn && fn(nullptr, &id) == CUDA_SUCCESS ? id : 0;
}

int materialize(snp_system* s) {
    if (s->materialized) return SNP_OK;
    if (!s->img) return fail(SNP_ERR_INVALID, "system has no host image");
    std::vector<Piece> plan;
    build_plan(s, plan);
    const size_t total = plan_bytes(plan);
    char* base = (char*)sys_alloc(s, total);
    if (!base) return fail(SNP_ERR_OOM, "device allocation of " + std::to_string(total) + " bytes failed");
    size_t off = 0;
    for (const Piece& p : plan) {
        *p.dst = base + off;
        cudaError_t e = cudaSuccess;
        if (p.src && p.bytes)
            e = cudaMemcpyAsync(base + off, p.src, p.bytes, cudaMemcpyHostToDevice, s->stream);
        else if (p.fill >= 0 && p.bytes)
            e = cudaMemsetAsync(base + off, p.fill, p.bytes, s->stream);
        if (e != cudaSuccess) return cuda_fail("upload");
        off += (p.bytes + 255) & ~(size_t)255;
    }
    DevSys& d = s->dev;
    d.step = reinterpret_cast<unsigned long long*>(reinterpret_cast<char*>(d.flags) + kStepOffset);
    const bool hp_hubs = (int64_t)s->img->hp.max_in * 32 >= s->q;
    d.rules_per_neuron = s->uniform_rules;
    d.identity = s->identity ? 1 : 0;
    d.compact = s->compact ? 1 : 0;
    d.hubs = hp_hubs ? 1 : 0;
    d.seed = s->opt.seed;
    philox_round_keys(d.seed, d.philox_rk);
    d.select = s->opt.select;
    d.max_p = s->max_p;
    if (cudaMemcpyAsync(s->d_self, &d, sizeof(DevSys), cudaMemcpyHostToDevice, s->stream) != cudaSuccess)
        return cuda_fail("descriptor upload");
    if (cudaStreamSynchronize(s->stream) != cudaSuccess) return cuda_fail("upload sync");
    s->img.reset();
    s->context = context_id();
    s->materialized = true;
    return SNP_OK;
}

bool is_device_ptr(const void* p) {
    cudaPointerAttributes a;
    if (cudaPointerGetAttributes(&a, p) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    return is_device_memory(a);
}

// Memory that a kernel on the current device may read in place.
static bool in_place_ptr(const void* p) {
    cudaPointerAttributes a;
    int dev = 0;
    if (cudaPointerGetAttributes(&a, p) != cudaSuccess || cudaGetDevice(&dev) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    return readable_in_place(a, dev);
}

// ---- chunk graphs of the grid-wide engines ------------------------------

// One pull launch of the system's grid-wide engine (L2-gather or tiled).
static cudaError_t launch_pull_any(snp_system* s, int kind, int32_t t, cudaStream_t st) {
    if (effective_engine(s) == SNP_ENGINE_TILED)
        return launch_tiled(s->dev, s->tiled, kind, t, st, s->compact, s->opt.select, s->tiled_smem,
                            s->tiled_threads);
    return launch_pull(s->dev, kind, t, st, s->compact, s->opt.select);
}

static int build_chunk_graph(snp_system* s) {
    if (s->chunk_exec) return SNP_OK;
    if (!s->cap_stream && cudaStreamCreateWithFlags(&s->cap_stream, cudaStreamNonBlocking) != cudaSuccess)
        return cuda_fail("stream create");
    cudaGraph_t g = nullptr;
    if (cudaStreamBeginCapture(s->cap_stream, cudaStreamCaptureModeThreadLocal) != cudaSuccess)
        return cuda_fail("begin capture");
    const bool compact = s->compact;
    const int sel = s->opt.select;
    for (int t = 0; t < kChunk; ++t) {
        if (s->opt.prop == SNP_PROP_PUSH)
            launch_push_step(s->dev, t, s->cap_stream, compact, sel);
        else
            launch_pull_any(s, kPullFused, t, s->cap_stream);
    }
    launch_advance(s->dev, kChunk, s->cap_stream);
    if (cudaStreamEndCapture(s->cap_stream, &g) != cudaSuccess) return cuda_fail("end capture");
    cudaError_t e = cudaGraphInstantiate(&s->chunk_exec, g, 0);
    cudaGraphDestroy(g);
    if (e != cudaSuccess) {
        s->chunk_exec = nullptr;
        return cuda_fail("graph instantiate");
    }
    return SNP_OK;
}

static int step_launch_engine(snp_system* s, int64_t n) {
    const bool compact = s->compact;
    const int sel = s->opt.select;
    cudaStream_t st = s->stream;
    if (launch_begin(s->dev, st) != cudaSuccess) return cuda_fail("begin");
    if (s->opt.prop == SNP_PROP_PUSH) {
        int64_t left = n;
        if (left >= kChunk) {
            int rc = build_chunk_graph(s);
            if (rc) return rc;
        }
        while (left >= kChunk) {
            if (cudaGraphLaunch(s->chunk_exec, st) != cudaSuccess) return cuda_fail("graph launch");
            left -= kChunk;
        }
        for (int64_t t = 0; t < left; ++t)
            if (launch_push_step(s->dev, (int32_t)t, st, compact, sel) != cudaSuccess) return cuda_fail("push step");
        if (launch_push_apply(s->dev, st) != cudaSuccess) return cuda_fail("push step");
        if (launch_finish(s->dev, (int32_t)left, st) != cudaSuccess) return cuda_fail("finish");
        return SNP_OK;
    }
    if (launch_pull_any(s, kPullSelectOnly, 0, st) != cudaSuccess) return cuda_fail("select");
    int64_t rem = n - 1;
    if (rem >= kChunk) {
        int rc = build_chunk_graph(s);
        if (rc) return rc;
    }
    while (rem >= kChunk) {
        if (cudaGraphLaunch(s->chunk_exec, st) != cudaSuccess) return cuda_fail("graph launch");
        rem -= kChunk;
    }
    for (int64_t t = 0; t < rem; ++t)
        if (launch_pull_any(s, kPullFused, (int32_t)t, st) != cudaSuccess) return cuda_fail("step");
    if (launch_pull_any(s, kPullGatherOnly, (int32_t)rem, st) != cudaSuccess) return cuda_fail("gather");
    if (launch_finish(s->dev, (int32_t)(rem + 1), st) != cudaSuccess) return cuda_fail("finish");
    return SNP_OK;
}

bool resident_fits(const snp_system* s, ResidentPlan* plan) {
    if (s->quad_lists) return plan == nullptr;  // on the cluster-resident engine
    if (!s->has_in_lists) return false;
    const int eb = resident_e_bits(s->max_p);
    const size_t smem = resident_smem_bytes(s->q, eb);
    if ((long long)smem + 1024 > (long long)resident_max_smem()) return false;
    if (plan) {
        plan->e_bits = eb;
        plan->max_q = s->q;
        plan->smem = smem;
        plan->threads = s->opt.threads > 0 ? s->opt.threads : 1024;
        plan->ctas = 1;
        plan->big = plan->threads == 1024;  // one CTA per system: the 64-register instance
    }
    return true;
}

bool cluster_plan(const snp_system* s, int T, ClusterPlan* plan) {
    if (T < 1 || T > kClusterMaxT || s->q > kMaxQuadQ) return false;
    const int ng = (s->q + kGroup - 1) / kGroup;
    const size_t cap = (size_t)resident_max_smem() - 1024;
    int lt = 0;
    while ((1 << lt) < T) ++lt;
    ClusterPlan p;
    p.mode = s->compiled    ? kClusterRec
             : s->tables    ? kClusterTable
             : s->test_recs ? (s->max_p < 256 ? kClusterTest8 : kClusterTest16)
                            : kClusterGeneral;
    p.T = T;
    // a warp per group, or several when a CTA has few groups: one for every
    // 16 columns (32 in-edges) of their lists at least, since meeting costs
    // what about ten columns do (128 neurons of 10 in-edges: 1.02 us per step
    // with one warp, 1.13 with two; the sorting system of 200 numbers, 100
    // columns: 7.2 with one, 6.2 with four)
    const int own = std::max(1, (ng + T - 1) / T);
    int S = 1;
    while (S < 8 && S * 32 <= s->cl_cols[lt] / own && 2 * S * own * 32 <= kClusterThreads) S *= 2;
    if (p.mode == kClusterRec && T <= 2 && 4 * own * 32 <= kClusterThreads) S = 4;  // a warp per neuron of the quads
    p.threads = s->opt.threads > 0 ? (s->opt.threads + 31) / 32 * 32 : S * own * 32;
    p.threads = std::max(kClusterMinThreads, std::min(kClusterThreads, p.threads));
    // what fits of lists and test records, the smaller first
    const bool test = p.mode == kClusterTest8 || p.mode == kClusterTest16;
    p.rules = test ? s->cl_rules[lt] : 0;
    auto bytes = [&] { return cluster_smem_bytes(p.mode, ng, T, p.lsm, s->cl_cols[lt], p.rules); };
    p.lsm = true;
    if ((p.smem = bytes()) > cap) {
        p.lsm = p.rules > 0 && (size_t)s->cl_cols[lt] * 512 < (size_t)p.rules * 16;
        if (p.lsm) p.rules = 0;
        p.smem = bytes();
    }
    if (p.smem > cap) {
        p.lsm = false;
        p.rules = 0;
        p.smem = bytes();
    }
    if (p.smem > cap) return false;
    *plan = p;
    return true;
}

static int step_resident(snp_system* s, int64_t n) {
    if (s->quad_lists) {
        // One system alone: as many CTAs as keep four groups (of 128 neurons)
        // each, since a CTA's step is a group's latency of about 1 us plus what
        // further groups add, and the cluster barrier costs less than either
        // (us per step with 1 / 8 CTAs: 8,192 neurons 9.7 / 2.1; 1,024 neurons
        // with 1 / 2 CTAs 1.61 / 1.50; 512 neurons and less: no gain).
        const int ng = (s->q + kGroup - 1) / kGroup;
        int T = 1;
        while (T < kClusterMaxT && ng > 4 * T) T *= 2;
        ClusterPlan cp;
        bool fits = cluster_plan(s, T, &cp);
        while (!fits && T < kClusterMaxT) fits = cluster_plan(s, T *= 2, &cp);
        if (!fits || launch_cluster(s->d_self, nullptr, n, 1, cp, s->opt.select, s->stream) != cudaSuccess)
            return cuda_fail("resident launch");
        return SNP_OK;
    }
    ResidentPlan plan;
    if (!resident_fits(s, &plan))
        return fail(SNP_ERR_UNSUPPORTED, "system too large for the resident engine (shared memory)");
    if (cudaMemcpyAsync(s->d_nsteps, &n, sizeof(long long), cudaMemcpyHostToDevice, s->stream) != cudaSuccess)
        return cuda_fail("nsteps upload");
    if (cudaMemsetAsync(s->d_work, 0, sizeof(unsigned int), s->stream) != cudaSuccess) return cuda_fail("work reset");
    if (launch_resident(s->d_self, s->d_nsteps, 1, s->d_work, plan, s->compact, s->opt.select, s->stream) != cudaSuccess)
        return cuda_fail("resident launch");
    return SNP_OK;
}

int effective_engine(const snp_system* s) {
    if (s->opt.form != SNP_FORM_OPT) return SNP_ENGINE_LAUNCH;
    if (s->opt.prop == SNP_PROP_PUSH) return SNP_ENGINE_LAUNCH;
    if (s->opt.engine == SNP_ENGINE_RESIDENT) return SNP_ENGINE_RESIDENT;
    if (s->opt.engine == SNP_ENGINE_LAUNCH) return SNP_ENGINE_LAUNCH;
    if (s->opt.engine == SNP_ENGINE_TILED) return SNP_ENGINE_TILED;
    if (s->q <= kAutoResidentMaxQ && s->m <= kAutoResidentMaxRules && resident_fits(s, nullptr))
        return SNP_ENGINE_RESIDENT;
    return s->has_tiled || s->has_grid ? SNP_ENGINE_TILED : SNP_ENGINE_LAUNCH;
}

static int step_grid(snp_system* s, int64_t n) {
    for (int64_t done = 0; done < n; done += kLaunchMaxSteps)
        if (launch_grid(s->dev, s->grid, std::min<int64_t>(n - done, kLaunchMaxSteps), done > 0, s->opt.select, s->stream) !=
            cudaSuccess)
            return cuda_fail("grid-resident launch");
    return SNP_OK;
}

// The grid-resident launch of an AUTO system in quad order (hp.quad_ptr32 given);
// false when the packed emissions and the state of a CTA's groups do not fit,
// the device cannot hold the grid at once, or a long in-list would keep one
// warp busy.
static bool grid_plan(snp_system* s, const HostPack& hp, int sms) {
    GridSys& gs = s->grid;
    const int ng = (hp.q + kGroup - 1) / kGroup;
    int coop = 0, dev = 0;
    cudaGetDevice(&dev);
    if (cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev) != cudaSuccess || !coop || sms < 1) return false;
    gs.mode = s->compiled ? kClusterRec : s->tables ? kClusterTable : s->test_recs ? kClusterTest8 : kClusterGeneral;
    gs.e_bits = tiled_e_bits(hp.max_p);
    gs.e_bytes = (int32_t)(((int64_t)ng * kGroup * gs.e_bits / 8 + 31) / 16 * 16);
    gs.G = std::min(sms, ng);
    gs.own = (ng + gs.G - 1) / gs.G;
    const std::vector<int32_t>& ptr = hp.quad_ptr32;
    int64_t most = 0;
    for (int r = 0; r < gs.G; ++r) {
        int64_t cols = 0;
        for (int g = r; g < ng; g += gs.G) cols += ptr[(size_t)g + 1] - ptr[(size_t)g];
        most = std::max(most, cols);
    }
    // several warps per group as in cluster_plan: one for every 16 columns
    int S = 1;
    while (S < 8 && S * 32 <= most / gs.own && 2 * S * gs.own * 32 <= kClusterThreads) S *= 2;
    gs.warps_per_group = S;
    // warps without a group help to copy the emissions, four 16-byte pieces a
    // thread: 65,000 neurons 4.75 -> 4.41 us per step; with fewer pieces a
    // larger CTA only meets later (32,768 neurons 3.85 -> 4.12)
    gs.threads = std::max(128, std::min(kClusterThreads, std::max(S * gs.own * 32, gs.e_bytes / 64 / 32 * 32)));
    // what fits of lists and test records, the lists first
    int64_t rules = 0;
    if (gs.mode == kClusterTest8)
        for (int r = 0; r < gs.G; ++r) {
            int64_t m = 0;
            for (int g = r; g < ng; g += gs.G)
                m += hp.rule_off[(size_t)std::min(hp.q, (g + 1) * kGroup)] - hp.rule_off[(size_t)g * kGroup];
            rules = std::max(rules, m);
        }
    const size_t cap = (size_t)resident_max_smem() - 1024;
    const int cols = (int)std::min<int64_t>(most, 1 << 20);
    gs.rules = (int32_t)rules;
    gs.lsm = 1;
    size_t b = grid_smem_bytes(gs.mode, gs, gs.lsm, cols, gs.rules);
    if (b > cap && gs.rules > 0) {
        gs.rules = 0;
        b = grid_smem_bytes(gs.mode, gs, gs.lsm, cols, 0);
    }
    if (b > cap && gs.lsm) {
        gs.lsm = 0;
        gs.rules = (int32_t)rules;
        b = grid_smem_bytes(gs.mode, gs, false, 0, gs.rules);
        if (b > cap) b = grid_smem_bytes(gs.mode, gs, false, 0, gs.rules = 0);
    }
    gs.smem = (int32_t)b;
    if (b > cap) return false;
    // A group's lists are as long as its longest one, and a few warps of one CTA
    // walk them, where the tiled engine deals all in-edges evenly to the chip's
    // threads.  From L2 a column costs a warp some 0.03 us (from shared memory a
    // third, and what fits there is short).  Without long lists a tiled step
    // takes 4 us more than a grid-resident one with compiled records, 6 at
    // 400,000 neurons, 12 to 15 more with test records or rule tables, 2 more
    // with the rule table itself.  us per step, grid / tiled, one neuron of 250,
    // 500, 1,000, 2,000 in-edges among neurons of 10: 32,768 neurons 4.0, 5.6, 7.9,
    // 12.5 / 7.1; 200,000 neurons 11.3, 18.8, 33, 62 / 8.6; 100,000 neurons with
    // test records 9.6, 13.4, 21, 37 / 17.4; 60,000 with rule tables 7.6, 10, 13.7,
    // 21.2 / 21.1.  100,000 neurons of power-law in-degrees (rank^-0.8, longest
    // list 19,745): 295 / 8.2.
    const int warps = gs.threads / 32;
    const int64_t even = hp.nsyn / ((int64_t)kGroup * gs.G * warps);
    const int spare = gs.mode == kClusterTest8 || gs.mode == kClusterTable ? 352 : 96;
    return gs.lsm || grid_longest_walk(ptr, gs.G, warps, S) - even <= spare + hp.q / 8192;
}

// Which layouts a system needs, from its options and size (before packing).
static void plan_layouts(const snp_options& o, int32_t q, int64_t m, bool* want_tiled, bool* want_in_lists) {
    if (o.form != SNP_FORM_OPT) {
        *want_tiled = *want_in_lists = false;
        return;
    }
    *want_tiled = o.prop == SNP_PROP_PULL &&
                  (o.engine == SNP_ENGINE_TILED ||
                   (o.engine == SNP_ENGINE_AUTO && (q > kAutoResidentMaxQ || m > kAutoResidentMaxRules)));
    // sliced ELL in-lists: the L2-gather and resident engines and the batch
    *want_in_lists = o.engine != SNP_ENGINE_TILED;
}

// ELL form (pull or push) and dense form: plain launches per step.
static int step_ell_forms(snp_system* s, int64_t n) {
    const bool compact = s->compact;
    const int sel = s->opt.select;
    cudaStream_t st = s->stream;
    const EllSys& e = s->ell;
    if (e.bit_ent) {
        for (int64_t done = 0; done < n; done += kLaunchMaxSteps)
            if (launch_ell_run(s->dev, e, std::min<int64_t>(n - done, kLaunchMaxSteps), done > 0, sel, st) != cudaSuccess)
                return cuda_fail("ell launch");
        return SNP_OK;
    }
    if (launch_begin(s->dev, st) != cudaSuccess) return cuda_fail("begin");
    if (s->opt.form == SNP_FORM_ELL && s->opt.prop == SNP_PROP_PULL) {
        if (launch_ell_pull(s->dev, e, kPullSelectOnly, 0, st, compact, sel) != cudaSuccess) return cuda_fail("select");
        for (int64_t t = 0; t + 1 < n; ++t)
            if (launch_ell_pull(s->dev, e, kPullFused, (int32_t)t, st, compact, sel) != cudaSuccess)
                return cuda_fail("ell step");
        if (launch_ell_pull(s->dev, e, kPullGatherOnly, (int32_t)(n - 1), st, compact, sel) != cudaSuccess)
            return cuda_fail("ell gather");
    } else if (s->opt.form == SNP_FORM_ELL) {
        for (int64_t t = 0; t < n; ++t) {
            if (launch_ell_select(s->dev, e, e.inflow != nullptr, true, (int32_t)t, st, compact, sel) != cudaSuccess ||
                launch_ell_push(s->dev, e, (int32_t)t, st) != cudaSuccess)
                return cuda_fail("ell push step");
        }
        if (e.inflow && launch_ell_select(s->dev, e, true, false, (int32_t)n, st, compact, sel) != cudaSuccess)
            return cuda_fail("ell push step");
    } else {
        if (launch_ell_select(s->dev, e, false, true, 0, st, compact, sel) != cudaSuccess) return cuda_fail("select");
        for (int64_t t = 0; t < n; ++t) {
            if (launch_dense_accum(s->dev, e, (int32_t)t, st) != cudaSuccess ||
                launch_ell_select(s->dev, e, true, t + 1 < n, (int32_t)(t + 1), st, compact, sel) != cudaSuccess)
                return cuda_fail("dense step");
        }
    }
    if (launch_finish(s->dev, (int32_t)n, st) != cudaSuccess) return cuda_fail("finish");
    return SNP_OK;
}

// Page-locked bytes for small reads back, one piece per thread and context for
// as long as both live: a copy into pageable memory is staged by the driver,
// about 5 us each time (a piece per system would cost its creation 100 us and
// its end 155).  NULL when there are none to be had.
struct PinnedWords {
    static constexpr int kContexts = 4;  // of one thread; beyond them, pageable copies
    unsigned long long ctx[kContexts] = {};
    void* p[kContexts] = {};
    ~PinnedWords() {
        // Only the current context's piece is known to exist still.  In the
        // relaxed capture mode: in the default one the call would fail, and
        // spoil the capture, while another thread captures a stream.
        const unsigned long long id = context_id();
        cudaStreamCaptureMode mode = cudaStreamCaptureModeRelaxed;
        for (int i = 0; i < kContexts && id != 0; ++i)
            if (ctx[i] == id && p[i]) {
                cudaThreadExchangeStreamCaptureMode(&mode);
                if (cudaFreeHost(p[i]) != cudaSuccess) cudaGetLastError();
                cudaThreadExchangeStreamCaptureMode(&mode);
            }
    }
};
// id: of the context whose memory is read.
static void* pinned_words(unsigned long long id) {
    static thread_local PinnedWords w;
    if (id == 0) return nullptr;
    for (int i = 0; i < PinnedWords::kContexts; ++i) {
        if (w.ctx[i] == id) return w.p[i];
        if (w.ctx[i] != 0) continue;
        if (context_id() != id) return nullptr;  // another context is current: not its own bytes
        w.ctx[i] = id;  // asked for once, whatever comes of it
        if (cudaHostAlloc(&w.p[i], kStatusBytes, cudaHostAllocDefault) != cudaSuccess) {
            cudaGetLastError();
            w.p[i] = nullptr;
        }
        return w.p[i];
    }
    return nullptr;
}

// Copies `bytes` (at most kStatusBytes) from the system's device memory and waits.
static bool read_small(const snp_system* s, void* dst, const void* src, size_t bytes) {
    void* pin = pinned_words(s->context);
    if (cudaMemcpyAsync(pin ? pin : dst, src, bytes, cudaMemcpyDeviceToHost, s->stream) != cudaSuccess ||
        cudaStreamSynchronize(s->stream) != cudaSuccess)
        return false;
    if (pin) std::memcpy(dst, pin, bytes);
    return true;
}

int read_flags(snp_system* s, int64_t* exec) {
    alignas(8) unsigned char words[kStatusBytes];
    if (!read_small(s, words, s->dev.flags, kStatusBytes)) return cuda_fail("flag read");
    uint32_t fl[kNumFlags];
    unsigned long long steps[kNumStepWords];
    std::memcpy(fl, words, sizeof(fl));
    std::memcpy(steps, words + kStepOffset, sizeof(steps));
    if (exec) *exec = (int64_t)steps[kStepExec];
    s->host_step = steps[kStepBase];
    if (fl[kFlagOverflow]) {
        const uint32_t zero = 0;
        cudaMemcpyAsync(s->dev.flags + kFlagOverflow, &zero, sizeof(zero), cudaMemcpyHostToDevice, s->stream);
        cudaStreamSynchronize(s->stream);
        return fail(SNP_ERR_OVERFLOW, "a spike count left the int32 range");
    }
    if (fl[kFlagBounds]) {
        char msg[96];
        snprintf(msg, sizeof(msg), "bounds check: an index out of range (sites 0x%x)", fl[kFlagBounds]);
        const uint32_t zero = 0;
        cudaMemcpyAsync(s->dev.flags + kFlagBounds, &zero, sizeof(zero), cudaMemcpyHostToDevice, s->stream);
        cudaStreamSynchronize(s->stream);
        return fail(SNP_ERR_INVALID, msg);
    }
    if (fl[kFlagTimeout]) return fail(SNP_ERR_TIMEOUT, "a bounded device wait gave up");
    if (fl[kFlagChoice]) {
        const uint32_t zero = 0;
        cudaMemcpyAsync(s->dev.flags + kFlagChoice, &zero, sizeof(zero), cudaMemcpyHostToDevice, s->stream);
        cudaStreamSynchronize(s->stream);
        return fail(SNP_ERR_INVALID, "a forced choice index was out of range for its neuron");
    }
    return SNP_OK;
}

int run_steps(snp_system* s, int64_t n) {
    if (n <= 0) return SNP_OK;
    if (s->opt.form != SNP_FORM_OPT) return step_ell_forms(s, n);
    if (s->has_grid) return step_grid(s, n);
    const int eng = effective_engine(s);
    if ((eng == SNP_ENGINE_LAUNCH || eng == SNP_ENGINE_RESIDENT) && s->opt.prop == SNP_PROP_PULL && !s->has_in_lists &&
        !s->quad_lists)
        return fail(SNP_ERR_UNSUPPORTED, "system was created for the tiled engine only");
    return eng == SNP_ENGINE_RESIDENT ? step_resident(s, n) : step_launch_engine(s, n);
}

// The launches of a pull call of n steps on a grid-wide engine, as
// step_launch_engine issues them but without its chunk graph (so without
// the base step's advances, which only bound the step index of the chunk
// graph's launches): begin, the first select, n - 1 fused steps, the last
// gather, finish.  Every parameter is a constant of the call, so the
// sequence can be captured once and replayed.
static cudaError_t enqueue_pull_call(snp_system* s, int64_t n, cudaStream_t st) {
    cudaError_t e = launch_begin(s->dev, st);
    if (e == cudaSuccess) e = launch_pull_any(s, kPullSelectOnly, 0, st);
    for (int64_t t = 0; t < n - 1 && e == cudaSuccess; ++t) e = launch_pull_any(s, kPullFused, (int32_t)t, st);
    if (e == cudaSuccess) e = launch_pull_any(s, kPullGatherOnly, (int32_t)(n - 1), st);
    if (e == cudaSuccess) e = launch_finish(s->dev, (int32_t)n, st);
    return e;
}

int run_steps_graphed(snp_system* s, int64_t n) {
    const int eng = s->opt.form == SNP_FORM_OPT ? effective_engine(s) : SNP_ENGINE_LAUNCH;
    if (n < 2 || n > kMaxGraphedCall || s->opt.form != SNP_FORM_OPT || s->opt.prop != SNP_PROP_PULL ||
        eng == SNP_ENGINE_RESIDENT || s->has_grid || (eng == SNP_ENGINE_LAUNCH && !s->has_in_lists))
        return run_steps(s, n);
    if (!s->call_exec || s->call_n != n) {
        if (s->call_exec) cudaGraphExecDestroy(s->call_exec);
        s->call_exec = nullptr;
        if (!s->cap_stream && cudaStreamCreateWithFlags(&s->cap_stream, cudaStreamNonBlocking) != cudaSuccess)
            return cuda_fail("stream create");
        cudaGraph_t g = nullptr;
        if (cudaStreamBeginCapture(s->cap_stream, cudaStreamCaptureModeThreadLocal) != cudaSuccess)
            return cuda_fail("begin capture");
        const cudaError_t le = enqueue_pull_call(s, n, s->cap_stream);
        if (cudaStreamEndCapture(s->cap_stream, &g) != cudaSuccess || le != cudaSuccess) {
            if (g) cudaGraphDestroy(g);
            return cuda_fail("call capture");
        }
        const cudaError_t e = cudaGraphInstantiate(&s->call_exec, g, 0);
        cudaGraphDestroy(g);
        if (e != cudaSuccess) {
            s->call_exec = nullptr;
            return cuda_fail("graph instantiate");
        }
        s->call_n = n;
    }
    if (cudaGraphLaunch(s->call_exec, s->stream) != cudaSuccess) return cuda_fail("graph launch");
    return SNP_OK;
}

}  // namespace snp

using namespace snp;

extern "C" {

const char* snp_strerror(int st) {
    switch (st) {
        case SNP_OK: return "ok";
        case SNP_ERR_INVALID: return "invalid argument or malformed system";
        case SNP_ERR_OOM: return "out of memory";
        case SNP_ERR_CUDA: return "CUDA runtime error";
        case SNP_ERR_TIMEOUT: return "bounded device wait timed out";
        case SNP_ERR_OVERFLOW: return "spike count overflowed int32";
        case SNP_ERR_BUSY: return "system is owned by an unfinished batch";
        case SNP_ERR_UNSUPPORTED: return "unsupported option combination";
        default: return "unknown status";
    }
}

const char* snp_last_error(void) { return snp::last_error(); }

int snp_create(const snp_desc* desc, const snp_options* opts, snp_system** out) {
    if (!out) return fail(SNP_ERR_INVALID, "out is NULL");
    *out = nullptr;
    int st = validate_desc(desc);
    if (st) return st;
    snp_options o;
    std::memset(&o, 0, sizeof(o));
    if (opts) o = *opts;
    if (o.form != SNP_FORM_OPT && o.form != SNP_FORM_ELL && o.form != SNP_FORM_DENSE)
        return fail(SNP_ERR_INVALID, "bad form");
    if (o.prop != SNP_PROP_PULL && o.prop != SNP_PROP_PUSH) return fail(SNP_ERR_INVALID, "bad prop");
    if (o.select != SNP_SELECT_FIRST && o.select != SNP_SELECT_PHILOX) return fail(SNP_ERR_INVALID, "bad select");
    if (o.engine < SNP_ENGINE_AUTO || o.engine > SNP_ENGINE_TILED) return fail(SNP_ERR_INVALID, "bad engine");
    if (o.prop == SNP_PROP_PUSH && (o.engine == SNP_ENGINE_RESIDENT || o.engine == SNP_ENGINE_TILED))
        return fail(SNP_ERR_UNSUPPORTED, "the resident and tiled engines are pull-only");
    if (o.form != SNP_FORM_OPT && o.engine != SNP_ENGINE_AUTO && o.engine != SNP_ENGINE_LAUNCH)
        return fail(SNP_ERR_UNSUPPORTED, "the ELL and dense forms run on the launch engine");
    if (o.form == SNP_FORM_DENSE && o.prop != SNP_PROP_PULL)
        return fail(SNP_ERR_UNSUPPORTED, "the dense form walks matrix columns (pull) only");

    snp_system* s = new (std::nothrow) snp_system();
    if (!s) return fail(SNP_ERR_OOM, "host allocation failed");
    s->opt = o;
    s->stream = (cudaStream_t)o.stream;
    if (o.alloc) s->alloc = *o.alloc;
    s->img.reset(new (std::nothrow) HostImage());
    if (!s->img) {
        delete s;
        return fail(SNP_ERR_OOM, "host allocation failed");
    }
    HostImage& im = *s->img;
    HostPack& hp = im.hp;
    bool want_tiled = false, want_in = false;
    plan_layouts(o, desc->q, desc->rule_offsets[desc->q], &want_tiled, &want_in);
    int dev = 0, sms = 0, optin = 0;
    if (want_tiled) {
        cudaGetDevice(&dev);
        if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
            cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) != cudaSuccess) {
            delete s;
            return cuda_fail("device query");
        }
    }
    // The tiled layout needs no in-degree order; without it slots are the
    // caller's neurons, and the select reads no slot-to-neuron map.  Under
    // AUTO the caller's order is kept as well when the system is too large
    // for one CTA (so no resident in-lists): if no tiled layout fits after
    // all, the system is packed again in the in-degree order that the
    // L2-gather engine's in-lists want.
    // The grid-resident form comes first where one CTA holds the packed
    // emissions beside its share of the state (some 690,000 neurons at 2 bits):
    // 450,000 neurons 9.4 us per step against the tiled engine's 12.8.
    const bool auto_large = o.engine == SNP_ENGINE_AUTO && want_tiled &&
                            resident_smem_bytes(desc->q, 2) + 1024 > (size_t)optin;
    bool grid_size = false;
    if (auto_large) {
        const int64_t m = desc->rule_offsets[desc->q];
        const int32_t max_p = m > 0 ? *std::max_element(desc->rule_p, desc->rule_p + m) : 0;
        const int64_t ng = ((int64_t)desc->q + kGroup - 1) / kGroup, own = (ng + sms - 1) / std::max(1, sms);
        GridSys gs{};
        gs.e_bytes = (int32_t)std::min<int64_t>(ng * kGroup * tiled_e_bits(max_p) / 8 + 32, INT32_MAX / 2);
        gs.own = (int32_t)own;
        gs.warps_per_group = 1;
        grid_size = grid_smem_bytes(kClusterRec, gs, false, 0, 0) + 2048 <= (size_t)optin;
    }
    int window = (o.form == SNP_FORM_OPT && (o.engine == SNP_ENGINE_TILED || (auto_large && !grid_size))) ? 0 : kSortWindow;
    // the cluster- and grid-resident engines want their slots in quad order
    const bool quads = o.form == SNP_FORM_OPT && o.prop == SNP_PROP_PULL && window > 0 &&
                       (o.engine == SNP_ENGINE_AUTO || (o.engine == SNP_ENGINE_RESIDENT && desc->q <= kMaxQuadQ));
    bool ell_bits = false;
    st = pack_system(desc, o.form == SNP_FORM_OPT && o.prop == SNP_PROP_PUSH, false, window, &hp, quads);
    if (!st && o.form == SNP_FORM_ELL && o.prop == SNP_PROP_PULL && hp.max_rules <= 4 && hp.max_p < 2048 &&
        hp.q <= kEllBitsMaxQ && (int64_t)hp.max_in * (int64_t)hp.max_p <= (int64_t)INT32_MAX) {
        // the one-launch form, where the device holds its grid at once
        EllSys& e = s->ell;
        int coop = 0, nsm = 0, d0 = 0;
        cudaGetDevice(&d0);
        if (cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, d0) == cudaSuccess && coop &&
            cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, d0) == cudaSuccess && nsm > 0) {
            const int nslices = (hp.q + kSlice - 1) / kSlice;
            e.bit_words = (nslices * 4 + 1 + 3) / 4 * 4;
            e.G = std::min(nsm, std::max(1, nslices));
            e.own = (nslices + e.G - 1) / e.G;
            ell_bits = ell_run_smem(e) + 1024 <= (size_t)resident_max_smem();
        }
        cudaGetLastError();
    }
    if (!st && o.form == SNP_FORM_ELL)
        st = pack_ell(desc, hp, o.prop == SNP_PROP_PULL, o.prop == SNP_PROP_PUSH, &im.ep, ell_bits);
    if (!st && o.form == SNP_FORM_DENSE) st = pack_dense(desc, hp, &im.dense);
    if (st) {
        delete s;
        return st;
    }
    // union expressions step through the compiled records when every neuron
    // fits one, else through union records in the general rule table
    s->unions = desc->rule_term_offsets != nullptr;

    s->q = hp.q;
    s->max_p = hp.max_p;
    s->compact = hp.compact;
    s->compiled = (s->opt.form == SNP_FORM_OPT || s->unions) && !hp.rec.empty();
    // the engines over quads: the first form that holds every rule, else the
    // rule table itself
    if (hp.quads && !s->compiled && !(s->tables = build_rule_tables(desc, &hp)))
        s->test_recs = build_test_records(desc, &hp);
    if (want_tiled && hp.quads && (int64_t)hp.max_in * (int64_t)hp.max_p <= (int64_t)INT32_MAX) {
        s->has_grid = quad_list_starts(hp, 1, &hp.quad_ptr32) && grid_plan(s, hp, sms);
        if (s->has_grid) {
            pack_in_quads32(desc, &hp, s->grid.e_bits);
            want_in = hp.q <= kBatchResidentMaxQ;  // for batches
        }
    }
    // not so after all: the caller's order for the tiled engine, unless batches
    // want the quads
    if (want_tiled && !s->has_grid && hp.quads && hp.q > kBatchResidentMaxQ) {
        hp = HostPack();
        s->tables = s->test_recs = false;
        window = 0;
        st = pack_system(desc, false, false, window, &hp);
        if (st) {
            delete s;
            return st;
        }
    }
    if (want_tiled && !s->has_grid) {
        // the gather sums a partition's in-flow in 32-bit shared accumulators,
        // read back as int32: a target must not be able to receive more than
        // INT32_MAX spikes from one partition in one step (the int64 sums of
        // the other engines carry any in-flow to the overflow check)
        if ((int64_t)hp.max_in * (int64_t)hp.max_p > (int64_t)INT32_MAX)
            st = fail(SNP_ERR_UNSUPPORTED, "in-degree x p can exceed the tiled engine's 32-bit accumulators");
        else {
            // clusters of P CTAs with about the largest shared memory per CTA
            int cpw[kTiledMaxCluster + 1] = {0};
            for (int P = 1; P <= kTiledMaxCluster; ++P) cpw[P] = tiled_clusters_per_wave(P, (size_t)optin - 2048);
            st = pack_tiled(desc, hp, sms, (size_t)optin - 2048, &im.tp, cpw);
        }
        // Under AUTO the tiled engine must pay for itself: every CTA copies a
        // whole emission partition into shared memory each step.  With one
        // wave of CTAs that copy overlaps the entry stream; with several
        // waves (large, low-degree systems with 32-bit accumulators: many
        // partitions) it can move more bytes than the gathers it replaces.
        // Keep it when it is one wave or the copies stay under half the
        // entry stream.
        if (st == SNP_OK && o.engine == SNP_ENGINE_AUTO && im.tp.G > sms &&
            (double)im.tp.G * im.tp.part_words * 4.0 > 0.5 * 4.0 * (double)im.tp.ent.size()) {
            im.tp = TiledPack();
            st = SNP_ERR_UNSUPPORTED;
        }
        if (st == SNP_OK) {
            s->has_tiled = true;
            // the resident engine (batches) still needs in-lists when the system fits one CTA
            if (o.engine == SNP_ENGINE_AUTO)
                want_in = hp.q <= kBatchResidentMaxQ &&
                          resident_smem_bytes(hp.q, resident_e_bits(hp.max_p)) + 1024 <= (size_t)optin;
        } else if (o.engine == SNP_ENGINE_TILED) {
            delete s;
            return st;
        } else {
            want_in = true;  // AUTO falls back to the L2-gather engine
            if (window != kSortWindow || hp.quads) {
                hp = HostPack();
                s->tables = s->test_recs = false;
                window = kSortWindow;
                st = pack_system(desc, false, false, window, &hp);
                if (st) {
                    delete s;
                    return st;
                }
            }
        }
    }
    if (want_in && hp.quads) {
        for (int T = 1; T <= kClusterMaxT && !s->quad_lists; T *= 2) {
            ClusterPlan cp;
            s->quad_lists = cluster_plan(s, T, &cp);
        }
    }
    // no cluster holds it (wide emissions, or more than 65,408 neurons): in a
    // batch one CTA does, where its packed emissions fit
    if (s->has_grid && !s->quad_lists)
        want_in = want_in && resident_smem_bytes(hp.q, resident_e_bits(hp.max_p)) + 1024 <= (size_t)optin;
    if (s->quad_lists)
        pack_in_quads(desc, &hp);
    else if (want_in)
        pack_in_lists(desc, &hp);
    s->has_in_lists = want_in && !s->quad_lists;
    for (int lt = 0; lt < 4 && s->quad_lists; ++lt) {  // group i goes to CTA i mod T of a cluster
        std::vector<int32_t> cols((size_t)1 << lt, 0), rules((size_t)1 << lt, 0);
        for (size_t i = 0; i + 1 < hp.quad_ptr.size(); ++i) {
            cols[i & (((size_t)1 << lt) - 1)] += hp.quad_ptr[i + 1] - hp.quad_ptr[i];
            rules[i & (((size_t)1 << lt) - 1)] +=
                hp.rule_off[std::min<size_t>((size_t)hp.q, (i + 1) * kGroup)] - hp.rule_off[i * kGroup];
        }
        s->cl_rules[lt] = *std::max_element(rules.begin(), rules.end());
        s->cl_cols[lt] = *std::max_element(cols.begin(), cols.end());
    }
    s->m = hp.m;
    s->nsyn = hp.nsyn;
    s->max_p = hp.max_p;
    s->max_rules = hp.max_rules;
    s->uniform_rules = hp.uniform_rules;
    s->identity = hp.identity;
    s->in_entries = s->quad_lists ? (int64_t)hp.in_quads.size() : (int64_t)hp.in_idx.size();
    s->out_entries = (int64_t)hp.out_idx.size();
    if (o.form == SNP_FORM_ELL) {
        s->in_entries = ell_bits ? (int64_t)im.ep.in_ptr.back() * kSlice : (int64_t)im.ep.in_ent.size() / 2;
        s->out_entries = (int64_t)im.ep.out_ent.size() / 2;
    }
    if (o.form == SNP_FORM_DENSE) s->in_entries = (int64_t)im.dense.size();
    s->grid_entries = (int64_t)hp.in_quads32.size();
    s->rule_words = (int64_t)hp.rules.size();
    s->perm = hp.perm;
    s->rule_offsets.assign(desc->rule_offsets, desc->rule_offsets + (size_t)desc->q + 1);
    if (s->has_tiled) {
        s->tiled_smem = tiled_smem_bytes(im.tp);
        s->tiled_entries = (int64_t)im.tp.ent.size();
        s->tiled_threads = kTiledThreads;  // fixed: the entry layout is dealt to this many threads
        s->tiled_P = im.tp.P;
        s->tiled_G = im.tp.G;
        s->tiled_layout = im.tp.rle ? 2 : (im.tp.pairs ? 1 : 0);
        s->tiled_acc_bits = im.tp.acc8 ? 8 : 32;
    }
    {
        std::vector<Piece> plan;
        build_plan(s, plan);
        s->planned_bytes = plan_bytes(plan);
    }
    if (!(o.flags & SNP_FLAG_DEFER_UPLOAD)) {
        st = materialize(s);
        if (st) {
            sys_free_all(s);
            delete s;
            return st;
        }
    }
    *out = s;
    return SNP_OK;
}

int snp_destroy(snp_system* s) {
    if (!s) return SNP_OK;
    if (s->busy.load()) return fail(SNP_ERR_BUSY, "system is owned by an unfinished batch");
    if (s->stream) cudaStreamSynchronize(s->stream);
    else cudaDeviceSynchronize();
    if (s->chunk_exec) cudaGraphExecDestroy(s->chunk_exec);
    if (s->call_exec) cudaGraphExecDestroy(s->call_exec);
    if (s->cap_stream) cudaStreamDestroy(s->cap_stream);
    batch_release(s);
    sys_free_all(s);
    if (s->own_stream) cudaStreamDestroy(s->stream);
    delete s;
    return SNP_OK;
}

// The system's descriptor with `forced` set (or cleared), also in its device
// copy (read by the CTA-resident engine).
static int set_forced(snp_system* s, const int32_t* forced) {
    s->dev.forced = forced;
    if (s->d_self &&
        cudaMemcpyAsync(s->d_self, &s->dev, sizeof(DevSys), cudaMemcpyHostToDevice, s->stream) != cudaSuccess)
        return cuda_fail("descriptor upload");
    return SNP_OK;
}

int snp_step(snp_system* s, int64_t n, int64_t* steps_done) {
    if (!s) return fail(SNP_ERR_INVALID, "system is NULL");
    if (s->busy.load()) return fail(SNP_ERR_BUSY, "system is owned by an unfinished batch");
    if (int rc_ = materialize(s)) return rc_;
    if (n < 0) return fail(SNP_ERR_INVALID, "n < 0");
    if (steps_done) *steps_done = 0;
    if (n == 0) return SNP_OK;
    if (s->choices_pending) {
        // the first step alone, with the forced choices, then the rest
        s->choices_pending = false;
        int rc = set_forced(s, s->d_forced);
        if (!rc) rc = run_steps(s, 1);
        const int rc2 = set_forced(s, nullptr);
        if (rc) return rc;
        if (rc2) return rc2;
        int64_t first = 0;
        if ((rc = read_flags(s, &first))) return rc;
        if (steps_done) *steps_done = first;
        if (n == 1 || first == 0) return SNP_OK;
        if ((rc = run_steps(s, n - 1))) return rc;
        int64_t rest = 0;
        if ((rc = read_flags(s, &rest))) return rc;
        if (steps_done) *steps_done += rest;
        return SNP_OK;
    }
    int rc = run_steps(s, n);
    if (rc) return rc;
    if (steps_done) return read_flags(s, steps_done);
    return SNP_OK;
}

// The message for the first invalid neuron a state check found; its three
// values are read back from the caller's arrays (host or device).
static int state_error(const snp_system* s, int32_t i, const int32_t* C, const int32_t* D, const int32_t* P,
                       const std::string& where = std::string()) {
    (void)s;
    int32_t c = 0, d = 0, p = 0;
    if (cudaMemcpy(&c, C + i, 4, cudaMemcpyDefault) != cudaSuccess ||
        cudaMemcpy(&d, D + i, 4, cudaMemcpyDefault) != cudaSuccess ||
        cudaMemcpy(&p, P + i, 4, cudaMemcpyDefault) != cudaSuccess)
        return cuda_fail("state read-back");
    const std::string at = " at neuron " + std::to_string(i);
    if (c < 0) return fail(SNP_ERR_INVALID, where + "negative spike count" + at);
    if (d < 0 || d > kMaxDelay) return fail(SNP_ERR_INVALID, where + "D out of range" + at);
    if (p == -1) return fail(SNP_ERR_INVALID, where + "D > 0 without a pending rule" + at);
    return fail(SNP_ERR_INVALID, where + "pending rule does not belong to neuron " + std::to_string(i));
}

int snp_branch_step(snp_system* s, int32_t nb, const int32_t* C, const int32_t* D, const int32_t* P,
                    const int32_t* choices, int32_t* C_out, int32_t* D_out, int32_t* P_out, int32_t* executed,
                    int32_t* bad, int32_t* counts) {
    if (!s) return fail(SNP_ERR_INVALID, "system is NULL");
    if (nb < 0) return fail(SNP_ERR_INVALID, "nb < 0");
    if (nb == 0) return SNP_OK;
    if (!C || !D || !P || !choices || !C_out || !D_out || !P_out || !executed || !bad)
        return fail(SNP_ERR_INVALID, "NULL argument");
    if (s->busy.load()) return fail(SNP_ERR_BUSY, "system is owned by an unfinished batch");
    if (int rc_ = materialize(s)) return rc_;
    if (s->opt.form != SNP_FORM_OPT || (!s->has_in_lists && !s->quad_lists) || s->q > kBranchMaxQ)
        return fail(SNP_ERR_UNSUPPORTED, "branch steps need the optimized form with in-lists and q <= 8192");
    const size_t n = (size_t)nb * (size_t)s->q;
    cudaStream_t st = s->stream;
    // Host buffers are staged on the device in one block from the system's
    // allocator, together with the word the input check reports into.
    struct Buf {
        const void* user;
        void* dev;
        size_t bytes;
        bool in, host;
    };
    Buf bufs[10] = {{C, nullptr, n * 4, true, false},      {D, nullptr, n * 4, true, false},
                    {P, nullptr, n * 4, true, false},      {choices, nullptr, n * 4, true, false},
                    {C_out, nullptr, n * 4, false, false}, {D_out, nullptr, n * 4, false, false},
                    {P_out, nullptr, n * 4, false, false}, {executed, nullptr, (size_t)nb * 4, false, false},
                    {bad, nullptr, (size_t)nb * 4, false, false}, {counts, nullptr, n * 4, false, false}};
    size_t stage = 256;  // the first 256 bytes hold the check's word
    for (Buf& b : bufs) {
        if (!b.user) continue;  // counts is optional
        b.host = !is_device_ptr(b.user);
        if (b.host) stage += (b.bytes + 255) & ~(size_t)255;
    }
    char* block = (char*)stage_alloc(s, stage);
    if (!block) return fail(SNP_ERR_OOM, "staging buffer for snp_branch_step");
    unsigned long long* d_first_bad = (unsigned long long*)block;
    size_t off = 256;
    int rc = SNP_OK;
    for (Buf& b : bufs) {
        if (!b.user) continue;
        if (!b.host) {
            b.dev = const_cast<void*>(b.user);
            continue;
        }
        b.dev = block + off;
        off += (b.bytes + 255) & ~(size_t)255;
        if (b.in && cudaMemcpyAsync(b.dev, b.user, b.bytes, cudaMemcpyHostToDevice, st) != cudaSuccess) {
            rc = cuda_fail("staging copy");
            break;
        }
    }
    // The input check runs, and is read back, before the step kernel is
    // launched: a configuration out of range never reaches k_branch_step.
    unsigned long long first_bad = ~0ull;
    if (!rc && (cudaMemsetAsync(d_first_bad, 0xff, sizeof(unsigned long long), st) != cudaSuccess ||
                launch_branch_check(s->dev, s->d_rule_base, nb, (const int32_t*)bufs[0].dev,
                                    (const int32_t*)bufs[1].dev, (const int32_t*)bufs[2].dev, d_first_bad,
                                    st) != cudaSuccess ||
                cudaMemcpyAsync(&first_bad, d_first_bad, sizeof(first_bad), cudaMemcpyDeviceToHost, st) !=
                    cudaSuccess ||
                cudaStreamSynchronize(st) != cudaSuccess))
        rc = cuda_fail("branch input check");
    if (!rc && first_bad != ~0ull) {
        const unsigned long long b = first_bad / (unsigned long long)s->q;
        const int32_t i = (int32_t)(first_bad % (unsigned long long)s->q);
        rc = state_error(s, i, C + b * (unsigned long long)s->q, D + b * (unsigned long long)s->q,
                         P + b * (unsigned long long)s->q, "configuration " + std::to_string(b) + ": ");
    }
    if (!rc && launch_branch_step(s->dev, s->d_rule_base, resident_e_bits(s->max_p), s->compact, nb,
                                  (const int32_t*)bufs[0].dev, (const int32_t*)bufs[1].dev, (const int32_t*)bufs[2].dev,
                                  (const int32_t*)bufs[3].dev, (int32_t*)bufs[4].dev, (int32_t*)bufs[5].dev,
                                  (int32_t*)bufs[6].dev, (int32_t*)bufs[7].dev, (int32_t*)bufs[8].dev,
                                  (int32_t*)bufs[9].dev, st) != cudaSuccess)
        rc = cuda_fail("branch step");
    for (Buf& b : bufs) {
        if (!b.host || !b.dev || b.in || rc) continue;
        if (cudaMemcpyAsync(const_cast<void*>(b.user), b.dev, b.bytes, cudaMemcpyDeviceToHost, st) != cudaSuccess)
            rc = cuda_fail("staging copy");
    }
    uint32_t over = 0;
    const bool synced = cudaMemcpyAsync(&over, s->dev.flags + kFlagOverflow, 4, cudaMemcpyDeviceToHost, st) ==
                            cudaSuccess &&
                        cudaStreamSynchronize(st) == cudaSuccess;
    stage_free(s, block, stage);
    if (!synced) return rc ? rc : cuda_fail("branch step");
    if (rc) return rc;
    if (over) {
        const uint32_t zero = 0;
        cudaMemcpyAsync(s->dev.flags + kFlagOverflow, &zero, 4, cudaMemcpyHostToDevice, st);
        cudaStreamSynchronize(st);
        return fail(SNP_ERR_OVERFLOW, "a spike count left the int32 range");
    }
    return SNP_OK;
}

int snp_set_choices(snp_system* s, const int32_t* idx, int64_t len) {
    if (!s || !idx) return fail(SNP_ERR_INVALID, "NULL argument");
    if (s->busy.load()) return fail(SNP_ERR_BUSY, "system is owned by an unfinished batch");
    if (int rc_ = materialize(s)) return rc_;
    if (len < s->q) return fail(SNP_ERR_INVALID, "choices shorter than q");
    std::vector<int32_t> host((size_t)s->q), slots((size_t)s->q);
    if (is_device_ptr(idx)) {
        if (cudaMemcpyAsync(host.data(), idx, sizeof(int32_t) * (size_t)s->q, cudaMemcpyDeviceToHost, s->stream) !=
                cudaSuccess ||
            cudaStreamSynchronize(s->stream) != cudaSuccess)
            return cuda_fail("choices copy");
    } else {
        std::memcpy(host.data(), idx, sizeof(int32_t) * (size_t)s->q);
    }
    for (int32_t slot = 0; slot < s->q; ++slot) slots[slot] = host[(size_t)s->perm[slot]];
    if (!s->d_forced) {
        s->d_forced = (int32_t*)sys_alloc(s, sizeof(int32_t) * (size_t)std::max(1, s->q));
        if (!s->d_forced) return fail(SNP_ERR_OOM, "device allocation for forced choices failed");
    }
    if (cudaMemcpyAsync(s->d_forced, slots.data(), sizeof(int32_t) * (size_t)s->q, cudaMemcpyHostToDevice,
                        s->stream) != cudaSuccess ||
        cudaStreamSynchronize(s->stream) != cudaSuccess)
        return cuda_fail("choices upload");
    s->choices_pending = true;
    return SNP_OK;
}

static int export_vec(const snp_system* sc, int what, int32_t* out, int64_t len) {
    snp_system* s = const_cast<snp_system*>(sc);
    if (!s || !out) return fail(SNP_ERR_INVALID, "NULL argument");
    if (s->busy.load()) return fail(SNP_ERR_BUSY, "system is owned by an unfinished batch");
    if (int rc_ = materialize(s)) return rc_;
    if (len < s->q) return fail(SNP_ERR_INVALID, "output shorter than q");
    const bool dev = is_device_ptr(out);
    int32_t* dst = dev ? out : s->scratch;
    if (launch_export(s->dev, s->d_rule_base, what, dst, -1, s->stream, s->compact) != cudaSuccess)
        return cuda_fail("export");
    if (!dev) {
        if (cudaMemcpyAsync(out, s->scratch, sizeof(int32_t) * (size_t)s->q, cudaMemcpyDeviceToHost, s->stream) != cudaSuccess ||
            cudaStreamSynchronize(s->stream) != cudaSuccess)
            return cuda_fail("export copy");
    }
    return SNP_OK;
}

int snp_get_config(const snp_system* s, int32_t* out, int64_t len) { return export_vec(s, kExportConfig, out, len); }
int snp_count_choices(const snp_system* s, int32_t* out, int64_t len) {
    return export_vec(s, kExportChoices, out, len);
}
int snp_get_spiking(const snp_system* s, int32_t* out, int64_t len) { return export_vec(s, kExportSpiking, out, len); }
int snp_get_status(const snp_system* s, int32_t* out, int64_t len) { return export_vec(s, kExportStatus, out, len); }
int snp_get_pending(const snp_system* s, int32_t* out, int64_t len) { return export_vec(s, kExportPending, out, len); }

int snp_get_state(const snp_system* s, int32_t* C, int32_t* D, int32_t* P, int64_t len, uint64_t* step) {
    if (!s) return fail(SNP_ERR_INVALID, "system is NULL");
    if (int rc_ = materialize(const_cast<snp_system*>(s))) return rc_;
    int rc;
    if (C && (rc = snp_get_config(s, C, len))) return rc;
    if (D && (rc = snp_get_status(s, D, len))) return rc;
    if (P && (rc = snp_get_pending(s, P, len))) return rc;
    if (step) {
        unsigned long long v = 0;
        if (!read_small(s, &v, s->dev.step + kStepBase, sizeof(v)))
            return cuda_fail("step read");
        *step = v;
    }
    return SNP_OK;
}

// Imports (C, D, P) on the device: arrays in this device's memory are read where
// they are (once: other streams may still write them), others (host memory,
// another GPU's) are copied, both into buffers whose contents set_state discards
// anyway (the spiking vectors and the export scratch).  One launch checks, a
// second writes in slot order if every neuron passed, and the host waits once
// for the verdict.
int snp_set_state(snp_system* s, const int32_t* C, const int32_t* D, const int32_t* P, int64_t len, uint64_t step) {
    if (!s || !C || !D || !P) return fail(SNP_ERR_INVALID, "NULL argument");
    if (s->busy.load()) return fail(SNP_ERR_BUSY, "system is owned by an unfinished batch");
    if (int rc_ = materialize(s)) return rc_;
    if (len < s->q) return fail(SNP_ERR_INVALID, "state shorter than q");
    cudaStream_t st = s->stream;
    const size_t bytes = sizeof(int32_t) * (size_t)s->q;
    const bool direct = ((uintptr_t)C | (uintptr_t)D | (uintptr_t)P) % sizeof(int32_t) == 0 && in_place_ptr(C) &&
                        in_place_ptr(D) && in_place_ptr(P);
    const int32_t *sc = C, *sd = D, *sp = P;
    if (!direct) {
        if (cudaMemcpyAsync(s->scratch, C, bytes, cudaMemcpyDefault, st) != cudaSuccess ||
            cudaMemcpyAsync(s->dev.S[0], D, bytes, cudaMemcpyDefault, st) != cudaSuccess ||
            cudaMemcpyAsync(s->dev.S[1], P, bytes, cudaMemcpyDefault, st) != cudaSuccess)
            return cuda_fail("state upload");
        sc = s->scratch;
        sd = s->dev.S[0];
        sp = s->dev.S[1];
    }
    uint32_t bad = 0xffffffffu;
    if (cudaMemsetAsync(s->dev.flags + kFlagImport, 0xff, sizeof(uint32_t), st) != cudaSuccess ||
        launch_import(s->dev, s->d_rule_base, sc, sd, sp, step, direct ? s->scratch : nullptr, st) != cudaSuccess)
        return cuda_fail("state import");
    // the spiking vectors held the staged D and P: all -1 again either way (in
    // place, the commit has done that)
    if (!direct && (cudaMemsetAsync(s->dev.S[0], 0xff, bytes, st) != cudaSuccess ||
                    cudaMemsetAsync(s->dev.S[1], 0xff, bytes, st) != cudaSuccess))
        return cuda_fail("state upload");
    if (!read_small(s, &bad, s->dev.flags + kFlagImport, sizeof(bad))) return cuda_fail("state import");
    if (bad != 0xffffffffu) {
        if (direct && (cudaMemsetAsync(s->dev.S[0], 0xff, bytes, st) != cudaSuccess ||
                       cudaMemsetAsync(s->dev.S[1], 0xff, bytes, st) != cudaSuccess ||
                       cudaStreamSynchronize(st) != cudaSuccess))
            return cuda_fail("state upload");
        return state_error(s, (int32_t)bad, C, D, P);
    }
    return SNP_OK;
}

int snp_check_bounded_wait(int32_t polls) {
    if (polls < 1 || polls > 1000000) return fail(SNP_ERR_INVALID, "polls must be in 1..1000000");
    cudaStream_t st = nullptr;
    uint32_t* d_out = nullptr;
    uint32_t h_out = 0;
    if (cudaStreamCreateWithFlags(&st, cudaStreamNonBlocking) != cudaSuccess) return cuda_fail("stream");
    int rc = SNP_OK;
    if (cudaMalloc(&d_out, sizeof(uint32_t)) != cudaSuccess || cudaMemsetAsync(d_out, 0, 4, st) != cudaSuccess ||
        launch_wait_check(polls, d_out, st) != cudaSuccess ||
        cudaMemcpyAsync(&h_out, d_out, 4, cudaMemcpyDeviceToHost, st) != cudaSuccess ||
        cudaStreamSynchronize(st) != cudaSuccess)
        rc = cuda_fail("bounded wait check");
    else if (h_out == 2u)
        rc = fail(SNP_ERR_TIMEOUT, "the bounded wait gave up after " + std::to_string(polls) + " polls");
    else if (h_out != 1u)
        rc = fail(SNP_ERR_CUDA, "the wait check did not report");
    if (d_out) cudaFree(d_out);
    cudaStreamDestroy(st);
    return rc;
}

int snp_get_info(const snp_system* s, snp_info* info) {
    if (!s || !info) return fail(SNP_ERR_INVALID, "NULL argument");
    std::memset(info, 0, sizeof(*info));
    info->q = s->q;
    info->form = s->opt.form;
    info->prop = s->opt.prop;
    info->select = s->opt.select;
    info->engine = effective_engine(s);
    info->m = s->m;
    info->num_syn = s->nsyn;
    info->in_entries = info->engine == SNP_ENGINE_TILED ? s->tiled_entries : s->in_entries;
    info->out_entries = s->out_entries;
    info->rule_words = s->rule_words;
    info->device_bytes = (int64_t)(s->materialized ? s->device_bytes : s->planned_bytes);
    info->max_rules = s->max_rules;
    info->max_p = s->max_p;
    info->compact_rules = s->compact ? 1 : 0;
    info->e_bits = info->engine != SNP_ENGINE_TILED ? resident_e_bits(s->max_p)
                   : s->has_grid                     ? s->grid.e_bits
                                                     : s->tiled.e_bits;
    info->step = s->host_step;
    info->compiled_rules = s->compiled ? 1 : 0;
    if (s->has_tiled) {
        info->tiled_partitions = s->tiled_P;
        info->tiled_ctas = s->tiled_G;
        info->tiled_layout = s->tiled_layout;
        info->tiled_acc_bits = s->tiled_acc_bits;
        info->tiled_smem_bytes = (int64_t)s->tiled_smem;
    }
    if (s->has_grid) {
        info->in_entries = s->grid_entries;
        info->tiled_partitions = 1;
        info->tiled_ctas = s->grid.G;
        info->tiled_layout = 3;
        info->tiled_acc_bits = 32;
        info->tiled_smem_bytes = s->grid.smem;
    }
    return SNP_OK;
}

}  // extern "C"
