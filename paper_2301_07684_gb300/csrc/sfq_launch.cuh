// sfq_launch.cuh -- launchers of one precision; included by sfq_launch_f32.cu and
// sfq_launch_f64.cu with SFQ_T set to float or double.
#pragma once
#include "sfq_internal.h"
#include "sfq_fused.cuh"
#include "sfq_push.cuh"
#include "sfq_step_tma.cuh"

namespace sfq {

template <typename T>
static Tables<T> tables_of(const sfq_ctx *ctx) {
    Tables<T> t;
    t.nlc_rate = static_cast<const T *>(ctx->d_nlc_rate);
    t.nbw_rate = static_cast<const T *>(ctx->d_nbw_rate);
    t.nlc_inv = static_cast<const T *>(ctx->d_nlc_inv);
    t.nbw_inv = static_cast<const T *>(ctx->d_nbw_inv);
    t.k23 = static_cast<const T *>(ctx->d_k23);
    t.ki13 = static_cast<const T *>(ctx->d_ki13);
    t.nlc_inv_r = static_cast<const T *>(ctx->d_nlc_inv_r);
    t.nbw_inv_r = static_cast<const T *>(ctx->d_nbw_inv_r);
    t.tr = ctx->inv_tr;
    return t;
}

template <typename T>
static cudaError_t launch_rate_t(const RateLaunch &L, bool pair) {
    if (L.n == 0) return cudaSuccess;
    const T *g = static_cast<const T *>(L.gamma), *x = static_cast<const T *>(L.chi);
    T *out = static_cast<T *>(L.rate);
    const T *tab = static_cast<const T *>(L.table);
    auto kern = pair ? (L.cheb ? rate_kernel<T, true, true> : rate_kernel<T, true, false>)
                     : (L.cheb ? rate_kernel<T, false, true> : rate_kernel<T, false, false>);
    kern<<<L.grid, L.block, 0, L.stream>>>(L.n, g, x, out, tab, (T)L.pref, L.counters, (T)L.pair_chi_min);
    return cudaGetLastError();
}

template <bool PAIR, int TR>
static cudaError_t launch_sample_tile(const SampleLaunch &L, const Tables<float> &tab) {
    auto kern = sample_tile_kernel<PAIR, TR>;
    const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)SAMP_SMEM);
    if (e != cudaSuccess) return e;
    const int64_t ntiles = (L.n + SAMP_TILE - 1) / SAMP_TILE, wave = (int64_t)SAMP_MINB * L.ctx->num_sms;
    kern<<<(unsigned)(ntiles < wave ? ntiles : wave), SAMP_BS, SAMP_SMEM, L.stream>>>(
        L.n, static_cast<const float *>(L.chi), static_cast<const float *>(L.r), static_cast<float *>(L.a),
        static_cast<float *>(L.b), tab, L.counters);
    return cudaGetLastError();
}

template <typename T, bool PAIR>
static cudaError_t launch_sample_k(const SampleLaunch &L, Tables<T> tab) {
    const T *x = static_cast<const T *>(L.chi), *r = static_cast<const T *>(L.r);
    T *a = static_cast<T *>(L.a), *b = static_cast<T *>(L.b);
    const bool clenshaw = L.ctx->eval == SFQ_EVAL_CLENSHAW;
    if constexpr (sizeof(T) == 4) {
        // sorted tiles once every SM has one (at that size 25 us one element per thread, under
        // 16 us sorted); smaller calls, which tiles would leave SMs idle in, and the comparison
        // evaluator take one element per thread
        if (!clenshaw && L.n >= (int64_t)SAMP_TILE * L.ctx->num_sms) {
            if (tab.tr == 2) return launch_sample_tile<PAIR, 2>(L, tab);
            if (tab.tr == 1) return launch_sample_tile<PAIR, 1>(L, tab);
            return launch_sample_tile<PAIR, 0>(L, tab);
        }
    }
    if (clenshaw) {
        // the comparison evaluator: Chebyshev pieces of the full tables, Clenshaw's recurrence
        tab.nlc_inv = static_cast<const T *>(L.ctx->d_nlc_inv_ch);
        tab.nbw_inv = static_cast<const T *>(L.ctx->d_nbw_inv_ch);
        sample_kernel<T, PAIR, false, true><<<L.grid, L.block, 0, L.stream>>>(L.n, x, r, a, b, tab, L.counters);
    } else if (tab.tr > 0) {
        sample_kernel<T, PAIR, true><<<L.grid, L.block, 0, L.stream>>>(L.n, x, r, a, b, tab, L.counters);
    } else {
        sample_kernel<T, PAIR, false><<<L.grid, L.block, 0, L.stream>>>(L.n, x, r, a, b, tab, L.counters);
    }
    return cudaGetLastError();
}

template <typename T>
static cudaError_t launch_sample_t(const SampleLaunch &L, bool pair) {
    if (L.n == 0) return cudaSuccess;
    const Tables<T> tab = tables_of<T>(L.ctx);
    return pair ? launch_sample_k<T, true>(L, tab) : launch_sample_k<T, false>(L, tab);
}

template <typename T>
static cudaError_t launch_uniforms_t(int64_t n, const uint64_t *id, uint32_t step, uint32_t tag, uint64_t seed,
                                     void *u, cudaStream_t s, int grid, int block) {
    if (n == 0) return cudaSuccess;
    uniforms_kernel<T><<<grid, block, 0, s>>>(n, id, step, tag, seed, static_cast<T *>(u));
    return cudaGetLastError();
}

// Dynamic shared-memory limits of the TMA-staged kernels, set once per process (and before
// any stream capture, where the launch itself is recorded).
template <typename T, bool TRUNC>
static cudaError_t prepare_step_t() {
    static bool done = false;
    if (done) return cudaSuccess;
    cudaError_t e = cudaSuccess;
#define SFQ_PREP(CWV)                                                                                         \
    if (e == cudaSuccess)                                                                                     \
        e = cudaFuncSetAttribute(mc_step_tma_kernel<T, FK_SOA, CWV, TRUNC>,                                  \
                                 cudaFuncAttributeMaxDynamicSharedMemorySize, (int)tma_smem_bytes<T, FK_SOA, CWV>()); \
    if (e == cudaSuccess)                                                                                     \
        e = cudaFuncSetAttribute(mc_step_tma_kernel<T, FK_PW, CWV, TRUNC>,                                   \
                                 cudaFuncAttributeMaxDynamicSharedMemorySize, (int)tma_smem_bytes<T, FK_PW, CWV>());
    if constexpr (TRUNC) {
        SFQ_PREP(TRUNC_CW)
    } else {
        SFQ_PREP(8)
        SFQ_PREP(16)
        SFQ_PREP(20)
        if (e == cudaSuccess)
            e = cudaFuncSetAttribute(mc_step_tma_kernel<T, FK_PW, TMA_CW_PW>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     (int)tma_smem_bytes<T, FK_PW, TMA_CW_PW>());
    }
#undef SFQ_PREP
    if (e == cudaSuccess) done = true;
    return e;
}

// Kernel arguments of one step (or of the first step of a fused run) from the C descriptors.
template <typename T>
static StepArgs<T> make_step_args(const StepLaunch &L) {
    const sfq_particles &p = *L.p;
    const sfq_fields &f = *L.f;
    const sfq_ctx *ctx = L.ctx;
    StepArgs<T> a{};
    a.n = p.n;
    a.n_dev = p.n_dev;
    a.px = static_cast<T *>(p.px); a.py = static_cast<T *>(p.py); a.pz = static_cast<T *>(p.pz);
    for (int k = 0; k < 3; ++k) {
        a.fprev[k] = static_cast<T *>(p.fprev[k]);
        a.dfprev[k] = static_cast<T *>(p.dfprev[k]);
    }
    a.lepton_model = p.lepton_model;
    a.tau = p.tau;
    a.id = p.id;
    a.id_base = p.id_base;
    a.flags = p.flags;
    a.ex = static_cast<const T *>(f.ex); a.ey = static_cast<const T *>(f.ey); a.ez = static_cast<const T *>(f.ez);
    a.bx = static_cast<const T *>(f.bx); a.by = static_cast<const T *>(f.by); a.bz = static_cast<const T *>(f.bz);
    a.k0 = f.k0;
    a.amp = static_cast<const T *>(f.amp);
    a.amp0 = (T)f.amp0;
    a.pw_table = static_cast<const T *>(f.table);
    a.n_table = f.n_table;
    a.pw_offset = f.kind == SFQ_FIELDS_PLANE_WAVE
                      ? (uint32_t)(((uint64_t)L.step * (uint64_t)f.k_step) % (uint64_t)f.n_table)
                      : 0u;
    a.cap = L.out->capacity;
    a.opx = static_cast<T *>(L.out->px); a.opy = static_cast<T *>(L.out->py); a.opz = static_cast<T *>(L.out->pz);
    a.opid = L.out->parent_id;
    a.ostep = L.out->step;
    a.ometa = L.out->meta;
    a.ocount = L.out->count;
    if (L.spawn) {
        const sfq_spawn &s = *L.spawn;
        a.scap = s.p.n;
        a.spx = static_cast<T *>(s.p.px); a.spy = static_cast<T *>(s.p.py); a.spz = static_cast<T *>(s.p.pz);
        a.stau = s.p.tau;
        a.sid = const_cast<uint64_t *>(s.p.id);
        a.sflags = s.p.flags;
        for (int k = 0; k < 3; ++k) {
            a.sfp[k] = static_cast<T *>(s.p.fprev[k]);
            a.sdf[k] = static_cast<T *>(s.p.dfprev[k]);
        }
        a.sk0 = s.k0;
        a.samp = static_cast<T *>(s.amp);
        a.scount = s.count;
    }
    a.step = L.step;
    a.seed = ctx->cfg.seed;
    a.prefdt = (T)(ctx->pref * ctx->cfg.dt);
    a.inv_rho = (T)(1.0 / ctx->rho);
    a.rho = (T)ctx->rho;
    a.inv_dt = (T)(1.0 / ctx->cfg.dt);
    a.dt = (T)ctx->cfg.dt;
    a.inv_dt2 = (T)(1.0 / (ctx->cfg.dt * ctx->cfg.dt));
    a.pair_chi_min = (T)ctx->pair_chi_min;
    a.tab = tables_of<T>(ctx);
    a.counters = L.counters;
    if (ctx->surr || ctx->defer_q.count) {
        const sfq_event_queue &q = ctx->surr ? ctx->surr_q : ctx->defer_q;
        a.qcap = q.capacity;
        a.qidx = q.index;
        a.qchi = q.chi; a.qr = q.r; a.qg = q.gamma;
        a.qpx = q.px; a.qpy = q.py; a.qpz = q.pz;
        a.qcount = q.count;
    }
    return a;
}

template <typename T, bool TRUNC>
static cudaError_t launch_step_t(const StepLaunch &L) {
    const sfq_particles &p = *L.p;
    const sfq_fields &f = *L.f;
    const sfq_ctx *ctx = L.ctx;
    if (p.n == 0) return cudaSuccess;
    const StepArgs<T> a = make_step_args<T>(L);
    const bool pw = f.kind == SFQ_FIELDS_PLANE_WAVE;
    // TMA-staged kernel: one persistent block per SM; `ppt` selects the consumer warps per block.
    // Chosen automatically (us per step in a graph, warp-streaming against TMA-staged):
    //  - binary32, fields in memory: from ten tiles per SM, where the pipeline has filled (150,000
    //    particles 13.0 / 14.0, 300,000 16.0 / 16.0, 10^6 22.0 / 23.8, 1.5*10^6 27.9 / 27.3,
    //    2*10^6 36.2 / 32.4);
    //  - binary32, plane wave: from a tile per SM (11.1 / 11.9 at 150,000, 13.8 / 13.6 at 300,000,
    //    31.6 / 30.6 at 2*10^6);
    //  - binary64: from 128 particles per SM (28 / 27 at 20,000, 80 / 44 at 160,000, 556 / 532 at
    //    4*10^6), with 8 consumer warps: the FP64 pipe takes two lanes per clock and SM whatever
    //    a warp's active lanes, 8 warps keep it busy and leave 8 partial event batches at the
    //    end instead of 16 (62 us at 160,000).  Only a plane wave of millions of
    //    particles gains from more (507 / 493 us at 4*10^6).
    const bool f64 = sizeof(T) == 8;
    const int dflt = f64 ? (pw && p.n >= (1ll << 21) ? TMA_CW_PW : 8) : (pw ? TMA_CW_PW : TMA_CW_SOA);
    const bool given = L.ppt == 8 || L.ppt == 16 || L.ppt == 20 || (pw && L.ppt == TMA_CW_PW);
    const int cw = TRUNC ? TRUNC_CW : (given ? L.ppt : dflt);
    const int tile = cw * (f64 ? 32 : 64);
    const int64_t tma_from = (int64_t)(TRUNC ? tile : (f64 ? 128 : (pw ? 1024 : 10 * 1024))) * ctx->num_sms;
    // the beyond-LCFA model runs on the warp-streaming kernel (its state is read directly)
    const bool tma = !L.cascade && p.lepton_model == SFQ_LEPTON_LCFA_OD &&
                     (L.variant == 2 || (L.variant == 0 && p.n >= tma_from));
    if (tma) {
        void (*kern)(const StepArgs<T>) = nullptr;
        size_t smem = 0;
#define SFQ_TMA_CASE(CWV)                                                                             \
    case CWV:                                                                                         \
        kern = pw ? mc_step_tma_kernel<T, FK_PW, CWV, TRUNC> : mc_step_tma_kernel<T, FK_SOA, CWV, TRUNC>; \
        smem = pw ? tma_smem_bytes<T, FK_PW, CWV>() : tma_smem_bytes<T, FK_SOA, CWV>();                 \
        break;
        if constexpr (TRUNC) {
            switch (cw) {
                default:
                SFQ_TMA_CASE(TRUNC_CW)
            }
        } else {
            switch (cw) {
                SFQ_TMA_CASE(8)
                SFQ_TMA_CASE(20)
                case TMA_CW_PW:
                    kern = mc_step_tma_kernel<T, FK_PW, TMA_CW_PW>;
                    smem = tma_smem_bytes<T, FK_PW, TMA_CW_PW>();
                    break;
                default:
                SFQ_TMA_CASE(16)
            }
        }
#undef SFQ_TMA_CASE
        cudaError_t e = prepare_step_t<T, TRUNC>();
        if (e != cudaSuccess) return e;
        (void)smem;
        const int64_t ntiles = (p.n + tile - 1) / tile;
        int grid = L.grid > 0 ? L.grid : ctx->num_sms;
        if (ntiles < grid) grid = (int)ntiles;
        kern<<<grid, 32 * (cw + 1), smem, L.stream>>>(a);
        return cudaGetLastError();
    }
    void (*kern)(const StepArgs<T>) = nullptr;
    if (L.cascade) {
        // the full cascade (plane-wave fields only) runs its own instance of this kernel
        kern = mc_step_kernel<T, FK_PW, TRUNC ? TRUNC_PPT : 2, TRUNC, true>;
    } else if constexpr (TRUNC) {
        kern = pw ? mc_step_kernel<T, FK_PW, TRUNC_PPT, true> : mc_step_kernel<T, FK_SOA, TRUNC_PPT, true>;
    } else if (p.lepton_model != SFQ_LEPTON_LCFA_OD) {
        // beyond-LCFA leptons: the instance of two particles per lane, in either precision
        kern = pw ? mc_step_kernel<T, FK_PW, 2> : mc_step_kernel<T, FK_SOA, 2>;
    } else {
        switch ((pw ? 10 : 0) + L.ppt) {
            case 1: kern = mc_step_kernel<T, FK_SOA, 1>; break;
            case 4: kern = mc_step_kernel<T, FK_SOA, 4>; break;
            case 11: kern = mc_step_kernel<T, FK_PW, 1>; break;
            case 12: kern = mc_step_kernel<T, FK_PW, 2>; break;
            case 14: kern = mc_step_kernel<T, FK_PW, 4>; break;
            default: kern = mc_step_kernel<T, FK_SOA, 2>; break;
        }
    }
    const int ppt = TRUNC ? TRUNC_PPT : ((L.cascade || p.lepton_model != SFQ_LEPTON_LCFA_OD) ? 2 : L.ppt);
    int grid = L.grid;
    if (grid <= 0) {
        // one wave of resident blocks: a multiple of the SM count
        int per_sm = 0;
        cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, STEP_BS, 0);
        if (e != cudaSuccess || per_sm < 1) per_sm = 1;
        grid = per_sm * ctx->num_sms;
        const int64_t chunks = (p.n + 32 * ppt - 1) / (32 * ppt);
        const int64_t need = (chunks + STEP_BS / 32 - 1) / (STEP_BS / 32);
        if (need < grid) grid = (int)(need > 0 ? need : 1);
    }
    if (L.cascade && grid > 65535) grid = 65535;       // the commit counts blocks in 16 bits
    kern<<<grid, STEP_BS, 0, L.stream>>>(a);
    return cudaGetLastError();
}

// nsteps steps from L.step on in one launch of the fused plane-wave kernel (sfq_fused.cuh).
template <typename T, bool TRUNC>
static cudaError_t launch_fused_t(const StepLaunch &L, uint32_t nsteps) {
    constexpr int PPL = sizeof(T) == 4 ? 4 : 2;
    using CFG = FusedCfg<T, PPL>;
    const sfq_particles &p = *L.p;
    const sfq_fields &f = *L.f;
    if (p.n == 0 || nsteps == 0) return cudaSuccess;
    const StepArgs<T> a = make_step_args<T>(L);
    auto kern = mc_fused_kernel<T, PPL, TRUNC>;
    static bool attr = false;
    if (!attr) {
        const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                   (int)CFG::smem(FUSED_TABLE_MAX));
        if (e != cudaSuccess) return e;
        attr = true;
    }
    const size_t smem = CFG::smem(f.n_table);
    int per_sm = 0;
    cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, FUSED_BS, smem);
    if (e != cudaSuccess || per_sm < 1) per_sm = 1;
    int grid = L.grid > 0 ? L.grid : per_sm * L.ctx->num_sms;
    const int64_t chunks = (p.n + 32 * PPL - 1) / (32 * PPL);
    const int64_t need = (chunks + CFG::WARPS - 1) / CFG::WARPS;
    if (need < grid) grid = (int)need;
    const uint32_t K = f.n_table;
    const uint32_t kstep = f.k_step % K;
    const uint32_t off0 = (uint32_t)(((uint64_t)L.step * (uint64_t)f.k_step) % (uint64_t)K);
    kern<<<grid, FUSED_BS, smem, L.stream>>>(a, L.step, nsteps, off0, kstep);
    return cudaGetLastError();
}

// One Boris push of the population at L.step (sfq_push.cuh).
template <typename T>
static cudaError_t launch_push_t(const StepLaunch &L, double dt) {
    if (L.p->n == 0) return cudaSuccess;
    const StepArgs<T> a = make_step_args<T>(L);
    const int64_t blocks = (L.p->n + 255) / 256;
    const int grid = (int)(blocks < (int64_t)L.ctx->num_sms * 8 ? blocks : (int64_t)L.ctx->num_sms * 8);
    if (L.f->kind == SFQ_FIELDS_PLANE_WAVE)
        push_kernel<T, FK_PW><<<grid, 256, 0, L.stream>>>(a, (T)dt);
    else
        push_kernel<T, FK_SOA><<<grid, 256, 0, L.stream>>>(a, (T)dt);
    return cudaGetLastError();
}

}  // namespace sfq
