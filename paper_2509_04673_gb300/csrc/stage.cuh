// stage.cuh — host-side launch sequence of one SSP-RK stage (Sec. 4.3 of
// the paper: element loop, udot solve, facet loop, element loop, SSP update).
#pragma once

#include <utility>

#include "fused.cuh"

namespace cgl {

// Device buffers of one state. R-typed arrays are void* here.
struct Bufs {
    void* u;      // state            [NC][NN]  (R)
    void* un;     // RK base u^n      [NC][NN]  (R)
    void* g;      // g_h              [2NC][NN] (R)
    void* g2;     // g_h ping-pong    [2NC][NN] (R)
    void* ud2;    // udot ping-pong   [NC][NN]  (R)
    void* bg;     // rhs of g_h       [2NC][NN] (R)
    void* r;      // target residual  [NC][NN]  (R)
    void* ud;     // udot             [NC][NN]  (R)
    void* ER;     // element residual [N2][NC][E]  (R)
    void* EW;     // SSP increments   [N2][NC][E]  (R)
    void* q;      // flux-limiter capacities [2][E] (scalar)  (R)
    void* fl;     // low-order facet fluxes [E][4][NC]         (R)
    float* cf;    // float copies for the Euler limiter certificate [1+NC][E]: s, ubar^{e,L}
    float* avg;   // float-float cell means [2NC][E] (FP32-mixed: k_avg for systems, k_lo for scalars)
    void* cq;     // systems: flux of the mean and speed parts per cell [2NC + 6][E]  (R) (k_avg), in EW
    void* fht;    // facet terms of f_i^e [NC][E]  (R) (k_facet -> k_update_el, k_upd_sys)
    cudaStream_t st2, st3, st4;  // side streams of a stage (run_stage)
    cudaEvent_t ev_fork0, ev_s, ev_w, ev_join;
    double *ue, *dte, *ubl, *gam, *nu, *ube, *beta;
    unsigned long long* cnt;     // CNT_N counters
    unsigned long long* dtbits;  // min dt_e as bits
    double *dt, *t, *t_end;
};

// kernel identifiers for per-kernel timing
enum KernelId {
    KID_AVG = 0, KID_PRE, KID_DT, KID_GRAD, KID_GATHER, KID_GRADF, KID_SWEEP, KID_RES,
    KID_UPDATE, KID_FINAL, KID_TADV, KID_UDOTF, KID_FACET, KID_RESW, KID_Q1F, KID_UDL, KID_SENS, KID_COUNT
};

// optional per-launch timing: CUDA events recorded around every launch on
// the launching stream (never used inside graph capture)
struct Prof {
    struct Rec { int id; cudaEvent_t a, b; };
    Rec* recs;
    int n, cap;
    void begin(int id, cudaStream_t st) {
        if (n < cap) {
            recs[n].id = id;
            cudaEventRecord(recs[n].a, st);
        }
    }
    void end(cudaStream_t st) {
        if (n < cap) cudaEventRecord(recs[n++].b, st);
    }
};

// (in run_stage: nothing is launched once a launch has failed, so that k_final
// never gathers what the others have left out)
#define CGL_LAUNCH(PROF, ID, ST, ...)             \
    do {                                          \
        if (err != cudaSuccess) break;            \
        if (PROF) (PROF)->begin((ID), (ST));      \
        __VA_ARGS__;                              \
        if (PROF) (PROF)->end((ST));              \
    } while (0)

// first: compute the global dt from this stage's dt_e (stage 1 of a step);
// dt_only: stop after the dt reduction (time-step query)
typedef cudaError_t (*StageFn)(const Bufs&, const MeshDev&, const ProbDev&, double a, double b,
                               bool first, bool dt_only, cudaStream_t st, Prof* prof);

inline unsigned nblk(long long n, int bs) { return (unsigned)((n + bs - 1) / bs); }

// Size of the stencils' tiles (StageTile): large ones unless they make fewer
// than four (p <= 2) or two blocks per SM, tiny ones (float64) where the small
// ones make fewer than one.  Euler 768 x 192 Q2 FP32-mixed, 325 large tiles: 548
// us/step with them, 531 with small ones; Burgers 301 x 199 Q4, 475 large
// tiles: 257 and 260.
template <class R, int P>
inline int tile_size(const MeshDev& m) {
    using TL = stage_tile_t<R, P, 0>;
    using TS = stage_tile_t<R, P, 1>;
    if ((long long)nblk(m.nnx, TL::NX) * nblk(m.nny, TL::NY) >= (P <= 2 ? 608 : 304)) return 0;
    if (sizeof(R) == 4) return 1;
    return (long long)nblk(m.nnx, TS::NX) * nblk(m.nny, TS::NY) >= 152 ? 1 : 2;
}
template <class R>
inline int tile_size_of(const MeshDev& m) {
    switch (m.p) {
        case 1: return tile_size<R, 1>(m);
        case 2: return tile_size<R, 2>(m);
        case 3: return tile_size<R, 3>(m);
        default: return tile_size<R, 4>(m);
    }
}
// The g_h right-hand side and the first sweep in one kernel: always in float;
// in float64 (rsz: bytes per value) only on tiny meshes, elsewhere the sweep's
// halo costs a fifth of the float64 operations of both kernels and their
// traffic less.
inline bool fuse_grad_sweep(size_t rsz, int size) { return rsz == 4 || size == 2; }

// Launch with programmatic stream serialisation (pdl): the kernel may be
// scheduled while the previous kernel of the stream drains and waits for it
// in pdl_begin(); inside a captured graph this becomes a programmatic edge.
template <typename... KArgs, typename... Args>
inline cudaError_t launch(bool pdl, void (*k)(KArgs...), dim3 grid, dim3 block, cudaStream_t st, Args... args) {
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = 0;
    cfg.stream = st;
    cfg.attrs = at;
    cfg.numAttrs = pdl ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, k, static_cast<KArgs>(args)...);
}

// the same with dynamic shared memory (opted in above the default 48 KB)
template <typename... KArgs, typename... Args>
inline cudaError_t launch_shared(bool pdl, void (*k)(KArgs...), dim3 grid, dim3 block, int smem, cudaStream_t st,
                                 Args... args) {
    if (smem > 48 * 1024) {
        const cudaError_t e = cudaFuncSetAttribute((const void*)k, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
        if (e != cudaSuccess) return e;
    }
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cfg.attrs = at;
    cfg.numAttrs = pdl ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, k, static_cast<KArgs>(args)...);
}

// the stencil kernels of a tile size
template <class R, int P, int NC>
struct Stencils {
    void (*grad)(MeshDev, const R*, R*, R*);
    void (*grad_sweep)(MeshDev, const R*, R*, R*);
    void (*udot)(MeshDev, const R*, R*, R*);
    void (*sweep_g)(MeshDev, const R*, const R*, R*);
    void (*sweep_u)(MeshDev, const R*, const R*, R*);
    dim3 grid_rhs, grid_grad, grid_udot, grid_g, grid_u, block;
    int ws_grad, ws_rhs, ws_udot, ws_sweep;
};
template <class R, int P, int NC, int SIZE>
Stencils<R, P, NC> stencils_of(const MeshDev& m) {
    using T = stage_tile_t<R, P, SIZE>;
    using H = stage_tile_t<R, P, SIZE, true>;
    // fields of a block: float launches over small tiles, which leave the GPU
    // partly idle, have a layer of the grid for each field (the udot sweep for
    // each udot_fields).  FP32-mixed Euler 60^2 Q3 with two sweeps: k_mass_sweep
    // 25 -> 10 us, the step 365 -> 199; with one sweep 208 -> 167.  In float64
    // the layers take the pipe from the sensor beside them (Euler 60^2 Q3 FP64
    // 0.8 of the speed with them).
    constexpr bool ONE = sizeof(R) == 4 && SIZE == 1;
    constexpr int FB = T::udot_fields(NC);
    const unsigned gx = nblk(m.nnx, T::NX), gy = nblk(m.nny, T::NY);
    Stencils<R, P, NC> s;
    s.grad = k_grad_rhs<R, P, NC, ONE ? 1 : NC, SIZE>;
    s.grad_sweep = nullptr;
    if constexpr (sizeof(R) == 4 || SIZE == 2) s.grad_sweep = k_grad_sweep<R, P, NC, ONE ? 1 : NC, SIZE>;
    s.udot = k_udot_sweep<R, P, NC, ONE ? FB : NC, SIZE>;
    s.sweep_g = k_mass_sweep<R, P, 2 * NC, ONE ? 1 : 2 * NC, SIZE>;
    s.sweep_u = k_mass_sweep<R, P, NC, ONE ? 1 : NC, SIZE>;
    s.grid_rhs = s.grid_u = dim3(gx, gy, ONE ? NC : 1);
    s.grid_grad = dim3(nblk(m.nnx, H::NX), nblk(m.nny, H::NY), ONE ? NC : 1);
    s.grid_udot = dim3(gx, gy, ONE ? NC / FB : 1);
    s.grid_g = dim3(gx, gy, ONE ? 2 * NC : 1);
    s.block = dim3(T::NT);
    s.ws_grad = (int)sizeof(R) * H::grad_ws;
    s.ws_rhs = (int)sizeof(R) * T::rhs_ws;
    s.ws_udot = (int)sizeof(R) * T::udot_ws(NC);
    s.ws_sweep = (int)sizeof(R) * T::sweep_ws;
    return s;
}

// Four streams, from the start of the stage: the main one carries the g_h
// solve, the residual, the udot solve, the element part of the update and the
// node gather; what needs only u runs beside it, the low-order part, dt and the
// facet part of the update (s2), the sensor (s3) and a scalar's Galerkin part
// of the residual (s4).  On small meshes a stage is as long as its longest
// chain of launches: KPP 256^2 Q2 FP32-mixed 125 us/step with the low-order
// part on the main stream and the rest on one other, 121 with four; advection
// 32^2 Q2 float64 186 and 168; KPP 256^2 Q2 LGL float64, whose streams fill the
// float64 pipe, 1296 and 1246.  On large meshes the order changes nothing.
// The streams are the state's own, and each is joined to the main stream
// before the last kernel of the stage.
template <class R, int P, class Ph>
cudaError_t run_stage(const Bufs& B, const MeshDev& m, const ProbDev& pr_in, double a, double b,
                      bool first, bool dt_only, cudaStream_t st, Prof* prof) {
    ProbDev pr = pr_in;
    if (dt_only) pr.mode = MODE_HO;  // no sensor needed for dt_e
    constexpr int NC = Ph::NC;
    constexpr bool F32 = sizeof(R) == 4;
    // element blocks: 64 threads on middle meshes, for an even spread over the
    // SMs (KPP 256^2: 6.7 blocks of 32 x 2 per SM); full blocks on tiny ones,
    // where the time is fetching instructions, once per SM (advection 32^2
    // float64: the step 6 % shorter with blocks of 128 than with 32)
    const int bex = m.E < (1 << 18) ? 32 : 64, bey = m.E < (1 << 14) ? 4 : 2;
    const dim3 be(bex, bey), bn(128, 1);
    const dim3 ge(nblk(m.nx, bex), nblk(m.ny, bey)), gn(nblk(m.nnx, 128), m.nny);
    const int size = tile_size<R, P>(m);
    Stencils<R, P, NC> S = size == 0 ? stencils_of<R, P, NC, 0>(m) : stencils_of<R, P, NC, 1>(m);
    if constexpr (!F32)
        if (size == 2) S = stencils_of<R, P, NC, 2>(m);
    // the element tiles of k_sens and k_lo: 32 by 8 in float, by 4 in float64
    // (24 modes of 340 elements are 65 KB there); lower ones on small meshes
    constexpr int STY = F32 ? 8 : 4, STS = F32 ? 4 : 1;
    const bool low = (long long)nblk(m.nx, K_TX) * nblk(m.ny, STY) < 304;
    const dim3 bs(K_TX, low ? STS : STY), gs(nblk(m.nx, K_TX), nblk(m.ny, low ? STS : STY));
    // the facet tiles of systems (k_lo_sys, k_facet_sys) and the rows of
    // k_res_sys and k_upd_sys
    const dim3 bf(F_TX, F_TY + 1), gf(nblk(m.nx, F_TX), nblk(m.ny, F_TY));
    const dim3 grs(nblk(m.nx, 32), m.ny), brs(32, NC);
    // per-launch timing records events between kernels: plain launches then
    const bool pdl = prof == nullptr;
    cudaError_t err = cudaSuccess;
    auto chk = [&](cudaError_t e) {
        if (e != cudaSuccess && err == cudaSuccess) err = e;
    };
    // the stage's own first error, and none left behind for the thread's next call
    auto done = [&] {
        if (err != cudaSuccess) cudaGetLastError();
        return err;
    };
    R* u = (R*)B.u;
    // the Q1 variant of eq. (aecQ1) needs neither g_h, nor the residual, nor udot
    const bool lo = pr.mode == MODE_LO, q1 = (pr.opts & OPT_AEC_Q1) != 0 && !lo;
    // per-launch timing serialises the stage on one stream, so that each
    // kernel's events bracket its own run and no overlap with the other streams
    const cudaStream_t s2 = prof || dt_only || q1 ? st : B.st2, s3 = prof ? st : B.st3, s4 = prof ? st : B.st4;
    auto fork = [&](cudaStream_t s) {
        if (s != st) chk(cudaStreamWaitEvent(s, B.ev_fork0, 0));
    };
    auto join = [&](cudaEvent_t e, cudaStream_t s) {
        if (s != st) {
            chk(cudaEventRecord(e, s));
            chk(cudaStreamWaitEvent(st, e, 0));
        }
    };
    chk(cudaEventRecord(B.ev_fork0, st));
    fork(s2);
    if (!dt_only) {
        fork(s3);
        auto* ksens = low ? k_sens<R, P, Ph, STS> : k_sens<R, P, Ph, STY>;
        if constexpr (NC == 1) {
            if (!q1 && !lo) {
                fork(s4);
                CGL_LAUNCH(prof, KID_RESW, s4,
                           chk(launch(false, k_res_w<R, P, Ph>, ge, be, s4, m, pr, (const R*)u, (R*)B.EW)));
            }
        }
        CGL_LAUNCH(prof, KID_SENS, s3, chk(launch(false, ksens, gs, bs, s3, m, pr, (const R*)u, B.gam, B.nu)));
    }
    const bool pdl2 = pdl && s2 == st;
    if constexpr (NC > 1) {
        CGL_LAUNCH(prof, KID_AVG, s2, chk(launch(pdl2, k_avg<R, P, Ph>, ge, be, s2, m, pr, (const R*)u, B.avg, B.ue, (R*)B.cq)));
        auto* klo = (pr.opts & OPT_SUBCELL_DT) ? k_lo_sys<R, P, Ph, true> : k_lo_sys<R, P, Ph, false>;
        CGL_LAUNCH(prof, KID_PRE, s2,
                   chk(launch(pdl, klo, gf, bf, s2, m, pr, (const R*)u, B.ue, B.dte, B.ubl, (R*)B.fl, B.cf,
                              (const float*)B.avg, (const R*)B.cq, first ? B.dtbits : nullptr)));
    } else {
        const bool sub = (pr.opts & OPT_SUBCELL_DT) != 0;
        auto* klo = low ? (sub ? k_lo<R, P, Ph, STS, true> : k_lo<R, P, Ph, STS, false>)
                        : (sub ? k_lo<R, P, Ph, STY, true> : k_lo<R, P, Ph, STY, false>);
        CGL_LAUNCH(prof, KID_PRE, s2,
                   chk(launch(pdl2, klo, gs, bs, s2, m, pr, (const R*)u, B.ue, B.dte, B.ubl, (R*)B.q, (R*)B.fl, B.cf, B.avg,
                              first ? B.dtbits : nullptr)));
    }
    if (first)
        CGL_LAUNCH(prof, KID_DT, s2,
                   chk(launch(pdl, k_dt_final, dim3(1), dim3(1), s2, B.dtbits, pr.cfl, (const double*)B.t,
                              (const double*)B.t_end, B.dt)));
    if (dt_only) return done();
    if (q1) {
        CGL_LAUNCH(prof, KID_Q1F, st,
                   chk(launch(pdl, k_q1_facet<R, P, Ph>, ge, be, st, m, pr, (const R*)u, (const double*)B.ue,
                              (const double*)B.dte, (const double*)B.ubl, (const R*)B.q, (const R*)B.fl,
                              (const float*)B.cf, (R*)B.ER, B.ube, B.cnt)));
        CGL_LAUNCH(prof, KID_UDL, st,
                   chk(launch(pdl, k_udl<R, P, NC>, gn, bn, st, m, (const R*)u, (const double*)B.ube,
                              (const double*)B.dte, (R*)B.ud)));
        join(B.ev_s, s3);  // gamma_e scales the contributions
        CGL_LAUNCH(prof, KID_UPDATE, st,
                   chk(launch(pdl, k_q1_update<R, P, Ph>, ge, be, st, m, pr, (const R*)u, (const R*)B.ud,
                              (const double*)B.ue, (const double*)B.dte, (const R*)B.ER, (const float*)B.cf,
                              (const float*)B.avg, (const double*)B.ube, (const double*)B.gam,
                              (const double*)B.dt, (R*)B.EW, B.beta, B.cnt)));
        CGL_LAUNCH(prof, KID_FINAL, st,
                   chk(launch(pdl, k_final<R, P, NC>, gn, bn, st, m, pr, (const R*)B.EW, (R*)B.un, u, R(a), R(b),
                              B.cnt, pr.last_stage ? B.t : (double*)nullptr, (const double*)B.dt)));
        return done();
    }
    // the facet part of the update
    if constexpr (NC > 1)
        CGL_LAUNCH(prof, KID_FACET, s2,
                   chk(launch(pdl, k_facet_sys<R, P, Ph>, gf, bf, s2, m, pr, (const R*)u, (const double*)B.ue,
                              B.dte, (const double*)B.ubl, (const R*)B.fl, B.cf, B.ube, (R*)B.fht, B.cnt)));
    else
        CGL_LAUNCH(prof, KID_FACET, s2,
                   chk(launch(pdl, k_facet<R, P, Ph>, ge, be, s2, m, pr, (const R*)u, (const double*)B.ue, B.dte,
                              (const double*)B.ubl, (const R*)B.q, (const R*)B.fl, B.cf, B.ube, (R*)B.fht, B.cnt)));
    R* ud = (R*)B.ud;
    if (!lo) {
        // g_h: right-hand side, lumped iterate and k_g sweeps (ping-pong), the
        // first sweep fused with the right-hand side where fuse_grad_sweep says
        R* g = (R*)B.g;
        R* g2 = (R*)B.g2;
        R* bg = (R*)B.bg;
        const bool fuse = !(pr.opts & OPT_UNFUSED_SWEEPS), fuse_g = fuse && fuse_grad_sweep(sizeof(R), size);
        int k0 = 0;
        if (fuse_g && pr.k_g >= 1) {
            CGL_LAUNCH(prof, KID_GRADF, st,
                       chk(launch_shared(pdl, S.grad_sweep, S.grid_grad, S.block, S.ws_grad, st, m, (const R*)u,
                                         pr.k_g > 1 ? bg : (R*)nullptr, g2)));
            std::swap(g, g2);
            k0 = 1;
        } else {
            CGL_LAUNCH(prof, KID_GRAD, st,
                       chk(launch_shared(pdl, S.grad, S.grid_rhs, S.block, S.ws_rhs, st, m, (const R*)u, bg, g)));
        }
        for (int k = k0; k < pr.k_g; ++k) {
            CGL_LAUNCH(prof, KID_SWEEP, st,
                       chk(launch_shared(pdl, S.sweep_g, S.grid_g, S.block, S.ws_sweep, st, m, (const R*)g, (const R*)bg, g2)));
            std::swap(g, g2);
        }
        R* ER = (R*)B.ER;
        R* r = (R*)B.r;
        R* ud2 = (R*)B.ud2;
        join(B.ev_s, s3);  // gamma_e and nu_e
        if (NC == 1) join(B.ev_w, s4);  // the Galerkin part
        if constexpr (NC > 1)
            CGL_LAUNCH(prof, KID_RES, st,
                       chk(launch_shared(pdl, k_res_sys<R, P, Ph>, grs, brs, (int)sizeof(R) * ResSys<R, P, NC>::ws, st, m,
                                         pr, (const R*)u, (const R*)g, (const double*)B.gam, (const double*)B.nu, ER)));
        else
            CGL_LAUNCH(prof, KID_RES, st,
                       chk(launch(pdl, k_res_s<R, P>, ge, be, st, m, (const R*)u, (const R*)g, (const double*)B.gam,
                                  (const double*)B.nu, (const R*)B.EW, ER)));
        int k1 = 0;
        if (fuse && pr.k_u >= 1) {
            CGL_LAUNCH(prof, KID_UDOTF, st,
                       chk(launch_shared(pdl, S.udot, S.grid_udot, S.block, S.ws_udot, st, m, (const R*)ER, r, ud2)));
            std::swap(ud, ud2);
            k1 = 1;
        } else {
            CGL_LAUNCH(prof, KID_GATHER, st,
                       chk(launch(pdl, k_gather_init<R, P, NC>, gn, bn, st, m, (const R*)ER, r, ud)));
        }
        for (int k = k1; k < pr.k_u; ++k) {
            CGL_LAUNCH(prof, KID_SWEEP, st,
                       chk(launch_shared(pdl, S.sweep_u, S.grid_u, S.block, S.ws_sweep, st, m, (const R*)ud, (const R*)r, ud2)));
            std::swap(ud, ud2);
        }
    }
    if (lo) join(B.ev_s, s3);
    join(B.ev_join, s2);
    if constexpr (NC > 1)
        CGL_LAUNCH(prof, KID_UPDATE, st,
                   chk(launch(pdl, k_upd_sys<R, P, Ph>, grs, brs, st, m, pr, (const R*)u, (const R*)ud,
                              (const double*)B.ue, (const double*)B.dte, (const R*)B.ER, (const float*)B.cf,
                              (const float*)B.avg, (const double*)B.ube, (const R*)B.fht, (const double*)B.dt,
                              (R*)B.EW, B.beta, B.cnt)));
    else
        CGL_LAUNCH(prof, KID_UPDATE, st,
                   chk(launch(pdl, k_update_el<R, P, Ph>, ge, be, st, m, pr, (const R*)u, (const R*)ud,
                              (const double*)B.ue, (const double*)B.dte, (const R*)B.ER, (const float*)B.cf,
                              (const float*)B.avg, (const double*)B.ube, (const R*)B.fht, (const double*)B.dt,
                              (R*)B.EW, B.beta, B.cnt)));
    CGL_LAUNCH(prof, KID_FINAL, st,
               chk(launch(pdl, k_final<R, P, NC>, gn, bn, st, m, pr, (const R*)B.EW, (R*)B.un, u, R(a), R(b),
                          B.cnt, pr.last_stage ? B.t : (double*)nullptr, (const double*)B.dt)));
    return done();
}

// stage of one precision R (float64: the FP64 form; float: FP32-mixed) for
// degrees 1..4; each physics compiles its two precisions in separate
// translation units (inst_*.cu, inst_*_f32.cu), built in parallel
template <class Ph, class R>
StageFn select_stage_r(int p) {
    switch (p) {
        case 1: return run_stage<R, 1, Ph>;
        case 2: return run_stage<R, 2, Ph>;
        case 3: return run_stage<R, 3, Ph>;
        case 4: return run_stage<R, 4, Ph>;
    }
    return nullptr;
}

// copy the host tables into this translation unit's constant memory
// (td: NTABD float64 tables, a2d: 2 A2_TOTAL values, both bases)
static inline cudaError_t upload_tables_here(const Tab<double>* td, const Tab<float>* tf,
                                             const double* a2d, const float* a2f) {
    cudaError_t e = cudaMemcpyToSymbol(c_tabd, td, sizeof(Tab<double>) * NTABD);
    if (e == cudaSuccess) e = cudaMemcpyToSymbol(c_tabf, tf, sizeof(Tab<float>) * (PMAX + 1));
    if (e == cudaSuccess) e = cudaMemcpyToSymbol(c_A2d, a2d, sizeof(double) * 2 * A2_TOTAL);
    if (e == cudaSuccess) e = cudaMemcpyToSymbol(c_A2f, a2f, sizeof(float) * A2_TOTAL);
    return e;
}

typedef cudaError_t (*UploadFn)(const Tab<double>*, const Tab<float>*, const double*, const float*);

StageFn stage_fn_adv(int prec, int p);
StageFn stage_fn_burgers(int prec, int p);
StageFn stage_fn_kpp(int prec, int p);
StageFn stage_fn_euler(int prec, int p);
StageFn stage_fn_adv32(int p);
StageFn stage_fn_burgers32(int p);
StageFn stage_fn_kpp32(int p);
StageFn stage_fn_euler32(int p);
cudaError_t upload_adv(const Tab<double>*, const Tab<float>*, const double*, const float*);
cudaError_t upload_burgers(const Tab<double>*, const Tab<float>*, const double*, const float*);
cudaError_t upload_kpp(const Tab<double>*, const Tab<float>*, const double*, const float*);
cudaError_t upload_euler(const Tab<double>*, const Tab<float>*, const double*, const float*);
cudaError_t upload_adv32(const Tab<double>*, const Tab<float>*, const double*, const float*);
cudaError_t upload_burgers32(const Tab<double>*, const Tab<float>*, const double*, const float*);
cudaError_t upload_kpp32(const Tab<double>*, const Tab<float>*, const double*, const float*);
cudaError_t upload_euler32(const Tab<double>*, const Tab<float>*, const double*, const float*);
cudaError_t upload_batch(const Tab<double>*, const Tab<float>*, const double*, const float*);

}  // namespace cgl
