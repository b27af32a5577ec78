// kernels.cuh — CUDA kernels of one SSP-RK stage of the element-based
// convex-limited CG-WENO scheme (Kuzmin, Hajduk, Vedral, arXiv 2509.04673),
// following the order of the algorithm summary in Sec. 4.3:
//
//   k_lo           scalars: cell averages u^e (eq. (ueold)), facet speeds,
//                  dt_e (eq. (dtmaxcell)), f^L, ubar^{e,L} (eq. (uelowFCT)),
//                  block minimum of dt_e; systems: k_avg (averages, their
//                  fluxes and speed parts), then k_lo_sys
//   k_dt_final     global dt = omega_CFL min_e dt_e (eq. (cflglob), Sec. 5)
//   k_sens         WENO sensor gamma_e (eqs. (WENO:alpha), (WENO:norm)), nu_e
//                  (eq. (stab:WENO))
//   k_grad_rhs     right-hand side of the g_h projection, int phi_i grad u_h,
//                  as a tiled separable stencil, and its lumped iterate
//   k_mass_sweep   lumped-preconditioned Richardson sweep with M_C applied
//                  as a tiled separable stencil; k_grad_sweep and
//                  k_udot_sweep carry the first one (fused.cuh)
//   k_res_w, k_res_s (scalars), k_res_sys (systems)
//                  element residual: Galerkin part of eq. (weak:stab2) with
//                  boundary terms (eqs. (aec), (aecb)) and s_h (eq. (stab:WENO))
//   k_gather_init  node-centric sum over E_i of the element residuals in a
//                  fixed order (deterministic), and its lumped iterate
//   k_facet (scalars), k_facet_sys (systems)
//                  facet fluxes f^H (eq. (hoflux)), flux limiter (eq. (fAlim),
//                  Appendix A), ubar^e (eq. (uelim))
//   k_update_el (scalars), k_upd_sys (systems)
//                  f_i^e (eq. (aec)), beta_e (eqs. (slimit1), (slimit2),
//                  Appendix A), element contributions of eq. (eq:SSPupdate)
//   k_final        node gather, SSP-RK combination, invariant-domain check;
//                  on the last stage of a step also t += dt
//
// One thread per element or node; per element and component in k_res_sys and
// k_upd_sys; the facets of systems once per facet; the stencils by segments
// of p nodes.
// Kernels are templated on the bulk precision R (double, or float in the
// mixed form), the degree P and the physics policy Ph. Cell averages, dt_e,
// the facet flux limiter, limiter bound gaps and positivity factors are
// float64 in both forms.
//
// Element vectors (ER, EW and the no-allocation scratch) are stored
// component-major, [local node i][field v][element e]: a warp of consecutive
// elements writes, and a warp of consecutive nodes reads, contiguous runs.
#pragma once

#include "modal.cuh"

namespace cgl {

// element-vector layout: value v of local node i of element e, NV values
DEV long long ev_at(long long E, int e, int i, int v, int NV) { return (long long)(i * NV + v) * E + e; }

// Value k of element e in an array of several values per element, [k][e].  A
// scalar state takes 192 bytes per element and more, so that three values of
// every element that fits one GPU can exceed 2^32; a system 592, so that eight
// cannot exceed 2^32 nor four 2^31 (those are indexed in 32 bits in place).
// 64-bit offsets throughout cost 2 % per step (Euler blast 2048^2 Q2 10.27 ->
// 10.49 ms).
template <int NC>
DEV auto off(int E, int k, int e) {
    if constexpr (NC == 1) return (long long)k * E + e;
    else return (unsigned)k * (unsigned)E + (unsigned)e;
}
// the values k of an array of more than eight
template <class T>
DEV T* field(T* p, int E, int k) { return p + (long long)k * E; }


// Programmatic dependent launch: every kernel of a stage first lets the next
// kernel of the stream be scheduled (it launches once all blocks of this one
// are resident) and then waits until the previous kernel has completed and
// its writes are visible.  Each kernel calls this first, in every thread,
// before any global memory access; for a kernel launched without the
// programmatic-serialisation attribute both instructions do nothing.
DEV void pdl_begin() {
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    asm volatile("griddepcontrol.wait;" ::: "memory");
}

// the batched kernels, whose phases run on one stream: the next is scheduled
// only once this one's predecessor has completed
DEV void pdl_wait_then_trigger() {
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}


template <int P>
struct Dim {
    static constexpr int N1 = P + 1, N2 = N1 * N1, NQ = P + 2;
};

// device counters: invariant-domain violations, rounding clamps, theta > 1,
// non-finite values, unlimited averages ubar^e outside G (flux limiter off),
// pseudo time steps reduced by the remark after eq. (dtmaxcell)
// (slot CNT_IMPORT: non-finite values of the last host copy into the state;
// CNT_REFUSED: pipelined host copies refused for a non-finite value since the
// last cgl_sync)
enum { CNT_VIOL = 0, CNT_CLAMP = 1, CNT_CFL = 2, CNT_NONFINITE = 3, CNT_UBAR = 4, CNT_DTE_RED = 5, CNT_IMPORT = 6,
       CNT_REFUSED = 7, CNT_N = 8 };

// global node of local (a, b) in element (ex, ey); periodic wrap at the far side
DEV long long node_of(const MeshDev& m, int ex, int ey, int a, int b) {
    int gx = ex * m.p + a, gy = ey * m.p + b;
    if (m.px && gx == m.nnx) gx = 0;
    if (m.py && gy == m.nny) gy = 0;
    return (long long)gy * m.nnx + gx;
}

// the coefficients of element (ex, ey) of one nodal field: one pointer per
// row, constant offsets along it, and the last column and row, the only ones
// that can wrap (in a periodic direction), at offsets of their own
template <class R, int P>
DEV void load_comp(const R* __restrict__ u, const MeshDev& m, int ex, int ey, R (&V)[(P + 1) * (P + 1)]) {
    constexpr int N1 = P + 1;
    const R* __restrict__ r0 = u + ((long long)(ey * P) * m.nnx + ex * P);
    const int dx = (m.px && ex == m.nx - 1) ? -ex * P : P;
    const int ry = (m.py && ey == m.ny - 1) ? -ey * P : P;
#pragma unroll
    for (int b = 0; b < N1; ++b) {
        const R* __restrict__ r = r0 + (long long)(b < P ? b : ry) * m.nnx;
#pragma unroll
        for (int a = 0; a < N1; ++a) V[b * N1 + a] = r[a < P ? a : dx];
    }
}

// face neighbour (0 W, 1 E, 2 S, 3 N) or -1 on a non-periodic boundary
DEV int neighbour(const MeshDev& m, int ex, int ey, int dir) {
    int jx = ex, jy = ey;
    if (dir == 0) jx = ex - 1;
    else if (dir == 1) jx = ex + 1;
    else if (dir == 2) jy = ey - 1;
    else jy = ey + 1;
    if (jx < 0 || jx >= m.nx) {
        if (!m.px) return -1;
        jx = (jx + m.nx) % m.nx;
    }
    if (jy < 0 || jy >= m.ny) {
        if (!m.py) return -1;
        jy = (jy + m.ny) % m.ny;
    }
    return jy * m.nx + jx;
}

// coordinates (jx, jy) of the face neighbour of element (ex, ey) in
// direction dir (0 W, 1 E, 2 S, 3 N), wrapped on periodic directions; only
// meaningful where neighbour() is >= 0 (no integer division)
DEV void neighbour_xy(const MeshDev& m, int ex, int ey, int dir, int& jx, int& jy) {
    jx = ex + (dir == 0 ? -1 : dir == 1 ? 1 : 0);
    jy = ey + (dir == 2 ? -1 : dir == 3 ? 1 : 0);
    jx = jx < 0 ? jx + m.nx : (jx >= m.nx ? jx - m.nx : jx);
    jy = jy < 0 ? jy + m.ny : (jy >= m.ny ? jy - m.ny : jy);
}

// ---------------------------------------------------------------------------
// boundary data u_hat on the sides d = 0..3 (W, E, S, N), Sec. 2.  The
// positions and the split are evaluated in float64 with explicit rounding
// (no contraction), so that a point that lies exactly on a split (a node at
// x = 1/6 on a mesh of width 1/192) takes the same side as the plain
// evaluation s0 + s1 (t + c dt) and x0 + k hn.
// ---------------------------------------------------------------------------
DEV bool side_plain(const ProbDev& pr, int d) { return (pr.plain_mask >> d) & 1; }
DEV bool side_split(const ProbDev& pr, int d) { return (pr.split_mask >> d) & 1; }

// slot (0 below the split, 1 at or above it) of a point at coordinate pos
// of a side with two parts
DEV int side_slot(const ProbDev& pr, int d, double pos) {
    const SideDev& sd = pr.side[d];
    double sp = sd.s0;
    if (sd.s1 != 0.0) {
        double ts = *pr.t_dev;
        if (pr.tc != 0.0) ts = __dadd_rn(ts, __dmul_rn(pr.tc, *pr.dt_dev));
        sp = __dadd_rn(sd.s0, __dmul_rn(sd.s1, ts));
    }
    return pos < sp ? 0 : 1;
}

// coordinate along side d of node k (0..p) of the face of element (ex, ey):
// x0 + g h/p (Bernstein), x_e + xn_k h (LGL)
DEV double side_node_pos(const MeshDev& m, int d, int ex, int ey, int k) {
    const int c = (d < 2) ? ey : ex;
    if (m.basis) {
        const double xk = c_tabd[PMAX + 1 + m.p].xn[k];
        return __dadd_rn(__dadd_rn((d < 2) ? m.y0 : m.x0, __dmul_rn((double)c, m.h)), __dmul_rn(xk, m.h));
    }
    const int g = c * m.p + k;
    return __dadd_rn((d < 2) ? m.y0 : m.x0, __dmul_rn((double)g, m.hn));
}

// coordinate along side d of the midpoint of the face of element (ex, ey)
DEV double side_mid_pos(const MeshDev& m, int d, int ex, int ey) {
    const int c = (d < 2) ? ey : ex;
    return __dadd_rn((d < 2) ? m.y0 : m.x0, __dmul_rn((double)c + 0.5, m.h));
}

// coordinate along side d of the Gauss point x_q (on [0,1]) of that face
DEV double side_quad_pos(const MeshDev& m, int d, int ex, int ey, double xq) {
    const int c = (d < 2) ? ey : ex;
    return __dadd_rn(__dadd_rn((d < 2) ? m.y0 : m.x0, __dmul_rn((double)c, m.h)), __dmul_rn(xq, m.h));
}

// u_hat from the interior state u: FIXED -> the side's state, OUTFLOW -> u,
// WALL -> u with the normal momentum reversed, m - 2 (m.n) n (Euler; the
// normals of the sides are +-x and +-y)
template <class T, int NC>
DEV void ext_state(const ProbDev& pr, int d, int slot, const T* u, T* uh) {
    const SideDev& sd = pr.side[d];
    const int kind = sd.kind[slot];
#pragma unroll
    for (int c = 0; c < NC; ++c) uh[c] = (kind == BC_FIXED) ? PV<T>::side_state(sd, slot, c) : u[c];
    if constexpr (NC == 4) {
        if (kind == BC_WALL) {
            if (d < 2) uh[1] = -u[1];
            else uh[2] = -u[2];
        }
    }
}

// 2D launches: elements as (x: ex, y: ey), nodes as (x: gx, y: gy); no
// integer division by runtime sizes in the kernels
DEV bool elem_of_thread(const MeshDev& m, int& ex, int& ey, int& e) {
    ex = blockIdx.x * blockDim.x + threadIdx.x;
    ey = blockIdx.y * blockDim.y + threadIdx.y;
    e = ey * m.nx + ex;
    return ex < m.nx && ey < m.ny;
}

DEV bool node_of_thread(const MeshDev& m, int& gx, int& gy, long long& node) {
    gx = blockIdx.x * blockDim.x + threadIdx.x;
    gy = blockIdx.y * blockDim.y + threadIdx.y;
    node = (long long)gy * m.nnx + gx;
    return gx < m.nnx && gy < m.nny;
}

template <class R, int P, int NC>
DEV void load_block(const R* __restrict__ u, const MeshDev& m, int ex, int ey,
                    R (&U)[NC][Dim<P>::N2]) {
#pragma unroll
    for (int c = 0; c < NC; ++c) load_comp<R, P>(u + c * m.NN, m, ex, ey, U[c]);
}

// element mean of the coefficients as float64: plain sum for double data;
// for float data a compensated (Neumaier) float sum widened once, accurate
// to ~1e-14 relative without per-node float64 arithmetic
template <int N>
DEV double block_mean(const double (&v)[N]) {
    double s = 0.0;
#pragma unroll
    for (int i = 0; i < N; ++i) s += v[i];
    return s * (1.0 / N);
}
template <int N>
DEV double block_mean(const float (&v)[N]) {
    float s = 0.f, c = 0.f;
#pragma unroll
    for (int i = 0; i < N; ++i) {
        float t = s + v[i];
        c += (fabsf(s) >= fabsf(v[i])) ? ((s - t) + v[i]) : ((v[i] - t) + s);
        s = t;
    }
    return ((double)s + (double)c) * (1.0 / N);
}

// u^e of eq. (ueold), (1/|K_e|) sum_i m_i^e u_i: the mean of the Bernstein
// coefficients, or on an LGL mesh (float64 form) the nodal values weighted
// by w_a w_b
template <class R, int P>
DEV double cell_mean(const MeshDev& m, const R (&v)[Dim<P>::N2]) {
    if constexpr (sizeof(R) == 8) {
        if (m.basis) {
            constexpr int N1 = P + 1;
            const Tab<double>& T = c_tabd[PMAX + 1 + P];
            double s = 0.0;
#pragma unroll
            for (int b = 0; b < N1; ++b) {
                double r = 0.0;
#pragma unroll
                for (int a = 0; a < N1; ++a) r += T.wl[a] * v[b * N1 + a];
                s += T.wl[b] * r;
            }
            return s;
        }
    }
    return block_mean<Dim<P>::N2>(v);
}

// b^e_i = (int phi_i d_x u_h, int phi_i d_y u_h), sum-factorised, into EV
// at ev_at(E, e, i, v, 2NC), v = dim*NC + c
template <class R, int P, int NC>
DEV void grad_vectors(const MeshDev& m, const R (&U)[NC][Dim<P>::N2], R h, long long E, int e,
                      R* __restrict__ EV) {
    constexpr int N1 = P + 1, N2 = Dim<P>::N2, NV = 2 * NC;
    const Tab<R>& T = tab_of<R>(m, P);
#pragma unroll
    for (int c = 0; c < NC; ++c) {
        R Y[N1][N1], Z[N1][N1];
#pragma unroll
        for (int d = 0; d < N1; ++d)
#pragma unroll
            for (int a = 0; a < N1; ++a) {
                R sx = R(0), sy = R(0);
#pragma unroll
                for (int k = 0; k < N1; ++k) {
                    sx += T.C[k][a] * U[c][d * N1 + k];
                    sy += T.M[a][k] * U[c][d * N1 + k];
                }
                Y[d][a] = sx;
                Z[d][a] = sy;
            }
#pragma unroll
        for (int b = 0; b < N1; ++b)
#pragma unroll
            for (int a = 0; a < N1; ++a) {
                R sx = R(0), sy = R(0);
#pragma unroll
                for (int d = 0; d < N1; ++d) {
                    sx += T.M[b][d] * Y[d][a];
                    sy += T.C[d][b] * Z[d][a];
                }
                EV[ev_at(E, e, b * N1 + a, c, NV)] = h * sx;
                EV[ev_at(E, e, b * N1 + a, NC + c, NV)] = h * sy;
            }
    }
}

// ---------------------------------------------------------------------------
// low-order facet quantities of element e on its four faces in the canonical
// orientation (normal +x for W/E, +y for S/N): lambda and F^L = F(u^L, u^R)
// with f^L of Sec. 4; on a non-periodic boundary the external state is
// u_hat (FIXED) or u^e itself (OUTFLOW) and the cell's outward normal is used.
// ---------------------------------------------------------------------------
// upper bound of the facet speed, evaluated in precision RS: float64, or in
// float with a 2^-20 relative inflation so that it stays an upper bound
template <class Ph, class RS>
DEV double facet_speed(const double* uL, const double* uR, double nx, double ny, const ProbDev& pr) {
    if (sizeof(RS) == 8) return Ph::template max_speed<double>(uL, uR, nx, ny, pr);
    float fL[Ph::NC], fR[Ph::NC];
#pragma unroll
    for (int c = 0; c < Ph::NC; ++c) {
        fL[c] = (float)uL[c];
        fR[c] = (float)uR[c];
    }
    float l = Ph::template max_speed<float>(fL, fR, (float)nx, (float)ny, pr);
    return (double)l * (1.0 + 0x1p-20);
}

template <class Ph, class R>
DEV void lo_facets(const MeshDev& m, const ProbDev& pr, const int (&nb)[4], int ex, int ey,
                   const double (&us)[Ph::NC], const double (&fxs)[Ph::NC], const double (&fys)[Ph::NC],
                   const double (&uo)[4][Ph::NC], const double (&fxo)[4][Ph::NC],
                   const double (&fyo)[4][Ph::NC], double (&lam)[4], double (&FL)[4][Ph::NC]) {
    constexpr int NC = Ph::NC;
#pragma unroll
    for (int d = 0; d < 4; ++d) {
        const double cnx = (d < 2) ? 1.0 : 0.0, cny = (d < 2) ? 0.0 : 1.0;
        const bool self_is_L = (d == 1 || d == 3);
        if (nb[d] >= 0) {
            const double* uL = self_is_L ? us : uo[d];
            const double* uR = self_is_L ? uo[d] : us;
            const double* fxL = self_is_L ? fxs : fxo[d];
            const double* fyL = self_is_L ? fys : fyo[d];
            const double* fxR = self_is_L ? fxo[d] : fxs;
            const double* fyR = self_is_L ? fyo[d] : fys;
            double l = facet_speed<Ph, R>(uL, uR, cnx, cny, pr);
            lam[d] = l;
#pragma unroll
            for (int c = 0; c < NC; ++c) {
                double nL = fxL[c] * cnx + fyL[c] * cny;
                double nR = fxR[c] * cnx + fyR[c] * cny;
                FL[d][c] = 0.5 * (nL + nR) - 0.5 * l * (uR[c] - uL[c]);
            }
        } else {
            // external state u_hat at the facet midpoint from the cell average
            const int slot = side_split(pr, d) ? side_slot(pr, d, side_mid_pos(m, d, ex, ey)) : 0;
            const int kind = pr.side[d].kind[slot];
            double ux[NC];
            ext_state<double, NC>(pr, d, slot, us, ux);
            const double sg = self_is_L ? 1.0 : -1.0;
            // f(u_hat) (FIXED, WALL) or the cell's own f(u^e) (OUTFLOW)
            double fxx[NC], fyx[NC];
            if (kind != BC_OUTFLOW) {
                R ubR[NC], fxR[NC], fyR[NC];
#pragma unroll
                for (int c = 0; c < NC; ++c) ubR[c] = R(ux[c]);
                Ph::template flux<R>(ubR, fxR, fyR, pr);
#pragma unroll
                for (int c = 0; c < NC; ++c) {
                    fxx[c] = (double)fxR[c];
                    fyx[c] = (double)fyR[c];
                }
            } else {
#pragma unroll
                for (int c = 0; c < NC; ++c) {
                    fxx[c] = fxs[c];
                    fyx[c] = fys[c];
                }
            }
            const double nx = sg * cnx, ny = sg * cny;
            double l = facet_speed<Ph, R>(us, ux, nx, ny, pr);
            lam[d] = l;
#pragma unroll
            for (int c = 0; c < NC; ++c) {
                double nL = fxs[c] * nx + fys[c] * ny;
                double nR = fxx[c] * nx + fyx[c] * ny;
                double F = 0.5 * (nL + nR) - 0.5 * l * (ux[c] - us[c]);
                FL[d][c] = sg * F;
            }
        }
    }
}

// the float64 Appendix-A factor where the float32 certificate could not show
// alpha = 1 (rare): out of line in the facet and slope limiters of systems, so
// that their loops carry a call instead of a copy of the float64 formula.  Only
// the eq. (aecQ1) variant has it inline: k_q1_facet behind the certificate,
// k_q1_update in float64, where it runs without one
static __device__ __noinline__ double euler_alpha_rare(const double* ub, const double* f, double m, double eps) {
    return euler_alpha<double>(ub, f, m, eps);
}
template <class R>
DEV double euler_alpha_of(const double* ub, const double* f, double m, double eps) {
    if constexpr (sizeof(R) == 4) return euler_alpha_rare(ub, f, m, eps);
    else return euler_alpha<double>(ub, f, m, eps);
}

// gamma_e of one component whose field is u (modal.cuh) from the element's own
// block, the neighbours' blocks loaded and transformed by this thread
template <class R, int P>
DEV R sensor_scalar(const MeshDev& m, const ProbDev& pr, const R* __restrict__ u, const R (&U)[Dim<P>::N2],
                    const int (&nb)[4], int ex, int ey) {
    constexpr int N2 = Dim<P>::N2;
    const Tab<R>& T = tab_of<R>(m, P);
    R own[N2];
    modal_block<R, P>(T, U, own);
    return modal_sensor<R, P, true>(T, a2_base<R>(m), pr, own, nb, [&](int d, R(&l)[N2]) {
        int jx, jy;
        neighbour_xy(m, ex, ey, d, jx, jy);
        R V[N2];
        load_comp<R, P>(u, m, jx, jy, V);
        modal_block<R, P>(T, V, l);
    });
}

// float-float mean of N floats: compensated (Neumaier) sum, then a division
// by N whose remainder is taken exactly with an FMA; hi + lo carries about
// 1e-14 relative accuracy without float64 arithmetic
// (explicit round-to-nearest intrinsics throughout: the compiler never
// contracts or reorders them, so every kernel that inlines these helpers
// computes the same bits)
template <int N>
DEV void ff_mean(const float (&v)[N], float& hi, float& lo) {
    float s = 0.f, c = 0.f;
#pragma unroll
    for (int i = 0; i < N; ++i) {
        const float t = __fadd_rn(s, v[i]);
        const float e = (fabsf(s) >= fabsf(v[i])) ? __fadd_rn(__fsub_rn(s, t), v[i])
                                                   : __fadd_rn(__fsub_rn(v[i], t), s);
        c = __fadd_rn(c, e);
        s = t;
    }
    const float h = __fadd_rn(s, c);
    const float l = __fsub_rn(c, __fsub_rn(h, s));
    const float k = 1.0f / N;
    const float q = __fmul_rn(h, k);
    const float r = __fmaf_rn(-q, (float)N, h);
    hi = q;
    lo = __fmul_rn(__fadd_rn(r, l), k);
}

// (ah + al) - (bh + bl) rounded to float (TwoSum on the high parts)
DEV float ff_diff(float ah, float al, float bh, float bl) {
    const float s = __fsub_rn(ah, bh);
    const float bb = __fsub_rn(s, ah);
    const float err = __fadd_rn(__fsub_rn(ah, __fsub_rn(s, bb)), __fsub_rn(-bh, bb));
    return __fadd_rn(s, __fadd_rn(err, __fsub_rn(al, bl)));
}

// error-free sum a + b = s + t (Knuth's TwoSum)
DEV void two_sum(float a, float b, float& s, float& t) {
    s = __fadd_rn(a, b);
    const float bb = __fsub_rn(s, a);
    t = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
}

// ((a - b) + c) - d as a float-float pair hi + lo (relative error ~2^-44)
DEV void ff_sum4(float a, float b, float c, float d, float& hi, float& lo) {
    float s1, t1, s2, t2, s3, t3;
    two_sum(a, -b, s1, t1);
    two_sum(s1, c, s2, t2);
    two_sum(s2, -d, s3, t3);
    hi = s3;
    lo = __fadd_rn(__fadd_rn(t1, t2), t3);
}

// sum of N floats as a float-float pair hi + lo: Knuth's TwoSum into a
// running sum with the rounding errors collected separately (relative error
// of hi + lo about N^2 2^-48 of the sum of magnitudes)
template <int N>
DEV void ff_sum(const float (&v)[N], float& hi, float& lo) {
    float s = 0.f, c = 0.f;
#pragma unroll
    for (int i = 0; i < N; ++i) {
        float t, e;
        two_sum(s, v[i], t, e);
        c = __fadd_rn(c, e);
        s = t;
    }
    two_sum(s, c, hi, lo);
}

// LLF flux value 0.5 (nL + nR) - 0.5 lambda jump, with a fixed evaluation order
DEV float llf_value(float nL, float nR, float lam, float jump) {
    return __fmaf_rn(__fmul_rn(-0.5f, lam), jump, __fmul_rn(0.5f, __fadd_rn(nL, nR)));
}

// the NC values of facet i of an array [4E][NC] of facet values (the four
// components of a system in 16-byte accesses: one by one they are stores of 4
// bytes at a stride of 64)
template <class R, int NC>
DEV void store_facet(R* __restrict__ f, long long i, const R (&v)[NC]) {
    if constexpr (NC == 4 && sizeof(R) == 4) {
        reinterpret_cast<float4*>(f)[i] = make_float4(v[0], v[1], v[2], v[3]);
    } else if constexpr (NC == 4) {
        reinterpret_cast<double2*>(f)[2 * i] = make_double2(v[0], v[1]);
        reinterpret_cast<double2*>(f)[2 * i + 1] = make_double2(v[2], v[3]);
    } else {
#pragma unroll
        for (int c = 0; c < NC; ++c) f[i * NC + c] = v[c];
    }
}
template <class R, int NC>
DEV void load_facet(const R* __restrict__ f, long long i, R (&v)[NC]) {
    if constexpr (NC == 4 && sizeof(R) == 4) {
        const float4 a = reinterpret_cast<const float4*>(f)[i];
        v[0] = a.x, v[1] = a.y, v[2] = a.z, v[3] = a.w;
    } else if constexpr (NC == 4) {
        const double2 a = reinterpret_cast<const double2*>(f)[2 * i], b = reinterpret_cast<const double2*>(f)[2 * i + 1];
        v[0] = a.x, v[1] = a.y, v[2] = b.x, v[3] = b.y;
    } else {
#pragma unroll
        for (int c = 0; c < NC; ++c) v[c] = f[i * NC + c];
    }
}

// ---------------------------------------------------------------------------
// the low-order part: dt_e, ubar^{e,L}
// ---------------------------------------------------------------------------
// block-wide minimum of positive doubles folded into *bits with an integer
// atomicMin on the bit pattern (order independent, hence deterministic)
DEV void block_min_to(double v, unsigned long long* bits) {
    __shared__ unsigned long long sm[32];
    const int t = threadIdx.y * blockDim.x + threadIdx.x;
    const int nt = blockDim.x * blockDim.y;
    unsigned long long b = (unsigned long long)__double_as_longlong(v);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        unsigned long long w = __shfl_down_sync(0xffffffffu, b, o);
        b = w < b ? w : b;
    }
    if ((t & 31) == 0) sm[t >> 5] = b;
    __syncthreads();
    if (t < 32) {
        b = (t < (nt >> 5)) ? sm[t] : 0x7ff0000000000000ull;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            unsigned long long w = __shfl_down_sync(0xffffffffu, b, o);
            b = w < b ? w : b;
        }
        if (t == 0) atomicMin(bits, b);
    }
}

// The low-order part of a stage: u^e of an element and its face neighbours (eq.
// (ueold)), the facet speeds and f^L, dt_e (eq. (dtmaxcell)), ubar^{e,L} (eq.
// (uelowFCT)), the flux-limiter capacities and, in stage 1, the block minimum of
// dt_e.  In the FP32-mixed form the cell means are float-float pairs and the
// low-order facet fluxes float (their flux part is float-accurate anyway, the
// jump comes from float-float differences), as are the capacities (rounded
// toward zero, so they stay admissible); u^e, the reciprocal of the speed sum,
// dt_e, ubar^{e,L} and the bound gaps are float64.

// values passed to and from the out-of-line functions
template <class R, int NC>
struct CompVec {
    R v[NC];
};

// pseudo time step dt_e^max of Lemma 1, eq. (dtmaxsubcell), for the
// unlimited-flux variant (option OPT_SUBCELL_DT with the flux limiter off):
//   dt_e = (1/s) min{ min_{i on dK_e} m_i^e / (|c_ie| lambda_0i),
//                     m_0^e / sum_{i on dK_e} |c_ie| lambda_0i }
// with u_0^e the mean of the interior coefficients (m_0^e their mass),
// c_ie = int_{dK_e} phi_i n ds = |S|/(p+1) times the sum of the outward
// normals of the faces through node i, lambda_0i the speed bound of
// (u_0^e, u_i) along c_ie/|c_ie|, s = 1; for Q1 (no interior node) u_0^e =
// u^e, m_0^e = |K_e| and s = 2.  A node term with zero speed is dropped and
// the sum is floored at lambda_floor |S|.  Float64 from the element's
// coefficients; out of line (not on the default path).
template <class R, int P, class Ph>
__device__ __noinline__ double subcell_dt(const R* __restrict__ u, const MeshDev& m, const ProbDev& pr, int ex,
                                          int ey) {
    constexpr int NC = Ph::NC, N1 = P + 1, N2 = N1 * N1;
    R Ub[NC][N2];
    load_block<R, P, NC>(u, m, ex, ey, Ub);
    double u0[NC];
    double m0, sfac;
    if constexpr (P >= 2) {
#pragma unroll
        for (int c = 0; c < NC; ++c) {
            double acc = 0.0;
            for (int b = 1; b < P; ++b)
                for (int a = 1; a < P; ++a) acc += (double)Ub[c][b * N1 + a];
            u0[c] = acc / (double)((P - 1) * (P - 1));
        }
        m0 = (double)((P - 1) * (P - 1)) * m.me;
        sfac = 1.0;
    } else {
#pragma unroll
        for (int c = 0; c < NC; ++c) {
            double acc = 0.0;
            for (int i = 0; i < N2; ++i) acc += (double)Ub[c][i];
            u0[c] = acc / (double)N2;
        }
        m0 = m.h * m.h;
        sfac = 2.0;
    }
    const double cface = m.h / (double)N1;
    double best = __longlong_as_double(0x7ff0000000000000LL), total = 0.0;
    for (int b = 0; b < N1; ++b)
        for (int a = 0; a < N1; ++a) {
            const double cx = (a == 0) ? -1.0 : (a == P) ? 1.0 : 0.0;
            const double cy = (b == 0) ? -1.0 : (b == P) ? 1.0 : 0.0;
            if (cx == 0.0 && cy == 0.0) continue;
            const double nrm = sqrt(cx * cx + cy * cy);
            double ui[NC];
#pragma unroll
            for (int c = 0; c < NC; ++c) ui[c] = (double)Ub[c][b * N1 + a];
            const double lam = Ph::template max_speed<double>(u0, ui, cx / nrm, cy / nrm, pr);
            const double w = (cface * nrm) * lam;
            total += w;
            if (w > 0.0) best = fmin(best, m.me / w);
        }
    total = fmax(total, pr.lambda_floor * m.h);
    return fmin(best, m0 / total) / sfac;
}

// low-order quantities of a boundary facet of the FP32-mixed form: the
// speed bound (inflated like the interior ones) and F(u^e, u_hat; n) in the
// canonical orientation, u_hat of side d at the facet midpoint in float-float
// (FIXED: the side's state; OUTFLOW: u^e; WALL: u^e with reversed normal
// momentum); uh, ul: the element's float-float mean, fn: its flux along the
// facet axis; returns [F_0 .. F_{NC-1}, lambda]
template <class Ph>
__device__ __noinline__ CompVec<float, Ph::NC + 1> boundary_facet_lo(const MeshDev& m, const ProbDev& pr, int d,
                                                                    int ex, int ey, float sg,
                                                                    CompVec<float, Ph::NC> uh,
                                                                    CompVec<float, Ph::NC> ul,
                                                                    CompVec<float, Ph::NC> fn) {
    constexpr int NC = Ph::NC;
    const bool xf = d < 2;
    const float inflate = 1.0f + 0x1p-20f;
    const float cnx = xf ? 1.f : 0.f, cny = xf ? 0.f : 1.f;
    const int slot = side_split(pr, d) ? side_slot(pr, d, side_mid_pos(m, d, ex, ey)) : 0;
    const SideDev& sd = pr.side[d];
    const int kind = sd.kind[slot];
    float xh[NC], xl[NC], xfx[NC], xfy[NC];
#pragma unroll
    for (int c = 0; c < NC; ++c) {
        xh[c] = (kind == BC_FIXED) ? sd.st_f[slot][c] : uh.v[c];
        xl[c] = (kind == BC_FIXED) ? sd.st_lo_f[slot][c] : ul.v[c];
    }
    if constexpr (NC == 4) {
        if (kind == BC_WALL) {
            const int cn = xf ? 1 : 2;
            xh[cn] = -xh[cn];
            xl[cn] = -xl[cn];
        }
    }
    Ph::template flux<float>(xh, xfx, xfy, pr);
    const float l = __fmul_rn(Ph::template max_speed<float>(uh.v, xh, sg * cnx, sg * cny, pr), inflate);
    CompVec<float, NC + 1> out;
    out.v[NC] = l;
#pragma unroll
    for (int c = 0; c < NC; ++c) {
        const float ns = sg * fn.v[c];
        const float nx = sg * (xf ? xfx[c] : xfy[c]);
        const float Fo = llf_value(ns, nx, l, ff_diff(xh[c], xl[c], uh.v[c], ul.v[c]));
        out.v[c] = sg * Fo;
    }
    return out;
}

// SUB: pseudo time steps from the subcell bound of Lemma 1 (a separate
// instantiation, so that the default kernels carry none of its code).
// What follows the four facets of an element in the FP32-mixed form: dt_e,
// ubar^{e,L}, the flux-limiter capacities (scalars) or the float copies for
// the limiter's certificate (systems), from the canonical facet fluxes F, the
// speeds lam and the float-float mean
template <int P, class Ph, bool SUB>
DEV double lo_outputs_mixed(const MeshDev& m, const ProbDev& pr, const float* __restrict__ u, const float (&lam)[4],
                            const float (&F)[4][Ph::NC], const float (&uh)[Ph::NC], const float (&ul)[Ph::NC],
                            double* __restrict__ ue_out, double* __restrict__ dte_out, double* __restrict__ ubl_out,
                            float* __restrict__ q_out, float* __restrict__ fl_out, float* __restrict__ cf_out,
                            float* __restrict__ avg, int ex, int ey, int e) {
    constexpr int NC = Ph::NC;
    float sf = __fadd_rn(__fadd_rn(__fadd_rn(lam[0], lam[1]), lam[2]), lam[3]);
    sf = fmaxf(sf, pr.lambda_floor_f);
    // dt_e / h = 1 / s: float reciprocal refined by one float64 Newton step
    // (relative error ~2^-46, far inside the 2^-20 inflation of the speeds;
    // GB300's float64 divide is a long sequence on its narrow float64 pipe)
    double s, rs;
    if constexpr (SUB) {
        // Lemma 1 bound; the float speed sum is rounded up (a float dt_e no
        // larger than the bound)
        rs = subcell_dt<float, P, Ph>(u, m, pr, ex, ey) * m.inv_h;
        s = 1.0 / rs;
        sf = __double2float_ru(s);
    } else {
        s = widen(sf);
        const double r0 = widen(__frcp_rn(sf));
        rs = fma(r0, fma(-s, r0, 1.0), r0);
    }
    const double dte = m.h * rs;
    dte_out[e] = dte;
    dte_out[off<NC>(m.E, 1, e)] = rs;
    dte_out[off<NC>(m.E, 2, e)] = s * m.inv_h;
#pragma unroll
    for (int d = 0; d < 4; ++d)
        store_facet<float, NC>(fl_out, (long long)e * 4 + d, F[d]);
    const float s4 = 0.25f * sf;  // |K| / (|dK| dt_e), exact
#pragma unroll
    for (int c = 0; c < NC; ++c) {
        // facet flux sum (F_E - F_W) + F_N - F_S as a float-float pair, widened once
        float osh, osl;
        ff_sum4(F[1][c], F[0][c], F[3][c], F[2][c], osh, osl);
        const double ued = widen(uh[c]) + widen(ul[c]);
        ue_out[c * m.E + e] = ued;
        const double bl = ued - rs * (widen(osh) + widen(osl));
        ubl_out[c * m.E + e] = bl;
        if (NC == 1) {
            // capacities (s/4)(umax - bl) >= 0 and (s/4)(umin - bl) <= 0: bound
            // gaps in float64, both factors and the product rounded toward zero
            // (smaller magnitudes stay admissible)
            q_out[e] = __fmul_rz(s4, fmaxf(0.f, narrow(pr.umax - bl)));
            q_out[off<NC>(m.E, 1, e)] = __fmul_rz(s4, fminf(0.f, narrow(pr.umin - bl)));
            // the float-float mean, for the element contributions of k_update_el
            avg[e] = uh[0];
            avg[off<NC>(m.E, 1, e)] = ul[0];
        } else {
            // float copies for the certificate of the facet limiter (euler_alpha_is_one)
            cf_out[off<NC>(m.E, 1 + c, e)] = cert_float(bl);
        }
    }
    cf_out[e] = sf;  // the float speed sum (dt_e in float for the update)
    return dte;
}

// FP32-mixed scalars, the arithmetic of k_lo and k_sens for one element (the
// batched stage)
template <int P, class Ph>
DEV double pre_at_mixed(const MeshDev& m, const ProbDev& pr, const float* __restrict__ u,
                        double* __restrict__ ue_out, double* __restrict__ dte_out,
                        double* __restrict__ ubl_out, double* __restrict__ gam_out,
                        double* __restrict__ nu_out, float* __restrict__ q_out,
                        float* __restrict__ fl_out, float* __restrict__ cf_out,
                        float* __restrict__ avg, int ex, int ey, int e) {
    constexpr int NC = 1, N2 = Dim<P>::N2;
    static_assert(Ph::NC == 1, "systems: k_lo_sys");
    int nb[4];
#pragma unroll
    for (int d = 0; d < 4; ++d) nb[d] = neighbour(m, ex, ey, d);
    float U[N2], uh[NC], ul[NC], fxs[NC], fys[NC];
    load_comp<float, P>(u, m, ex, ey, U);
    ff_mean<N2>(U, uh[0], ul[0]);
    Ph::template flux<float>(uh, fxs, fys, pr);
    // neighbours: means and fluxes
    float oh[4][NC], ol[4][NC], ofx[4][NC], ofy[4][NC];
#pragma unroll
    for (int d = 0; d < 4; ++d) {
        if (nb[d] >= 0) {
            int jx, jy;
            neighbour_xy(m, ex, ey, d, jx, jy);
            float B[N2];
            load_comp<float, P>(u, m, jx, jy, B);
            ff_mean<N2>(B, oh[d][0], ol[d][0]);
            Ph::template flux<float>(oh[d], ofx[d], ofy[d], pr);
        } else {
            oh[d][0] = ol[d][0] = ofx[d][0] = ofy[d][0] = 0.f;
        }
    }
    // canonical facet fluxes F(u^L, u^R; n), n = +x (W, E) or +y (S, N)
    const float inflate = 1.0f + 0x1p-20f;
    float lam[4], F[4][NC];
#pragma unroll
    for (int d = 0; d < 4; ++d) {
        const bool xf = d < 2;
        const float cnx = xf ? 1.f : 0.f, cny = xf ? 0.f : 1.f;
        const bool self_is_L = (d == 1 || d == 3);
        if (nb[d] >= 0) {
            const float* Lh = self_is_L ? uh : oh[d];
            const float* Ll = self_is_L ? ul : ol[d];
            const float* Rh = self_is_L ? oh[d] : uh;
            const float* Rl = self_is_L ? ol[d] : ul;
            const float* fL = xf ? (self_is_L ? fxs : ofx[d]) : (self_is_L ? fys : ofy[d]);
            const float* fR = xf ? (self_is_L ? ofx[d] : fxs) : (self_is_L ? ofy[d] : fys);
            const float l = __fmul_rn(Ph::template max_speed<float>(Lh, Rh, cnx, cny, pr), inflate);
            lam[d] = l;
            F[d][0] = llf_value(fL[0], fR[0], l, ff_diff(Rh[0], Rl[0], Lh[0], Ll[0]));
        } else {
            // boundary facet: out of line (rare; keeps the hot code small)
            CompVec<float, NC> vh, vl, vf;
            vh.v[0] = uh[0];
            vl.v[0] = ul[0];
            vf.v[0] = xf ? fxs[0] : fys[0];
            const CompVec<float, NC + 1> o =
                boundary_facet_lo<Ph>(m, pr, d, ex, ey, self_is_L ? 1.f : -1.f, vh, vl, vf);
            lam[d] = o.v[NC];
            F[d][0] = o.v[0];
        }
    }
    const double dte = lo_outputs_mixed<P, Ph, false>(m, pr, u, lam, F, uh, ul, ue_out, dte_out, ubl_out, q_out, fl_out,
                                                      cf_out, avg, ex, ey, e);
    float gam;
    if (pr.mode == MODE_WENO || pr.mode == MODE_WENO_L) {
        gam = sensor_scalar<float, P>(m, pr, u, U, nb, ex, ey);
    } else {
        gam = (pr.mode == MODE_HO) ? 1.f : 0.f;
    }
    gam_out[e] = widen(gam);
    float lm = 0.f;
#pragma unroll
    for (int i = 0; i < N2; ++i) lm = fmaxf(lm, Ph::template node_speed<float>(&U[i], pr));
    nu_out[e] = widen(lm * (m.h_f * (0.5f / P)));
    return dte;
}

// the same in float64: dt_e, ubar^{e,L} and the capacities or certificate
// copies from the facets
template <int P, class Ph, bool SUB>
DEV double lo_outputs_fp64(const MeshDev& m, const ProbDev& pr, const double* __restrict__ u, const double (&lam)[4],
                           const double (&FL)[4][Ph::NC], const double (&us)[Ph::NC], double* __restrict__ dte_out,
                           double* __restrict__ ubl_out, double* __restrict__ q_out, double* __restrict__ fl_out,
                           float* __restrict__ cf_out, int ex, int ey, int e) {
    constexpr int NC = Ph::NC;
    double s = ((lam[0] + lam[1]) + lam[2]) + lam[3];
    s = fmax(s, pr.lambda_floor);
    // dt_e = |K| / (|S| sum lambda) = h / s; dt_e / h = 1 / s
    double rs = 1.0 / s;
    if constexpr (SUB) {
        // Lemma 1 bound instead (the unlimited-flux variant)
        rs = subcell_dt<double, P, Ph>(u, m, pr, ex, ey) * m.inv_h;
        s = 1.0 / rs;
    }
    const double dte = m.h * rs;
    dte_out[e] = dte;
    dte_out[off<NC>(m.E, 1, e)] = rs;              // dt_e / h
    dte_out[off<NC>(m.E, 2, e)] = s * m.inv_h; // 1 / dt_e
#pragma unroll
    for (int d = 0; d < 4; ++d)
        store_facet<double, NC>(fl_out, (long long)e * 4 + d, FL[d]);
#pragma unroll
    for (int c = 0; c < NC; ++c) {
        const double os = ((FL[1][c] - FL[0][c]) + FL[3][c]) - FL[2][c];
        const double bl = us[c] - rs * os;
        ubl_out[c * m.E + e] = bl;
        if (NC == 1) {
            // admissible antidiffusive capacities of eq. (fAlim):
            // (|K|/|dK|)(umax - ubar^{e,L})/dt_e = (s/4)(umax - ubar^{e,L}) >= 0, and
            // (s/4)(umin - ubar^{e,L}) <= 0
            q_out[e] = fmax(0.0, (0.25 * s) * (pr.umax - bl));
            q_out[off<NC>(m.E, 1, e)] = fmin(0.0, (0.25 * s) * (pr.umin - bl));
        } else {
            cf_out[off<NC>(m.E, 1 + c, e)] = cert_float(bl);  // for the certificate of the facet limiter
        }
    }
    if (NC > 1) cf_out[e] = cert_float(s);
    return dte;
}

// k_avg (systems): cell means of every element, read by k_lo_sys for the facets
// of the cell instead of its coefficient block: float-float in the FP32-mixed
// form (avg[(2c) E + e] high, avg[(2c+1) E + e] low part of component c), u^e
// itself in float64.  Beside them the quantities of the mean's state that
// every facet of the cell needs, formed once per cell: cq[c E + e] = f_x(u^e)
// and cq[(NC + c) E + e] = f_y(u^e) (the flux of the high parts), then the
// speed parts of the two-rarefaction bound.
template <class R, int P, class Ph>
__global__ void k_avg(MeshDev m, ProbDev pr, const R* __restrict__ u, float* __restrict__ avg, double* __restrict__ ue_out,
                      R* __restrict__ cq) {
    pdl_begin();
    int ex, ey, e;
    if (!elem_of_thread(m, ex, ey, e)) return;
    constexpr int NC = Ph::NC, N2 = Dim<P>::N2;
    R uh[NC];
#pragma unroll
    for (int c = 0; c < NC; ++c) {
        R U[N2];
        load_comp<R, P>(u + c * m.NN, m, ex, ey, U);
        if constexpr (sizeof(R) == 4) {
            float hi, lo;
            ff_mean<N2>(U, hi, lo);
            avg[off<NC>(m.E, 2 * c, e)] = hi;
            avg[off<NC>(m.E, 2 * c + 1, e)] = lo;
            uh[c] = hi;
        } else {
            uh[c] = cell_mean<R, P>(m, U);
            ue_out[c * m.E + e] = uh[c];
        }
    }
    R fx[NC], fy[NC], q[Ph::NPART];
    Ph::template flux<R>(uh, fx, fy, pr);
    Ph::speed_parts(uh, PV<R>::gam(pr), q);
#pragma unroll
    for (int c = 0; c < NC; ++c) {
        field(cq, m.E, c)[e] = fx[c];
        field(cq, m.E, NC + c)[e] = fy[c];
    }
#pragma unroll
    for (int k = 0; k < Ph::NPART; ++k) field(cq, m.E, 2 * NC + k)[e] = q[k];
}

// element of position i of a tile's halo rows (tiles of K_TX x TY elements, one
// element of halo): false where it does not exist or no element of the tile
// reads it (wrapped once on periodic directions)
constexpr int K_TX = 32;
template <int TY>
DEV bool halo_elem(const MeshDev& m, int ex0, int ey0, int i, int& jx, int& jy) {
    constexpr int HX = K_TX + 2;
    const int hy = i / HX, hx = i - hy * HX;
    jx = ex0 + hx - 1;
    jy = ey0 + hy - 1;
    if ((hx == 0 || hx == HX - 1) && (hy == 0 || hy == TY + 1)) return false;
    if (jx > m.nx || jy > m.ny) return false;
    if (m.px) jx = jx < 0 ? m.nx - 1 : (jx == m.nx ? 0 : jx);
    if (m.py) jy = jy < 0 ? m.ny - 1 : (jy == m.ny ? 0 : jy);
    return jx >= 0 && jx < m.nx && jy >= 0 && jy < m.ny;
}
// halo position of the face neighbour d of the tile element (tx, ty) (-1: its own)
DEV int halo_pos(int tx, int ty, int d) {
    return (ty + 1 + (d == 2 ? -1 : d == 3 ? 1 : 0)) * (K_TX + 2) + tx + 1 + (d == 0 ? -1 : d == 1 ? 1 : 0);
}

// scalars: the low-order part of the stage (cell means, facet speeds and f^L,
// dt_e, ubar^{e,L}, the flux-limiter capacities); gamma_e and nu_e come from
// k_sens, which runs beside it.  The means and their fluxes of a tile of 32 x
// TY elements and its halo are formed once in shared memory, instead of five
// times per element.  pre_at_mixed is the same arithmetic for one element of a
// batch.
template <class R, int P, class Ph, int TY, bool SUB = false>
__global__ void __launch_bounds__(K_TX * TY) k_lo(MeshDev m, ProbDev pr, const R* __restrict__ u,
                                                  double* __restrict__ ue_out, double* __restrict__ dte_out,
                                                  double* __restrict__ ubl_out, R* __restrict__ q_out,
                                                  R* __restrict__ fl_out, float* __restrict__ cf_out,
                                                  float* __restrict__ avg, unsigned long long* __restrict__ dtbits) {
    constexpr int N2 = Dim<P>::N2, HE = (K_TX + 2) * (TY + 2), NT = K_TX * TY;
    __shared__ R sA[HE], sL[sizeof(R) == 4 ? HE : 1], sX[HE], sY[HE];  // mean (high, low part), its fluxes
    pdl_begin();
    const int tx = threadIdx.x, ty = threadIdx.y, ex0 = blockIdx.x * K_TX, ey0 = blockIdx.y * TY;
    for (int i = ty * K_TX + tx; i < HE; i += NT) {
        int jx, jy;
        if (!halo_elem<TY>(m, ex0, ey0, i, jx, jy)) continue;
        R B[N2], a[1], fx[1], fy[1];
        load_comp<R, P>(u, m, jx, jy, B);
        if constexpr (sizeof(R) == 4) ff_mean<N2>(B, a[0], sL[i]);
        else a[0] = cell_mean<R, P>(m, B);
        Ph::template flux<R>(a, fx, fy, pr);
        sA[i] = a[0];
        sX[i] = fx[0];
        sY[i] = fy[0];
    }
    __syncthreads();
    const int ex = ex0 + tx, ey = ey0 + ty, e = ey * m.nx + ex;
    double dte = __longlong_as_double(0x7ff0000000000000LL);
    if (ex < m.nx && ey < m.ny) {
        int nb[4];
#pragma unroll
        for (int d = 0; d < 4; ++d) nb[d] = neighbour(m, ex, ey, d);
        const int own = halo_pos(tx, ty, -1);
        R us[1] = {sA[own]}, lam[4], F[4][1];
        const R fxs[1] = {sX[own]}, fys[1] = {sY[own]};
        if constexpr (sizeof(R) == 4) {
            const float ul[1] = {sL[own]};
            const float inflate = 1.0f + 0x1p-20f;
#pragma unroll
            for (int d = 0; d < 4; ++d) {
                const bool xf = d < 2, self_is_L = (d == 1 || d == 3);
                if (nb[d] >= 0) {
                    const int j = halo_pos(tx, ty, d);
                    const float oh = sA[j], ol = sL[j], of = xf ? sX[j] : sY[j], sf = xf ? fxs[0] : fys[0];
                    const float Lh = self_is_L ? us[0] : oh, Rh = self_is_L ? oh : us[0];
                    const float Ll = self_is_L ? ul[0] : ol, Rl = self_is_L ? ol : ul[0];
                    const float l = __fmul_rn(
                        Ph::template max_speed<float>(&Lh, &Rh, xf ? 1.f : 0.f, xf ? 0.f : 1.f, pr), inflate);
                    lam[d] = l;
                    F[d][0] = llf_value(self_is_L ? sf : of, self_is_L ? of : sf, l, ff_diff(Rh, Rl, Lh, Ll));
                } else {
                    // boundary facet: out of line (rare; keeps the hot code small)
                    CompVec<float, 1> vh, vl, vf;
                    vh.v[0] = us[0];
                    vl.v[0] = ul[0];
                    vf.v[0] = xf ? fxs[0] : fys[0];
                    const CompVec<float, 2> o =
                        boundary_facet_lo<Ph>(m, pr, d, ex, ey, self_is_L ? 1.f : -1.f, vh, vl, vf);
                    lam[d] = o.v[1];
                    F[d][0] = o.v[0];
                }
            }
            dte = lo_outputs_mixed<P, Ph, SUB>(m, pr, u, lam, F, us, ul, ue_out, dte_out, ubl_out, q_out, fl_out, cf_out,
                                               avg, ex, ey, e);
        } else {
            ue_out[e] = us[0];
            double uo[4][1], fxo[4][1], fyo[4][1];
#pragma unroll
            for (int d = 0; d < 4; ++d) {
                const int j = halo_pos(tx, ty, d);
                uo[d][0] = nb[d] >= 0 ? sA[j] : 0.0;
                fxo[d][0] = nb[d] >= 0 ? sX[j] : 0.0;
                fyo[d][0] = nb[d] >= 0 ? sY[j] : 0.0;
            }
            lo_facets<Ph, R>(m, pr, nb, ex, ey, us, fxs, fys, uo, fxo, fyo, lam, F);
            dte = lo_outputs_fp64<P, Ph, SUB>(m, pr, u, lam, F, us, dte_out, ubl_out, q_out, fl_out, cf_out, ex, ey, e);
        }
    }
    if (dtbits) block_min_to(dte, dtbits);
}

// The facets of a tile of F_TX x F_TY elements (systems).  A block of F_TX x
// (F_TY + 1) threads evaluates each once, where one thread per element
// evaluated its four (every interior facet twice), and the elements take them
// from shared memory.  Two rounds: the vertical facets, a row of threads the
// facets left of a row of elements (aligned, as all arrays of elements are),
// the last row the far ends; then the F_TY + 1 rows of horizontal ones.
// Bound by latency (six blocks of loads per facet and few instructions): four
// rows of threads taking the 292 facets in turn left a third round of 36 and
// split addresses, 489 us for k_lo_sys and 407 for k_facet_sys on 2048^2
// elements of degree 2 (FP32-mixed); five rows, and f^L in 16-byte accesses,
// 319 and 348.
constexpr int F_TX = 32, F_TY = 4;
struct FacetItem {
    int axis, slot;        // x (0) or y (1); position in the tile's facets (facet_of)
    int eL, eR;            // cells left and right (below and above), -1 outside the domain
    int ex, ey, d;         // a cell of the facet and its side there (the one inside on the boundary)
};
// the facet of thread (tx, ty) in the round of an axis: false where it has none
DEV bool facet_item(const MeshDev& m, int ex0, int ey0, int axis, FacetItem& f) {
    const int tx = threadIdx.x, ty = threadIdx.y;
    int c = tx, r = ty;
    if (axis == 0 && ty == F_TY) {
        c = F_TX, r = tx;
        if (r >= F_TY) return false;
    }
    f.axis = axis;
    f.slot = axis == 0 ? r * (F_TX + 1) + c : (F_TX + 1) * F_TY + r * F_TX + c;
    // the cell right of (above) the facet, and the one left of (below) it
    const int xR = ex0 + c, yR = ey0 + r, xL = axis == 0 ? xR - 1 : xR, yL = axis == 0 ? yR : yR - 1;
    const bool inR = xR < m.nx && yR < m.ny, inL = xL >= 0 && yL >= 0 && xL < m.nx && yL < m.ny;
    // a cell of the tile itself: the right one unless it is the far end's
    const bool tR = axis == 0 ? c < F_TX : r < F_TY, tL = axis == 0 ? c > 0 : r > 0;
    if (!((tR && inR) || (tL && inL))) return false;
    if (inR) {
        f.eR = yR * m.nx + xR;
        f.ex = xR, f.ey = yR, f.d = axis == 0 ? 0 : 2;
        f.eL = neighbour(m, xR, yR, f.d);
    } else {
        f.eL = yL * m.nx + xL;
        f.ex = xL, f.ey = yL, f.d = axis == 0 ? 1 : 3;
        f.eR = neighbour(m, xL, yL, f.d);
    }
    return true;
}
// slots of the element (tx, ty)'s facets W, E (x) and S, N (y)
DEV int facet_of(int tx, int ty, int d) {
    return d < 2 ? ty * (F_TX + 1) + tx + d : (F_TX + 1) * F_TY + (ty + d - 2) * F_TX + tx;
}
constexpr int F_NT = F_TX * (F_TY + 1), F_N = (F_TX + 1) * F_TY + F_TX * (F_TY + 1);

// low-order quantities of a boundary facet in float64, as boundary_facet_lo
template <class Ph>
__device__ __noinline__ CompVec<double, Ph::NC + 1> boundary_facet_lo64(const MeshDev& m, const ProbDev& pr, int d,
                                                                       int ex, int ey, CompVec<double, Ph::NC> us,
                                                                       CompVec<double, Ph::NC> fn) {
    constexpr int NC = Ph::NC;
    const bool xf = d < 2;
    const double sg = (d & 1) ? 1.0 : -1.0, nx = xf ? sg : 0.0, ny = xf ? 0.0 : sg;
    // external state u_hat at the facet midpoint from the cell average
    const int slot = side_split(pr, d) ? side_slot(pr, d, side_mid_pos(m, d, ex, ey)) : 0;
    double ux[NC], fx[NC];
    ext_state<double, NC>(pr, d, slot, us.v, ux);
    if (pr.side[d].kind[slot] != BC_OUTFLOW) {
        Ph::template normal<double>(ux, xf ? 0 : 1, fx, pr);
    } else {
#pragma unroll
        for (int c = 0; c < NC; ++c) fx[c] = fn.v[c];
    }
    const double l = Ph::template max_speed<double>(us.v, ux, nx, ny, pr);
    CompVec<double, NC + 1> out;
    out.v[NC] = l;
#pragma unroll
    for (int c = 0; c < NC; ++c)
        out.v[c] = sg * (0.5 * (sg * fn.v[c] + sg * fx[c]) - 0.5 * l * (ux[c] - us.v[c]));
    return out;
}

// systems: the low-order part of the stage from the cell states of k_avg
// (facet speeds and f^L, dt_e, ubar^{e,L}, the float copies for the facet
// limiter's certificate); gamma_e and nu_e come from k_sens
template <class R, int P, class Ph, bool SUB = false>
__global__ void __launch_bounds__(F_NT, sizeof(R) == 4 ? (SUB ? 5 : 6) : (SUB ? 2 : 3))
    k_lo_sys(MeshDev m, ProbDev pr, const R* __restrict__ u, double* __restrict__ ue_io, double* __restrict__ dte_out,
             double* __restrict__ ubl_out, R* __restrict__ fl_out, float* __restrict__ cf_out,
             const float* __restrict__ avg, const R* __restrict__ cq, unsigned long long* __restrict__ dtbits) {
    constexpr int NC = Ph::NC;
    __shared__ R sF[NC + 1][F_N];  // f^L, speed
    pdl_begin();
    const int tx = threadIdx.x, ty = threadIdx.y, ex0 = blockIdx.x * F_TX, ey0 = blockIdx.y * F_TY;
    const int E = m.E;
    const R g = PV<R>::gam(pr);
#pragma unroll 1
    for (int axis = 0; axis < 2; ++axis) {
        FacetItem f;
        if (!facet_item(m, ex0, ey0, axis, f)) continue;
        R F[NC], lam;
        const R* __restrict__ fa = field(cq, E, f.axis * NC);  // the means' fluxes along the facet's axis
        if (f.eL >= 0 && f.eR >= 0) {
            const R* __restrict__ q = field(cq, E, 2 * NC + 2);
            const R* __restrict__ qv = field(cq, E, 2 * NC + f.axis);
            const R l = Ph::facet_speed_parts(qv[f.eL], q[f.eL], q[E + f.eL], q[2 * E + f.eL], q[3 * E + f.eL], qv[f.eR],
                                              q[f.eR], q[E + f.eR], q[2 * E + f.eR], q[3 * E + f.eR], g);
            if constexpr (sizeof(R) == 4) {
                lam = __fmul_rn(l, 1.0f + 0x1p-20f);
#pragma unroll
                for (int c = 0; c < NC; ++c) {
                    const float* __restrict__ ah = field(avg, E, 2 * c);
                    F[c] = llf_value(fa[c * E + f.eL], fa[c * E + f.eR], lam,
                                     ff_diff(ah[f.eR], ah[E + f.eR], ah[f.eL], ah[E + f.eL]));
                }
            } else {
                lam = l;
#pragma unroll
                for (int c = 0; c < NC; ++c)
                    F[c] = 0.5 * (fa[c * E + f.eL] + fa[c * E + f.eR]) -
                           0.5 * l * (ue_io[c * E + f.eR] - ue_io[c * E + f.eL]);
            }
        } else {
            // a facet on the domain boundary: out of line (rare)
            const int e = f.ey * m.nx + f.ex;
            if constexpr (sizeof(R) == 4) {
                CompVec<float, NC> vh, vl, vf;
#pragma unroll
                for (int c = 0; c < NC; ++c) {
                    vh.v[c] = avg[off<NC>(E, 2 * c, e)];
                    vl.v[c] = avg[off<NC>(E, 2 * c + 1, e)];
                    vf.v[c] = fa[c * E + e];
                }
                const CompVec<float, NC + 1> o =
                    boundary_facet_lo<Ph>(m, pr, f.d, f.ex, f.ey, (f.d & 1) ? 1.f : -1.f, vh, vl, vf);
                lam = o.v[NC];
#pragma unroll
                for (int c = 0; c < NC; ++c) F[c] = o.v[c];
            } else {
                CompVec<double, NC> us, vf;
#pragma unroll
                for (int c = 0; c < NC; ++c) {
                    us.v[c] = ue_io[c * E + e];
                    vf.v[c] = fa[c * E + e];
                }
                const CompVec<double, NC + 1> o = boundary_facet_lo64<Ph>(m, pr, f.d, f.ex, f.ey, us, vf);
                lam = o.v[NC];
#pragma unroll
                for (int c = 0; c < NC; ++c) F[c] = o.v[c];
            }
        }
#pragma unroll
        for (int c = 0; c < NC; ++c) sF[c][f.slot] = F[c];
        sF[NC][f.slot] = lam;
    }
    __syncthreads();
    const int ex = ex0 + tx, ey = ey0 + ty, e = ey * m.nx + ex;
    double dte = __longlong_as_double(0x7ff0000000000000LL);
    if (ty < F_TY && ex < m.nx && ey < m.ny) {
        R lam[4], F[4][NC];
#pragma unroll
        for (int d = 0; d < 4; ++d) {
            const int s = facet_of(tx, ty, d);
            lam[d] = sF[NC][s];
#pragma unroll
            for (int c = 0; c < NC; ++c) F[d][c] = sF[c][s];
        }
        R us[NC];
        if constexpr (sizeof(R) == 4) {
            float ul[NC];
#pragma unroll
            for (int c = 0; c < NC; ++c) {
                us[c] = avg[off<NC>(E, 2 * c, e)];
                ul[c] = avg[off<NC>(E, 2 * c + 1, e)];
            }
            dte = lo_outputs_mixed<P, Ph, SUB>(m, pr, u, lam, F, us, ul, ue_io, dte_out, ubl_out, nullptr, fl_out, cf_out,
                                               nullptr, ex, ey, e);
        } else {
#pragma unroll
            for (int c = 0; c < NC; ++c) us[c] = ue_io[c * E + e];
            dte = lo_outputs_fp64<P, Ph, SUB>(m, pr, u, lam, F, us, dte_out, ubl_out, nullptr, fl_out, cf_out, ex, ey, e);
        }
    }
    if (dtbits) block_min_to(dte, dtbits);
}

// the WENO sensor gamma_e (eqs. (WENO:alpha), (WENO:norm)) and nu_e (eq.
// (stab:WENO)).  A block of K_TX x TY threads holds a tile of K_TX x TY
// elements; component by component it puts the modal coefficients of the tile
// and its one-element halo in shared memory (modal.cuh), so that each block of
// coefficients is loaded and transformed 1.3 to 1.6 times instead of five,
// and one thread per element evaluates the sensor from them.
// The node speeds of nu_e are formed once per node of the tile (an element
// has (p+1)^2 nodes but brings p^2 new ones) and pass through the same
// shared memory.
template <class R, int P, class Ph, int TY>
__global__ void __launch_bounds__(K_TX * TY) k_sens(MeshDev m, ProbDev pr, const R* __restrict__ u,
                                                    double* __restrict__ gam_out, double* __restrict__ nu_out) {
    constexpr int NC = Ph::NC, N2 = Dim<P>::N2, HE = (K_TX + 2) * (TY + 2), NT = K_TX * TY;
    constexpr int NH = (HE + NT - 1) / NT;                        // halo positions per thread
    constexpr int SX = K_TX * P + 1, SY = TY * P + 1, NS = SX * SY;  // the tile's nodes
    // four continued candidates in registers where they leave two blocks per SM
    constexpr bool KEEP = (N2 - 1) * sizeof(R) <= 128;
    constexpr int WS = (N2 - 1) * HE > NS ? (N2 - 1) * HE : NS;
    __shared__ R ws[WS];
    R(*sM)[HE] = reinterpret_cast<R(*)[HE]>(ws);
    R(*sS)[SX] = reinterpret_cast<R(*)[SX]>(ws);
    pdl_begin();
    const int tx = threadIdx.x, ty = threadIdx.y, tid = ty * K_TX + tx;
    const int ex0 = blockIdx.x * K_TX, ey0 = blockIdx.y * TY;
    const int ex = ex0 + tx, ey = ey0 + ty;
    const bool valid = ex < m.nx && ey < m.ny;
    const Tab<R>& T = tab_of<R>(m, P);
    R gam = R(1);
    if (pr.mode == MODE_WENO || pr.mode == MODE_WENO_L) {
        int nb[4], hx[NH], hy[NH];
        bool hv[NH];
#pragma unroll
        for (int d = 0; d < 4; ++d) nb[d] = neighbour(m, ex, ey, d);
#pragma unroll
        for (int j = 0; j < NH; ++j)
            hv[j] = tid + j * NT < HE && halo_elem<TY>(m, ex0, ey0, tid + j * NT, hx[j], hy[j]);
#pragma unroll 1
        for (int c = 0; c < NC; ++c) {
            if (c > 0) __syncthreads();  // the previous component is consumed
#pragma unroll
            for (int j = 0; j < NH; ++j) {
                if (!hv[j]) continue;
                R V[N2], l[N2];
                load_comp<R, P>(u + c * m.NN, m, hx[j], hy[j], V);
                modal_block<R, P>(T, V, l);
#pragma unroll
                for (int k = 1; k < N2; ++k) sM[k - 1][tid + j * NT] = l[k];
            }
            __syncthreads();
            if (valid) {
                R own[N2];
                const int at = halo_pos(tx, ty, -1);
                own[0] = R(0);
#pragma unroll
                for (int k = 1; k < N2; ++k) own[k] = sM[k - 1][at];
                const R g = modal_sensor<R, P, KEEP>(T, a2_base<R>(m), pr, own, nb, [&](int d, R(&l)[N2]) {
                    const int j = halo_pos(tx, ty, d);
                    l[0] = R(0);
#pragma unroll
                    for (int k = 1; k < N2; ++k) l[k] = sM[k - 1][j];
                });
                gam = fmin(gam, g);
            }
        }
        __syncthreads();  // the modes are consumed
    } else {
        gam = (pr.mode == MODE_HO) ? R(1) : R(0);
    }
    for (int i = tid; i < NS; i += NT) {
        const int r = i / SX, q = i - r * SX;
        int gx = ex0 * P + q, gy = ey0 * P + r;
        if (m.px && gx == m.nnx) gx = 0;
        if (m.py && gy == m.nny) gy = 0;
        if (gx < m.nnx && gy < m.nny) {
            const R* __restrict__ un = u + ((long long)gy * m.nnx + gx);
            R ui[NC];
#pragma unroll
            for (int c = 0; c < NC; ++c) ui[c] = un[c * m.NN];
            ws[i] = Ph::template node_speed<R>(ui, pr);
        }
    }
    __syncthreads();
    if (!valid) return;
    R lm = R(0);
#pragma unroll
    for (int b = 0; b <= P; ++b)
#pragma unroll
        for (int a = 0; a <= P; ++a) lm = fmax(lm, sS[ty * P + b][tx * P + a]);
    const int e = ey * m.nx + ex;
    if constexpr (sizeof(R) == 4) gam_out[e] = widen(gam);
    else gam_out[e] = gam;
    if constexpr (sizeof(R) == 4) nu_out[e] = widen(lm * (m.h_f * (0.5f / P)));
    else nu_out[e] = lm * (m.h * (0.5 / P));
}

// global dt from the block minima folded into the bit pattern by k_lo
// dt = min(cfl * min_e dt_e, t_end - t), never negative
static __global__ void k_dt_final(unsigned long long* bits, double cfl, const double* t,
                                  const double* t_end, double* dt) {
    pdl_begin();
    double d = cfl * __longlong_as_double((long long)*bits);
    *bits = 0x7ff0000000000000ull;  // ready for the next reduction
    double rem = *t_end - *t;
    if (rem < d) d = rem > 0.0 ? rem : 0.0;
    *dt = d;
}

// ---------------------------------------------------------------------------
// node-centric gathers over E_i in a fixed order (lower neighbour first in
// each direction): deterministic, no atomics.
// ---------------------------------------------------------------------------
// elements containing node (gx, gy): at most two per direction (lower one
// first), with the node's local index in each; compile-time P
template <int P>
struct NodeC {
    int ex0, ex1, a0, a1, nxc;
    int ey0, ey1, b0, b1, nyc;
};

template <int P>
DEV NodeC<P> node_c(const MeshDev& m, int gx, int gy) {
    NodeC<P> c;
    int ex = gx / P, a = gx - ex * P;
    if (a == 0) {
        const bool lo = (ex > 0) || m.px, hi = ex < m.nx;
        c.ex0 = lo ? (ex == 0 ? m.nx - 1 : ex - 1) : ex;
        c.a0 = lo ? P : 0;
        c.ex1 = ex;
        c.a1 = 0;
        c.nxc = (int)lo + (int)hi;
    } else {
        c.ex0 = c.ex1 = ex;
        c.a0 = c.a1 = a;
        c.nxc = 1;
    }
    int ey = gy / P, b = gy - ey * P;
    if (b == 0) {
        const bool lo = (ey > 0) || m.py, hi = ey < m.ny;
        c.ey0 = lo ? (ey == 0 ? m.ny - 1 : ey - 1) : ey;
        c.b0 = lo ? P : 0;
        c.ey1 = ey;
        c.b1 = 0;
        c.nyc = (int)lo + (int)hi;
    } else {
        c.ey0 = c.ey1 = ey;
        c.b0 = c.b1 = b;
        c.nyc = 1;
    }
    return c;
}

// 1/|E_i| for |E_i| in {1, 2, 4} (exact powers of two)
template <class R>
DEV R inv_count(int n) {
    return n == 4 ? R(0.25) : (n == 2 ? R(0.5) : R(1));
}

// 1 / m_i on an LGL mesh (float64 form): m_i = sum over the cnt elements
// containing node i of h^2 w_a w_b, with the node's local indices (a0, b0)
// in the first of them; the LGL weights are symmetric (w_0 = w_p), so a
// shared node has the same weight in every element containing it
template <int P>
DEV double inv_lumped_lgl(const MeshDev& m, int cnt, int a0, int b0) {
    const Tab<double>& T = c_tabd[PMAX + 1 + P];
    return inv_count<double>(cnt) * (m.inv_h2 * (T.iwl[a0] * T.iwl[b0]));
}


// s[v] = sum over E_i of the element vectors at node (gx, gy), fixed order
template <class R, int P, int NV>
DEV void gather_at(const MeshDev& m, const R* __restrict__ EV, const NodeC<P>& c, R (&s)[NV]) {
    constexpr int N1 = P + 1, N2 = N1 * N1;
#pragma unroll
    for (int v = 0; v < NV; ++v) s[v] = R(0);
#pragma unroll
    for (int j = 0; j < 2; ++j) {
        if (j < c.nyc) {
            const int ey = j ? c.ey1 : c.ey0, b = j ? c.b1 : c.b0;
#pragma unroll
            for (int i = 0; i < 2; ++i) {
                if (i < c.nxc) {
                    const int ex = i ? c.ex1 : c.ex0, a = i ? c.a1 : c.a0;
                    const int e = ey * m.nx + ex;
#pragma unroll
                    for (int v = 0; v < NV; ++v) s[v] += EV[ev_at(m.E, e, b * N1 + a, v, NV)];
                }
            }
        }
    }
}

// sum over E_i of element vectors; out[v*NN + node]; if xout, also x = sum / m_i
template <class R, int P, int NV>
DEV void gather_init_at(MeshDev m, const R* __restrict__ EV, R* __restrict__ bout,
                              R* __restrict__ xout, int gx, int gy, long long node) {
    const NodeC<P> c = node_c<P>(m, gx, gy);
    R s[NV];
    gather_at<R, P, NV>(m, EV, c, s);
    const R inv_mi = is_lgl<R>(m) ? R(inv_lumped_lgl<P>(m, c.nxc * c.nyc, c.a0, c.b0))
                                  : PV<R>::inv_me(m) * inv_count<R>(c.nxc * c.nyc);
#pragma unroll
    for (int v = 0; v < NV; ++v) {
        if (bout) bout[v * m.NN + node] = s[v];
        if (xout) xout[v * m.NN + node] = s[v] * inv_mi;
    }
}

template <class R, int P, int NV>
__global__ void k_gather_init(MeshDev m, const R* __restrict__ EV, R* __restrict__ bout,
                              R* __restrict__ xout) {
    pdl_begin();
    int gx, gy;
    long long node;
    if (!node_of_thread(m, gx, gy, node)) return;
    gather_init_at<R, P, NV>(m, EV, bout, xout, gx, gy, node);
}




// Richardson update x + (b - h^2 s) / m_i with s = (M (x) M) x at the node
template <class R>
DEV R sweep_value(R x, R b, R s, R h2, R inv_mi) {
    return fma_r(fma_r(-h2, s, b), inv_mi, x);
}

// ---------------------------------------------------------------------------
// node-centric application of the assembled linear operators. On a uniform
// mesh, sum_{e in E_i} of an element operator A^e = Ax (x) Ay is a separable
// stencil over the (2p+1)^2 nodes around node i: along x the weight of offset
// k is sum over the (at most two) elements containing i of Ax[a_e][k + a_e]
// (a_e = local index of i in e); likewise along y.
// ---------------------------------------------------------------------------
// entries of the 1D tables: the assembled mass (WHICH 0: M[a][c]) or the
// derivative on the trial index (WHICH 1: C[c][a] = int B_c' B_a)
template <class R, int P, int WHICH>
DEV R wtab(const Tab<R>& T, int a, int c) {
    return (WHICH == 0) ? T.M[a][c] : T.C[c][a];
}

// an index on a periodic direction of n taken into [0, n): one period covers
// every node of a tile and its halo on meshes at least a tile wide; a
// narrower mesh (down to one element) takes the remainder, so a staged halo
// value is always a node of the mesh
DEV int wrap_periodic(int g, int n) {
    g = g < 0 ? g + n : (g >= n ? g - n : g);
    if ((unsigned)g >= (unsigned)n) g = ((g % n) + n) % n;
    return g;
}

// runtime-degree candidate list (diagnostics only)
struct NodeCands {
    int nxc, nyc;
    int ex[2], a[2], ey[2], b[2];
};

DEV NodeCands node_cands(const MeshDev& m, int gx, int gy) {
    NodeCands nc;
    const int p = m.p;
    int ex = gx / p, a = gx - ex * p;
    nc.nxc = 0;
    if (a == 0) {
        if (ex > 0 || m.px) {
            nc.ex[nc.nxc] = (ex - 1 + m.nx) % m.nx;
            nc.a[nc.nxc++] = p;
        }
        if (ex < m.nx) {
            nc.ex[nc.nxc] = ex;
            nc.a[nc.nxc++] = 0;
        }
    } else {
        nc.ex[0] = ex;
        nc.a[0] = a;
        nc.nxc = 1;
    }
    int ey = gy / p, b = gy - ey * p;
    nc.nyc = 0;
    if (b == 0) {
        if (ey > 0 || m.py) {
            nc.ey[nc.nyc] = (ey - 1 + m.ny) % m.ny;
            nc.b[nc.nyc++] = p;
        }
        if (ey < m.ny) {
            nc.ey[nc.nyc] = ey;
            nc.b[nc.nyc++] = 0;
        }
    } else {
        nc.ey[0] = ey;
        nc.b[0] = b;
        nc.nyc = 1;
    }
    return nc;
}

// ---------------------------------------------------------------------------
// The element residual R^e_i = W^e_i - s^e_i with
//   W^e_i = int grad phi_i . f(u_h) - sum_{interior faces} int phi_i f_h.n
//           - sum_{faces on dOmega} int phi_i F(u_h, u_hat; n)
//   s^e_i = nu_e int grad phi_i . (grad u_h - gamma_e g_h)      eq. (stab:WENO)
// (p+2)-point Gauss rule for nonlinear integrands; exact face mass for f_h.
// ER layout ev_at(E, e, i, c, NC).
// ---------------------------------------------------------------------------
// boundary-face part of the weak form of element (ex, ey) on face d: the
// (p+2)-point quadrature of phi_i F(u_h, u_hat; n), u_hat of the side at
// each Gauss point, or of phi_i f(u_h).n on a side that is OUTFLOW
// everywhere; per unit of h; Uf and term are [NC][p+1]
template <class R, int P, class Ph>
__device__ __noinline__ void boundary_face_term(const MeshDev& m, const ProbDev& pr, int d, int ex, int ey,
                                                const R* Uf, R* term) {
    constexpr int NC = Ph::NC, N1 = P + 1, NQ = Dim<P>::NQ;
    const Tab<R>& T = tab_of<R>(m, P);
    const Tab<double>& Td = tab_of<double>(m, P);
    const R nxo = (d == 0) ? R(-1) : (d == 1) ? R(1) : R(0);
    const R nyo = (d == 2) ? R(-1) : (d == 3) ? R(1) : R(0);
    const bool plain = side_plain(pr, d);
    // a FIXED side with one part: one external state, its flux evaluated once
    const bool fixed1 = !plain && !side_split(pr, d) && pr.side[d].kind[0] == BC_FIXED;
    R ub1[NC], fxb[NC], fyb[NC];
    if (fixed1) {
#pragma unroll
        for (int c = 0; c < NC; ++c) ub1[c] = PV<R>::side_state(pr.side[d], 0, c);
        Ph::template flux<R>(ub1, fxb, fyb, pr);
    }
    R acc[NC][N1];
#pragma unroll
    for (int c = 0; c < NC; ++c)
#pragma unroll
        for (int b = 0; b < N1; ++b) acc[c][b] = R(0);
#pragma unroll
    for (int r = 0; r < NQ; ++r) {
        R uq[NC], F[NC];
#pragma unroll
        for (int c = 0; c < NC; ++c) {
            R s = R(0);
#pragma unroll
            for (int k = 0; k < N1; ++k) s += Uf[c * N1 + k] * T.Bq[r][k];
            uq[c] = s;
        }
        if (fixed1) {
            llf_given_fR<Ph, R>(uq, ub1, fxb, fyb, nxo, nyo, pr, F);
        } else if (!plain) {
            const int slot = side_split(pr, d) ? side_slot(pr, d, side_quad_pos(m, d, ex, ey, Td.xq[r])) : 0;
            R ub[NC];
            ext_state<R, NC>(pr, d, slot, uq, ub);
            llf<Ph, R>(uq, ub, nxo, nyo, pr, F, (R*)nullptr);
        } else {
            R fx[NC], fy[NC];
            Ph::template flux<R>(uq, fx, fy, pr);
#pragma unroll
            for (int c = 0; c < NC; ++c) F[c] = fx[c] * nxo + fy[c] * nyo;
        }
#pragma unroll
        for (int c = 0; c < NC; ++c)
#pragma unroll
            for (int b = 0; b < N1; ++b) acc[c][b] += F[c] * T.wB[r][b];
    }
#pragma unroll
    for (int c = 0; c < NC; ++c)
#pragma unroll
        for (int b = 0; b < N1; ++b) term[c * N1 + b] = acc[c][b];
}

// local node k of face d (W, E, S, N)
template <int P>
DEV constexpr int face_node(int d, int k) {
    return d == 0 ? k * (P + 1) : d == 1 ? k * (P + 1) + P : d == 2 ? k : P * (P + 1) + k;
}

// volume integral of one component from its fluxes at the quadrature points
// of row q2 (fx(q1), fy(q1)), added to W (per unit of h): the weights are
// folded into the tables
template <class R, int P, class FX, class FY>
DEV void volume_row(const Tab<R>& T, int q2, const FX& fx, const FY& fy, R (&W)[Dim<P>::N2]) {
    constexpr int N1 = P + 1, NQ = P + 2;
    R Tx[N1], Ty[N1];
#pragma unroll
    for (int a = 0; a < N1; ++a) Tx[a] = Ty[a] = R(0);
#pragma unroll
    for (int q1 = 0; q1 < NQ; ++q1) {
        const R x = fx(q1), y = fy(q1);
#pragma unroll
        for (int a = 0; a < N1; ++a) {
            Tx[a] += T.wdB[q1][a] * x;
            Ty[a] += T.wB[q1][a] * y;
        }
    }
#pragma unroll
    for (int b = 0; b < N1; ++b)
#pragma unroll
        for (int a = 0; a < N1; ++a) W[b * N1 + a] += T.wB[q2][b] * Tx[a] + T.wdB[q2][b] * Ty[a];
}

// Galerkin part W^e of the element residual of a scalar: volume and face terms
// of the weak form (needs only u)
template <class R, int P, class Ph>
DEV void w_part(const MeshDev& m, const ProbDev& pr, const R (&U)[Dim<P>::N2], int ex, int ey, R (&W)[Dim<P>::N2]) {
    constexpr int N1 = P + 1, N2 = Dim<P>::N2, NQ = Dim<P>::NQ;
    static_assert(Ph::NC == 1, "systems: k_res_sys");
    const Tab<R>& T = tab_of<R>(m, P);
#pragma unroll
    for (int i = 0; i < N2; ++i) W[i] = R(0);
    // volume term: interpolate along x first
    R X[N1][NQ];
#pragma unroll
    for (int d = 0; d < N1; ++d)
#pragma unroll
        for (int q1 = 0; q1 < NQ; ++q1) {
            R s = R(0);
#pragma unroll
            for (int a = 0; a < N1; ++a) s += T.Bq[q1][a] * U[d * N1 + a];
            X[d][q1] = s;
        }
#pragma unroll 1
    for (int q2 = 0; q2 < NQ; ++q2) {
        R fx[NQ], fy[NQ];
#pragma unroll
        for (int q1 = 0; q1 < NQ; ++q1) {
            R s = R(0);
#pragma unroll
            for (int d = 0; d < N1; ++d) s += T.Bq[q2][d] * X[d][q1];
            Ph::template flux<R>(&s, &fx[q1], &fy[q1], pr);
        }
        volume_row<R, P>(T, q2, [&](int q) { return fx[q]; }, [&](int q) { return fy[q]; }, W);
    }
    // face terms
#pragma unroll
    for (int d = 0; d < 4; ++d) {
        R Uf[N1], term[N1];
#pragma unroll
        for (int k = 0; k < N1; ++k) Uf[k] = U[face_node<P>(d, k)];
        if (neighbour(m, ex, ey, d) >= 0) {
            R fn[N1];
#pragma unroll
            for (int k = 0; k < N1; ++k) {
                Ph::template normal<R>(&Uf[k], d >> 1, &fn[k], pr);
                if ((d & 1) == 0) fn[k] = -fn[k];
            }
#pragma unroll
            for (int b = 0; b < N1; ++b) {
                R s = R(0);
#pragma unroll
                for (int k = 0; k < N1; ++k) s += fn[k] * T.M[b][k];
                term[b] = s;
            }
        } else {
            // a face on the domain boundary: out of line, so the common
            // interior path stays compact in the instruction cache
            boundary_face_term<R, P, Ph>(m, pr, d, ex, ey, Uf, term);
        }
#pragma unroll
        for (int k = 0; k < N1; ++k) W[face_node<P>(d, k)] -= term[k];
    }
    const R h = PV<R>::h(m);
#pragma unroll
    for (int i = 0; i < N2; ++i) W[i] = mul_r(W[i], h);
}

// a per-element float64 scalar in the bulk precision (gamma_e, nu_e)
template <class R>
DEV R bulk(double v) {
    if constexpr (sizeof(R) == 4) return narrow(v);
    else return v;
}

// coefficients of h u_h' along a line
template <class R, int P>
DEV void deriv_line(const MeshDev& m, const Tab<R>& T, const R (&u)[P + 1], R (&d)[P + 1]) {
    if (is_lgl<R>(m)) {
#pragma unroll
        for (int i = 0; i <= P; ++i) {
            R s = R(0);
#pragma unroll
            for (int k = 0; k <= P; ++k) s += T.dn[i][k] * u[k];
            d[i] = s;
        }
        return;
    }
    // Bernstein: differences raised to degree p
    R D[P];
#pragma unroll
    for (int i = 0; i < P; ++i) D[i] = u[i + 1] - u[i];
#pragma unroll
    for (int i = 0; i <= P; ++i)
        d[i] = i == 0 ? R(P) * D[0] : i == P ? R(P) * D[P - 1] : R(i) * D[i - 1] + R(P - i) * D[i];
}

// stabilisation s^e = nu_e int grad phi_i . (grad u_h - gamma_e g_h) of one
// component.  The integrand's coefficients w_d = h d_d u_h - gamma_e h g_d are
// formed first (u_h' in the basis itself), so that one application of the
// tensor operators C (x) M and M (x) C serves both terms: at p = 2 144
// multiply-adds instead of the 234 of separate stiffness and gradient terms.
template <class R, int P>
DEV void stab_comp(const MeshDev& m, const Tab<R>& T, const R (&U)[Dim<P>::N2], const R (&GX)[Dim<P>::N2],
                   const R (&GY)[Dim<P>::N2], R gh, R nue, R (&s)[Dim<P>::N2]) {
    constexpr int N1 = P + 1;
    R Z[N1][N1];
#pragma unroll
    for (int dir = 0; dir < 2; ++dir) {
        // w along the direction's lines, then C along it
#pragma unroll
        for (int t = 0; t < N1; ++t) {
            R l[N1], d[N1];
#pragma unroll
            for (int k = 0; k < N1; ++k) l[k] = U[dir == 0 ? t * N1 + k : k * N1 + t];
            deriv_line<R, P>(m, T, l, d);
#pragma unroll
            for (int k = 0; k < N1; ++k) {
                const int i = dir == 0 ? t * N1 + k : k * N1 + t;
                d[k] -= gh * (dir == 0 ? GX[i] : GY[i]);
            }
#pragma unroll
            for (int a = 0; a < N1; ++a) {
                R z = R(0);
#pragma unroll
                for (int k = 0; k < N1; ++k) z += T.C[a][k] * d[k];
                Z[t][a] = z;  // line t, index a along the direction
            }
        }
        // M across the lines
#pragma unroll
        for (int t = 0; t < N1; ++t)
#pragma unroll
            for (int a = 0; a < N1; ++a) {
                R z = R(0);
#pragma unroll
                for (int k = 0; k < N1; ++k) z += T.M[t][k] * Z[k][a];
                const int i = dir == 0 ? t * N1 + a : a * N1 + t;
                s[i] = dir == 0 ? z : mul_r(nue, add_r(s[i], z));
            }
    }
}

// stabilisation and the residual R^e = W^e - s^e of a scalar into ER (W^e and
// s^e rounded on their own, so that the residual in one kernel and in two
// gives the same bits)
template <class R, int P>
DEV void stab_part(const MeshDev& m, const R (&U)[Dim<P>::N2], const R* __restrict__ g,
                   const double* __restrict__ gam, const double* __restrict__ nu, const R (&W)[Dim<P>::N2],
                   R* __restrict__ ER, int ex, int ey, int e) {
    constexpr int N2 = Dim<P>::N2;
    R GX[N2], GY[N2], s[N2];
    load_comp<R, P>(g, m, ex, ey, GX);
    load_comp<R, P>(g + m.NN, m, ex, ey, GY);
    stab_comp<R, P>(m, tab_of<R>(m, P), U, GX, GY, bulk<R>(gam[e]) * PV<R>::h(m), bulk<R>(nu[e]), s);
#pragma unroll
    for (int i = 0; i < N2; ++i) ER[ev_at(m.E, e, i, 0, 1)] = sub_r(W[i], s[i]);
}

template <class R, int P, class Ph>
DEV void res_at(const MeshDev& m, const ProbDev& pr, const R* __restrict__ u, const R* __restrict__ g,
                         const double* __restrict__ gam, const double* __restrict__ nu,
                         R* __restrict__ ER, int ex, int ey, int e) {
    constexpr int N2 = Dim<P>::N2;
    R U[N2], W[N2];
    load_comp<R, P>(u, m, ex, ey, U);
    w_part<R, P, Ph>(m, pr, U, ex, ey, W);
    stab_part<R, P>(m, U, g, gam, nu, W, ER, ex, ey, e);
}

// The residual of systems with one thread per element and component: a block
// holds 32 elements of a row, a warp each component.  The threads interpolate
// and integrate their own component; only the fluxes couple the components,
// so the states at the quadrature points and the face nodes pass through
// shared memory, where the block's warps share the points and leave the
// fluxes in the states' place.  One thread per element held 4 (p+1)^2
// coefficients and residuals at 128 registers with the rest in local memory
// and 16 warps per SM.
template <class R, int P, int NC>
struct ResSys {
    static constexpr int NQ = P + 2, QP = NQ * NQ, PTS = QP + 4 * P, TX = 32;  // quadrature points, then face nodes
    static constexpr int points = PTS * 2 * NC * TX;    // [point][f_x, f_y][component][element]
    static constexpr int faces = 4 * NC * (P + 1) * TX;  // boundary terms [face][component][node][element]
    static constexpr int ws = points + faces;
};
// slot of node k of face d among the 4 p face nodes: the rows below and above,
// then the sides between
template <int P>
DEV constexpr int face_slot(int d, int k) {
    return d == 2 ? k
                  : d == 3 ? P + 1 + k
                           : k == 0 ? (d == 0 ? 0 : P)
                                    : k == P ? P + 1 + (d == 0 ? 0 : P) : 2 * (P + 1) + 2 * (k - 1) + d;
}
template <class R, int P, class Ph>
__global__ void __launch_bounds__(32 * Ph::NC, sizeof(R) == 4 ? (P <= 2 ? 6 : P == 3 ? 4 : 3) : (P <= 2 ? 3 : 2))
    k_res_sys(MeshDev m, ProbDev pr, const R* __restrict__ u, const R* __restrict__ g, const double* __restrict__ gam,
              const double* __restrict__ nu, R* __restrict__ ER) {
    constexpr int NC = Ph::NC, N1 = P + 1, N2 = Dim<P>::N2, NQ = Dim<P>::NQ, TX = 32, NF = 2 * NC;
    using WS = ResSys<R, P, NC>;
    extern __shared__ __align__(16) unsigned char dyn_smem[];
    R(*sF)[NF][TX] = reinterpret_cast<R(*)[NF][TX]>(dyn_smem);
    R(*sB)[NC * N1][TX] = reinterpret_cast<R(*)[NC * N1][TX]>(reinterpret_cast<R*>(dyn_smem) + WS::points);
    pdl_begin();
    const int tx = threadIdx.x, c = threadIdx.y;
    const int ex = min(blockIdx.x * TX + tx, m.nx - 1), ey = blockIdx.y;  // a lane past the row repeats its last element
    const int e = ey * m.nx + ex;
    const Tab<R>& T = tab_of<R>(m, P);
    R W[N2], s[N2];
    {
        R U[N2];
        load_comp<R, P>(u + c * m.NN, m, ex, ey, U);
        R X[N1][NQ];
#pragma unroll
        for (int d = 0; d < N1; ++d)
#pragma unroll
            for (int q1 = 0; q1 < NQ; ++q1) {
                R v = R(0);
#pragma unroll
                for (int a = 0; a < N1; ++a) v += T.Bq[q1][a] * U[d * N1 + a];
                X[d][q1] = v;
            }
#pragma unroll
        for (int q2 = 0; q2 < NQ; ++q2)
#pragma unroll
            for (int q1 = 0; q1 < NQ; ++q1) {
                R v = R(0);
#pragma unroll
                for (int d = 0; d < N1; ++d) v += T.Bq[q2][d] * X[d][q1];
                sF[q2 * NQ + q1][c][tx] = v;
            }
#pragma unroll
        for (int d = 0; d < 4; ++d)
#pragma unroll
            for (int k = 0; k < N1; ++k)
                if (d >= 2 || (k > 0 && k < P)) sF[WS::QP + face_slot<P>(d, k)][c][tx] = U[face_node<P>(d, k)];
        // the component's stabilisation needs no other
        R GX[N2], GY[N2];
        load_comp<R, P>(g + c * m.NN, m, ex, ey, GX);
        load_comp<R, P>(g + (NC + c) * m.NN, m, ex, ey, GY);
        stab_comp<R, P>(m, T, U, GX, GY, bulk<R>(gam[e]) * PV<R>::h(m), bulk<R>(nu[e]), s);
    }
    // terms on the domain boundary: warp c takes face c, all components
    if (neighbour(m, ex, ey, c) < 0) {
        R Uf[NC][N1], term[NC][N1];
#pragma unroll
        for (int k = 0; k < NC; ++k) {
            const R* __restrict__ uk = u + k * m.NN;
#pragma unroll
            for (int j = 0; j < N1; ++j)
                Uf[k][j] = uk[node_of(m, ex, ey, c == 0 ? 0 : c == 1 ? P : j, c == 2 ? 0 : c == 3 ? P : j)];
        }
        boundary_face_term<R, P, Ph>(m, pr, c, ex, ey, &Uf[0][0], &term[0][0]);
#pragma unroll
        for (int k = 0; k < NC; ++k)
#pragma unroll
            for (int j = 0; j < N1; ++j) sB[c][k * N1 + j][tx] = term[k][j];
    }
    __syncthreads();
#pragma unroll 2
    for (int pt = c; pt < WS::PTS; pt += NC) {
        R uq[NC], fx[NC], fy[NC];
#pragma unroll
        for (int k = 0; k < NC; ++k) uq[k] = sF[pt][k][tx];
        Ph::template flux<R>(uq, fx, fy, pr);
#pragma unroll
        for (int k = 0; k < NC; ++k) {
            sF[pt][k][tx] = fx[k];
            sF[pt][NC + k][tx] = fy[k];
        }
    }
    __syncthreads();
#pragma unroll
    for (int i = 0; i < N2; ++i) W[i] = R(0);
#pragma unroll
    for (int q2 = 0; q2 < NQ; ++q2)
        volume_row<R, P>(T, q2, [&](int q) { return sF[q2 * NQ + q][c][tx]; },
                         [&](int q) { return sF[q2 * NQ + q][NC + c][tx]; }, W);
#pragma unroll
    for (int d = 0; d < 4; ++d) {
        if (neighbour(m, ex, ey, d) >= 0) {
            R fn[N1];
#pragma unroll
            for (int k = 0; k < N1; ++k) fn[k] = sF[WS::QP + face_slot<P>(d, k)][(d >> 1) * NC + c][tx];
#pragma unroll
            for (int b = 0; b < N1; ++b) {
                R t = R(0);
#pragma unroll
                for (int k = 0; k < N1; ++k) t += fn[k] * T.M[b][k];
                W[face_node<P>(d, b)] += (d & 1) ? -t : t;
            }
        } else {
#pragma unroll
            for (int b = 0; b < N1; ++b) W[face_node<P>(d, b)] -= sB[d][c * N1 + b][tx];
        }
    }
    const R h = PV<R>::h(m);
    if (blockIdx.x * TX + tx < m.nx) {
        R* __restrict__ out = ER + ((long long)c * m.E + e);
        const long long step = (long long)NC * m.E;
#pragma unroll
        for (int i = 0; i < N2; ++i, out += step) *out = h * W[i] - s[i];
    }
}

// ---------------------------------------------------------------------------
// The update: facet fluxes and flux limiter, ubar^e, f_i^e, beta_e and the
// element increments of eq. (eq:SSPupdate),
//   m_i u_i^SSP = sum_e m_i^e [(1 - theta_e) u_i + theta_e ubar_i^e]
//   <=> u_i^SSP = u_i + sum_e (m_i^e/m_i) theta_e (ubar^e - u_i + beta_e f_i^e/m_i^e),
// theta_e = dt/dt_e; the increment theta_e (...) is stored per (e, i).
// Per-node arithmetic is in R (float in the mixed form, the float64 values
// ubar^e and u^e enter as hi + lo float pairs); per-facet and per-element
// quantities are float64.
// ---------------------------------------------------------------------------
template <class T>
DEV void split(double v, T& hi, T& lo) {
    hi = T(v);
    lo = T(v - (double)hi);
}

// sum over the face nodes of F(u_j, u_hat_j; n) on a boundary face of side
// d that is not OUTFLOW everywhere (f^H of eq. (hoflux) before the division
// by p+1; on an LGL mesh the sum weighted by w_j, f^H itself), u_hat_j of
// the side at node j; Uf is [NC][p+1]
template <class R, int P, class Ph>
__device__ __noinline__ CompVec<R, Ph::NC> bnd_face_llf_sum(const MeshDev& m, const ProbDev& pr, int d, int e,
                                                           R nx, R ny, const R* Uf) {
    constexpr int NC = Ph::NC, N1 = P + 1;
    const bool split = side_split(pr, d);
    int ex = 0, ey = 0;
    if (split) {
        ey = e / m.nx;
        ex = e - ey * m.nx;
    }
    CompVec<R, NC> out;
    R* acc = out.v;
#pragma unroll
    for (int c = 0; c < NC; ++c) acc[c] = R(0);
    // a FIXED side with one part: one external state, its flux evaluated once
    const bool fixed1 = !split && pr.side[d].kind[0] == BC_FIXED;
    R ub1[NC], fxb[NC], fyb[NC];
    if (fixed1) {
#pragma unroll
        for (int c = 0; c < NC; ++c) ub1[c] = PV<R>::side_state(pr.side[d], 0, c);
        Ph::template flux<R>(ub1, fxb, fyb, pr);
    }
#pragma unroll
    for (int k = 0; k < N1; ++k) {
        R uk[NC], ub[NC], F[NC];
#pragma unroll
        for (int c = 0; c < NC; ++c) uk[c] = Uf[c * N1 + k];
        if (fixed1) {
            llf_given_fR<Ph, R>(uk, ub1, fxb, fyb, nx, ny, pr, F);
        } else {
            const int slot = split ? side_slot(pr, d, side_node_pos(m, d, ex, ey, k)) : 0;
            ext_state<R, NC>(pr, d, slot, uk, ub);
            llf<Ph, R>(uk, ub, nx, ny, pr, F, (R*)nullptr);
        }
        if (is_lgl<R>(m)) {
            const R wk = R(c_tabd[PMAX + 1 + P].wl[k]);
#pragma unroll
            for (int c = 0; c < NC; ++c) acc[c] += wk * F[c];
        } else {
#pragma unroll
            for (int c = 0; c < NC; ++c) acc[c] += F[c];
        }
    }
    return out;
}

// ubar^e in G: scalars umin <= ubar <= umax, Euler rho > 0 and
// rho E - |m|^2/2 > 0 (explicit float64 roundings, the same decision in
// every kernel)
template <class Ph>
DEV bool average_in_G(const ProbDev& pr, const double (&ub)[Ph::NC]) {
    if constexpr (Ph::NC == 1) {
        return ub[0] >= pr.umin && ub[0] <= pr.umax;
    } else {
        const double kin = __dmul_rn(0.5, __dadd_rn(__dmul_rn(ub[1], ub[1]), __dmul_rn(ub[2], ub[2])));
        return ub[0] > 0.0 && __dsub_rn(__dmul_rn(ub[0], ub[3]), kin) > 0.0;
    }
}

// An unlimited average ubar^e = u^e - r S_e (eq. (uebar), r = dt_e / h, S_e
// the outward sum of f^H) that left G: counted; with OPT_DTE_REDUCE the
// strategy of the remark after eq. (dtmaxcell): the largest r in [0, rs]
// with ubar^e in G (scalars: the crossed bound solved exactly; Euler: the
// Appendix-A criterion for u^e moved by -rs S_e, r = rs alpha).  Returns
// [ubar^e .., r].
template <class Ph>
__device__ __noinline__ CompVec<double, Ph::NC + 1> reduce_pseudo_step(const ProbDev& pr,
                                                                      const double (&ue)[Ph::NC],
                                                                      const double (&os)[Ph::NC], double rs,
                                                                      unsigned long long* __restrict__ cnt) {
    constexpr int NC = Ph::NC;
    atomicAdd(&cnt[CNT_UBAR], 1ull);
    CompVec<double, NC + 1> out;
    double r = rs;
    if (pr.opts & OPT_DTE_REDUCE) {
        if constexpr (NC == 1) {
            const double d = os[0];
            if (d < 0.0) r = fmin(r, (pr.umax - ue[0]) / (-d));
            if (d > 0.0) r = fmin(r, (ue[0] - pr.umin) / d);
            r = fmax(r, 0.0);
        } else {
            double g[NC];
#pragma unroll
            for (int c = 0; c < NC; ++c) g[c] = (-rs) * os[c];
            r = rs * euler_alpha<double>(ue, g, 1.0, pr.pos_eps);
        }
        if (r < rs) atomicAdd(&cnt[CNT_DTE_RED], 1ull);
    }
#pragma unroll
    for (int c = 0; c < NC; ++c) out.v[c] = ue[c] - r * os[c];
    out.v[NC] = r;
    return out;
}

// a pseudo time step decreased by the remark after eq. (dtmaxcell): the float
// speed sum that the element part reads is rounded up (its float dt_e never
// exceeds the reduced one)
DEV void store_reduced_step(const MeshDev& m, double* dte_a, float* cf, double rs2, int e) {
    const double dte2 = m.h * rs2;
    dte_a[e] = dte2;
    dte_a[off<1>(m.E, 1, e)] = rs2;
    dte_a[off<1>(m.E, 2, e)] = 1.0 / dte2;
    cf[e] = __double2float_ru(1.0 / rs2);
}

// facet part of the element update (scalars, and systems in the eq. (aecQ1)
// variant; k_facet_sys holds that of systems): canonical f^H, the flux limiter and
// ubar^e (eqs. (hoflux), (fAlim)/(uelim), Appendix A), and the facet term
// (h/(p+1)^2) sum_d +-f^H_d of the element contributions f_i^e (eq. (aec))
template <class R, int P, class Ph>
DEV void facet_part(const MeshDev& m, const ProbDev& pr, const R (&U)[Ph::NC][Dim<P>::N2], const int (&nb)[4],
                    const double (&uec)[Ph::NC], const double (&ublc)[Ph::NC], double rs,
                    const double* __restrict__ dte_a, const double* __restrict__ ubl,
                    const R* __restrict__ qcap, const R* __restrict__ fl_in, const float* cf, int e,
                    double (&ubec)[Ph::NC], R (&fh)[Ph::NC], double& rs_out,
                    unsigned long long* __restrict__ cnt) {
    constexpr int NC = Ph::NC, N1 = P + 1;
    rs_out = rs;
    // FP32-mixed systems: the limited facet fluxes enter ubar^e as float-float
    // terms (below), so f^H stays in float and no float64 copy is formed
    constexpr bool mixed_sys = sizeof(R) == 4 && NC > 1;
    const double h = m.h;
    // canonical high-order facet fluxes f^H (eq. (hoflux)): face average of
    // f(u_j).n (or of F(u_j, u_hat; n) on a FIXED boundary), summed along the
    // face in a fixed order so both cells of a facet get the same value
    double FH[4][NC];
    R FHr[4][NC];
    const bool need_fh = !(pr.mode == MODE_LO && pr.fl == FL_LOW);
    if (need_fh) {
#pragma unroll
        for (int d = 0; d < 4; ++d) {
            const R cnx = (d < 2) ? R(1) : R(0), cny = (d < 2) ? R(0) : R(1);
            const bool fixed_b = (nb[d] < 0) && !side_plain(pr, d);
            const R sg = (d == 1 || d == 3) ? R(1) : R(-1);
            R acc[NC];
#pragma unroll
            for (int c = 0; c < NC; ++c) acc[c] = R(0);
            if (fixed_b) {
                // boundary face with u_hat data: out of line (rare; keeps the hot code small)
                R Uf[NC * N1];
#pragma unroll
                for (int k = 0; k < N1; ++k) {
                    const int li = (d == 0) ? k * N1 : (d == 1) ? k * N1 + P : (d == 2) ? k : P * N1 + k;
#pragma unroll
                    for (int c = 0; c < NC; ++c) Uf[c * N1 + k] = U[c][li];
                }
                const CompVec<R, NC> fs = bnd_face_llf_sum<R, P, Ph>(m, pr, d, e, sg * cnx, sg * cny, Uf);
#pragma unroll
                for (int c = 0; c < NC; ++c) acc[c] = fs.v[c];  // acc was 0: same sums
            } else {
#pragma unroll
                for (int k = 0; k < N1; ++k) {
                    const int li = (d == 0) ? k * N1 : (d == 1) ? k * N1 + P : (d == 2) ? k : P * N1 + k;
                    R uk[NC], fn[NC];
#pragma unroll
                    for (int c = 0; c < NC; ++c) uk[c] = U[c][li];
                    Ph::template normal<R>(uk, d >> 1, fn, pr);
                    if (is_lgl<R>(m)) {
                        // LGL: the face mean weights node k by w_k
                        const R wk = R(c_tabd[PMAX + 1 + P].wl[k]);
#pragma unroll
                        for (int c = 0; c < NC; ++c) acc[c] += wk * fn[c];
                    } else {
#pragma unroll
                        for (int c = 0; c < NC; ++c) acc[c] += fn[c];
                    }
                }
            }
#pragma unroll
            for (int c = 0; c < NC; ++c) {
                const R a = is_lgl<R>(m) ? acc[c] : mul_r(acc[c], R(1.0 / N1));
                FHr[d][c] = fixed_b ? sg * a : a;
                if constexpr (!mixed_sys) FH[d][c] = (double)FHr[d][c];
            }
        }
    }
    // limited cell average ubar^e
    if (pr.fl == FL_LOW) {
#pragma unroll
        for (int c = 0; c < NC; ++c) ubec[c] = ublc[c];
    } else if (pr.fl == FL_NONE) {
        double osv[NC];
#pragma unroll
        for (int c = 0; c < NC; ++c) {
            double os;
            if constexpr (mixed_sys) {
                float osh, osl;
                ff_sum4(FHr[1][c], FHr[0][c], FHr[3][c], FHr[2][c], osh, osl);
                os = widen(osh) + widen(osl);
            } else {
                os = ((FH[1][c] - FH[0][c]) + FH[3][c]) - FH[2][c];
            }
            osv[c] = os;
            ubec[c] = uec[c] - rs * os;
        }
        // eq. (uebar) with the macrocell dt_e need not stay in G: count such
        // averages, and with the option decrease dt_e as the remark after
        // eq. (dtmaxcell) says (out of line: rare)
        if (!average_in_G<Ph>(pr, ubec)) {
            const CompVec<double, NC + 1> red = reduce_pseudo_step<Ph>(pr, uec, osv, rs, cnt);
#pragma unroll
            for (int c = 0; c < NC; ++c) ubec[c] = red.v[c];
            rs_out = red.v[NC];
        }
    } else {
        R FLr[4][NC];
#pragma unroll
        for (int d = 0; d < 4; ++d)
#pragma unroll
            for (int c = 0; c < NC; ++c) FLr[d][c] = fl_in[((long long)e * 4 + d) * NC + c];
        double FB[4][NC];
        R FBr[4];  // scalar limited fluxes in the bulk precision
        // mixed systems: facet d enters as the float pair (TH, TL) per
        // component: (f^L, -f^H) where alpha = 1 (certified in float, or
        // computed as 1 in float64: the same terms either way, so the
        // certificate changes no bit), else alpha f^A split into two floats
        float TH[mixed_sys ? 4 : 1][mixed_sys ? NC : 1], TL[mixed_sys ? 4 : 1][mixed_sys ? NC : 1];
#pragma unroll
        for (int d = 0; d < 4; ++d) {
            const bool self_is_L = (d == 1 || d == 3);
            const int Lc = self_is_L ? e : nb[d];
            const int Rc = self_is_L ? nb[d] : e;
            if (Ph::NC == 1) {
                // eq. (fAlim) with the capacities of both cells (R-typed; in the
                // mixed form they were rounded toward zero, so still admissible)
                const R fA = FLr[d][0] - FHr[d][0];
                const R inf = R(__int_as_float(0x7f800000));
                R fmaxv = inf, fminv = -inf;
                if (Lc >= 0) {
                    fmaxv = fmin(fmaxv, qcap[Lc]);
                    fminv = fmax(fminv, qcap[off<NC>(m.E, 1, Lc)]);
                }
                if (Rc >= 0) {
                    fmaxv = fmin(fmaxv, -qcap[off<NC>(m.E, 1, Rc)]);
                    fminv = fmax(fminv, -qcap[Rc]);
                }
                FBr[d] = (fA >= R(0)) ? fmin(fA, fmaxv) : fmax(fA, fminv);
                if constexpr (sizeof(R) == 8) FB[d][0] = FBr[d];
            } else {
                double fA[NC];
#pragma unroll
                for (int c = 0; c < NC; ++c) fA[c] = (double)FLr[d][c] - (double)FHr[d][c];
                // float32 certificate first: where both cells certainly give
                // alpha = 1 the float64 formula is skipped (same result; in
                // the float64 form too, where it is 100 float64 instructions
                // a facet against 4 conversions)
                if (!(pr.opts & OPT_FP64_LIMITER)) {
                    float fAf[NC], fAm[NC], ub[NC];
#pragma unroll
                    for (int c = 0; c < NC; ++c) {
                        fAf[c] = sizeof(R) == 4 ? __fsub_rn((float)FLr[d][c], (float)FHr[d][c]) : cert_float(fA[c]);
                        fAm[c] = -fAf[c];
                    }
                    bool one = true;
                    if (Lc >= 0) {
#pragma unroll
                        for (int c = 0; c < NC; ++c) ub[c] = cf[off<NC>(m.E, 1 + c, Lc)];
                        one = euler_alpha_is_one<R>(ub, fAf, 0.25f * cf[Lc], pr.ome_f);
                    }
                    if (one && Rc >= 0) {
#pragma unroll
                        for (int c = 0; c < NC; ++c) ub[c] = cf[off<NC>(m.E, 1 + c, Rc)];
                        one = euler_alpha_is_one<R>(ub, fAm, 0.25f * cf[Rc], pr.ome_f);
                    }
                    if (one) {
#pragma unroll
                        for (int c = 0; c < NC; ++c) {
                            if constexpr (mixed_sys) {
                                TH[d][c] = FLr[d][c];
                                TL[d][c] = -FHr[d][c];
                            } else {
                                FB[d][c] = fA[c];
                            }
                        }
                        continue;
                    }
                }
                double alpha = 1.0;
                if (Lc >= 0) {
                    double ub[NC];
#pragma unroll
                    for (int c = 0; c < NC; ++c) ub[c] = ubl[c * m.E + Lc];
                    double mL = (0.25 * h) * dte_a[off<NC>(m.E, 2, Lc)];
                    alpha = fmin(alpha, euler_alpha<double>(ub, fA, mL, pr.pos_eps));
                }
                if (Rc >= 0) {
                    double ub[NC], fm[NC];
#pragma unroll
                    for (int c = 0; c < NC; ++c) {
                        ub[c] = ubl[c * m.E + Rc];
                        fm[c] = -fA[c];
                    }
                    double mR = (0.25 * h) * dte_a[off<NC>(m.E, 2, Rc)];
                    alpha = fmin(alpha, euler_alpha<double>(ub, fm, mR, pr.pos_eps));
                }
                if constexpr (mixed_sys) {
#pragma unroll
                    for (int c = 0; c < NC; ++c) {
                        if (alpha == 1.0) {
                            TH[d][c] = FLr[d][c];
                            TL[d][c] = -FHr[d][c];
                        } else {
                            const double v = alpha * fA[c];
                            TH[d][c] = __double2float_rn(v);
                            TL[d][c] = __double2float_rn(v - (double)TH[d][c]);
                        }
                    }
                } else {
#pragma unroll
                    for (int c = 0; c < NC; ++c) FB[d][c] = alpha * fA[c];
                }
            }
        }
#pragma unroll
        for (int c = 0; c < NC; ++c) {
            double os;
            if constexpr (sizeof(R) == 4 && Ph::NC == 1) {
                // float limited fluxes summed as a float-float pair, widened once
                float osh, osl;
                ff_sum4(FBr[1], FBr[0], FBr[3], FBr[2], osh, osl);
                os = widen(osh) + widen(osl);
            } else if constexpr (mixed_sys) {
                // (fbar_E - fbar_W) + fbar_N - fbar_S from the eight float terms,
                // compensated, widened once
                const float t[8] = {TH[1][c], TL[1][c], -TH[0][c], -TL[0][c],
                                    TH[3][c], TL[3][c], -TH[2][c], -TL[2][c]};
                float osh, osl;
                ff_sum<8>(t, osh, osl);
                os = widen(osh) + widen(osl);
            } else {
                os = ((FB[1][c] - FB[0][c]) + FB[3][c]) - FB[2][c];
            }
            ubec[c] = ublc[c] + rs * os;
        }
    }
    // (m_i^e / |K_e|) |S| times the outward sum of f^H, the facet term of
    // eq. (aecb): h / (p+1)^2 for every node (Bernstein); on an LGL mesh h,
    // weighted by w_a w_b per node in element_part
    const R h_over_n2R = (sizeof(R) == 4) ? R(m.h_over_n2_f) : (is_lgl<R>(m) ? R(m.h) : R(m.h_over_n2));
#pragma unroll
    for (int c = 0; c < NC; ++c)
        fh[c] = need_fh ? h_over_n2R * (((FHr[1][c] - FHr[0][c]) + FHr[3][c]) - FHr[2][c]) : R(0);
}

// element part of the update: theta, f_i^e (eq. (aec)), the slope limiter
// beta_e (eqs. (slimit1), (slimit2), Appendix A) and the SSP increments
// Q1: the variant of eq. (aecQ1); the caller passes ER = -D_i (the
// divergence term), ud = udot^L and fh = 0, and the contributions are scaled
// by gamma_e (gq)
template <class R, int P, class Ph, bool Q1 = false>
DEV void element_part(const MeshDev& m, const ProbDev& pr, const R (&U)[Ph::NC][Dim<P>::N2],
                      const R* __restrict__ ud, const R* __restrict__ ER, const float* __restrict__ cf,
                      const float* __restrict__ avg, const double (&uec)[Ph::NC], double dt, double dte, double rdte,
                      const double (&ubec)[Ph::NC], const R (&fh)[Ph::NC], R* __restrict__ EW,
                      double* __restrict__ beta_out, unsigned long long* __restrict__ cnt, int ex, int ey, int e,
                      double gq = 1.0) {
    constexpr int NC = Ph::NC, N1 = P + 1, N2 = Dim<P>::N2;
    const Tab<R>& T = tab_of<R>(m, P);
    const double me = m.me;
    // theta = dt / dt_e = dt s / h; FP32-mixed: in float from the float
    // speed sum of the low-order part (it weights float increments; the check counts only)
    R thR;
    if constexpr (sizeof(R) == 4) {
        thR = __fmul_rn((float)dt, __fmul_rn(cf[e], m.inv_h_f));
        if (thR > 1.f) atomicAdd(&cnt[CNT_CFL], 1ull);
    } else {
        const double theta = dt * rdte;
        if (theta > 1.0) atomicAdd(&cnt[CNT_CFL], 1ull);
        thR = R(theta);
    }
    R ubh[NC], ubo[NC];
#pragma unroll
    for (int c = 0; c < NC; ++c) split<R>(ubec[c], ubh[c], ubo[c]);
    if (pr.mode == MODE_LO) {
#pragma unroll
        for (int c = 0; c < NC; ++c)
#pragma unroll
            for (int i = 0; i < N2; ++i)
                EW[ev_at(m.E, e, i, c, NC)] = thR * ((ubh[c] - U[c][i]) + ubo[c]);
        beta_out[e] = 0.0;
        return;
    }
    // f_i^e, eq. (aec) with eq. (aecb) folded into the residual
    const R meR = PV<R>::me(m), h2 = PV<R>::h2(m), inv_meR = PV<R>::inv_me(m);
    // LGL mesh (float64 form): m_i^e = h^2 w_a w_b and 1/m_i^e per node, the
    // facet term fh weighted by w_a w_b (see facet_part)
    const bool lgl = is_lgl<R>(m);
    const Tab<double>& TL = c_tabd[PMAX + 1 + P];
    R dteR;
    if constexpr (sizeof(R) == 4) dteR = __fmul_rn(m.h_f, __frcp_rn(cf[e]));  // h / s in float
    else dteR = R(dte);
    R F[NC][N2];
    // components unrolled for p >= 3 (registers); at p <= 2 the rolled loop
    // keeps occupancy higher (measured on the Euler workloads)
#pragma unroll (P >= 3 ? Ph::NC : 1)
    for (int c = 0; c < NC; ++c) {
        R UD[N2];
        load_comp<R, P>(ud + c * m.NN, m, ex, ey, UD);
        R Y[N1][N1];
#pragma unroll
        for (int d = 0; d < N1; ++d)
#pragma unroll
            for (int a = 0; a < N1; ++a) {
                R s = R(0);
#pragma unroll
                for (int k = 0; k < N1; ++k) s += T.M[a][k] * UD[d * N1 + k];
                Y[d][a] = s;
            }
        const R fh_term = fh[c];
        R ueh, uel;
        if constexpr (sizeof(R) == 4) {
            // the float-float mean itself (k_lo for scalars, k_avg for systems)
            ueh = avg[off<NC>(m.E, 2 * c, e)];
            uel = avg[off<NC>(m.E, 2 * c + 1, e)];
        } else {
            split<R>(uec[c], ueh, uel);
        }
#pragma unroll
        for (int b = 0; b < N1; ++b)
#pragma unroll
            for (int a = 0; a < N1; ++a) {
                R s = R(0);
#pragma unroll
                for (int d = 0; d < N1; ++d) s += T.M[b][d] * Y[d][a];
                const int i = b * N1 + a;
                R Ri = ER[ev_at(m.E, e, i, c, NC)];
                R dev = (U[c][i] - ueh) - uel;
                if (lgl) {
                    const R w2 = R(TL.wl[a] * TL.wl[b]);
                    const R mi = h2 * w2;
                    F[c][i] = mi * dev + dteR * (((Ri + fh_term * w2) - h2 * s) + mi * UD[i]);
                } else {
                    F[c][i] = meR * dev + dteR * (((Ri + fh_term) - h2 * s) + meR * UD[i]);
                }
                if constexpr (Q1) F[c][i] = R(gq) * F[c][i];
            }
    }
    // slope limiter beta_e
    R beta = R(1);
    if (pr.mode == MODE_WENO_L) {
        if (Ph::NC == 1) {
            // bound gaps in float64 per element, ratios per node in R
            R gp, gm;
            if constexpr (sizeof(R) == 4) {
                // gaps in float64; m_i^e, the gaps and the products rounded
                // toward zero (smaller magnitudes stay admissible)
                gp = __fmul_rz(m.me_rz_f, __double2float_rz(pr.umax - ubec[0]));
                gm = __fmul_rz(m.me_rz_f, __double2float_rz(pr.umin - ubec[0]));
            } else {
                gp = R(me * (pr.umax - ubec[0]));
                gm = R(me * (pr.umin - ubec[0]));
            }
            R b = R(1);
            if (!lgl) {
                // the gaps are the same for every node and the quotients
                // monotone: the smallest comes from the extreme contributions
                R hi = R(0), lo = R(0);
#pragma unroll
                for (int i = 0; i < N2; ++i) {
                    hi = fmax(hi, F[0][i]);
                    lo = fmin(lo, F[0][i]);
                }
                if (hi > R(0)) b = fmin(b, gp / hi);
                if (lo < R(0)) b = fmin(b, gm / lo);
            } else {
#pragma unroll
                for (int i = 0; i < N2; ++i) {
                    const R f = F[0][i];
                    // m_i^e of this node (the gaps scale with it)
                    const double mi = m.h * m.h * (TL.wl[i % N1] * TL.wl[i / N1]);
                    R bi = R(1);
                    if (f > R(0)) bi = fmin(R(1), R(mi * (pr.umax - ubec[0])) / f);
                    else if (f < R(0)) bi = fmin(R(1), R(mi * (pr.umin - ubec[0])) / f);
                    b = fmin(b, bi);
                }
            }
            beta = fmin(fmax(b, R(0)), R(1));
        } else {
            double b = 1.0;
            float ubf[NC];
            const bool cert = (sizeof(R) == 4) && !(pr.opts & OPT_FP64_LIMITER);
#pragma unroll
            for (int c = 0; c < NC; ++c) ubf[c] = cert ? (float)ubec[c] : 0.f;
#pragma unroll
            for (int i = 0; i < N2; ++i) {
                // float32 certificate first; the float64 formula only where
                // it cannot show alpha_i = 1 (min(b, 1) = b: same result)
                if (cert) {
                    float ff[NC];
#pragma unroll
                    for (int c = 0; c < NC; ++c) ff[c] = (float)F[c][i];
                    if (euler_alpha_is_one<R>(ubf, ff, m.me_f, pr.ome_f)) continue;
                }
                double f[NC];
#pragma unroll
                for (int c = 0; c < NC; ++c) f[c] = (double)F[c][i];
                const double mi = lgl ? m.h * m.h * (TL.wl[i % N1] * TL.wl[i / N1]) : me;
                b = fmin(b, euler_alpha_of<R>(ubec, f, mi, pr.pos_eps));
            }
            beta = R(b);
        }
    }
    if constexpr (sizeof(R) == 4) beta_out[e] = widen(beta);
    else beta_out[e] = beta;
#pragma unroll
    for (int c = 0; c < NC; ++c)
#pragma unroll
        for (int i = 0; i < N2; ++i) {
            const R inv_mi = lgl ? R(m.inv_h2 * (TL.iwl[i % N1] * TL.iwl[i / N1])) : inv_meR;
            EW[ev_at(m.E, e, i, c, NC)] = thR * (((ubh[c] - U[c][i]) + ubo[c]) + (beta * F[c][i]) * inv_mi);
        }
}

template <class R, int P, class Ph>
DEV void update_at(const MeshDev& m, const ProbDev& pr, const R* __restrict__ u, const R* __restrict__ ud,
                            const double* __restrict__ ue, double* dte_a,
                            const double* __restrict__ ubl,
                            const R* __restrict__ qcap, const R* __restrict__ fl_in,
                            const R* __restrict__ ER, const float* __restrict__ cf,
                            const float* __restrict__ avg,
                            const double* __restrict__ dtp, R* __restrict__ EW,
                            double* __restrict__ ube_out, double* __restrict__ beta_out,
                            unsigned long long* __restrict__ cnt, int ex, int ey, int e) {
    constexpr int NC = Ph::NC, N1 = P + 1, N2 = Dim<P>::N2;
    const Tab<R>& T = tab_of<R>(m, P);
    const double h = m.h;
    const double me = m.me;
    const double dt = *dtp;
    const double dte = dte_a[e];
    const double rs = dte_a[off<NC>(m.E, 1, e)];       // dt_e / h
    const double rdte = dte_a[off<NC>(m.E, 2, e)]; // 1 / dt_e
    int nb[4];
#pragma unroll
    for (int d = 0; d < 4; ++d) nb[d] = neighbour(m, ex, ey, d);
    R U[NC][N2];
    load_block<R, P, NC>(u, m, ex, ey, U);
    double uec[NC], ublc[NC];
#pragma unroll
    for (int c = 0; c < NC; ++c) {
        uec[c] = ue[c * m.E + e];
        ublc[c] = ubl[c * m.E + e];
    }
    double ubec[NC];
    R fh[NC];
    double rs2;
    facet_part<R, P, Ph>(m, pr, U, nb, uec, ublc, rs, dte_a, ubl, qcap, fl_in, cf, e, ubec, fh, rs2, cnt);
#pragma unroll
    for (int c = 0; c < NC; ++c) ube_out[c * m.E + e] = ubec[c];
    if (rs2 != rs) {
        // a pseudo time step decreased by the remark after eq. (dtmaxcell)
        const double dte2 = h * rs2;
        dte_a[e] = dte2;
        dte_a[off<NC>(m.E, 1, e)] = rs2;
        dte_a[off<NC>(m.E, 2, e)] = 1.0 / dte2;
        element_part<R, P, Ph>(m, pr, U, ud, ER, cf, avg, uec, dt, dte2, 1.0 / dte2, ubec, fh, EW, beta_out, cnt, ex,
                               ey, e);
        return;
    }
    element_part<R, P, Ph>(m, pr, U, ud, ER, cf, avg, uec, dt, dte, rdte, ubec, fh, EW, beta_out, cnt, ex, ey, e);
}

// ---------------------------------------------------------------------------
// The Q1 variant, eq. (aecQ1) (option OPT_AEC_Q1):
//   f_i^e = gamma_e ( m_i^e (u_i - u^e) - dt_e [ D_i + (M udot^L)_i - m_i^e udot^L_i ] ),
//   D_i = int (phi_i - m_i^e/|K_e|) div f_h,  f_h = sum_j f(u_j) phi_j,
// udot^L from the low-order scheme, eq. (weak:low2).  Three kernels replace
// the g_h, residual and udot kernels: k_q1_facet (ubar^e and -D_i),
// k_udl (udot^L at the nodes) and k_q1_update (the element part of the
// update with ER = -D_i, udot := udot^L, no facet term, scaled by gamma_e).
// ---------------------------------------------------------------------------
template <class R, int P, class Ph>
__global__ void __launch_bounds__(128) k_q1_facet(MeshDev m, ProbDev pr, const R* __restrict__ u,
                                                  const double* __restrict__ ue, const double* __restrict__ dte_a,
                                                  const double* __restrict__ ubl, const R* __restrict__ qcap,
                                                  const R* __restrict__ fl_in, const float* __restrict__ cf,
                                                  R* __restrict__ ER, double* __restrict__ ube_out,
                                                  unsigned long long* __restrict__ cnt) {
    pdl_begin();
    int ex, ey, e;
    if (!elem_of_thread(m, ex, ey, e)) return;
    constexpr int NC = Ph::NC, N1 = P + 1, N2 = Dim<P>::N2;
    const Tab<R>& T = tab_of<R>(m, P);
    int nb[4];
#pragma unroll
    for (int d = 0; d < 4; ++d) nb[d] = neighbour(m, ex, ey, d);
    R U[NC][N2];
    load_block<R, P, NC>(u, m, ex, ey, U);
    double uec[NC], ublc[NC];
#pragma unroll
    for (int c = 0; c < NC; ++c) {
        uec[c] = ue[c * m.E + e];
        ublc[c] = ubl[c * m.E + e];
    }
    double ubec[NC];
    R fh[NC];
    double rs2;  // eq. (aecQ1) is not combined with the pseudo-time-step reduction
    facet_part<R, P, Ph>(m, pr, U, nb, uec, ublc, dte_a[off<NC>(m.E, 1, e)], dte_a, ubl, qcap, fl_in, cf, e, ubec, fh, rs2,
                         cnt);
#pragma unroll
    for (int c = 0; c < NC; ++c) ube_out[c * m.E + e] = ubec[c];
    // nodal fluxes f(u_j)
    R FX[NC][N2], FY[NC][N2];
#pragma unroll
    for (int j = 0; j < N2; ++j) {
        R uj[NC], fx[NC], fy[NC];
#pragma unroll
        for (int c = 0; c < NC; ++c) uj[c] = U[c][j];
        Ph::template flux<R>(uj, fx, fy, pr);
#pragma unroll
        for (int c = 0; c < NC; ++c) {
            FX[c][j] = fx[c];
            FY[c][j] = fy[c];
        }
    }
    // int phi_i d_x phi_j = h int B_a B_c' int B_b B_d (C[c][a] = int B_c' B_a),
    // int d_x phi_j = sum_i of it; the same with x and y exchanged
    const R h = PV<R>::h(m);
    R csum[N1], msum[N1];
#pragma unroll
    for (int c = 0; c < N1; ++c) {
        R s1 = R(0), s2 = R(0);
#pragma unroll
        for (int a = 0; a < N1; ++a) {
            s1 += T.C[c][a];
            s2 += T.M[a][c];
        }
        csum[c] = s1;
        msum[c] = s2;
    }
    const R inv_n2 = R(1) / R(N2);
#pragma unroll
    for (int c = 0; c < NC; ++c) {
        // mean term (m_i^e/|K_e|) sum_j c_j . f(u_j), the same for every i
        R mean = R(0);
#pragma unroll
        for (int d = 0; d < N1; ++d)
#pragma unroll
            for (int cc = 0; cc < N1; ++cc)
                mean += (csum[cc] * msum[d]) * FX[c][d * N1 + cc] + (msum[cc] * csum[d]) * FY[c][d * N1 + cc];
        mean = h * mean * inv_n2;
#pragma unroll
        for (int b = 0; b < N1; ++b)
#pragma unroll
            for (int a = 0; a < N1; ++a) {
                R s = R(0);
#pragma unroll
                for (int d = 0; d < N1; ++d)
#pragma unroll
                    for (int cc = 0; cc < N1; ++cc)
                        s += (T.C[cc][a] * T.M[b][d]) * FX[c][d * N1 + cc] + (T.M[a][cc] * T.C[d][b]) * FY[c][d * N1 + cc];
                ER[ev_at(m.E, e, b * N1 + a, c, NC)] = -(h * s - mean);
            }
    }
}

// udot^L_i = (1/|E_i|) sum_{e in E_i} (ubar^e - u_i) / dt_e, eq. (weak:low2)
// with m_i = |E_i| m_i^e (float64 sums, fixed order)
template <class R, int P, int NC>
__global__ void k_udl(MeshDev m, const R* __restrict__ u, const double* __restrict__ ube,
                      const double* __restrict__ dte_a, R* __restrict__ ud) {
    pdl_begin();
    int gx, gy;
    long long node;
    if (!node_of_thread(m, gx, gy, node)) return;
    const NodeC<P> c = node_c<P>(m, gx, gy);
    const double w = inv_count<double>(c.nxc * c.nyc);
#pragma unroll
    for (int k = 0; k < NC; ++k) {
        const double ui = (double)u[(long long)k * m.NN + node];
        double s = 0.0;
#pragma unroll
        for (int j = 0; j < 2; ++j) {
            if (j < c.nyc) {
                const int ey = j ? c.ey1 : c.ey0;
#pragma unroll
                for (int i = 0; i < 2; ++i) {
                    if (i < c.nxc) {
                        const int e = ey * m.nx + (i ? c.ex1 : c.ex0);
                        s += (ube[k * m.E + e] - ui) * dte_a[off<NC>(m.E, 2, e)];
                    }
                }
            }
        }
        ud[(long long)k * m.NN + node] = R(s * w);
    }
}

template <class R, int P, class Ph>
__global__ void __launch_bounds__(128) k_q1_update(MeshDev m, ProbDev pr, const R* __restrict__ u,
                                                   const R* __restrict__ udl, const double* __restrict__ ue,
                                                   const double* __restrict__ dte_a, const R* __restrict__ ER,
                                                   const float* __restrict__ cf, const float* __restrict__ avg,
                                                   const double* __restrict__ ube, const double* __restrict__ gam,
                                                   const double* __restrict__ dtp, R* __restrict__ EW,
                                                   double* __restrict__ beta_out, unsigned long long* __restrict__ cnt) {
    pdl_begin();
    int ex, ey, e;
    if (!elem_of_thread(m, ex, ey, e)) return;
    constexpr int NC = Ph::NC, N2 = Dim<P>::N2;
    R U[NC][N2];
    load_block<R, P, NC>(u, m, ex, ey, U);
    double uec[NC], ubec[NC];
    R fh[NC];
#pragma unroll
    for (int c = 0; c < NC; ++c) {
        uec[c] = ue[c * m.E + e];
        ubec[c] = ube[c * m.E + e];
        fh[c] = R(0);
    }
    element_part<R, P, Ph, true>(m, pr, U, udl, ER, cf, avg, uec, *dtp, dte_a[e], dte_a[off<NC>(m.E, 2, e)], ubec, fh, EW,
                                 beta_out, cnt, ex, ey, e, gam[e]);
}

// Scalars: the update in two kernels.  k_facet needs only u and the outputs of
// k_lo, so it runs on the low-order stream beside the g_h and udot kernels;
// k_update_el then reads its ubar^e and facet terms.  The bodies are
// device functions of one element, also run by the batched stage.
template <class R, int P, class Ph>
DEV void facet_el_at(const MeshDev& m, const ProbDev& pr, const R* __restrict__ u,
                     const double* __restrict__ ue, double* dte_a, const double* __restrict__ ubl,
                     const R* __restrict__ qcap, const R* __restrict__ fl_in, float* cf,
                     double* __restrict__ ube_out, R* __restrict__ fht, unsigned long long* __restrict__ cnt,
                     int ex, int ey, int e) {
    constexpr int N2 = Dim<P>::N2;
    int nb[4];
#pragma unroll
    for (int d = 0; d < 4; ++d) nb[d] = neighbour(m, ex, ey, d);
    R U[1][N2];
    load_block<R, P, 1>(u, m, ex, ey, U);
    double uec[1], ublc[1], ubec[1];
    R fh[1];
    uec[0] = pr.fl == FL_NONE ? ue[e] : 0.0;  // u^e enters ubar^e only without the flux limiter
    ublc[0] = ubl[e];
    const double rs = dte_a[off<1>(m.E, 1, e)];
    double rs2;
    facet_part<R, P, Ph>(m, pr, U, nb, uec, ublc, rs, dte_a, ubl, qcap, fl_in, cf, e, ubec, fh, rs2, cnt);
    ube_out[e] = ubec[0];
    fht[e] = fh[0];
    if (rs2 != rs) store_reduced_step(m, dte_a, cf, rs2, e);
}

template <class R, int P, class Ph>
DEV void update_el_at(const MeshDev& m, const ProbDev& pr, const R* __restrict__ u,
                      const R* __restrict__ ud, const double* __restrict__ ue, const double* __restrict__ dte_a,
                      const R* __restrict__ ER, const float* __restrict__ cf,
                      const float* __restrict__ avg, const double* __restrict__ ube,
                      const R* __restrict__ fht, const double* __restrict__ dtp, R* __restrict__ EW,
                      double* __restrict__ beta_out, unsigned long long* __restrict__ cnt, int ex, int ey, int e) {
    constexpr int N2 = Dim<P>::N2;
    R U[1][N2];
    load_block<R, P, 1>(u, m, ex, ey, U);
    const double ubec[1] = {ube[e]};
    const R fh[1] = {fht[e]};
    // the float path of element_part takes dt_e and theta from the float
    // speed sum and the mean from the float-float pair
    if constexpr (sizeof(R) == 4) {
        const double uec[1] = {0.0};
        element_part<R, P, Ph>(m, pr, U, ud, ER, cf, avg, uec, *dtp, 0.0, 0.0, ubec, fh, EW, beta_out, cnt, ex, ey, e);
    } else {
        const double uec[1] = {ue[e]};
        element_part<R, P, Ph>(m, pr, U, ud, ER, cf, avg, uec, *dtp, dte_a[e], dte_a[off<1>(m.E, 2, e)], ubec, fh, EW, beta_out,
                               cnt, ex, ey, e);
    }
}

template <class R, int P, class Ph>
__global__ void __launch_bounds__(128) k_facet(MeshDev m, ProbDev pr, const R* __restrict__ u,
                                               const double* __restrict__ ue, double* dte_a,
                                               const double* __restrict__ ubl, const R* __restrict__ qcap,
                                               const R* __restrict__ fl_in, float* cf,
                                               double* __restrict__ ube_out, R* __restrict__ fht,
                                               unsigned long long* __restrict__ cnt) {
    pdl_begin();
    int ex, ey, e;
    if (!elem_of_thread(m, ex, ey, e)) return;
    facet_el_at<R, P, Ph>(m, pr, u, ue, dte_a, ubl, qcap, fl_in, cf, ube_out, fht, cnt, ex, ey, e);
}

template <class R, int P, class Ph>
__global__ void __launch_bounds__(128)
    k_update_el(MeshDev m, ProbDev pr, const R* __restrict__ u, const R* __restrict__ ud,
                const double* __restrict__ ue, const double* __restrict__ dte_a, const R* __restrict__ ER,
                const float* __restrict__ cf, const float* __restrict__ avg, const double* __restrict__ ube,
                const R* __restrict__ fht, const double* __restrict__ dtp, R* __restrict__ EW,
                double* __restrict__ beta_out, unsigned long long* __restrict__ cnt) {
    pdl_begin();
    int ex, ey, e;
    if (!elem_of_thread(m, ex, ey, e)) return;
    update_el_at<R, P, Ph>(m, pr, u, ud, ue, dte_a, ER, cf, avg, ube, fht, dtp, EW, beta_out, cnt, ex, ey, e);
}

// The facet part of the update of systems: f^H (eq. (hoflux)), the facet
// limiter of Appendix A, ubar^e (eqs. (uebar), (uelim), (uebar2)) and the
// facet terms of f_i^e.  As in k_lo_sys each facet of a tile is evaluated once
// (f^H from its p + 1 nodes, the positivity factors of its two cells) and the
// elements take its terms from shared memory.  A limited facet enters ubar^e
// as two terms T0 + T1: (f^L, -f^H) where alpha = 1 (certified in float, or
// computed as 1 in float64: the same terms either way, so the certificate
// changes no bit), else alpha f^A, split into two floats in the FP32-mixed
// form; the eight float terms are summed as a compensated pair.
template <class R, int P, class Ph>
__global__ void __launch_bounds__(F_NT, sizeof(R) == 4 ? 6 : 3)
    k_facet_sys(MeshDev m, ProbDev pr, const R* __restrict__ u, const double* __restrict__ ue, double* dte_a,
                const double* __restrict__ ubl, const R* __restrict__ fl_in, float* cf, double* __restrict__ ube_out,
                R* __restrict__ fht, unsigned long long* __restrict__ cnt) {
    constexpr int NC = Ph::NC, N1 = P + 1, NFC = F_N;
    constexpr int NTERM = sizeof(R) == 4 ? 3 : 2;  // f^H, and T0, T1 (float64: their sum)
    __shared__ R sT[NTERM][NC][NFC];
    pdl_begin();
    const int tx = threadIdx.x, ty = threadIdx.y, ex0 = blockIdx.x * F_TX, ey0 = blockIdx.y * F_TY;
    const int E = m.E;
    const bool need_fh = !(pr.mode == MODE_LO && pr.fl == FL_LOW);
    if (need_fh) {
#pragma unroll 1
        for (int axis = 0; axis < 2; ++axis) {
            FacetItem f;
            if (!facet_item(m, ex0, ey0, axis, f)) continue;
            const int i = f.slot;
            // the face's coefficients
            R Uf[NC * N1];
            {
                const int gx0 = f.ex * P + (f.d == 1 ? P : 0), gy0 = f.ey * P + (f.d == 3 ? P : 0);
#pragma unroll
                for (int k = 0; k < N1; ++k) {
                    int gx = gx0 + (f.axis == 0 ? 0 : k), gy = gy0 + (f.axis == 0 ? k : 0);
                    if (m.px && gx == m.nnx) gx = 0;
                    if (m.py && gy == m.nny) gy = 0;
                    const R* __restrict__ un = u + ((long long)gy * m.nnx + gx);
#pragma unroll
                    for (int c = 0; c < NC; ++c) Uf[c * N1 + k] = un[c * m.NN];
                }
            }
            const bool bnd = f.eL < 0 || f.eR < 0;
            R FH[NC];
            if (bnd && !side_plain(pr, f.d)) {
                // boundary data u_hat: out of line (rare)
                const R sg = (f.d & 1) ? R(1) : R(-1);
                const CompVec<R, NC> fs = bnd_face_llf_sum<R, P, Ph>(m, pr, f.d, f.ey * m.nx + f.ex, f.axis == 0 ? sg : R(0),
                                                                     f.axis == 0 ? R(0) : sg, Uf);
#pragma unroll
                for (int c = 0; c < NC; ++c) FH[c] = sg * (is_lgl<R>(m) ? fs.v[c] : mul_r(fs.v[c], R(1.0 / N1)));
            } else {
#pragma unroll
                for (int c = 0; c < NC; ++c) FH[c] = R(0);
#pragma unroll
                for (int k = 0; k < N1; ++k) {
                    R uk[NC], fn[NC];
#pragma unroll
                    for (int c = 0; c < NC; ++c) uk[c] = Uf[c * N1 + k];
                    Ph::template normal<R>(uk, f.axis, fn, pr);
                    const R wk = is_lgl<R>(m) ? R(c_tabd[PMAX + 1 + P].wl[k]) : R(1);
#pragma unroll
                    for (int c = 0; c < NC; ++c) FH[c] += is_lgl<R>(m) ? wk * fn[c] : fn[c];
                }
                if (!is_lgl<R>(m)) {
#pragma unroll
                    for (int c = 0; c < NC; ++c) FH[c] = mul_r(FH[c], R(1.0 / N1));
                }
            }
#pragma unroll
            for (int c = 0; c < NC; ++c) sT[0][c][i] = FH[c];
            if (pr.fl != FL_LIMITED) continue;
            R FL[NC], T0[NC], T1[NC];
            load_facet<R, NC>(fl_in, (long long)(f.ey * m.nx + f.ex) * 4 + f.d, FL);
#pragma unroll
            for (int c = 0; c < NC; ++c) {
                T0[c] = FL[c];
                T1[c] = -FH[c];
            }
            // float32 certificate first: where both cells certainly give alpha
            // = 1 the float64 formula is skipped (same result; in the float64
            // form it is some 100 float64 instructions a facet)
            bool one = !(pr.opts & OPT_FP64_LIMITER);
            if (one) {
                float fA[NC], ub[NC];
#pragma unroll
                for (int c = 0; c < NC; ++c)
                    fA[c] = sizeof(R) == 4 ? __fsub_rn((float)FL[c], (float)FH[c]) : cert_float((double)FL[c] - (double)FH[c]);
                if (f.eL >= 0) {
#pragma unroll
                    for (int c = 0; c < NC; ++c) ub[c] = cf[off<NC>(E, 1 + c, f.eL)];
                    one = euler_alpha_is_one<R>(ub, fA, 0.25f * cf[f.eL], pr.ome_f);
                }
                if (one && f.eR >= 0) {
#pragma unroll
                    for (int c = 0; c < NC; ++c) {
                        ub[c] = cf[off<NC>(E, 1 + c, f.eR)];
                        fA[c] = -fA[c];
                    }
                    one = euler_alpha_is_one<R>(ub, fA, 0.25f * cf[f.eR], pr.ome_f);
                }
            }
            if (!one) {
                double alpha = 1.0, fA[NC], ub[NC];
#pragma unroll
                for (int c = 0; c < NC; ++c) fA[c] = (double)FL[c] - (double)FH[c];
                if (f.eL >= 0) {
#pragma unroll
                    for (int c = 0; c < NC; ++c) ub[c] = ubl[c * E + f.eL];
                    alpha = fmin(alpha, euler_alpha_rare(ub, fA, (0.25 * m.h) * dte_a[off<NC>(E, 2, f.eL)], pr.pos_eps));
                }
                if (f.eR >= 0) {
                    double fm[NC];
#pragma unroll
                    for (int c = 0; c < NC; ++c) {
                        ub[c] = ubl[c * E + f.eR];
                        fm[c] = -fA[c];
                    }
                    alpha = fmin(alpha, euler_alpha_rare(ub, fm, (0.25 * m.h) * dte_a[off<NC>(E, 2, f.eR)], pr.pos_eps));
                }
                if (alpha != 1.0) {
#pragma unroll
                    for (int c = 0; c < NC; ++c) {
                        const double v = alpha * fA[c];
                        if constexpr (sizeof(R) == 4) {
                            T0[c] = __double2float_rn(v);
                            T1[c] = __double2float_rn(v - (double)T0[c]);
                        } else {
                            T0[c] = v;
                            T1[c] = 0.0;
                        }
                    }
                }
            }
#pragma unroll
            for (int c = 0; c < NC; ++c) {
                if constexpr (sizeof(R) == 4) {
                    sT[1][c][i] = T0[c];
                    sT[2][c][i] = T1[c];
                } else {
                    sT[1][c][i] = T0[c] + T1[c];
                }
            }
        }
    }
    __syncthreads();
    const int ex = ex0 + tx, ey = ey0 + ty, e = ey * m.nx + ex;
    if (ty >= F_TY || ex >= m.nx || ey >= m.ny) return;
    int at[4];
#pragma unroll
    for (int d = 0; d < 4; ++d) at[d] = facet_of(tx, ty, d);
    const double rs = dte_a[off<NC>(E, 1, e)];
    double rs2 = rs, ub[NC];
    R fh[NC];
    // (m_i^e / |K_e|) |S| times the outward sum of f^H, the facet term of eq.
    // (aecb): h / (p+1)^2 for every node (Bernstein); on an LGL mesh h,
    // weighted by w_a w_b per node in k_upd_sys
    const R hw = (sizeof(R) == 4) ? R(m.h_over_n2_f) : (is_lgl<R>(m) ? R(m.h) : R(m.h_over_n2));
    // outward sum (E - W) + N - S of a facet term, in float as a pair
    auto outward = [&](int k, int c) {
        const R w = sT[k][c][at[0]], ea = sT[k][c][at[1]], so = sT[k][c][at[2]], no = sT[k][c][at[3]];
        if constexpr (sizeof(R) == 4) {
            float hi, lo;
            ff_sum4(ea, w, no, so, hi, lo);
            return widen(hi) + widen(lo);
        } else {
            return ((ea - w) + no) - so;
        }
    };
#pragma unroll
    for (int c = 0; c < NC; ++c)
        fh[c] = need_fh ? hw * (((sT[0][c][at[1]] - sT[0][c][at[0]]) + sT[0][c][at[3]]) - sT[0][c][at[2]]) : R(0);
    if (pr.fl == FL_LOW) {
#pragma unroll
        for (int c = 0; c < NC; ++c) ub[c] = ubl[c * E + e];
    } else if (pr.fl == FL_NONE) {
        double uec[NC], osv[NC];
#pragma unroll
        for (int c = 0; c < NC; ++c) {
            uec[c] = ue[c * E + e];
            osv[c] = outward(0, c);
            ub[c] = uec[c] - rs * osv[c];
        }
        // eq. (uebar) with the macrocell dt_e need not stay in G: count such
        // averages, and with the option decrease dt_e as the remark after
        // eq. (dtmaxcell) says (out of line: rare)
        if (!average_in_G<Ph>(pr, ub)) {
            const CompVec<double, NC + 1> red = reduce_pseudo_step<Ph>(pr, uec, osv, rs, cnt);
#pragma unroll
            for (int c = 0; c < NC; ++c) ub[c] = red.v[c];
            rs2 = red.v[NC];
        }
    } else {
#pragma unroll
        for (int c = 0; c < NC; ++c) {
            double os;
            if constexpr (sizeof(R) == 4) {
                // (fbar_E - fbar_W) + fbar_N - fbar_S from the eight float
                // terms, compensated, widened once
                const float t[8] = {sT[1][c][at[1]], sT[2][c][at[1]], -sT[1][c][at[0]], -sT[2][c][at[0]],
                                    sT[1][c][at[3]], sT[2][c][at[3]], -sT[1][c][at[2]], -sT[2][c][at[2]]};
                float hi, lo;
                ff_sum<8>(t, hi, lo);
                os = widen(hi) + widen(lo);
            } else {
                os = outward(1, c);
            }
            ub[c] = ubl[c * E + e] + rs * os;
        }
    }
#pragma unroll
    for (int c = 0; c < NC; ++c) {
        ube_out[c * E + e] = ub[c];
        fht[c * E + e] = fh[c];
    }
    if (rs2 != rs) store_reduced_step(m, dte_a, cf, rs2, e);
}

// The element part of the update of systems (f_i^e, the slope limiter beta_e,
// the SSP increments) with one thread per element and component, as k_res_sys:
// the contributions f_i^e pass through shared memory for the positivity
// factors, which couple the components, the block's warps sharing the nodes.
// One thread per element waited on its 27 loads a component one component
// after the other, at 128 registers and 16 warps per SM.
template <class R, int P, class Ph>
__global__ void __launch_bounds__(32 * Ph::NC, sizeof(R) == 4 ? (P <= 2 ? 8 : P == 3 ? 5 : 4) : (P <= 2 ? 4 : P == 3 ? 3 : 2))
    k_upd_sys(MeshDev m, ProbDev pr, const R* __restrict__ u, const R* __restrict__ ud, const double* __restrict__ ue,
              const double* __restrict__ dte_a, const R* __restrict__ ER, const float* __restrict__ cf,
              const float* __restrict__ avg, const double* __restrict__ ube, const R* __restrict__ fht,
              const double* __restrict__ dtp, R* __restrict__ EW, double* __restrict__ beta_out,
              unsigned long long* __restrict__ cnt) {
    constexpr int NC = Ph::NC, N1 = P + 1, N2 = Dim<P>::N2, TX = 32;
    __shared__ R sF[N2][NC][TX];
    __shared__ R sB[NC][TX];
    __shared__ float sU[NC][TX];
    pdl_begin();
    const int tx = threadIdx.x, c = threadIdx.y;
    const bool valid = blockIdx.x * TX + tx < m.nx;
    const int ex = valid ? blockIdx.x * TX + tx : m.nx - 1, ey = blockIdx.y;  // a lane past the row repeats its last element
    const int e = ey * m.nx + ex;
    const Tab<R>& T = tab_of<R>(m, P);
    // theta = dt / dt_e and dt_e; FP32-mixed: in float from the float speed sum
    R thR, dteR;
    if constexpr (sizeof(R) == 4) {
        const float s = cf[e];
        float dth, dtl;
        split_ff(*dtp, dth, dtl);
        thR = __fmul_rn(__fadd_rn(dth, dtl), __fmul_rn(s, m.inv_h_f));
        dteR = __fmul_rn(m.h_f, __frcp_rn(s));
    } else {
        thR = *dtp * dte_a[off<NC>(m.E, 2, e)];
        dteR = dte_a[e];
    }
    if (valid && c == 0 && thR > R(1)) atomicAdd(&cnt[CNT_CFL], 1ull);
    const double ubd = ube[c * m.E + e];
    R ubh, ubo;
    if constexpr (sizeof(R) == 4) split_ff(ubd, ubh, ubo);
    else split<R>(ubd, ubh, ubo);
    R U[N2], F[N2];
    load_comp<R, P>(u + c * m.NN, m, ex, ey, U);
    if (pr.mode == MODE_LO) {
        if (!valid) return;
#pragma unroll
        for (int i = 0; i < N2; ++i) EW[ev_at(m.E, e, i, c, NC)] = thR * ((ubh - U[i]) + ubo);
        if (c == 0) beta_out[e] = 0.0;
        return;
    }
    // f_i^e, eq. (aec) with eq. (aecb) folded into the residual
    const R meR = PV<R>::me(m), h2 = PV<R>::h2(m), inv_meR = PV<R>::inv_me(m);
    const bool lgl = is_lgl<R>(m);
    const Tab<double>& TL = c_tabd[PMAX + 1 + P];
    {
        R UD[N2];
        load_comp<R, P>(ud + c * m.NN, m, ex, ey, UD);
        const R* __restrict__ r = ER + ((long long)c * m.E + e);
#pragma unroll
        for (int i = 0; i < N2; ++i) F[i] = r[(long long)(i * NC) * m.E];
        R ueh, uel;
        if constexpr (sizeof(R) == 4) {
            ueh = avg[off<NC>(m.E, 2 * c, e)];
            uel = avg[off<NC>(m.E, 2 * c + 1, e)];
        } else {
            split<R>(ue[c * m.E + e], ueh, uel);
        }
        const R fh = fht[c * m.E + e];
        R Y[N1][N1];
#pragma unroll
        for (int d = 0; d < N1; ++d)
#pragma unroll
            for (int a = 0; a < N1; ++a) {
                R s = R(0);
#pragma unroll
                for (int k = 0; k < N1; ++k) s += T.M[a][k] * UD[d * N1 + k];
                Y[d][a] = s;
            }
#pragma unroll
        for (int b = 0; b < N1; ++b)
#pragma unroll
            for (int a = 0; a < N1; ++a) {
                R s = R(0);
#pragma unroll
                for (int d = 0; d < N1; ++d) s += T.M[b][d] * Y[d][a];
                const int i = b * N1 + a;
                const R dev = (U[i] - ueh) - uel;
                if (lgl) {
                    const R w2 = R(TL.wl[a] * TL.wl[b]);
                    const R mi = h2 * w2;
                    F[i] = mi * dev + dteR * (((F[i] + fh * w2) - h2 * s) + mi * UD[i]);
                } else {
                    F[i] = meR * dev + dteR * (((F[i] + fh) - h2 * s) + meR * UD[i]);
                }
            }
    }
    R beta = R(1);
    if (pr.mode == MODE_WENO_L) {
#pragma unroll
        for (int i = 0; i < N2; ++i) sF[i][c][tx] = F[i];
        sU[c][tx] = cert_float(ubd);
        __syncthreads();
        float ubf[NC];
        const bool cert = !(pr.opts & OPT_FP64_LIMITER);
#pragma unroll
        for (int k = 0; k < NC; ++k) ubf[k] = sU[k][tx];
#pragma unroll 1
        for (int i = c; i < N2; i += NC) {
            // float32 certificate first; the float64 formula only where it
            // cannot show alpha_i = 1 (min(b, 1) = b: same result)
            if (cert) {
                float ff[NC];
#pragma unroll
                for (int k = 0; k < NC; ++k) ff[k] = sizeof(R) == 4 ? (float)sF[i][k][tx] : cert_float((double)sF[i][k][tx]);
                float mi = m.me_f;
                if (lgl) mi = (float)(m.h * m.h * (TL.wl[i % N1] * TL.wl[i / N1]));
                if (euler_alpha_is_one<R>(ubf, ff, mi, pr.ome_f)) continue;
            }
            double f[NC], ub[NC];
#pragma unroll
            for (int k = 0; k < NC; ++k) {
                f[k] = (double)sF[i][k][tx];
                ub[k] = ube[k * m.E + e];
            }
            const double mi = lgl ? m.h * m.h * (TL.wl[i % N1] * TL.wl[i / N1]) : m.me;
            beta = fmin(beta, R(euler_alpha_rare(ub, f, mi, pr.pos_eps)));  // rounding keeps the order
        }
        sB[c][tx] = beta;
        __syncthreads();
#pragma unroll
        for (int k = 0; k < NC; ++k) beta = fmin(beta, sB[k][tx]);
    }
    if (!valid) return;
    if (c == 0) {
        if constexpr (sizeof(R) == 4) beta_out[e] = widen(beta);
        else beta_out[e] = beta;
    }
    R* __restrict__ out = EW + ((long long)c * m.E + e);
#pragma unroll
    for (int i = 0; i < N2; ++i) {
        const R inv_mi = lgl ? R(m.inv_h2 * (TL.iwl[i % N1] * TL.iwl[i / N1])) : inv_meR;
        out[(long long)(i * NC) * m.E] = thR * (((ubh - U[i]) + ubo) + (beta * F[i]) * inv_mi);
    }
}

// Scalars: the residual in two kernels.  k_res_w (the Galerkin part W^e, needs
// only u) runs on a stream of its own from the start of the stage, beside k_lo
// and the g_h kernels; k_res_s adds the stabilisation, which needs g_h,
// gamma_e and nu_e.  W^e passes through the increment buffer, which is free
// until k_update_el.
template <class R, int P, class Ph>
DEV void res_w_at(const MeshDev& m, const ProbDev& pr, const R* __restrict__ u, R* __restrict__ WV, int ex, int ey,
                  int e) {
    constexpr int N2 = Dim<P>::N2;
    R U[N2], W[N2];
    load_comp<R, P>(u, m, ex, ey, U);
    w_part<R, P, Ph>(m, pr, U, ex, ey, W);
#pragma unroll
    for (int i = 0; i < N2; ++i) WV[ev_at(m.E, e, i, 0, 1)] = W[i];
}

template <class R, int P>
DEV void res_s_at(const MeshDev& m, const R* __restrict__ u, const R* __restrict__ g,
                  const double* __restrict__ gam, const double* __restrict__ nu, const R* __restrict__ WV,
                  R* __restrict__ ER, int ex, int ey, int e) {
    constexpr int N2 = Dim<P>::N2;
    R U[N2], W[N2];
    load_comp<R, P>(u, m, ex, ey, U);
#pragma unroll
    for (int i = 0; i < N2; ++i) W[i] = WV[ev_at(m.E, e, i, 0, 1)];
    stab_part<R, P>(m, U, g, gam, nu, W, ER, ex, ey, e);
}

template <class R, int P, class Ph>
__global__ void __launch_bounds__(128) k_res_w(MeshDev m, ProbDev pr, const R* __restrict__ u, R* __restrict__ WV) {
    pdl_begin();
    int ex, ey, e;
    if (!elem_of_thread(m, ex, ey, e)) return;
    res_w_at<R, P, Ph>(m, pr, u, WV, ex, ey, e);
}

template <class R, int P>
__global__ void __launch_bounds__(128) k_res_s(MeshDev m, const R* __restrict__ u, const R* __restrict__ g,
                                               const double* __restrict__ gam, const double* __restrict__ nu,
                                               const R* __restrict__ WV, R* __restrict__ ER) {
    pdl_begin();
    int ex, ey, e;
    if (!elem_of_thread(m, ex, ey, e)) return;
    res_s_at<R, P>(m, u, g, gam, nu, WV, ER, ex, ey, e);
}

// ---------------------------------------------------------------------------
// k_final: u_i^SSP = u_i + (sum_{e in E_i} increment_i^e) / |E_i| (m_i^e/m_i
// = 1/|E_i| on a uniform mesh), SSP-RK combination a u^n + b u^SSP, the
// invariant-domain check and clamp (scalar IDP modes, bounds rounded inward
// to the storage precision) or the positivity count (Euler), non-finite count.
// ---------------------------------------------------------------------------
// Float certificate of the positivity check of a stored state (rho, m, E):
// true only when rho > 0 and rho E - |m|^2/2 > 0 hold for these values
// exactly, so p = (gamma - 1)(E - |m|^2 / (2 rho)) > 0 as well (and the
// float64 check agrees).  The float evaluation t = fma(rho, E, -kin), kin =
// 0.5 fma(mx, mx, my^2), differs from the exact value by at most about
// 3.1 2^-24 A, A = |rho E| + kin, so t > 2^-21 A certifies it; A is kept in
// [2^-100, 2^100] (no underflow or overflow in the products).  Otherwise
// (near-vacuum or near-zero pressure states, NaN) the float64 check decides.
template <class R>
DEV bool euler_positive_certified(const R* u) {
    if constexpr (sizeof(R) == 4) {
        const float rho = u[0], mx = u[1], my = u[2], E = u[3];
        if (!(rho > 0.f)) return false;
        const float kin = __fmul_rn(0.5f, __fmaf_rn(mx, mx, __fmul_rn(my, my)));
        const float t = __fmaf_rn(rho, E, -kin);
        const float A = __fadd_rn(fabsf(__fmul_rn(rho, E)), kin);
        return t > 0x1p-21f * A && A > 0x1p-100f && A < 0x1p100f;
    } else {
        // the same in float64: t differs from the exact value by at most about
        // 3.1 2^-53 (rho E + kin), and kin < rho E where t > 0, so t > 2^-40 rho
        // E certifies it; integer tests of the high words (rho and the
        // difference positive and finite, rho E away from under- and overflow)
        const double A = __dmul_rn(u[0], u[3]);
        const double t = __fma_rn(u[0], u[3], -(0.5 * __fma_rn(u[1], u[1], __dmul_rn(u[2], u[2]))));
        const int hr = __double2hiint(u[0]), ha = __double2hiint(A), hd = __double2hiint(__fma_rn(-0x1p-40, A, t));
        return hr > 0 && hr < 0x7ff00000 && ha > (123 << 20) && ha < (1923 << 20) && hd > 0 && hd < 0x7ff00000;
    }
}

template <class R, int P, int NC>
DEV void final_at(const MeshDev& m, const ProbDev& pr, const R* __restrict__ EW,
                        R* __restrict__ un, R* __restrict__ u, R a, R b,
                        unsigned long long* __restrict__ cnt, int gx, int gy, long long node) {
    const NodeC<P> nc = node_c<P>(m, gx, gy);
    R s[NC];
    gather_at<R, P, NC>(m, EW, nc, s);
    const R inv_cnt = inv_count<R>(nc.nxc * nc.nyc);
    R out[NC];
    bool bad = false;
#pragma unroll
    for (int c = 0; c < NC; ++c) {
        const R uold = u[c * m.NN + node];
        R ufe = uold + s[c] * inv_cnt;
        if (a != R(0)) {
            out[c] = a * un[c * m.NN + node] + b * ufe;
        } else {
            out[c] = b * ufe;
            un[c * m.NN + node] = uold;  // first stage: keep u^n for the later stages
        }
        bad |= !is_finite(out[c]);
    }
    if (bad) atomicAdd(&cnt[CNT_NONFINITE], 1ull);
    if (NC == 1) {
        if (pr.mode == MODE_LO || pr.mode == MODE_WENO_L) {
            const R lo = PV<R>::lo(pr), hi = PV<R>::hi(pr);
            const R v = out[0];
            if (v < PV<R>::lo_tol(pr) || v > PV<R>::hi_tol(pr))
                atomicAdd(&cnt[CNT_VIOL], 1ull);
            if (v < lo || v > hi) {
                atomicAdd(&cnt[CNT_CLAMP], 1ull);
                out[0] = fmin(fmax(v, lo), hi);
            }
        }
    } else {
        if (!euler_positive_certified(out)) {
            double dd[NC];
#pragma unroll
            for (int c = 0; c < NC; ++c) dd[c] = (double)out[c];
            double pres = PhysEuler::pressure<double>(dd, pr.gam);
            if (!(dd[0] > 0.0) || !(pres > 0.0)) atomicAdd(&cnt[CNT_VIOL], 1ull);
        }
    }
#pragma unroll
    for (int c = 0; c < NC; ++c) u[c * m.NN + node] = out[c];
}

template <class R, int P, int NC>
__global__ void k_final(MeshDev m, ProbDev pr, const R* __restrict__ EW,
                        R* __restrict__ un, R* __restrict__ u, R a, R b,
                        unsigned long long* __restrict__ cnt, double* __restrict__ t_adv,
                        const double* __restrict__ dtp) {
    pdl_begin();
    // last stage of a step: one thread advances the time (nothing in this
    // kernel reads it)
    if (t_adv && blockIdx.x == 0 && blockIdx.y == 0 && threadIdx.x == 0 && threadIdx.y == 0) *t_adv += *dtp;
    int gx, gy;
    long long node;
    if (!node_of_thread(m, gx, gy, node)) return;
    final_at<R, P, NC>(m, pr, EW, un, u, a, b, cnt, gx, gy, node);
}


}  // namespace cgl
