// modal.cuh — the WENO sensor gamma_e (eqs. (WENO:alpha), (WENO:norm) of the
// paper) in a modal basis.
//
// The semi-norm of eq. (WENO:norm) is a quadratic form on the (p+1)^2
// coefficients of a polynomial.  On products of Legendre polynomials it is
// nearly diagonal: derivatives of P_k contain only Legendre polynomials of
// the other parity, so two 1D modes k < l interact only when l = k + 2 and k
// >= 1, which leaves no off-diagonal entry for p <= 2, 10 pairs at p = 3 and
// 28 at p = 4 (against 28, 105 and 276 pairs of nodal coefficients).  The
// neighbour's polynomial continued onto the element, m_j(x +- 1) = m_j + sum
// over k < j, is unit upper triangular.  The modal coefficients of an element
// serve its own candidate and those of its four neighbours, so the tile
// kernels form them once per element in shared memory.
//
// A line v_0 .. v_p goes to modes by its even and odd pairs v_j + v_{p-j} and
// v_{p-j} - v_j; the modes are scaled so that the outer pair enters with
// weight 1 (p = 2: four operations a line).  Every block is shifted by its
// first coefficient first (constants do not change any semi-norm: flat data
// give exact zeros, nearly flat data no cancellation), and the constant mode
// (0, 0) is never formed.
//
// Explicitly rounded operations throughout, so that every kernel that
// inlines these functions computes the same bits.
#pragma once

#include "common.cuh"

namespace cgl {

// explicitly rounded arithmetic (no contraction choices left to the compiler)
DEV float fma_r(float a, float b, float c) { return __fmaf_rn(a, b, c); }
DEV double fma_r(double a, double b, double c) { return __fma_rn(a, b, c); }
DEV float mul_r(float a, float b) { return __fmul_rn(a, b); }
DEV double mul_r(double a, double b) { return __dmul_rn(a, b); }
DEV float add_r(float a, float b) { return __fadd_rn(a, b); }
DEV double add_r(double a, double b) { return __dadd_rn(a, b); }
DEV float sub_r(float a, float b) { return __fsub_rn(a, b); }
DEV double sub_r(double a, double b) { return __dsub_rn(a, b); }

// x^e for the exponents other than the defaults r = 2, q = 1 of the sensor
// (eqs. (WENO:alpha), (stab:WENO)): out of line, so that the sensor's hot
// code, which the default exponents take, stays small in the instruction
// cache (the same powf / pow as an inlined call)
static __device__ __noinline__ float pow_rare(float x, float e) { return powf(x, e); }
static __device__ __noinline__ double pow_rare(double x, double e) { return pow(x, e); }

// 1 / x, x >= 0, of a weight or a norm: float by the hardware's approximation
// (within one unit in the last place), float64 by rcp_nr where x and 1 / x are
// normal and by the division, out of line, elsewhere.  Both give infinity at 0
// (a flat element's norm with gamma_eps = 0) and 0 at infinity, as the division
// does.
static __device__ __noinline__ double rcp_rare(double x) { return 1.0 / x; }
DEV float recip(float x) {
    float r;
    asm("rcp.approx.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}
DEV double recip(double x) {
    // the biased exponent in 1 .. 2044: x < 2^1022
    if ((((unsigned)__double2hiint(x) >> 20) & 0x7ffu) - 1u >= 2044u) return rcp_rare(x);
    return rcp_nr(x);
}

// square root of a squared norm, x >= 0: float by the hardware's approximation
// (within one unit in the last place; gamma_e is as exact with it as without)
DEV float norm_root(float x) {
    float r;
    asm("sqrt.approx.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}
DEV double norm_root(double x) { return root(x); }

// modal coefficients of one line
template <class R, int P>
DEV void modal_line(const Tab<R>& T, const R (&v)[P + 1], R (&l)[P + 1]) {
    constexpr int NP = (P + 1) / 2, NE = P / 2 + 1;
    R e[NE], o[NP];
#pragma unroll
    for (int j = 0; j < NP; ++j) {
        e[j] = add_r(v[j], v[P - j]);
        o[j] = sub_r(v[P - j], v[j]);
    }
    if constexpr (P % 2 == 0) e[NE - 1] = v[P / 2];
#pragma unroll
    for (int k = 0; k <= P; ++k) {
        R s = (k % 2 == 0) ? e[0] : o[0];
#pragma unroll
        for (int j = 1; j < 3; ++j) {
            if (k % 2 == 0 && j < NE) s = fma_r(T.mf[k][j - 1], e[j], s);
            if (k % 2 == 1 && j < NP) s = fma_r(T.mf[k][j - 1], o[j], s);
        }
        l[k] = s;
    }
}

// modal coefficients [ky (p+1) + kx] of a coefficient block ([b (p+1) + a]);
// entry 0, the constant, is set to 0
template <class R, int P>
DEV void modal_block(const Tab<R>& T, const R (&v)[(P + 1) * (P + 1)], R (&l)[(P + 1) * (P + 1)]) {
    constexpr int N1 = P + 1;
    R X[N1][N1];
#pragma unroll
    for (int b = 0; b < N1; ++b) {
        R line[N1];
#pragma unroll
        for (int a = 0; a < N1; ++a) line[a] = (a == 0 && b == 0) ? R(0) : sub_r(v[b * N1 + a], v[0]);
        modal_line<R, P>(T, line, X[b]);
    }
#pragma unroll
    for (int k = 0; k < N1; ++k) {
        R line[N1], m[N1];
#pragma unroll
        for (int b = 0; b < N1; ++b) line[b] = X[b][k];
        modal_line<R, P>(T, line, m);
#pragma unroll
        for (int b = 0; b < N1; ++b) l[b * N1 + k] = m[b];
    }
    l[0] = R(0);
}

// the neighbour's polynomial (modal coefficients l) continued onto the
// element: dir 0 W and 2 S take m_j(x + 1), dir 1 E and 3 N m_j(x - 1), whose
// odd steps change sign
template <class R, int P, int dir>
DEV void modal_continue(const Tab<R>& T, const R (&l)[(P + 1) * (P + 1)], R (&w)[(P + 1) * (P + 1)]) {
    constexpr int N1 = P + 1;
    constexpr bool lower = (dir & 1) == 0;
#pragma unroll
    for (int t = 0; t < N1; ++t)
#pragma unroll
        for (int k = 0; k < N1; ++k) {
            const int i = (dir < 2) ? t * N1 + k : k * N1 + t;
            R s = l[i];
            if (i > 0) {
#pragma unroll
                for (int j = k + 1; j < N1; ++j) {
                    const R c = (lower || (j - k) % 2 == 0) ? T.mc[k][j] : -T.mc[k][j];
                    s = fma_r(c, l[(dir < 2) ? t * N1 + j : j * N1 + t], s);
                }
            }
            w[i] = i > 0 ? s : R(0);
        }
}

// squared semi-norm of eq. (WENO:norm) of a polynomial in modal coefficients
// (a2b: offset of the basis in the packed matrices, a2_base): each mode
// (k1, k2) with itself and with the later ones it couples to, k1 + 2 and
// k2 + 2 where the lower of the two is at least 1
template <class R, int P>
DEV R modal_norm(const R (&l)[(P + 1) * (P + 1)], int a2b) {
    constexpr int N1 = P + 1, N2 = N1 * N1, off = A2_OFF[P];
    R s = R(0);
#pragma unroll
    for (int k2 = 0; k2 < N1; ++k2)
#pragma unroll
        for (int k1 = 0; k1 < N1; ++k1) {
            const int i = k2 * N1 + k1;
            if (i == 0) continue;
            const int row = a2b + off + i * N2;
            R t = mul_r(TabSel<R>::A2(row + i), l[i]);
            if (k1 >= 1 && k1 + 2 < N1) t = fma_r(TabSel<R>::A2(row + i + 2), l[i + 2], t);
            if (k2 >= 1 && k2 + 2 < N1) {
                const int j = i + 2 * N1;
                if (k1 >= 3) t = fma_r(TabSel<R>::A2(row + j - 2), l[j - 2], t);
                t = fma_r(TabSel<R>::A2(row + j), l[j], t);
                if (k1 >= 1 && k1 + 2 < N1) t = fma_r(TabSel<R>::A2(row + j + 2), l[j + 2], t);
            }
            s = fma_r(l[i], t, s);
        }
    return s;
}

// a direction as a compile-time value: with the four directions in a loop the
// compiler left the candidates in local memory
template <int D> struct Dir {
    static constexpr int value = D;
};
template <class F>
DEV void each_dir(const F& f) {
    f(Dir<0>{});
    f(Dir<1>{});
    f(Dir<2>{});
    f(Dir<3>{});
}

// gamma_e of one component from the modal coefficients own of the element and
// those of its face neighbours, nbr(d, l) (d = W, E, S, N, called where nb[d]
// >= 0).  u_h^e - u_h^{e,*} is formed as sum_{l>=1} omega_l (u_h^e -
// u_{h,l}^e), using sum_l omega_l = 1.  The continued candidates are needed
// twice (their norms give the weights of their sum); KEEP holds them in
// registers, otherwise they are formed again.
template <class R, int P, bool KEEP, class Nbr>
DEV R modal_sensor(const Tab<R>& T, int a2b, const ProbDev& pr, const R (&own)[(P + 1) * (P + 1)],
                   const int (&nb)[4], const Nbr& nbr) {
    constexpr int N2 = (P + 1) * (P + 1);
    const R wl = PV<R>::w_lin(pr), eps = PV<R>::weno_eps(pr), geps = PV<R>::gamma_eps(pr);
    const bool r2 = pr.r2 != 0;
    const R rh = PV<R>::rh(pr);
    int ne = 0;
#pragma unroll
    for (int d = 0; d < 4; ++d) ne += (nb[d] >= 0);
    const R sig0 = fmax(modal_norm<R, P>(own, a2b), R(0));
    R wt[5];
    wt[0] = (R(1) - R(ne) * wl) * recip((r2 ? sig0 : pow_rare(sig0, rh)) + eps);
    R W[KEEP ? 4 : 1][N2];
    each_dir([&](auto dir) {
        constexpr int d = decltype(dir)::value;
        wt[d + 1] = R(0);
        if (nb[d] >= 0) {
            R l[N2];
            nbr(d, l);
            modal_continue<R, P, d>(T, l, W[KEEP ? d : 0]);
            const R sg = fmax(modal_norm<R, P>(W[KEEP ? d : 0], a2b), R(0));
            wt[d + 1] = wl * recip((r2 ? sg : pow_rare(sg, rh)) + eps);
        }
    });
    const R tot = (((wt[0] + wt[1]) + wt[2]) + wt[3]) + wt[4];
    const R rtot = recip(tot);
    R D[N2];
#pragma unroll
    for (int i = 0; i < N2; ++i) D[i] = R(0);
    each_dir([&](auto dir) {
        constexpr int d = decltype(dir)::value;
        if (nb[d] >= 0) {
            if constexpr (!KEEP) {
                R l[N2];
                nbr(d, l);
                modal_continue<R, P, d>(T, l, W[0]);
            }
            const R wd = mul_r(wt[d + 1], rtot);
#pragma unroll
            for (int i = 1; i < N2; ++i) D[i] = fma_r(wd, sub_r(own[i], W[KEEP ? d : 0][i]), D[i]);
        }
    });
    const R num = norm_root(fmax(modal_norm<R, P>(D, a2b), R(0)));
    const R den = norm_root(sig0);
    const R ratio = num * recip(den + geps);
    return R(1) - (pr.q1 ? fmin(R(1), ratio) : pow_rare(fmin(R(1), ratio), PV<R>::q(pr)));
}

}  // namespace cgl
