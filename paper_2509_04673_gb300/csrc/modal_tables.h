// modal_tables.h — host computation of the sensor's modal tables (modal.cuh).
//
// With P_k the Legendre polynomials on [0, 1] and L[k][a] the P_k coefficient
// of the basis function a, a line v has the modal coefficients l_k = (sum_a
// L[k][a] v_a) / L[k][p], so that u = sum_k l_k m_k with m_k = L[k][p] P_k.
//   mf[k][j - 1] = L[k][p - j] / L[k][p], the weights of the pairs (v_j, v_{p-j})
//   mc[k][j]     the expansion of m_j(x + 1) in m_k
//   m2           the semi-norm matrix of eq. (WENO:norm) over the products
//                m_k1 m_k2, off-diagonal entries doubled
// Everything that cancels is a sum of integers below 2^53 (over a common
// denominator), so every entry is off by a few roundings of its last operations
// only: gamma_e multiplies errors of the tables by up to 10^5 where a semi-norm
// is small beside the coefficients.
#pragma once

#include "common.cuh"

namespace cgl {

struct ModalTables {
    double mf[N1MAX][2], mc[N1MAX][N1MAX];
    double m2[N1MAX * N1MAX * N1MAX * N1MAX];  // [i][j], (p + 1)^2 x (p + 1)^2
};

inline double exact_binom(int n, int k) {
    double r = 1.0;
    for (int i = 1; i <= k; ++i) r = r * (n - k + i) / i;  // an integer after every step
    return r;
}

// 2520 int_0^1 a b of polynomials with integer coefficients, degree 8 at most
// in all (2520: the least common multiple of 1 .. 9)
inline double integral_2520(const double* a, int da, const double* b, int db) {
    double s = 0.0;
    for (int i = 0; i <= da; ++i)
        for (int m = 0; m <= db; ++m) s += a[i] * b[m] * (2520 / (i + m + 1));
    return s;
}

// xn: the LGL points on [0, 1] (basis LGL), or null (Bernstein)
inline void modal_tables(int p, const double* xn, ModalTables& T) {
    const int n = p + 1, n2 = n * n;
    // monomial coefficients of P_k(2x - 1)
    double P[N1MAX][N1MAX];
    for (int k = 0; k < n; ++k)
        for (int i = 0; i < n; ++i)
            P[k][i] = i <= k ? ((k + i) % 2 ? -1.0 : 1.0) * exact_binom(k, i) * exact_binom(k + i, i) : 0.0;
    // end[k] = L[k][p] and mf.  Bernstein: int x^i B_a = C(p,a) (a+i)! (p-a)! /
    // (p+i+1)!.  LGL: l_a is interpolated by its P_k-coefficients (2k+1) w_a
    // P_k(x_a) for k < p and p w_a P_p(x_a) (the rule integrates P_p^2 to 1/p in
    // place of 1/(2p+1)), w_a = 1 / (p (p+1) P_p(x_a)^2)
    double end[N1MAX];
    for (int k = 0; k < n; ++k) {
        double num[3] = {0.0, 0.0, 0.0};  // of a = p, p - 1, p - 2
        if (!xn) {
            double whole = 1.0;  // (2p + 1)!
            for (int i = 2; i <= 2 * p + 1; ++i) whole *= i;
            for (int j = 0; j < 3 && j <= p; ++j) {
                const int a = p - j;
                double fj = 1.0;
                for (int i = 2; i <= j; ++i) fj *= i;
                for (int i = 0; i <= k; ++i) {
                    double t = P[k][i] * exact_binom(p, a) * fj;
                    for (int q = 2; q <= a + i; ++q) t *= q;
                    for (int q = p + i + 2; q <= 2 * p + 1; ++q) t *= q;
                    num[j] += t;
                }
            }
            end[k] = (2 * k + 1) * num[0] / whole;
        } else {
            end[k] = (k < p ? 2.0 * k + 1.0 : (double)p) / (p * (p + 1.0));
            for (int j = 0; j < 3 && j <= p; ++j) {
                double z = 2.0 * xn[p - j] - 1.0, q[N1MAX] = {1.0, z};
                for (int i = 2; i <= p; ++i) q[i] = ((2.0 * i - 1.0) * z * q[i - 1] - (i - 1.0) * q[i - 2]) / i;
                num[j] = j == 0 ? 1.0 : q[k] / (q[p] * q[p]);
            }
        }
        const int pairs = (p + 1) / 2;  // (v_j, v_{p-j}), j < pairs; an even p has the middle value too
        for (int j = 1; j < 3; ++j) {
            const bool used = (k % 2 == 0) ? j < pairs + (p % 2 == 0) : j < pairs;
            T.mf[k][j - 1] = used ? num[j] / num[0] : 0.0;
        }
    }
    for (int j = 0; j < n; ++j) {
        double sh[N1MAX] = {0.0};  // P_j at x + 1
        for (int i = 0; i <= j; ++i)
            for (int m = 0; m <= i; ++m) sh[m] += P[j][i] * exact_binom(i, m);
        for (int k = 0; k < n; ++k) {
            const double e = (2 * k + 1) * integral_2520(sh, j, P[k], k) / 2520.0;
            T.mc[k][j] = j > k ? e * (end[j] / end[k]) : (j == k ? 1.0 : 0.0);
        }
    }
    double S[N1MAX][N1MAX][N1MAX];  // int P_k^(d) P_l^(d)
    for (int d = 0; d <= p; ++d)
        for (int k = 0; k < n; ++k)
            for (int l = 0; l < n; ++l) {
                double dk[N1MAX] = {0.0}, dl[N1MAX] = {0.0};
                for (int i = d; i < n; ++i) {
                    double f = 1.0;
                    for (int q = 0; q < d; ++q) f *= i - q;
                    dk[i - d] = f * P[k][i];
                    dl[i - d] = f * P[l][i];
                }
                S[d][k][l] = integral_2520(dk, p - d, dl, p - d) / 2520.0;
            }
    for (int i = 0; i < n2; ++i)
        for (int j = 0; j < n2; ++j) {
            const int k1 = i % n, k2 = i / n, l1 = j % n, l2 = j / n;
            double s = 0.0;
            for (int d1 = 0; d1 <= p; ++d1)
                for (int d2 = 0; d2 <= p - d1; ++d2)
                    if (d1 + d2 >= 1) s += S[d1][k1][l1] * S[d2][k2][l2];
            T.m2[i * n2 + j] = (i == j ? s : 2.0 * s) * (end[k1] * end[l1]) * (end[k2] * end[l2]);
        }
}

}  // namespace cgl
