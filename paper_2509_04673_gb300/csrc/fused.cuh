// fused.cuh — the separable node stencils of the g_h and udot solves on tiles
// of whole elements, and the first Richardson sweep fused into the kernel
// that builds its right-hand side.
//
// k_grad_sweep: g_h right-hand side b = int phi_i grad u_h, lumped iterate
//   g0 = b / m_i and the first sweep g1 = g0 + (b - M_C g0) / m_i (Sec. 2.2,
//   Richardson reading of the consistent L2 projection) in one pass.
// k_udot_sweep: node gather r_i = sum_e R^e_i, lumped iterate udot0 = r / m_i
//   and the first sweep (Sec. 4.3, step 2) in one pass.
// k_mass_sweep: one further sweep.
// k_grad_rhs: b and g0 alone (no sweeps, CGL_OPT_UNFUSED_SWEEPS).
//
// What bounds them is the shared-memory pipe and instruction issue, not DRAM,
// so a thread owns a segment, the vertex v and the p - 1 interior nodes after
// it, instead of a node: one read of the 2p + 1 values v - p .. v + p gives
// the p outputs of every 1D operator applied to them (p = 2: 2.5 reads per
// node in place of 5), the interior nodes skip the p weights that are zero
// for them, and every weight is a table constant, except the vertex's own,
// which differs at the ends of a non-periodic mesh.
//
// Tiles start at vertices.  A field is staged by local index: plane a holds
// the nodes of index a of every segment, so the segment reads of a warp along
// x fall on consecutive words; planes are padded so that a warp running over
// nodes (along y, and at the global accesses) hits distinct banks as well.
//
// A tile (with the halo it works on) is LX segments wide, and so is the block:
// in the x passes a thread keeps one segment and steps over rows, in the y passes and
// at the global accesses one node column and steps over y segments.  Columns,
// plane offsets, weights and masses are formed once per thread, and the loops
// add constants (with the items of a pass numbered through, index arithmetic
// was 40 % of k_grad_sweep's instructions, 64 of 161 warp instructions per
// element of the Euler form at p = 2).
//
// The sums run over the offsets -p .. p in order with explicit rounding, so
// the fused and the separate kernels, and every tile size, give the same bits.
#pragma once

#include "kernels.cuh"

namespace cgl {

// A tile of TEX x TEY elements (NX x NY nodes) worked by NT threads: LX
// segments wide in the x passes, RX rows of them per step; LY node columns
// wide in the y passes, RY y segments per step, KY steps.  HALO: the passes
// run on the tile and one element around it (the fused g_h kernel, whose
// first iterate is needed there).
template <class R, int P, int LX_, int KY_, int NT_, bool HALO_>
struct SegTile {
    static constexpr int LX = LX_, KY = KY_, NT = NT_, HALO = HALO_;
    static constexpr int LY = LX * P, RX = NT / LX, RY = NT / LY;
    static constexpr int TEX = HALO ? LX - 2 : LX, TEY = HALO ? RY * KY - 2 : RY * KY;
    static_assert(NT % LX == 0 && NT % LY == 0 && TEY >= 1, "whole rows of threads");
    static constexpr int NX = TEX * P, NY = TEY * P;
    // nodes along x and y of the tile with one (1) and two (2) elements of halo
    // (one less on the high side, where the last vertex suffices), segments
    static constexpr int W1 = NX + P + 1, H1 = NY + P + 1, S1 = TEX + 2;
    static constexpr int W2 = NX + 3 * P + 1, H2 = NY + 3 * P + 1, S2 = TEX + 4;
    static constexpr int K1 = (H1 + RX - 1) / RX, K2 = (H2 + RX - 1) / RX;  // steps of the x passes
    // plane stride: n words or more, congruent to a p-th of the banks
    static constexpr int plane(int n) {
        constexpr int B = 128 / (int)sizeof(R), want = P == 1 ? 0 : (B + P - 1) / P;
        int k = n;
        while (P > 1 && k % B != want % B) ++k;
        return k;
    }
    static constexpr int PU = plane(H2 * S2);  // u on the two-element halo
    static constexpr int PT = plane(H2 * S1);  // its x pass
    static constexpr int PG = plane(H1 * S1);  // a field on the one-element halo, or its x pass
    static constexpr int PR = plane(NY * S1);  // a field on the tile
    // shared words of grad_sweep_seg, grad_rhs_seg, mass_sweep_seg
    static constexpr int grad_ws = (P * PU > 2 * P * PG ? P * PU : 2 * P * PG) + 2 * P * PT;
    static constexpr int rhs_ws = 3 * P * PG;
    static constexpr int sweep_ws = 2 * P * PG;
    // fields of a udot sweep staged together: two where they take 32 KB at most
    static constexpr int udot1 = P * (2 * PG + PR);
    static constexpr int udot_fields(int nc) { return (nc % 2 == 0 && 2 * udot1 * (int)sizeof(R) <= 32768) ? 2 : 1; }
    static constexpr int udot_ws(int nc) { return udot_fields(nc) * udot1; }
};

// kind of a vertex along a direction of n nodes: 0 shared by two elements, 1
// and 2 the lower and upper end of a non-periodic mesh
DEV int vertex_kind(int g, int n, int periodic) { return periodic ? 0 : (g == 0 ? 1 : (g == n - 1 ? 2 : 0)); }

// the vertex's own weight in the assembled operator (WHICH 0 mass, 1
// derivative on the trial index)
template <class R, int P, int WHICH>
DEV R vertex_weight(const Tab<R>& T, int kind) {
    const R lo = wtab<R, P, WHICH>(T, P, P), hi = wtab<R, P, WHICH>(T, 0, 0);
    return kind == 0 ? add_r(lo, hi) : (kind == 1 ? hi : lo);
}

// the 1D operator on a segment: x[k] the value at offset k - P from its vertex
template <class R, int P, int WHICH>
DEV void seg_apply(const Tab<R>& T, const R (&x)[2 * P + 1], R w0, R (&out)[P]) {
    R s = R(0);
#pragma unroll
    for (int k = 0; k <= 2 * P; ++k) {
        const R w = k < P ? wtab<R, P, WHICH>(T, P, k) : (k == P ? w0 : wtab<R, P, WHICH>(T, 0, k - P));
        s = fma_r(w, x[k], s);
    }
    out[0] = s;
#pragma unroll
    for (int a = 1; a < P; ++a) {
        s = R(0);
#pragma unroll
        for (int c = 0; c <= P; ++c) s = fma_r(wtab<R, P, WHICH>(T, a, c), x[P + c], s);
        out[a] = s;
    }
}

// a segment's values along x (f: its vertex in plane 0, planes of stride PL)
// and along y (f: its vertex, rows of stride S)
template <class R, int P>
DEV void seg_x(const R* f, int PL, R (&x)[2 * P + 1]) {
#pragma unroll
    for (int k = 0; k <= 2 * P; ++k) x[k] = f[(k % P) * PL + k / P - 1];
}
template <class R, int P>
DEV void seg_y(const R* f, int S, R (&x)[2 * P + 1]) {
#pragma unroll
    for (int k = 0; k <= 2 * P; ++k) x[k] = f[(k - P) * S];
}

// 1 / m_i of node (gx, gy) with local indices a, b in its segments
template <class R, int P>
DEV R seg_inv_mass(const MeshDev& m, int a, int kx, int b, int ky) {
    const int cnt = (a == 0 && kx == 0 ? 2 : 1) * (b == 0 && ky == 0 ? 2 : 1);
    if (is_lgl<R>(m)) {
        const int a0 = a != 0 ? a : (kx == 1 ? 0 : P), b0 = b != 0 ? b : (ky == 1 ? 0 : P);
        return R(inv_lumped_lgl<P>(m, cnt, a0, b0));
    }
    return mul_r(PV<R>::inv_me(m), inv_count<R>(cnt));
}

// what a thread keeps of its place in a tile: segment xs and first row xr of
// the x passes, node column q (counted from one element below the tile), its
// local index a and segment s, and first y segment yr of the y passes.  FULL:
// the tile and its halo lie inside the mesh (all but the tiles at its edge),
// so that no index wraps, every vertex is shared and no node is left out.
template <class R, int P, class TL, bool FULL>
struct SegThread {
    int xr, xs, yr, q, a, s, gx, kx, xkind;
    bool act, own_seg, own_x;
    DEV SegThread(const MeshDev& m, int gx0, int tid) {
        act = tid < TL::NT;  // a block may have more threads than the tile takes
        xr = tid / TL::LX;
        xs = tid - xr * TL::LX + (TL::HALO ? 0 : 1);
        yr = tid / TL::LY;
        q = tid - yr * TL::LY + (TL::HALO ? 0 : P);
        yr += TL::HALO ? 0 : 1;
        a = q % P;
        s = q / P;
        gx = gx0 - P + q;
        kx = FULL ? 0 : vertex_kind(gx, m.nnx, m.px);
        xkind = FULL ? 0 : vertex_kind(gx0 + (xs - 1) * P, m.nnx, m.px);
        own_seg = act && (!TL::HALO || (xs >= 1 && xs <= TL::TEX));
        own_x = act && (!TL::HALO || (q >= P && q < P + TL::NX)) && (FULL || gx < m.nnx);
    }
    DEV int ykind(const MeshDev& m, int gyv) const { return FULL ? 0 : vertex_kind(gyv, m.nny, m.py); }
    DEV R inv_mass(const MeshDev& m, int b, int ky) const { return seg_inv_mass<R, P>(m, a, kx, b, ky); }
};

// Staging of a field on the tile and HALO elements around it (W nodes by H
// rows, plane stride PL, row stride S): a thread takes one column and every
// RY-th row, the few columns beyond the block's width go round the block.
// load() reads into registers, so that it can run ahead of the barrier that
// frees the planes, store() writes them.  Values outside a non-periodic mesh
// are 0, and the 1D operators rely on it: they give a vertex at the end of the
// mesh the same weights beyond it as any other.
template <class R, int P, class TL, int HALO, int W, int H, int PL, int S, bool FULL>
struct Stage {
    static constexpr int K = (H + TL::RY - 1) / TL::RY;
    static constexpr int XC = W > TL::LY ? W - TL::LY : 1, KE = W > TL::LY ? (XC * H + TL::NT - 1) / TL::NT : 0;
    int q, r, gx, gxt, gyt;  // the thread's column and first row, its node column; the tile's first node
    bool vx;
    R v[K], e[KE > 0 ? KE : 1];

    DEV Stage(const MeshDev& m, int gx0, int gy0, int tid) {
        r = tid / TL::LY;
        q = tid - r * TL::LY;
        if (tid >= TL::NT) r = H;  // a thread beyond the tile's stages nothing
        gxt = gx0 - HALO * P;
        gyt = gy0 - HALO * P;
        gx = gxt + q;
        vx = q < W && inside(gx, m.nnx, m.px);
    }
    static DEV bool inside(int& g, int n, int periodic) {
        if (FULL) return true;
        if (periodic) g = wrap_periodic(g, n);
        return g >= 0 && g < n;
    }
    // CG: through L2 (ld.global.cg).  u, which k_final reads and writes: it may
    // still run when the kernel behind it starts (and waits), so that lines of u
    // in an SM's L1 can be older than the other SMs' writes.  The fields that the
    // kernel before has only written are read the ordinary way
    template <bool CG>
    static DEV R get(const R* __restrict__ p) {
        if constexpr (CG) return __ldcg(p);
        else return *p;
    }
    template <bool CG>
    DEV void load(const MeshDev& m, const R* __restrict__ x, int tid) {
        if constexpr (FULL) {
            const R* __restrict__ p = x + ((long long)(gyt + r) * m.nnx + gx);
            const long long step = (long long)TL::RY * m.nnx;
#pragma unroll
            for (int k = 0; k < K; ++k, p += step) v[k] = (r + k * TL::RY < H && vx) ? get<CG>(p) : R(0);
        } else {
#pragma unroll
            for (int k = 0; k < K; ++k) {
                const int row = r + k * TL::RY;
                int gy = gyt + row;
                v[k] = (row < H && vx && inside(gy, m.nny, m.py)) ? get<CG>(&x[(long long)gy * m.nnx + gx]) : R(0);
            }
        }
#pragma unroll
        for (int k = 0; k < KE; ++k) {
            const int i = tid + k * TL::NT, row = tid < TL::NT ? i / XC : H;
            int g = gxt + TL::LY + i - row * XC, gy = gyt + row;
            e[k] = (row < H && inside(g, m.nnx, m.px) && inside(gy, m.nny, m.py)) ? get<CG>(&x[(long long)gy * m.nnx + g])
                                                                                  : R(0);
        }
    }
    DEV void store(R* f, int tid) const {
        R* p = f + (q % P) * PL + q / P + r * S;
#pragma unroll
        for (int k = 0; k < K; ++k)
            if (q < W && r + k * TL::RY < H) p[k * TL::RY * S] = v[k];
#pragma unroll
        for (int k = 0; k < KE; ++k) {
            const int i = tid + k * TL::NT, row = i / XC, c = TL::LY + i - row * XC;
            if (tid < TL::NT && row < H) f[(c % P) * PL + row * S + c / P] = e[k];
        }
    }
};

// x pass with the mass operator over the rows of a field staged at X (planes
// PG, rows of S1), into Y of the same shape: the thread's segment, its rows
template <class R, int P, class TL>
DEV void mass_x(const Tab<R>& T, const R* X, R* Y, int xs, int xr, R w0) {
    X += xr * TL::S1 + xs;
    Y += xr * TL::S1 + xs;
#pragma unroll 2
    for (int k = 0; k < TL::K1; ++k) {
        if (k * TL::RX + xr < TL::H1) {
            R x[2 * P + 1], o[P];
            seg_x<R, P>(X + k * TL::RX * TL::S1, TL::PG, x);
            seg_apply<R, P, 0>(T, x, w0, o);
#pragma unroll
            for (int a = 0; a < P; ++a) Y[a * TL::PG + k * TL::RX * TL::S1] = o[a];
        }
    }
}

// whether a tile with n elements of halo lies inside the mesh, away from its
// ends
template <int P, class TL, int N>
DEV bool tile_full(const MeshDev& m, int gx0, int gy0) {
    return gx0 >= N * P + 1 && gy0 >= N * P + 1 && gx0 + TL::NX + N * P < m.nnx && gy0 + TL::NY + N * P < m.nny;
}

// Right-hand side of the g_h projection, its lumped iterate and the first
// sweep on the tile at (gx0, gy0), one component after the other: u on a
// two-element halo (the next component's loads run under this one's passes),
// x pass with the derivative and the mass operator, y pass to b and g0 on the
// one-element halo, then the sweep's x and y passes.  A thread keeps b and g0
// of its own nodes in registers from the first y pass to the second.
template <class R, int P, int NC, int NF, class TL, bool FULL>
DEV void grad_sweep_body(const MeshDev& m, const R* __restrict__ u, R* __restrict__ bout, R* __restrict__ gout, int gx0,
                         int gy0, int tid, R* ws) {
    constexpr int TEY = TL::TEY, S1 = TL::S1, KY = TL::KY, RY = TL::RY, RX = TL::RX;
    R* B = ws;                   // the x passes
    R* A = ws + 2 * P * TL::PT;  // u, then g0 (x and y parts)
    const Tab<R>& T = tab_of<R>(m, P);
    const R h = PV<R>::h(m), h2 = PV<R>::h2(m);
    const SegThread<R, P, TL, FULL> t(m, gx0, tid);
    const R w0c = vertex_weight<R, P, 1>(T, t.xkind), w0m = vertex_weight<R, P, 0>(T, t.xkind);
    const bool inx = FULL || m.px || (t.gx >= 0 && t.gx < m.nnx);
    const bool feeds_x = t.act && t.q < TL::W1 && (FULL || t.gx < m.nnx + P);
    const bool feeds_seg = t.act && (FULL || gx0 + (t.xs - 1) * P < m.nnx + P);
    Stage<R, P, TL, 2, TL::W2, TL::H2, TL::PU, TL::S2, FULL> in(m, gx0, gy0, tid);
    in.template load<true>(m, u, tid);
#pragma unroll 1
    for (int c = 0; c < NF; ++c) {
        in.store(A, tid);
        __syncthreads();
        if (c + 1 < NF) in.template load<true>(m, u + (c + 1) * m.NN, tid);
        if (feeds_seg) {
            const R* X = A + t.xr * TL::S2 + t.xs + 1;
            R* Y = B + t.xr * S1 + t.xs;
#pragma unroll 2
            for (int k = 0; k < TL::K2; ++k) {
                if (k * RX + t.xr < TL::H2) {
                    R x[2 * P + 1], o[P];
                    seg_x<R, P>(X + k * RX * TL::S2, TL::PU, x);
                    seg_apply<R, P, 1>(T, x, w0c, o);
#pragma unroll
                    for (int i = 0; i < P; ++i) Y[i * TL::PT + k * RX * S1] = o[i];
                    seg_apply<R, P, 0>(T, x, w0m, o);
#pragma unroll
                    for (int i = 0; i < P; ++i) Y[(P + i) * TL::PT + k * RX * S1] = o[i];
                }
            }
        }
        __syncthreads();
        R ob[KY][2][P], og[KY][2][P];  // b and g0 of the thread's nodes
        if (feeds_x) {
            const R* X = B + t.a * TL::PT + (t.yr + 1) * P * S1 + t.s;
            R* Y = A + t.a * TL::PG + t.yr * P * S1 + t.s;
#pragma unroll
            for (int k = 0; k < KY; ++k) {
                const int sy = t.yr + k * RY;  // 0: the segment below the tile
                const int gyv = gy0 + (sy - 1) * P, ky = t.ykind(m, gyv);
                R x[2 * P + 1];
                seg_y<R, P>(X + k * RY * P * S1, S1, x);
                seg_apply<R, P, 0>(T, x, vertex_weight<R, P, 0>(T, ky), ob[k][0]);
                seg_y<R, P>(X + P * TL::PT + k * RY * P * S1, S1, x);
                seg_apply<R, P, 1>(T, x, vertex_weight<R, P, 1>(T, ky), ob[k][1]);
#pragma unroll
                for (int b = 0; b < P; ++b) {
                    const bool in_mesh = FULL || (inx && (m.py || (gyv + b >= 0 && gyv + b < m.nny)));
                    const R inv = t.inv_mass(m, b, ky);
#pragma unroll
                    for (int f = 0; f < 2; ++f) {
                        ob[k][f][b] = mul_r(h, ob[k][f][b]);
                        og[k][f][b] = in_mesh ? mul_r(ob[k][f][b], inv) : R(0);
                        if (sy <= TEY || b == 0) Y[f * P * TL::PG + (k * RY * P + b) * S1] = og[k][f][b];
                    }
                }
            }
        }
        __syncthreads();
        if (t.own_seg) {
            mass_x<R, P, TL>(T, A, B, t.xs, t.xr, w0m);
            mass_x<R, P, TL>(T, A + P * TL::PG, B + P * TL::PG, t.xs, t.xr, w0m);
        }
        __syncthreads();
        if (t.own_x) {
            const R* X = B + t.a * TL::PG + t.yr * P * S1 + t.s;
#pragma unroll
            for (int k = 0; k < KY; ++k) {
                const int sy = t.yr + k * RY, gyv = gy0 + (sy - 1) * P, ky = t.ykind(m, gyv);
                if (sy < 1 || sy > TEY || (!FULL && gyv >= m.nny)) continue;
#pragma unroll
                for (int f = 0; f < 2; ++f) {
                    R x[2 * P + 1], o[P];
                    seg_y<R, P>(X + f * P * TL::PG + k * RY * P * S1, S1, x);
                    seg_apply<R, P, 0>(T, x, vertex_weight<R, P, 0>(T, ky), o);
                    const long long node = (long long)(f * NC + c) * m.NN + (long long)gyv * m.nnx + t.gx;
#pragma unroll
                    for (int b = 0; b < P; ++b)
                        if (FULL || gyv + b < m.nny) {
                            const long long n = node + (long long)b * m.nnx;
                            gout[n] = sweep_value(og[k][f][b], ob[k][f][b], o[b], h2, t.inv_mass(m, b, ky));
                            if (bout) bout[n] = ob[k][f][b];
                        }
                }
            }
        }
    }
}

// b and g0 alone, from u on a one-element halo
template <class R, int P, int NC, int NF, class TL, bool FULL>
DEV void grad_rhs_body(const MeshDev& m, const R* __restrict__ u, R* __restrict__ bout, R* __restrict__ gout, int gx0,
                       int gy0, int tid, R* ws) {
    constexpr int TEY = TL::TEY, S1 = TL::S1, RX = TL::RX, RY = TL::RY;
    R* A = ws;
    R* B = ws + P * TL::PG;
    const Tab<R>& T = tab_of<R>(m, P);
    const R h = PV<R>::h(m);
    const SegThread<R, P, TL, FULL> t(m, gx0, tid);
    const R w0c = vertex_weight<R, P, 1>(T, t.xkind), w0m = vertex_weight<R, P, 0>(T, t.xkind);
    Stage<R, P, TL, 1, TL::W1, TL::H1, TL::PG, S1, FULL> in(m, gx0, gy0, tid);
    in.template load<true>(m, u, tid);
#pragma unroll 1
    for (int c = 0; c < NF; ++c) {
        in.store(A, tid);
        __syncthreads();
        if (c + 1 < NF) in.template load<true>(m, u + (c + 1) * m.NN, tid);
        if (t.own_seg) {
            const R* X = A + t.xr * S1 + t.xs;
            R* Y = B + t.xr * S1 + t.xs;
#pragma unroll 2
            for (int k = 0; k < TL::K1; ++k) {
                if (k * RX + t.xr < TL::H1) {
                    R x[2 * P + 1], o[P];
                    seg_x<R, P>(X + k * RX * S1, TL::PG, x);
                    seg_apply<R, P, 1>(T, x, w0c, o);
#pragma unroll
                    for (int i = 0; i < P; ++i) Y[i * TL::PG + k * RX * S1] = o[i];
                    seg_apply<R, P, 0>(T, x, w0m, o);
#pragma unroll
                    for (int i = 0; i < P; ++i) Y[(P + i) * TL::PG + k * RX * S1] = o[i];
                }
            }
        }
        __syncthreads();
        if (t.own_x) {
#pragma unroll 2
            for (int k = 0; k < TL::KY; ++k) {
                const int sy = t.yr + k * RY, gyv = gy0 + (sy - 1) * P, ky = t.ykind(m, gyv);
                if (sy < 1 || sy > TEY || (!FULL && gyv >= m.nny)) continue;
                const R* X = B + t.a * TL::PG + sy * P * S1 + t.s;
#pragma unroll
                for (int f = 0; f < 2; ++f) {
                    R x[2 * P + 1], o[P];
                    seg_y<R, P>(X + f * P * TL::PG, S1, x);
                    if (f == 0) seg_apply<R, P, 0>(T, x, vertex_weight<R, P, 0>(T, ky), o);
                    else seg_apply<R, P, 1>(T, x, vertex_weight<R, P, 1>(T, ky), o);
                    const long long node = (long long)(f * NC + c) * m.NN + (long long)gyv * m.nnx + t.gx;
#pragma unroll
                    for (int b = 0; b < P; ++b)
                        if (FULL || gyv + b < m.nny) {
                            const long long n = node + (long long)b * m.nnx;
                            const R v = mul_r(h, o[b]);
                            bout[n] = v;
                            gout[n] = mul_r(v, t.inv_mass(m, b, ky));
                        }
                }
            }
        }
    }
}

// one Richardson sweep for NV fields on the tile
template <class R, int P, int NV, class TL, bool FULL>
DEV void mass_sweep_body(const MeshDev& m, const R* __restrict__ xin, const R* __restrict__ b, R* __restrict__ xout,
                         int gx0, int gy0, int tid, R* ws) {
    constexpr int TEY = TL::TEY, S1 = TL::S1, RY = TL::RY;
    R* A = ws;
    R* B = ws + P * TL::PG;
    const Tab<R>& T = tab_of<R>(m, P);
    const R h2 = PV<R>::h2(m);
    const SegThread<R, P, TL, FULL> t(m, gx0, tid);
    const R w0 = vertex_weight<R, P, 0>(T, t.xkind);
    Stage<R, P, TL, 1, TL::W1, TL::H1, TL::PG, S1, FULL> in(m, gx0, gy0, tid);
    in.template load<false>(m, xin, tid);
#pragma unroll 1
    for (int v = 0; v < NV; ++v) {
        in.store(A, tid);
        __syncthreads();
        if (v + 1 < NV) in.template load<false>(m, xin + (v + 1) * m.NN, tid);
        if (t.own_seg) mass_x<R, P, TL>(T, A, B, t.xs, t.xr, w0);
        __syncthreads();
        if (t.own_x) {
#pragma unroll 2
            for (int k = 0; k < TL::KY; ++k) {
                const int sy = t.yr + k * RY, gyv = gy0 + (sy - 1) * P, ky = t.ykind(m, gyv);
                if (sy < 1 || sy > TEY || (!FULL && gyv >= m.nny)) continue;
                const int at = t.a * TL::PG + sy * P * S1 + t.s;
                R x[2 * P + 1], o[P];
                seg_y<R, P>(B + at, S1, x);
                seg_apply<R, P, 0>(T, x, vertex_weight<R, P, 0>(T, ky), o);
                const long long node = v * m.NN + (long long)gyv * m.nnx + t.gx;
#pragma unroll
                for (int c = 0; c < P; ++c)
                    if (FULL || gyv + c < m.nny) {
                        const long long n = node + (long long)c * m.nnx;
                        xout[n] = sweep_value(A[at + c * S1], b[n], o[c], h2, t.inv_mass(m, c, ky));
                    }
            }
        }
        if (v + 1 < NV) __syncthreads();  // the iterate is consumed
    }
}

// Gather of the element residuals, lumped iterate and first sweep on the
// tile.  A thread gathers the p x p nodes of one vertex segment pair: each of
// the (p+1)^2 element values it needs is read once, a warp's reads of one
// value are consecutive in the element index, and no lane branches on its
// node's position in the element.  r = sum over E_i (stored for further sweeps
// and diagnostics), udot0 = r / m_i, udot1 = udot0 + (r - M_C udot0) / m_i.
template <class R, int P, int NC, int NF, class TL, bool FULL>
DEV void udot_sweep_body(const MeshDev& m, const R* __restrict__ ER, R* __restrict__ rout, R* __restrict__ xout,
                         int gx0, int gy0, int tid, R* ws) {
    constexpr int TEX = TL::TEX, TEY = TL::TEY, S1 = TL::S1, RY = TL::RY, N1 = P + 1;
    constexpr int FB = TL::udot_fields(NC), NI = S1 * (TEY + 2);
    R* A = ws;                   // udot0 on the one-element halo
    R* B = A + FB * P * TL::PG;  // its x pass
    R* C = B + FB * P * TL::PG;  // r on the tile
    const Tab<R>& T = tab_of<R>(m, P);
    const R h2 = PV<R>::h2(m);
    const int E = m.E, nx = m.nx;
    const SegThread<R, P, TL, FULL> t(m, gx0, tid);
    const R w0 = vertex_weight<R, P, 0>(T, t.xkind);
#pragma unroll 1
    for (int v0 = 0; v0 < NF; v0 += FB) {
        if (v0 > 0) __syncthreads();  // the previous fields are consumed
#pragma unroll 1
        for (int it = tid; it < NI && t.act; it += TL::NT) {
            const int sy = it / S1, xs = it - sy * S1;
            // the elements before (l) and after (h) the vertex along x and y;
            // hx, hy false: the segment has its vertex only (or lies outside)
            int xl = gx0 / P + xs - 2, xh = xl + 1, yl = gy0 / P + sy - 2, yh = yl + 1;
            if (!FULL) {
                if (xl > nx || yl > m.ny) continue;  // feeds no node of the mesh
                if (m.px) xl = wrap_periodic(xl, nx), xh = wrap_periodic(xh, nx);
                if (m.py) yl = wrap_periodic(yl, m.ny), yh = wrap_periodic(yh, m.ny);
            }
            const bool lx = FULL || (xl >= 0 && xl < nx), hx = FULL || (xh >= 0 && xh < nx);
            const bool ly = FULL || (yl >= 0 && yl < m.ny), hy = FULL || (yh >= 0 && yh < m.ny);
            const int xkind = m.px || FULL ? 0 : (!lx ? 1 : !hx ? 2 : 0);
            const int ykind = m.py || FULL ? 0 : (!ly ? 1 : !hy ? 2 : 0);
            const bool tile = xs >= 1 && xs <= TEX && sy >= 1 && sy <= TEY;
            const int ell = yl * nx + xl, ehl = yl * nx + xh, elh = yh * nx + xl, ehh = yh * nx + xh;
#pragma unroll
            for (int f = 0; f < FB; ++f) {
                auto val = [&](bool in, int e, int i, int j) {
                    return in ? (ER + (long long)((j * N1 + i) * NC + v0 + f) * E)[e] : R(0);
                };
#pragma unroll
                for (int j = 0; j < P; ++j)
#pragma unroll
                    for (int i = 0; i < P; ++i) {
                        // past the last vertex of the halo
                        if ((i > 0 && xs == TEX + 1) || (j > 0 && sy == TEY + 1)) continue;
                        R sum;
                        bool in;
                        if (i == 0 && j == 0) {
                            sum = ((val(lx && ly, ell, P, P) + val(hx && ly, ehl, 0, P)) + val(lx && hy, elh, P, 0)) +
                                  val(hx && hy, ehh, 0, 0);
                            in = (lx || hx) && (ly || hy);
                        } else if (j == 0) {
                            sum = val(hx && ly, ehl, i, P) + val(hx && hy, ehh, i, 0);
                            in = hx && (ly || hy);
                        } else if (i == 0) {
                            sum = val(lx && hy, elh, P, j) + val(hx && hy, ehh, 0, j);
                            in = (lx || hx) && hy;
                        } else {
                            sum = val(hx && hy, ehh, i, j);
                            in = hx && hy;
                        }
                        const int row = sy * P + j;
                        A[(f * P + i) * TL::PG + row * S1 + xs] =
                            in ? mul_r(sum, seg_inv_mass<R, P>(m, i, xkind, j, ykind)) : R(0);
                        if (tile) C[(f * P + i) * TL::PR + (row - P) * S1 + xs] = sum;
                    }
            }
        }
        __syncthreads();
        if (t.own_seg) {
#pragma unroll
            for (int f = 0; f < FB; ++f) mass_x<R, P, TL>(T, A + f * P * TL::PG, B + f * P * TL::PG, t.xs, t.xr, w0);
        }
        __syncthreads();
        if (t.own_x) {
#pragma unroll 2
            for (int k = 0; k < TL::KY; ++k) {
                const int sy = t.yr + k * RY, gyv = gy0 + (sy - 1) * P, ky = t.ykind(m, gyv);
                if (sy < 1 || sy > TEY || (!FULL && gyv >= m.nny)) continue;
#pragma unroll
                for (int f = 0; f < FB; ++f) {
                    const int at = (f * P + t.a) * TL::PG + sy * P * S1 + t.s;
                    R x[2 * P + 1], o[P];
                    seg_y<R, P>(B + at, S1, x);
                    seg_apply<R, P, 0>(T, x, vertex_weight<R, P, 0>(T, ky), o);
                    const long long node = (v0 + f) * m.NN + (long long)gyv * m.nnx + t.gx;
#pragma unroll
                    for (int c = 0; c < P; ++c)
                        if (FULL || gyv + c < m.nny) {
                            const long long n = node + (long long)c * m.nnx;
                            const R r = C[(f * P + t.a) * TL::PR + ((sy - 1) * P + c) * S1 + t.s];
                            rout[n] = r;
                            xout[n] = sweep_value(A[at + c * S1], r, o[c], h2, t.inv_mass(m, c, ky));
                        }
                }
            }
        }
    }
}

// The same on any tile, inside the mesh or at its edge, for NF of the fields
// (pointers to the first of them; of the udot sweep a multiple of
// udot_fields(NC)).  ws: TL::grad_ws, rhs_ws, sweep_ws or udot_ws(NC) values.
// All threads of the block call them together.
template <class R, int P, int NC, int NF, class TL>
DEV void grad_sweep_seg(const MeshDev& m, const R* u, R* bout, R* gout, int gx0, int gy0, int tid, R* ws) {
    if (tile_full<P, TL, 2>(m, gx0, gy0)) grad_sweep_body<R, P, NC, NF, TL, true>(m, u, bout, gout, gx0, gy0, tid, ws);
    else grad_sweep_body<R, P, NC, NF, TL, false>(m, u, bout, gout, gx0, gy0, tid, ws);
}
template <class R, int P, int NC, int NF, class TL>
DEV void grad_rhs_seg(const MeshDev& m, const R* u, R* bout, R* gout, int gx0, int gy0, int tid, R* ws) {
    if (tile_full<P, TL, 1>(m, gx0, gy0)) grad_rhs_body<R, P, NC, NF, TL, true>(m, u, bout, gout, gx0, gy0, tid, ws);
    else grad_rhs_body<R, P, NC, NF, TL, false>(m, u, bout, gout, gx0, gy0, tid, ws);
}
template <class R, int P, int NV, class TL>
DEV void mass_sweep_seg(const MeshDev& m, const R* xin, const R* b, R* xout, int gx0, int gy0, int tid, R* ws) {
    if (tile_full<P, TL, 1>(m, gx0, gy0)) mass_sweep_body<R, P, NV, TL, true>(m, xin, b, xout, gx0, gy0, tid, ws);
    else mass_sweep_body<R, P, NV, TL, false>(m, xin, b, xout, gx0, gy0, tid, ws);
}
template <class R, int P, int NC, int NF, class TL>
DEV void udot_sweep_seg(const MeshDev& m, const R* ER, R* rout, R* xout, int gx0, int gy0, int tid, R* ws) {
    if (tile_full<P, TL, 2>(m, gx0, gy0)) udot_sweep_body<R, P, NC, NF, TL, true>(m, ER, rout, xout, gx0, gy0, tid, ws);
    else udot_sweep_body<R, P, NC, NF, TL, false>(m, ER, rout, xout, gx0, gy0, tid, ws);
}

// The tiles of the single-state kernels (HALO: of the fused g_h kernel, by two
// elements smaller in each direction).  SIZE 0, large: 32 (p <= 2) or 16
// elements wide and 16 or 8 high, in float64 16 by 16 (p = 3) and 16 by 12 (p =
// 4), where the float64 pipe pays for every operation on the halo.  1, for
// meshes whose large tiles leave SMs idle: 16 (p = 1: 32) by 8 or 6.  2, for
// tiny meshes in float64, where a block's work is long against a launch: 8 by
// 4 to 8.
template <class R, int P, int SIZE, bool HALO>
struct StageTile {
    static constexpr bool F = sizeof(R) == 4;
    static constexpr int LX = SIZE == 2 ? 8 : SIZE == 1 ? (P == 1 ? 32 : 16) : (P <= 2 ? 32 : 16);
    static constexpr int NT = SIZE == 2 ? (P == 3 ? 72 : 64) : SIZE == 1 ? (P == 3 ? 96 : 128) : (P == 3 ? 192 : 256);
    static constexpr int RY = NT / (LX * P);
    static constexpr int ROWS = SIZE == 2 ? (RY >= 8 ? 8 : RY == 4 ? 4 : 6)
                                : SIZE == 1 ? (RY == 4 ? 8 : 6)
                                            : (P <= 2 ? 16 : F ? 8 : P == 3 ? 16 : 12);  // y segments
    using type = SegTile<R, P, LX, ROWS / RY, NT, HALO>;
};
template <class R, int P, int SIZE, bool HALO = false>
using stage_tile_t = typename StageTile<R, P, SIZE, HALO>::type;

// dynamic shared memory as an array of R (more than 48 KB in float64)
template <class R>
DEV R* dyn_shared() {
    extern __shared__ __align__(16) unsigned char dyn_smem[];
    return reinterpret_cast<R*>(dyn_smem);
}

// The stencil kernels.  A block takes NF of the fields: all of them, one after
// the other with the next one's loads under the passes of this one, where the
// tiles alone fill the GPU; else one (of the udot sweep udot_fields(NC)), and
// the grid has a layer for each.
template <int NF, int N>
DEV long long first_field(const MeshDev& m) {
    return NF == N ? 0 : (long long)(blockIdx.z * NF) * m.NN;
}

template <class R, int P, int NC, int NF, int SIZE>
__global__ void __launch_bounds__(stage_tile_t<R, P, SIZE>::NT, SIZE ? 1 : (P == 3 ? 4 : 3))
    k_grad_sweep(MeshDev m, const R* __restrict__ u, R* __restrict__ bout, R* __restrict__ gout) {
    using TL = stage_tile_t<R, P, SIZE, true>;
    pdl_begin();
    const long long at = first_field<NF, NC>(m);
    grad_sweep_seg<R, P, NC, NF, TL>(m, u + at, bout ? bout + at : bout, gout + at, blockIdx.x * TL::NX, blockIdx.y * TL::NY,
                                     threadIdx.x, dyn_shared<R>());
}

template <class R, int P, int NC, int NF, int SIZE>
__global__ void __launch_bounds__(stage_tile_t<R, P, SIZE>::NT)
    k_grad_rhs(MeshDev m, const R* __restrict__ u, R* __restrict__ bout, R* __restrict__ gout) {
    using TL = stage_tile_t<R, P, SIZE>;
    pdl_begin();
    const long long at = first_field<NF, NC>(m);
    grad_rhs_seg<R, P, NC, NF, TL>(m, u + at, bout + at, gout + at, blockIdx.x * TL::NX, blockIdx.y * TL::NY, threadIdx.x,
                                   dyn_shared<R>());
}

template <class R, int P, int NC, int NF, int SIZE>
__global__ void __launch_bounds__(stage_tile_t<R, P, SIZE>::NT)
    k_udot_sweep(MeshDev m, const R* __restrict__ ER, R* __restrict__ rout, R* __restrict__ xout) {
    using TL = stage_tile_t<R, P, SIZE>;
    pdl_begin();
    const long long at = first_field<NF, NC>(m);
    const R* __restrict__ er = ER + (NF == NC ? 0 : (long long)(blockIdx.z * NF) * m.E);
    udot_sweep_seg<R, P, NC, NF, TL>(m, er, rout + at, xout + at, blockIdx.x * TL::NX, blockIdx.y * TL::NY, threadIdx.x,
                                     dyn_shared<R>());
}

// (NV: the fields of a launch)
template <class R, int P, int NV, int NF, int SIZE>
__global__ void __launch_bounds__(stage_tile_t<R, P, SIZE>::NT)
    k_mass_sweep(MeshDev m, const R* __restrict__ xin, const R* __restrict__ b, R* __restrict__ xout) {
    using TL = stage_tile_t<R, P, SIZE>;
    pdl_begin();
    const long long at = first_field<NF, NV>(m);
    mass_sweep_seg<R, P, NF, TL>(m, xin + at, b + at, xout + at, blockIdx.x * TL::NX, blockIdx.y * TL::NY, threadIdx.x,
                                 dyn_shared<R>());
}

}  // namespace cgl
