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
// nodes (along y, and at the global stores) hits distinct banks as well.
//
// The sums run over the offsets -p .. p in order with explicit rounding, so
// the fused and the separate kernels, and every tile size, give the same bits.
#pragma once

#include "kernels.cuh"

namespace cgl {

// wrap (gx, gy) on periodic directions (wrap_periodic: any number of
// periods); false outside a non-periodic mesh
DEV bool wrap_node(const MeshDev& m, int& gx, int& gy) {
    bool in = true;
    if (m.py) gy = wrap_periodic(gy, m.nny);
    else in = gy >= 0 && gy < m.nny;
    if (m.px) gx = wrap_periodic(gx, m.nnx);
    else in = in && gx >= 0 && gx < m.nnx;
    return in;
}

// a tile of TEX x TEY elements (NX x NY nodes) worked by NT threads
template <class R, int P, int TEX_, int TEY_, int NT_>
struct SegTile {
    static constexpr int TEX = TEX_, TEY = TEY_, NT = NT_;
    static constexpr int NX = TEX * P, NY = TEY * P;
    // nodes and segments of the tile with one (1) and two (2) elements of halo
    // on the low side and one, two vertices' reach on the high side
    static constexpr int W1 = (TEX + 1) * P + 1, H1 = (TEY + 1) * P + 1, S1 = TEX + 2;
    static constexpr int W2 = (TEX + 3) * P + 1, H2 = (TEY + 3) * P + 1, S2 = TEX + 4;
    // plane stride: n words or more, congruent to a p-th of the banks
    static constexpr int plane(int n) {
        constexpr int B = 128 / (int)sizeof(R), want = P == 1 ? 0 : (B + P - 1) / P;
        int k = n;
        while (P > 1 && k % B != want % B) ++k;
        return k;
    }
    static constexpr int PU = plane(H2 * S2);   // u on the two-element halo
    static constexpr int PT = plane(H2 * S1);   // its x pass
    static constexpr int PG = plane(H1 * S1);   // an iterate on the one-element halo
    static constexpr int PS = plane(H1 * TEX);  // its x pass
    static constexpr int PR = plane(NY * TEX);  // a field on the tile
    static constexpr int NOWN = NX * TEY, NJ = (NOWN + NT - 1) / NT;  // (column, y segment) items
    static constexpr int grad_a = P * PU > 2 * P * PG ? P * PU : 2 * P * PG;
    static constexpr int grad_b = 2 * P * (PT > PS ? PT : PS);
    static constexpr int grad_ws = grad_a + grad_b;
    static constexpr int sweep_ws = P * (PG + PS);
    // fields of a udot sweep staged together: two where they take 32 KB at most
    static constexpr int udot1 = P * (PG + PS + PR);
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

// a segment's values along x (planes of stride PL, at: its row and segment)
// and along y (rows of stride S, at: its column, row the vertex's)
template <class R, int P>
DEV void seg_x(const R* f, int PL, int at, R (&x)[2 * P + 1]) {
#pragma unroll
    for (int k = 0; k <= 2 * P; ++k) x[k] = f[(k % P) * PL + at + k / P - 1];
}
template <class R, int P>
DEV void seg_y(const R* f, int S, int at, int row, R (&x)[2 * P + 1]) {
#pragma unroll
    for (int k = 0; k <= 2 * P; ++k) x[k] = f[at + (row + k - P) * S];
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

// Right-hand side of the g_h projection, its lumped iterate and the first
// sweep on the tile at (gx0, gy0), one component after the other: u on a
// two-element halo (the next component's loads run under this one's passes),
// x pass with the derivative and the mass operator, y pass to b and g0 on the
// one-element halo, then the sweep's x and y passes.  A thread keeps b and g0
// of its own nodes in registers from the first y pass to the second.  ws:
// TL::grad_ws values.  All threads of the block call it together.
// SWEEP false: b and g0 of the tile's nodes only.
template <class R, int P, int NC, class TL, bool SWEEP = true>
DEV void grad_sweep_seg(const MeshDev& m, const R* __restrict__ u, R* __restrict__ bout, R* __restrict__ gout, int gx0,
                        int gy0, int tid, R* ws) {
    constexpr int NT = TL::NT, NJ = TL::NJ, NX = TL::NX, TEX = TL::TEX, TEY = TL::TEY;
    constexpr int NA = (TL::W2 * TL::H2 + NT - 1) / NT;
    R* A = ws;                // u, then g0 (x and y parts)
    R* B = ws + TL::grad_a;   // the x passes
    const Tab<R>& T = tab_of<R>(m, P);
    const R h = PV<R>::h(m), h2 = PV<R>::h2(m);
    // segments and rows that feed nodes of the mesh (ragged tiles stop there)
    const int ns = min(TL::S1, (m.nnx - gx0 + P - 1) / P + 2), nr = min(TL::H2, m.nny - gy0 + 4 * P);
    long long off[NA];
    R next[NA];
#pragma unroll
    for (int j = 0; j < NA; ++j) {
        const int i = tid + j * NT, r = i / TL::W2, q = i - r * TL::W2;
        int gx = gx0 - 2 * P + q, gy = gy0 - 2 * P + r;
        const bool in = r < nr && wrap_node(m, gx, gy);
        off[j] = in ? (long long)gy * m.nnx + gx : -1;
        // through L2 (ld.global.cg): this runs before the kernel launched just
        // before it has completed
        next[j] = in ? __ldcg(&u[off[j]]) : R(0);
    }
#pragma unroll 1
    for (int c = 0; c < NC; ++c) {
#pragma unroll
        for (int j = 0; j < NA; ++j) {
            const int i = tid + j * NT, r = i / TL::W2, q = i - r * TL::W2;
            if (i < TL::W2 * TL::H2) A[(q % P) * TL::PU + r * TL::S2 + q / P] = next[j];
        }
        __syncthreads();
        if (c + 1 < NC) {
            const R* __restrict__ uc = u + (c + 1) * m.NN;
#pragma unroll
            for (int j = 0; j < NA; ++j)
                if (off[j] >= 0) next[j] = __ldcg(&uc[off[j]]);
        }
        for (int i = tid; i < TL::H2 * TL::S1; i += NT) {
            const int r = i / TL::S1, s = i - r * TL::S1;
            if (s >= ns || r >= nr) continue;
            if (!SWEEP && (s == 0 || s > TEX || r < P || r >= TL::H2 - P)) continue;  // feeds the halo only
            R x[2 * P + 1], o[P];
            seg_x<R, P>(A, TL::PU, r * TL::S2 + s + 1, x);
            const int kind = vertex_kind(gx0 + (s - 1) * P, m.nnx, m.px);
            seg_apply<R, P, 1>(T, x, vertex_weight<R, P, 1>(T, kind), o);
#pragma unroll
            for (int a = 0; a < P; ++a) B[a * TL::PT + i] = o[a];
            seg_apply<R, P, 0>(T, x, vertex_weight<R, P, 0>(T, kind), o);
#pragma unroll
            for (int a = 0; a < P; ++a) B[(P + a) * TL::PT + i] = o[a];
        }
        __syncthreads();
        // b and g0 = b / m_i (zero outside the mesh) on column q of the halo
        // tile and the rows of y segment sy
        R ob[NJ][2][P], og[NJ][2][P];
        auto column = [&](int q, int sy, R(&bx)[P], R(&by)[P], R(&vx)[P], R(&vy)[P]) {
            const int a = q % P, s = q / P;
            const int gx = gx0 - P + q, gyv = gy0 + (sy - 1) * P;
            const int kx = vertex_kind(gx, m.nnx, m.px), ky = vertex_kind(gyv, m.nny, m.py);
            R t[2 * P + 1];
            seg_y<R, P>(B + a * TL::PT, TL::S1, s, (sy + 1) * P, t);
            seg_apply<R, P, 0>(T, t, vertex_weight<R, P, 0>(T, ky), bx);
            seg_y<R, P>(B + (P + a) * TL::PT, TL::S1, s, (sy + 1) * P, t);
            seg_apply<R, P, 1>(T, t, vertex_weight<R, P, 1>(T, ky), by);
            const bool inx = m.px || (gx >= 0 && gx < m.nnx);
#pragma unroll
            for (int b = 0; b < P; ++b) {
                const int gy = gyv + b;
                const bool in = inx && (m.py || (gy >= 0 && gy < m.nny));
                const R inv = seg_inv_mass<R, P>(m, a, kx, b, ky);
                bx[b] = mul_r(h, bx[b]);
                by[b] = mul_r(h, by[b]);
                vx[b] = in ? mul_r(bx[b], inv) : R(0);
                vy[b] = in ? mul_r(by[b], inv) : R(0);
                if (SWEEP && (sy <= TEY || b == 0)) {
                    const int at = a * TL::PG + (sy * P + b) * TL::S1 + s;
                    A[at] = vx[b];
                    A[P * TL::PG + at] = vy[b];
                }
            }
        };
#pragma unroll
        for (int j = 0; j < NJ; ++j) {
            const int i = tid + j * NT, sy = i / NX, q = i - sy * NX;
            if (i < TL::NOWN && gx0 + q < m.nnx + P && gy0 + sy * P < m.nny + P)
                column(q + P, sy + 1, ob[j][0], ob[j][1], og[j][0], og[j][1]);
        }
        if constexpr (!SWEEP) {
#pragma unroll
            for (int j = 0; j < NJ; ++j) {
                const int i = tid + j * NT, sy = i / NX, q = i - sy * NX;
                const int gx = gx0 + q, gyv = gy0 + sy * P;
                if (i >= TL::NOWN || gx >= m.nnx || gyv >= m.nny) continue;
#pragma unroll
                for (int f = 0; f < 2; ++f) {
                    const long long node = (long long)(f * NC + c) * m.NN + (long long)gyv * m.nnx + gx;
#pragma unroll
                    for (int b = 0; b < P; ++b)
                        if (gyv + b < m.nny) {
                            bout[node + (long long)b * m.nnx] = ob[j][f][b];
                            gout[node + (long long)b * m.nnx] = og[j][f][b];
                        }
                }
            }
            continue;  // the next staging writes u, which no one reads any more
        }
        // the halo: the rows below and above the tile, then its sides
        constexpr int NROW = 2 * TL::W1, NEXT = NROW + (P + 1) * TEY;
        for (int i = tid; i < NEXT; i += NT) {
            int q, sy;
            if (i < NROW) {
                sy = i < TL::W1 ? 0 : TEY + 1;
                q = i < TL::W1 ? i : i - TL::W1;
            } else {
                const int k = i - NROW, w = k % (P + 1);
                sy = k / (P + 1) + 1;
                q = w < P ? w : TL::W1 - 1;
            }
            R b0[P], b1[P], v0[P], v1[P];
            column(q, sy, b0, b1, v0, v1);
        }
        __syncthreads();
        const int ns0 = ns - 2, nr1 = min(TL::H1, m.nny - gy0 + 2 * P);
        for (int i = tid; i < 2 * TL::H1 * TEX; i += NT) {
            const int f = i / (TL::H1 * TEX), k = i - f * (TL::H1 * TEX), r = k / TEX, s = k - r * TEX;
            if (s >= ns0 || r >= nr1) continue;
            R x[2 * P + 1], o[P];
            seg_x<R, P>(A + f * P * TL::PG, TL::PG, r * TL::S1 + s + 1, x);
            seg_apply<R, P, 0>(T, x, vertex_weight<R, P, 0>(T, vertex_kind(gx0 + s * P, m.nnx, m.px)), o);
#pragma unroll
            for (int a = 0; a < P; ++a) B[(f * P + a) * TL::PS + k] = o[a];
        }
        __syncthreads();
#pragma unroll
        for (int j = 0; j < NJ; ++j) {
            const int i = tid + j * NT, sy = i / NX, q = i - sy * NX;
            const int gx = gx0 + q, gyv = gy0 + sy * P;
            if (i >= TL::NOWN || gx >= m.nnx || gyv >= m.nny) continue;
            const int a = q % P, kx = vertex_kind(gx, m.nnx, m.px), ky = vertex_kind(gyv, m.nny, m.py);
#pragma unroll
            for (int f = 0; f < 2; ++f) {
                R t[2 * P + 1], o[P];
                seg_y<R, P>(B + (f * P + a) * TL::PS, TEX, q / P, (sy + 1) * P, t);
                seg_apply<R, P, 0>(T, t, vertex_weight<R, P, 0>(T, ky), o);
                const long long node = (long long)(f * NC + c) * m.NN + (long long)gyv * m.nnx + gx;
#pragma unroll
                for (int b = 0; b < P; ++b)
                    if (gyv + b < m.nny) {
                        const long long k = node + (long long)b * m.nnx;
                        gout[k] = sweep_value(og[j][f][b], ob[j][f][b], o[b], h2, seg_inv_mass<R, P>(m, a, kx, b, ky));
                        if (bout) bout[k] = ob[j][f][b];
                    }
            }
        }
    }
}

// x pass of a mass sweep for FB iterates staged at X (planes PG), into Y
template <class R, int P, int FB, class TL>
DEV void sweep_x(const MeshDev& m, const Tab<R>& T, const R* X, R* Y, int gx0, int gy0, int tid) {
    constexpr int TEX = TL::TEX;
    const int ns = (m.nnx - gx0 + P - 1) / P, nr = min(TL::H1, m.nny - gy0 + 2 * P);
    for (int i = tid; i < FB * TL::H1 * TEX; i += TL::NT) {
        const int f = i / (TL::H1 * TEX), k = i - f * (TL::H1 * TEX), r = k / TEX, s = k - r * TEX;
        if (s >= ns || r >= nr) continue;
        R x[2 * P + 1], o[P];
        seg_x<R, P>(X + f * P * TL::PG, TL::PG, r * TL::S1 + s + 1, x);
        seg_apply<R, P, 0>(T, x, vertex_weight<R, P, 0>(T, vertex_kind(gx0 + s * P, m.nnx, m.px)), o);
#pragma unroll
        for (int a = 0; a < P; ++a) Y[(f * P + a) * TL::PS + k] = o[a];
    }
}

// one Richardson sweep for NV fields on the tile; ws: TL::sweep_ws values
template <class R, int P, int NV, class TL>
DEV void mass_sweep_seg(const MeshDev& m, const R* __restrict__ xin, const R* __restrict__ b, R* __restrict__ xout,
                        int gx0, int gy0, int tid, R* ws) {
    constexpr int NT = TL::NT, NX = TL::NX;
    constexpr int NA = (TL::W1 * TL::H1 + NT - 1) / NT;
    R* A = ws;
    R* B = ws + P * TL::PG;
    const Tab<R>& T = tab_of<R>(m, P);
    const R h2 = PV<R>::h2(m);
    long long off[NA];
    R next[NA];
#pragma unroll
    for (int j = 0; j < NA; ++j) {
        const int i = tid + j * NT, r = i / TL::W1, q = i - r * TL::W1;
        int gx = gx0 - P + q, gy = gy0 - P + r;
        const bool in = r < TL::H1 && wrap_node(m, gx, gy);
        off[j] = in ? (long long)gy * m.nnx + gx : -1;
        next[j] = in ? xin[off[j]] : R(0);
    }
#pragma unroll 1
    for (int v = 0; v < NV; ++v) {
#pragma unroll
        for (int j = 0; j < NA; ++j) {
            const int i = tid + j * NT, r = i / TL::W1, q = i - r * TL::W1;
            if (i < TL::W1 * TL::H1) A[(q % P) * TL::PG + r * TL::S1 + q / P] = next[j];
        }
        __syncthreads();
        if (v + 1 < NV) {
            const R* __restrict__ xv = xin + (v + 1) * m.NN;
#pragma unroll
            for (int j = 0; j < NA; ++j)
                if (off[j] >= 0) next[j] = xv[off[j]];
        }
        sweep_x<R, P, 1, TL>(m, T, A, B, gx0, gy0, tid);
        __syncthreads();
        for (int i = tid; i < TL::NOWN; i += NT) {
            const int sy = i / NX, q = i - sy * NX, gx = gx0 + q, gyv = gy0 + sy * P;
            if (gx >= m.nnx || gyv >= m.nny) continue;
            const int a = q % P, kx = vertex_kind(gx, m.nnx, m.px), ky = vertex_kind(gyv, m.nny, m.py);
            R t[2 * P + 1], o[P];
            seg_y<R, P>(B + a * TL::PS, TL::TEX, q / P, (sy + 1) * P, t);
            seg_apply<R, P, 0>(T, t, vertex_weight<R, P, 0>(T, ky), o);
            const long long node = v * m.NN + (long long)gyv * m.nnx + gx;
#pragma unroll
            for (int c = 0; c < P; ++c)
                if (gyv + c < m.nny) {
                    const long long k = node + (long long)c * m.nnx;
                    xout[k] = sweep_value(A[a * TL::PG + ((sy + 1) * P + c) * TL::S1 + q / P + 1], b[k], o[c], h2,
                                          seg_inv_mass<R, P>(m, a, kx, c, ky));
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
// ws: TL::udot_ws(NC) values.
template <class R, int P, int NC, class TL>
DEV void udot_sweep_seg(const MeshDev& m, const R* __restrict__ ER, R* __restrict__ rout, R* __restrict__ xout, int gx0,
                        int gy0, int tid, R* ws) {
    constexpr int NT = TL::NT, NX = TL::NX, TEX = TL::TEX, TEY = TL::TEY, N1 = P + 1;
    constexpr int FB = TL::udot_fields(NC);
    R* A = ws;                    // udot0 on the one-element halo
    R* B = A + FB * P * TL::PG;   // its x pass
    R* C = B + FB * P * TL::PS;   // r on the tile
    const Tab<R>& T = tab_of<R>(m, P);
    const R h2 = PV<R>::h2(m);
    const int ex0 = gx0 / P, ey0 = gy0 / P;
    const long long E = m.E;
#pragma unroll 1
    for (int v0 = 0; v0 < NC; v0 += FB) {
        if (v0 > 0) __syncthreads();  // the previous fields are consumed
        for (int i = tid; i < (TEX + 2) * (TEY + 2); i += NT) {
            const int sy = i / (TEX + 2), sx = i - sy * (TEX + 2);
            // the elements before (l) and after (h) the vertex along x and y;
            // hx, hy false: the segment has its vertex only (or lies outside)
            int xl = ex0 + sx - 2, xh = xl + 1, yl = ey0 + sy - 2, yh = yl + 1;
            if (xl > m.nx || yl > m.ny) continue;  // feeds no node of the mesh
            if (m.px) xl = wrap_periodic(xl, m.nx), xh = wrap_periodic(xh, m.nx);
            if (m.py) yl = wrap_periodic(yl, m.ny), yh = wrap_periodic(yh, m.ny);
            const bool lx = xl >= 0 && xl < m.nx, hx = xh >= 0 && xh < m.nx;
            const bool ly = yl >= 0 && yl < m.ny, hy = yh >= 0 && yh < m.ny;
            const int kx = m.px ? 0 : (!lx ? 1 : !hx ? 2 : 0), ky = m.py ? 0 : (!ly ? 1 : !hy ? 2 : 0);
            const bool tile = sx >= 1 && sx <= TEX && sy >= 1 && sy <= TEY;
            const long long ell = (long long)yl * m.nx + xl, ehl = (long long)yl * m.nx + xh;
            const long long elh = (long long)yh * m.nx + xl, ehh = (long long)yh * m.nx + xh;
#pragma unroll
            for (int f = 0; f < FB; ++f) {
                const R* __restrict__ Ev = ER + (v0 + f) * E;
                auto val = [&](bool in, long long e, int a, int b) {
                    return in ? Ev[(long long)((b * N1 + a) * NC) * E + e] : R(0);
                };
#pragma unroll
                for (int b = 0; b < P; ++b)
#pragma unroll
                    for (int a = 0; a < P; ++a) {
                        // past the last vertex of the halo
                        if ((a > 0 && sx == TEX + 1) || (b > 0 && sy == TEY + 1)) continue;
                        R s;
                        bool in;
                        if (a == 0 && b == 0) {
                            s = ((val(lx && ly, ell, P, P) + val(hx && ly, ehl, 0, P)) + val(lx && hy, elh, P, 0)) +
                                val(hx && hy, ehh, 0, 0);
                            in = (lx || hx) && (ly || hy);
                        } else if (b == 0) {
                            s = val(hx && ly, ehl, a, P) + val(hx && hy, ehh, a, 0);
                            in = hx && (ly || hy);
                        } else if (a == 0) {
                            s = val(lx && hy, elh, P, b) + val(hx && hy, ehh, 0, b);
                            in = (lx || hx) && hy;
                        } else {
                            s = val(hx && hy, ehh, a, b);
                            in = hx && hy;
                        }
                        const int q = sx, row = sy * P + b;
                        A[(f * P + a) * TL::PG + row * TL::S1 + q] =
                            in ? mul_r(s, seg_inv_mass<R, P>(m, a, kx, b, ky)) : R(0);
                        if (tile) C[(f * P + a) * TL::PR + (row - P) * TEX + q - 1] = s;
                    }
            }
        }
        __syncthreads();
        sweep_x<R, P, FB, TL>(m, T, A, B, gx0, gy0, tid);
        __syncthreads();
        for (int i = tid; i < TL::NOWN; i += NT) {
            const int sy = i / NX, q = i - sy * NX, gx = gx0 + q, gyv = gy0 + sy * P;
            if (gx >= m.nnx || gyv >= m.nny) continue;
            const int a = q % P, kx = vertex_kind(gx, m.nnx, m.px), ky = vertex_kind(gyv, m.nny, m.py);
#pragma unroll
            for (int f = 0; f < FB; ++f) {
                R t[2 * P + 1], o[P];
                seg_y<R, P>(B + (f * P + a) * TL::PS, TEX, q / P, (sy + 1) * P, t);
                seg_apply<R, P, 0>(T, t, vertex_weight<R, P, 0>(T, ky), o);
                const long long node = (v0 + f) * m.NN + (long long)gyv * m.nnx + gx;
#pragma unroll
                for (int c = 0; c < P; ++c)
                    if (gyv + c < m.nny) {
                        const long long k = node + (long long)c * m.nnx;
                        const R r = C[(f * P + a) * TL::PR + (sy * P + c) * TEX + q / P];
                        rout[k] = r;
                        xout[k] = sweep_value(A[(f * P + a) * TL::PG + ((sy + 1) * P + c) * TL::S1 + q / P + 1], r, o[c],
                                              h2, seg_inv_mass<R, P>(m, a, kx, c, ky));
                    }
            }
        }
    }
}

// The tiles of the single-state kernels.  Large: about 1024 nodes and 256
// threads (float64 with fewer rows at p >= 3, where 48 KB of shared memory
// ends); small: 4 x 4 elements (8 x 8 at p = 1) and 64 threads, for meshes
// whose large tiles leave SMs idle.
template <class R, int P, bool SMALL>
struct StageTile {
    static constexpr bool F = sizeof(R) == 4;
    static constexpr int X = SMALL ? (P == 1 ? 8 : 4) : (P == 1 ? 32 : P == 2 ? 16 : P == 3 ? 12 : 8);
    static constexpr int Y = SMALL ? (P == 1 ? 8 : 4) : (P <= 2 ? 16 : P == 3 ? (F ? 12 : 7) : (F ? 8 : 6));
    using type = SegTile<R, P, X, Y, SMALL ? 64 : 256>;
};
template <class R, int P, bool SMALL>
using stage_tile_t = typename StageTile<R, P, SMALL>::type;

template <class R, int P, int NC, bool SMALL>
__global__ void __launch_bounds__(SMALL ? 64 : 256, SMALL ? 1 : (sizeof(R) == 4 ? 3 : 2))
    k_grad_sweep(MeshDev m, const R* __restrict__ u, R* __restrict__ bout, R* __restrict__ gout) {
    using TL = stage_tile_t<R, P, SMALL>;
    // like k_grad_rhs: runs beside k_pre, waits for it before exiting
    pdl_trigger();
    __shared__ R ws[TL::grad_ws];
    grad_sweep_seg<R, P, NC, TL>(m, u, bout, gout, blockIdx.x * TL::NX, blockIdx.y * TL::NY, threadIdx.x, ws);
    pdl_wait();
}

template <class R, int P, int NC, bool SMALL>
__global__ void __launch_bounds__(SMALL ? 64 : 256)
    k_grad_rhs(MeshDev m, const R* __restrict__ u, R* __restrict__ bout, R* __restrict__ gout) {
    using TL = stage_tile_t<R, P, SMALL>;
    // needs only u, whose last writer completed before k_pre let this kernel
    // start (pdl_wait_then_trigger), so it runs beside k_pre and waits for it
    // only before exiting
    pdl_trigger();
    __shared__ R ws[TL::grad_ws];
    grad_sweep_seg<R, P, NC, TL, false>(m, u, bout, gout, blockIdx.x * TL::NX, blockIdx.y * TL::NY, threadIdx.x, ws);
    pdl_wait();
}

template <class R, int P, int NC, bool SMALL>
__global__ void __launch_bounds__(SMALL ? 64 : 256)
    k_udot_sweep(MeshDev m, const R* __restrict__ ER, R* __restrict__ rout, R* __restrict__ xout) {
    using TL = stage_tile_t<R, P, SMALL>;
    pdl_begin();
    __shared__ R ws[TL::udot_ws(NC)];
    udot_sweep_seg<R, P, NC, TL>(m, ER, rout, xout, blockIdx.x * TL::NX, blockIdx.y * TL::NY, threadIdx.x, ws);
}

template <class R, int P, int NV, bool SMALL>
__global__ void __launch_bounds__(SMALL ? 64 : 256)
    k_mass_sweep(MeshDev m, const R* __restrict__ xin, const R* __restrict__ b, R* __restrict__ xout) {
    using TL = stage_tile_t<R, P, SMALL>;
    pdl_begin();
    __shared__ R ws[TL::sweep_ws];
    mass_sweep_seg<R, P, NV, TL>(m, xin, b, xout, blockIdx.x * TL::NX, blockIdx.y * TL::NY, threadIdx.x, ws);
}

}  // namespace cgl
