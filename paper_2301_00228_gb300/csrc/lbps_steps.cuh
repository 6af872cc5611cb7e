// Device functions of one time step, shared by the kernels of the
// translation units: the boundary rules of one boundary point, and the strips
// of interior points that a warp advances by one step or by two.
#pragma once

#include "lbps_launch.h"

namespace lbps {

namespace {

// ------------------------------------------------------------- boundary

// One warp's FP64 instruction holds its sub-partition's FP64 pipe for about 64
// cycles (2 lanes a clock and SM), so the boundary passes are bound by the
// number of FP64 instructions on their chains.  Hence: the stencils of every
// point and its neighbours are settled at creation (BNode::kinds, no node-type
// loads, no weights in local memory); terms whose weight is 0 or 1 are left
// out; the x and y components of the Newmark pass, and a point's own reset and
// its neighbours' stresses, are separate tasks of separate warps; first
// moments stay in the populations' type (FP32 - FP32 rounded through FP64 is
// the FP32 difference).

// Where boundary point b lies, its difference stencils (BNode::kinds) and the
// interior neighbours it streams into (BNode::smask).  A rectangle's follow
// from its place in the perimeter list: computed, so that the loads of u do
// not wait for the table's (an interior neighbour's stencils are central).
struct BPoint {
    int i, j, kinds, smask;
};
__device__ __forceinline__ BPoint point_of(const Geo& g, const BNode* __restrict__ bn, int b) {
    BPoint p;
    if (g.general) {
        p.i = LBPS_LD(&bn[b].i);
        p.j = LBPS_LD(&bn[b].j);
        p.kinds = LBPS_LD(&bn[b].kinds);
        p.smask = LBPS_LD(&bn[b].smask);
        return p;
    }
    const int rows = g.periodic_y ? 0 : 2 * g.nx;   // the inverse of perim_index
    if (b < rows) {
        p.i = b < g.nx ? b : b - g.nx;
        p.j = b < g.nx ? 0 : g.ny - 1;
    } else {
        const int jlo = g.periodic_y ? 0 : 1, len = g.ny - 2 * jlo, q = b - rows;
        p.i = q < len ? 0 : g.nx - 1;
        p.j = jlo + (q < len ? q : q - len);
    }
    const bool l = !g.periodic_x && p.i == 0, r = !g.periodic_x && p.i == g.nx - 1;
    const bool d = !g.periodic_y && p.j == 0, u = !g.periodic_y && p.j == g.ny - 1;
    p.kinds = (l ? DIFF_FORWARD : r ? DIFF_BACKWARD : DIFF_CENTRAL) |
              (d ? DIFF_FORWARD : u ? DIFF_BACKWARD : DIFF_CENTRAL) << 2;
    p.smask = (l || r) && (d || u) ? 0 : l ? 1 : r ? 4 : d ? 2 : 8;   // none at corners
    return p;
}

// Differences of u at (i, j): xx = du_x/dx, yx = du_y/dx, xy = du_x/dy, yy = du_y/dy.
struct Grad {
    double xx, yx, xy, yy;
};
__device__ __forceinline__ Grad grad_at(const Geo& g, const Consts& c, const double* ux, const double* uy, int i,
                                        int j, int kx, int ky) {
    const size_t p = (size_t)j * g.px + i;
    Grad d;
    d.xx = mul_rn(diff3(ux + p, kx, i, g.nx, 1), c.inv2h);
    d.yx = mul_rn(diff3(uy + p, kx, i, g.nx, 1), c.inv2h);
    d.xy = mul_rn(diff3(ux + p, ky, j, g.ny, g.px), c.inv2h);
    d.yy = mul_rn(diff3(uy + p, ky, j, g.ny, g.px), c.inv2h);
    return d;
}

// Cauchy stress (Eq. hooke with the strain of Eq. strain) from the differences
// of u at a point; s = {xx, yy, xy}.
__device__ __forceinline__ void stress_of(const Consts& c, const Grad& d, double s[3]) {
    const double tr = mul_rn(c.lam, add_rn(d.xx, d.yy));
    s[0] = add_rn(tr, mul_rn(c.two_mu, d.xx));
    s[1] = add_rn(tr, mul_rn(c.two_mu, d.yy));
    s[2] = mul_rn(c.mu, add_rn(d.xy, d.yx));
}

// Component Q (0 x, 1 y) of Eq. acc_neumann for the boundary cell of (i, j):
// the square of side dh clipped to the rectangle; one face per existing
// neighbour r with normal pointing to r, length l_kr, stress (sigma_k +
// sigma_r)/2; external force F = int t* da (component f) supplied per point.
// The stresses come from the stress pass: slot b at boundary point b, slot nb
// + b at its interior neighbour.
// General geometry (reading R14): the cell's side lengths and 1/(rho V_C)
// come with the point; sigma at b is in slot 5b and at its body neighbour in
// direction d in slot 5b + 1 + d; a side facing no
// body neighbour but lying partly in the body carries sigma_k.
template <int Q>
__device__ __forceinline__ double accel_neumann(const Geo& g, const Consts& c, const BNode* __restrict__ bn,
                                                const double* __restrict__ sig, int nb, int b, int i, int j,
                                                double f) {
    // the stress component that a face across x, across y contributes
    constexpr int CX = Q == 0 ? 0 : 2, CY = Q == 0 ? 2 : 1;
    if (g.general) {
        const int nbm = LBPS_LD(&bn[b].nbmask);
        const double kx = LBPS_LD(&sig[(size_t)b * 15 + CX]), ky = LBPS_LD(&sig[(size_t)b * 15 + CY]);
#pragma unroll
        for (int d = 0; d < 4; ++d) {   // E, N, W, S
            const double len = LBPS_LD(&bn[b].l[d]);
            const bool has = (nbm >> d) & 1;
            if (!has && !(len > 0.0)) continue;
            const double k = (d & 1) ? ky : kx;
            const double r = has ? LBPS_LD(&sig[(size_t)b * 15 + 3 * (1 + d) + ((d & 1) ? CY : CX)]) : k;
            f = add_rn(f, mul_rn(add_rn(k, r), mul_rn(d < 2 ? 0.5 : -0.5, len)));
        }
        return mul_rn(f, LBPS_LD(&bn[b].inv_m));
    }
    const bool hE = g.periodic_x || i < g.nx - 1, hN = g.periodic_y || j < g.ny - 1;
    const bool hW = g.periodic_x || i > 0, hS = g.periodic_y || j > 0;
    const bool fullx = hE && hW, fully = hN && hS;
    // half the length of a face across x, across y
    const double lx = fully ? c.half_dh : c.quarter_dh, ly = fullx ? c.half_dh : c.quarter_dh;
    const double kx = LBPS_LD(&sig[(size_t)b * 3 + CX]), ky = LBPS_LD(&sig[(size_t)b * 3 + CY]);
    auto slot = [&](int ri, int rj) {
        return is_boundary(ri, rj, g) ? (size_t)perim_index(ri, rj, g) : (size_t)nb + b;
    };
    if (hE) f = add_rn(f, mul_rn(add_rn(kx, LBPS_LD(&sig[slot(wrap(i + 1, g.nx), j) * 3 + CX])), lx));
    if (hN) f = add_rn(f, mul_rn(add_rn(ky, LBPS_LD(&sig[slot(i, wrap(j + 1, g.ny)) * 3 + CY])), ly));
    if (hW) f = sub_rn(f, mul_rn(add_rn(kx, LBPS_LD(&sig[slot(wrap(i - 1, g.nx), j) * 3 + CX])), lx));
    if (hS) f = sub_rn(f, mul_rn(add_rn(ky, LBPS_LD(&sig[slot(i, wrap(j - 1, g.ny)) * 3 + CY])), ly));
    // 1 / (rho V_C): V_C is dh^2, dh^2/2 or dh^2/4 (exact powers of two)
    return mul_rn(f, mul_rn(c.inv_rho_dh2, fullx ? (fully ? 1.0 : 2.0) : (fully ? 2.0 : 4.0)));
}

// Value streamed out of a boundary source (Eq. LBE_mod).  f-hat is the mean
// of the stored (a5, copy A) and reset (b5, copy B) populations of the
// source; the equilibrium is taken from f-hat (mode 0) or from f(x_k, t)
// (mode 1).  ALPHA is the direction of travel (1..4), OPP its reverse.
template <int ALPHA, int OPP, typename V>
__device__ __forceinline__ V stream_from_boundary(const V (&a5)[5], const V (&b5)[5], const KC<V>& k, int set, int mode) {
    V h5[5];
#pragma unroll
    for (int q = 0; q < 5; ++q) h5[q] = mul_rn((V)0.5, add_rn(a5[q], b5[q]));
    if (mode == 0) {
        V sh = sum5(h5[0], h5[1], h5[2], h5[3], h5[4]);
        return fma_rn(k.two_a[set], sh, -h5[OPP]);  // 2 f_eq(f-hat) - f-hat = 2 a s-hat - f-hat^opp
    }
    V sa = sum5(a5[0], a5[1], a5[2], a5[3], a5[4]);
    V ej = sub_rn(a5[ALPHA], a5[OPP]);              // e_alpha . Jbar(x_k, t)
    return sub_rn(add_rn(mul_rn(k.two_a[set], sa), ej), h5[ALPHA]);
}

// The boundary work of a step runs in two passes over the perimeter list,
// each one thread per boundary point b at (i, j) and part:
//   newmark  acceleration of b (Eq. acc_neumann, from the stresses of copy A,
//            or Eq. acc_dirichlet) and u(t + dt) at b; parts: x, y;
//   (the interior kernel runs here: u(t + dt) at every interior point)
//   reset    phi, psi from differences of u(t + dt) (Eq. psi_phi_at_bound),
//            populations by Eq. correction-f, the value b streams into its
//            interior neighbour (Eq. LBE_mod), written over the population the
//            interior kernel put there, and the stresses of u(t + dt) that
//            the next step's Eq. acc_neumann reads, into copy B; parts: the
//            point itself, the stresses at its neighbours.
// Each copy thus carries the stresses of its own u; the stress pass below
// computes them where u was set otherwise (initialisation).

// sigma at b (slot b of a rectangle, 5b of a general geometry).
__device__ __forceinline__ void store_point_stress(const Geo& g, double* __restrict__ sig, int b,
                                                   const double s[3]) {
    const size_t o = (size_t)b * (g.general ? 15 : 3);
#pragma unroll
    for (int q = 0; q < 3; ++q) LBPS_ST(&sig[o + q], s[q]);
}

// sigma at the neighbours of b that its Eq. acc_neumann reads besides the
// boundary points: the interior neighbour of a rectangle's edge point (slot
// nb + b), the body neighbours of a general boundary point (slot 5b + 1 + d).
__device__ __forceinline__ void neighbour_stresses(const Geo& g, const Consts& c, const double* ux, const double* uy,
                                                   const BNode* __restrict__ bn, int nb, double* __restrict__ sig,
                                                   int b) {
    const BPoint pt = point_of(g, bn, b);
    const int mask = g.general ? LBPS_LD(&bn[b].nbmask) : pt.smask;
    for (int d = 0; d < 4; ++d) {   // E, N, W, S
        if (!((mask >> d) & 1)) continue;
        const int ni = wrap(pt.i + (d == 0) - (d == 2), g.nx), nj = wrap(pt.j + (d == 1) - (d == 3), g.ny);
        double s[3];
        stress_of(c, grad_at(g, c, ux, uy, ni, nj, (pt.kinds >> (4 + 4 * d)) & 3, (pt.kinds >> (6 + 4 * d)) & 3), s);
        const size_t o = g.general ? (size_t)b * 15 + 3 * (1 + d) : ((size_t)nb + b) * 3;
#pragma unroll
        for (int q = 0; q < 3; ++q) LBPS_ST(&sig[o + q], s[q]);
    }
}

__device__ __forceinline__ void boundary_stress(const Geo& g, const Consts& c, const double* ux, const double* uy,
                                       const BNode* __restrict__ bn, int nb, double* __restrict__ sig, int b) {
    const BPoint pt = point_of(g, bn, b);
    double s[3];
    stress_of(c, grad_at(g, c, ux, uy, pt.i, pt.j, pt.kinds & 3, (pt.kinds >> 2) & 3), s);
    store_point_stress(g, sig, b, s);
    neighbour_stresses(g, c, ux, uy, bn, nb, sig, b);
}

// Component Q of the Newmark pass.  n: the steps done so far; time-dependent
// data take the Neumann force at t_n and the Dirichlet target at t_{n+1}.
template <int Q, typename P>
__device__ __forceinline__ void boundary_newmark_q(const Geo& g, const Consts& c, const View<P>& A, const View<P>& B,
                                                   const BNode* __restrict__ bn, int nb,
                                                   const double* __restrict__ sig, double n, int b) {
    const BPoint pt = point_of(g, bn, b);
    const int i = pt.i, j = pt.j;
    const bool fixed = LBPS_LD(&bn[b].type) == DIRICHLET;
    const size_t p = (size_t)j * g.px + i;
    const double u = LBPS_LD(&A.u[Q * g.plane + p]), v = LBPS_LD(&A.u[(2 + Q) * g.plane + p]);
    double data = LBPS_LD(Q == 0 ? &bn[b].bx : &bn[b].by);
    if (c.load_rate[fixed] > 0.0) data = mul_rn(load_factor(c, fixed, (fixed ? n + 1.0 : n) * c.dt), data);
    double a;
    if (fixed)
        a = sub_rn(mul_rn(c.two_dt2, sub_rn(data, u)), mul_rn(c.two_dt, v));
    else
        a = accel_neumann<Q>(g, c, bn, sig, nb, b, i, j, data);
    double u1, v1;
    newmark(u, v, a, c, u1, v1);
    LBPS_ST(&B.u[Q * g.plane + p], u1);
    LBPS_ST(&B.u[(2 + Q) * g.plane + p], v1);
}

// Part 0 (x) or 1 (y) of it; the part is uniform over a warp.
template <typename P>
__device__ __forceinline__ void boundary_newmark(const Geo& g, const Consts& c, const View<P>& A, const View<P>& B,
                                        const BNode* __restrict__ bn, int nb, const double* __restrict__ sig,
                                        double n, int b, int part) {
    if (part == 0)
        boundary_newmark_q<0, P>(g, c, A, B, bn, nb, sig, n, b);
    else
        boundary_newmark_q<1, P>(g, c, A, B, bn, nb, sig, n, b);
}

// bc_j_mode 1: J(x_k, t) of Eq. correction-f is the first moment of the
// populations the plain LBE (Eq. LBE, from copy A) streams into (i, j):
// direction alpha arrives from the body neighbour at x - e_alpha as
// 2 a s - f^opp there (tau = dt/2); a direction whose source is outside the
// body keeps the point's own stored population (own5).
template <typename P>
__device__ __forceinline__ void partial_stream_moment(const Geo& g, const KCof<P>& k, const View<P>& A, int i, int j,
                                             const typename P::V (&own5)[2][5], typename P::V (&jx)[2],
                                             typename P::V (&jy)[2]) {
    using V = typename P::V;
    const int SX[5] = {0, -1, 0, 1, 0};  // source offset x - e_alpha
    const int SY[5] = {0, 0, -1, 0, 1};
    const int OPP[5] = {0, 3, 4, 1, 2};
    V in5[2][5];
#pragma unroll
    for (int set = 0; set < 2; ++set)
#pragma unroll
        for (int q = 1; q < 5; ++q) in5[set][q] = own5[set][q];
#pragma unroll
    for (int q = 1; q < 5; ++q) {
        const int si = i + SX[q], sj = j + SY[q];
        if (!body_at(g, si, sj)) continue;
        typename P::Raw r;
        P::template load_raw<false>(A.f, g.plane, (size_t)wrap(sj, g.ny) * g.px + wrap(si, g.nx), true, r);
#pragma unroll
        for (int set = 0; set < 2; ++set) {
            V f5[5];
            P::decode(r, set, k, f5);
            in5[set][q] = fma_rn(k.two_a[set], sum5(f5[0], f5[1], f5[2], f5[3], f5[4]), -f5[OPP[q]]);
        }
    }
#pragma unroll
    for (int set = 0; set < 2; ++set) {
        jx[set] = sub_rn(in5[set][1], in5[set][3]);
        jy[set] = sub_rn(in5[set][2], in5[set][4]);
    }
}

// The populations boundary point (i, j) streams into its interior
// neighbours, the directions d (0: +x, 1: +y, 2: -x, 3: -y) set in mask, from
// its populations at t (a5s) and after the reset (b5s) (Eq. LBE_mod).
template <typename P>
__device__ __forceinline__ void stream_out(const Geo& g, const Consts& c, const KCof<P>& k, const View<P>& B, int i, int j,
                                  int mask, const typename P::V (&a5s)[2][5], const typename P::V (&b5s)[2][5]) {
    using V = typename P::V;
    const int DXS[4] = {1, 0, -1, 0};
    const int DYS[4] = {0, 1, 0, -1};
#pragma unroll
    for (int d = 0; d < 4; ++d) {
        if (!((mask >> d) & 1)) continue;
        V v[2];
#pragma unroll
        for (int set = 0; set < 2; ++set) {
            switch (d) {
            case 0: v[set] = stream_from_boundary<1, 3>(a5s[set], b5s[set], k, set, c.bc_feq_mode); break;
            case 1: v[set] = stream_from_boundary<2, 4>(a5s[set], b5s[set], k, set, c.bc_feq_mode); break;
            case 2: v[set] = stream_from_boundary<3, 1>(a5s[set], b5s[set], k, set, c.bc_feq_mode); break;
            default: v[set] = stream_from_boundary<4, 2>(a5s[set], b5s[set], k, set, c.bc_feq_mode); break;
            }
        }
        const size_t pin = (size_t)wrap(j + DYS[d], g.ny) * g.px + wrap(i + DXS[d], g.nx);
        P::store1_both(B.f, g.plane, pin, d + 1, v, k);
    }
}

// The reset of point b itself; with NEIGHBOURS also the stresses at its
// neighbours (otherwise a part of its own, neighbour_stresses).
template <typename P, bool NEIGHBOURS = false>
__device__ __forceinline__ bool boundary_reset(const Geo& g, const Consts& c, const KCof<P>& k, const View<P>& A,
                                               const View<P>& B, const BNode* __restrict__ bn, int nb, int b) {
    using V = typename P::V;
    const BPoint pt = point_of(g, bn, b);
    const int i = pt.i, j = pt.j, smask = pt.smask;
    const size_t p = (size_t)j * g.px + i;
    // The populations at t (copy A's boundary mirror, entry b, coalesced
    // along the boundary list) and every difference are loaded before the
    // first store: no load may pass a store, and together their latencies
    // overlap.
    typename P::Raw ra, rb;
    P::template load_raw<false>(A.m, g.mplane, (size_t)b, true, ra);
    // Eq. psi_phi_at_bound: differences of u(t + dt) at (i, j).
    const Grad d = grad_at(g, c, B.u, B.u + g.plane, i, j, pt.kinds & 3, (pt.kinds >> 2) & 3);
    if (NEIGHBOURS) {
        if (g.general) {
            neighbour_stresses(g, c, B.u, B.u + g.plane, bn, nb, B.s, b);
        } else if (smask) {   // the one interior neighbour of an edge point
            const Grad e = grad_at(g, c, B.u, B.u + g.plane, i + (smask == 1) - (smask == 4),
                                   j + (smask == 2) - (smask == 8), DIFF_CENTRAL, DIFF_CENTRAL);
            double s[3];
            stress_of(c, e, s);
#pragma unroll
            for (int q = 0; q < 3; ++q) LBPS_ST(&B.s[((size_t)nb + b) * 3 + q], s[q]);
        }
    }
    const double phi = add_rn(d.xx, d.yy);
    const double psi = sub_rn(d.yx, d.xy);
    // Eq. correction-f with J(x_k, t) of the stored populations, then the value
    // this point streams into each interior neighbour (Eq. LBE_mod): the
    // population travelling that way, replacing what the interior kernel
    // wrote there (a rectangle's edge point has one such neighbour, a corner
    // none; next to a hole a point may have several).
    // The reset populations go to the lattice and to copy B's mirror.
    V a5s[2][5], b5s[2][5];
    const double sv[2] = {phi, psi};
    V jx[2], jy[2];
#pragma unroll
    for (int set = 0; set < 2; ++set) {
        P::decode(ra, set, k, a5s[set]);
        jx[set] = sub_rn(a5s[set][1], a5s[set][3]);
        jy[set] = sub_rn(a5s[set][2], a5s[set][4]);
    }
    if (c.bc_j_mode == 1) partial_stream_moment<P>(g, k, A, i, j, a5s, jx, jy);
    P::eq_raw(p, c, sv, jx, jy, k, rb);
    P::store_raw(B.f, g.plane, p, rb);
    P::store_raw(B.m, g.mplane, (size_t)b, rb);
    if (smask)
#pragma unroll
        for (int set = 0; set < 2; ++set) P::decode(rb, set, k, b5s[set]);
    // a policy whose words hold both pairs of a point leaves the y streams to
    // a second pass (boundary_stream_y): two boundary points may stream into
    // one point along x and along y
    stream_out<P>(g, c, k, B, i, j, P::kSplitStream ? (smask & 5) : smask, a5s, b5s);
    // sigma of u(t + dt) at b (from the same differences), for the next step
    double s[3];
    stress_of(c, d, s);
    store_point_stress(g, B.s, b, s);
    return !isfinite((V)phi + (V)psi);
}

// The y streams of the reset for PopBfp13 (P::kSplitStream), in a pass after
// the one that wrote everything else: the values depend only on the boundary
// point's populations at t (copy A's mirror) and those the reset stored for
// t + dt (copy B's mirror), which that pass left as they are.
template <typename P>
__device__ __forceinline__ void boundary_stream_y(const Geo& g, const Consts& c, const KCof<P>& k, const View<P>& A,
                                         const View<P>& B, const BNode* __restrict__ bn, int b) {
    using V = typename P::V;
    const BPoint pt = point_of(g, bn, b);
    const int smask = pt.smask & 10, i = pt.i, j = pt.j;
    if (!smask) return;
    typename P::Raw ra, rb;
    P::template load_raw<false>(A.m, g.mplane, (size_t)b, true, ra);
    P::template load_raw<false>(B.m, g.mplane, (size_t)b, true, rb);
    V a5s[2][5], b5s[2][5];
#pragma unroll
    for (int set = 0; set < 2; ++set) {
        P::decode(ra, set, k, a5s[set]);
        P::decode(rb, set, k, b5s[set]);
    }
    stream_out<P>(g, c, k, B, i, j, smask, a5s, b5s);
}

// ---------------------------------------------------------------- bulk

// Bulk kernel: each warp owns a strip of kStripCols output columns and marches
// along y over kRowsPerWarp rows.  Lane l holds column xs - 1 + l, so lanes 0
// and 31 are halo lanes whose values reach their neighbours by shuffles; the
// rows above and below stay in registers, and the populations are prefetched
// two rows ahead (in their stored form, decoded when the row window shifts).
// Every lattice point's words are read once per launch (plus the two halo
// columns and two halo rows of each strip).
constexpr int kStripCols = 30;
static_assert(kStripCols == kBatchStripCols, "one strip width for the single-lattice and batched kernels");
constexpr int kWarpsPerBlock = 4;

template <typename P>
__device__ __forceinline__ void decode_row(const typename P::Raw& r, const KCof<P>& k,
                                           typename P::V (&f)[2][5]) {
#pragma unroll
    for (int s = 0; s < 2; ++s) P::decode(r, s, k, f[s]);
}

template <bool NC = true>
__device__ __forceinline__ void load_uv(const double* __restrict__ U, size_t plane, size_t p, bool ok,
                                        double (&u)[4]) {
#pragma unroll
    for (int q = 0; q < 4; ++q) u[q] = ok ? LBPS_LDX(NC, U + (size_t)q * plane + p) : 0.0;
}

// An output window of the interior kernel: columns [x0, x1), rows [y0, y1).
struct Win {
    int x0, x1, y0, y1;
};

// The moving populations of interior point (i, j) (plane offset p) that
// stream in from boundary points and that the reset pass overwrites: 1 f^1
// (from i - 1), 2 f^3 (from i + 1), 4 f^2 (from j - 1), 8 f^4 (from j + 1).
// A rectangle's boundary points are its non-periodic edges; a general
// geometry marks them in its node-type plane.
template <bool RECT>
__device__ __forceinline__ int streamed_in(const Geo& g, int i, int j, size_t p) {
    if (RECT || !g.general) {
        int m = 0;
        if (!g.periodic_x) m |= (i == 1 ? 1 : 0) | (i == g.nx - 2 ? 2 : 0);
        if (!g.periodic_y) m |= (j == 1 ? 4 : 0) | (j == g.ny - 2 ? 8 : 0);
        return m;
    }
    auto bnd = [&](size_t q) {
        const int t = LBPS_LDG(&g.type[q]);
        return t == NEUMANN || t == DIRICHLET;
    };
    const size_t row = p - (size_t)i;
    return (bnd(row + (size_t)wrap(i - 1, g.nx)) ? 1 : 0) | (bnd(row + (size_t)wrap(i + 1, g.nx)) ? 2 : 0) |
           (bnd((size_t)wrap(j - 1, g.ny) * g.px + (size_t)i) ? 4 : 0) |
           (bnd((size_t)wrap(j + 1, g.ny) * g.px + (size_t)i) ? 8 : 0);
}

// One warp's strip: output columns [xs, xs + kStripCols) of rows [j0, j1).
// Returns true in lanes that produced a non-finite value.  All 32 lanes of
// the warp must call it together (warp shuffles).  UVD: how many rows ahead u
// and du/dt are prefetched (1 or 2; the populations always 2).  WIN: writes
// only columns [w.x0, w.x1) of its rows, which lie inside the window (the
// frame passes of sweeps of several steps).
// NC = false: copy A may have been written earlier in the same launch (the
// many-step kernel, which is bound by FP64 instructions and has registers to
// spare: it widens the accelerations with integer operations).  GEN, with NC =
// false: a general geometry.
template <typename P, int UVD, bool WIN = false, bool NC = true, bool GEN = false>
__device__ __forceinline__ bool bulk_strip(const Geo& g, const Consts& c, const KCof<P>& k, const View<P>& A,
                                           const View<P>& B, int xs, int j0, int j1, Win w = Win{0, 0, 0, 0}) {
    using V = typename P::V;
    const unsigned FULL = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    const int xl = xs - 1 + lane;
    const bool col_ok = g.periodic_x ? (xl <= g.nx) : (xl >= 0 && xl < g.nx);
    const int col = col_ok ? wrap(xl, g.nx) : 0;
    const bool out_lane = lane >= 1 && lane <= kStripCols && xl < g.nx &&
                          (g.periodic_x || (xl > 0 && xl < g.nx - 1)) && (!WIN || (xl >= w.x0 && xl < w.x1));
    const size_t PL = g.plane;

    auto row_ok = [&](int j) { return g.periodic_y || (j >= 0 && j < g.ny); };
    auto row_of = [&](int j) { return g.periodic_y ? wrap(j, g.ny) : j; };
    // Offsets are formed only for rows inside the lattice (rows outside are
    // clamped; their loads are masked), so no address ever leaves the planes
    // even where a masked load is issued unconditionally.
    auto at = [&](int j) { return (size_t)min(max(row_of(j), 0), g.ny - 1) * (size_t)g.px + (size_t)col; };

    V Ps[2], Pf4[2];                          // row j - 1: moment and f^4
    V Cf[2][5], Cs[2], Cm[2];                 // row j
    V Nf[2][5];                               // row j + 1
    typename P::Raw Qr;                       // row j + 2 (in flight, stored form)
    double Cu[4], Nu[4], Qu[4];               // u, du/dt of rows j, j + 1, j + 2
    {
        V t[2][5];
        P::template load_raw<NC>(A.f, PL, at(j0 - 1), col_ok && row_ok(j0 - 1), Qr);
        decode_row<P>(Qr, k, t);
#pragma unroll
        for (int s = 0; s < 2; ++s) {
            Ps[s] = sum5(t[s][0], t[s][1], t[s][2], t[s][3], t[s][4]);
            Pf4[s] = t[s][4];
        }
    }
    P::template load_raw<NC>(A.f, PL, at(j0), col_ok, Qr);
    decode_row<P>(Qr, k, Cf);
    P::template load_raw<NC>(A.f, PL, at(j0 + 1), col_ok && row_ok(j0 + 1), Qr);
    decode_row<P>(Qr, k, Nf);
    load_uv<NC>(A.u, PL, at(j0), out_lane, Cu);
    if (UVD == 2) load_uv<NC>(A.u, PL, at(j0 + 1), out_lane && j0 + 1 < j1, Nu);
#pragma unroll
    for (int s = 0; s < 2; ++s) {
        Cm[s] = add_rn(add_rn(Cf[s][1], Cf[s][2]), add_rn(Cf[s][3], Cf[s][4]));
        Cs[s] = add_rn(Cf[s][0], Cm[s]);
    }
    // GEN: the node types, one row ahead too (loaded where they are used, their
    // latency is in every row's chain: 1024^2 with a hole 41.8 us a step, now 40)
    unsigned Ct = 0, Nt = 0;
    if (GEN) Ct = LBPS_LDG(&g.type[at(j0)]);
    bool bad = false;
    for (int j = j0; j < j1; ++j) {
        // prefetch: populations two rows ahead, u and du/dt one row ahead
        if (GEN) Nt = LBPS_LDG(&g.type[at(j + 1)]);
        P::template load_raw<NC>(A.f, PL, at(j + 2), col_ok && row_ok(j + 2) && j + 2 <= j1, Qr);
        if (UVD == 2)
            load_uv<NC>(A.u, PL, at(j + 2), out_lane && j + 2 < j1, Qu);
        else
            load_uv<NC>(A.u, PL, at(j + 1), out_lane && j + 1 < j1, Nu);
        V Nm[2], Ns[2];
#pragma unroll
        for (int s = 0; s < 2; ++s) {
            Nm[s] = add_rn(add_rn(Nf[s][1], Nf[s][2]), add_rn(Nf[s][3], Nf[s][4]));
            Ns[s] = add_rn(Nf[s][0], Nm[s]);
        }
        // (a window's rows are interior ones of the lattice: j0 .. j1 lie in it)
        const bool row_interior = g.periodic_y || (j > 0 && j < g.ny - 1);
        if (row_interior) {  // warp-uniform
            V sW[2], sE[2], out[2][5];
#pragma unroll
            for (int s = 0; s < 2; ++s) {
                sW[s] = __shfl_up_sync(FULL, Cs[s], 1);
                sE[s] = __shfl_down_sync(FULL, Cs[s], 1);
                V f3W = __shfl_up_sync(FULL, Cf[s][3], 1);
                V f1E = __shfl_down_sync(FULL, Cf[s][1], 1);
                // rest population: 2 a0 s - f0 = f0 + (2 a0 m - 8 a f0)
                out[s][0] = add_rn(Cf[s][0], fma_rn(k.two_a0[s], Cm[s], -mul_rn(k.eight_a[s], Cf[s][0])));
                // moving populations: f^alpha(x) = 2 a s(x - e_alpha) - f^opp(x - e_alpha)
                // (for sources on the boundary the reset pass overwrites them)
                out[s][1] = fma_rn(k.two_a[s], sW[s], -f3W);
                out[s][3] = fma_rn(k.two_a[s], sE[s], -f1E);
                out[s][2] = fma_rn(k.two_a[s], Ps[s], -Pf4[s]);
                out[s][4] = fma_rn(k.two_a[s], Ns[s], -Nf[s][2]);
            }
            const size_t p = at(j);
            // general geometry: only interior points (boundary and void points
            // are the boundary passes' or stay zero)
            if (out_lane && (GEN ? Ct == 0 : WIN || !g.general || LBPS_LDG(&g.type[p]) == 0)) {
                double ax, ay;
                accel_interior<V, !NC>(sW[0], sE[0], Ps[0], Ns[0], sW[1], sE[1], Ps[1], Ns[1], k, ax, ay);
                double u1[4];
                newmark(Cu[0], Cu[2], ax, c, u1[0], u1[2]);
                newmark(Cu[1], Cu[3], ay, c, u1[1], u1[3]);
                if constexpr (P::kSplitStream)
                    P::store_point_pins(B.f, PL, p, out, k, streamed_in<WIN>(g, col, j, p));
                else
                    P::store_point(B.f, PL, p, out, k);
#pragma unroll
                for (int q = 0; q < 4; ++q) LBPS_ST(&B.u[(size_t)q * PL + p], u1[q]);
                bad |= !isfinite(out[0][0] + out[1][0]);
            }
        }
        // shift the row window
#pragma unroll
        for (int s = 0; s < 2; ++s) {
            Ps[s] = Cs[s];
            Pf4[s] = Cf[s][4];
            Cs[s] = Ns[s];
            Cm[s] = Nm[s];
#pragma unroll
            for (int q = 0; q < 5; ++q) Cf[s][q] = Nf[s][q];
        }
        decode_row<P>(Qr, k, Nf);
        if (GEN) Ct = Nt;
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            Cu[q] = Nu[q];
            if (UVD == 2) Nu[q] = Qu[q];
        }
    }
    return bad;
}

// The interior kernel on a few columns [x0, x1) next to a left or right edge of
// a rectangle: the warp is 32 / W groups of W lanes, each marching down its own
// `rows` rows of [j0, je) (group q from j0 + q rows) over the W columns from xb
// on, which hold [x0 - 1, x1].  A strip of 32 columns there would have a handful
// of its lanes in the window and pay each row's FP64 instructions (64 cycles
// each) and loads for them; here one instruction serves 32 / W rows.  The
// arithmetic of bulk_strip.
template <typename P, int W>
__device__ __forceinline__ bool side_strip(const Geo& g, const Consts& c, const KCof<P>& k, const View<P>& A,
                                           const View<P>& B, int xb, int x0, int x1, int j0, int je, int rows) {
    using V = typename P::V;
    const unsigned FULL = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    const int col = xb + lane % W;                       // inside the lattice (sides >= W)
    const int jb = min(j0 + lane / W * rows, je), jend = min(jb + rows, je);
    const bool out_col = col >= x0 && col < x1;
    const size_t PL = g.plane;
    // rows up to jend (at most ny - 1) are read, further ones clamped and masked
    auto at = [&](int j) { return (size_t)min(j, jend) * (size_t)g.px + (size_t)col; };

    V Ps[2], Pf4[2];
    V Cf[2][5], Nf[2][5];
    typename P::Raw Qr;
    double Cu[4], Nu[4];
    {
        V t[2][5];
        P::load_raw(A.f, PL, at(jb - 1), true, Qr);
        decode_row<P>(Qr, k, t);
#pragma unroll
        for (int s = 0; s < 2; ++s) {
            Ps[s] = sum5(t[s][0], t[s][1], t[s][2], t[s][3], t[s][4]);
            Pf4[s] = t[s][4];
        }
    }
    P::load_raw(A.f, PL, at(jb), true, Qr);
    decode_row<P>(Qr, k, Cf);
    P::load_raw(A.f, PL, at(jb + 1), true, Qr);
    decode_row<P>(Qr, k, Nf);
    load_uv(A.u, PL, at(jb), out_col && jb < jend, Cu);
    bool bad = false;
    for (int r = 0; r < rows; ++r) {
        const int j = jb + r;
        P::load_raw(A.f, PL, at(j + 2), j + 2 <= jend, Qr);
        load_uv(A.u, PL, at(j + 1), out_col && j + 1 < jend, Nu);
        V sW[2], sE[2], Cs[2], Ns[2], out[2][5];
#pragma unroll
        for (int s = 0; s < 2; ++s) {
            const V Cm = add_rn(add_rn(Cf[s][1], Cf[s][2]), add_rn(Cf[s][3], Cf[s][4]));
            Cs[s] = add_rn(Cf[s][0], Cm);
            Ns[s] = sum5(Nf[s][0], Nf[s][1], Nf[s][2], Nf[s][3], Nf[s][4]);
            sW[s] = __shfl_up_sync(FULL, Cs[s], 1, W);
            sE[s] = __shfl_down_sync(FULL, Cs[s], 1, W);
            const V f3W = __shfl_up_sync(FULL, Cf[s][3], 1, W);
            const V f1E = __shfl_down_sync(FULL, Cf[s][1], 1, W);
            out[s][0] = add_rn(Cf[s][0], fma_rn(k.two_a0[s], Cm, -mul_rn(k.eight_a[s], Cf[s][0])));
            out[s][1] = fma_rn(k.two_a[s], sW[s], -f3W);
            out[s][3] = fma_rn(k.two_a[s], sE[s], -f1E);
            out[s][2] = fma_rn(k.two_a[s], Ps[s], -Pf4[s]);
            out[s][4] = fma_rn(k.two_a[s], Ns[s], -Nf[s][2]);
        }
        if (out_col && j < jend) {
            const size_t p = at(j);
            double ax, ay, u1[4];
            accel_interior<V, true>(sW[0], sE[0], Ps[0], Ns[0], sW[1], sE[1], Ps[1], Ns[1], k, ax, ay);
            newmark(Cu[0], Cu[2], ax, c, u1[0], u1[2]);
            newmark(Cu[1], Cu[3], ay, c, u1[1], u1[3]);
            if constexpr (P::kSplitStream)
                P::store_point_pins(B.f, PL, p, out, k, streamed_in<true>(g, col, j, p));
            else
                P::store_point(B.f, PL, p, out, k);
#pragma unroll
            for (int q = 0; q < 4; ++q) LBPS_ST(&B.u[(size_t)q * PL + p], u1[q]);
            bad |= !isfinite(out[0][0] + out[1][0]);
        }
#pragma unroll
        for (int s = 0; s < 2; ++s) {
            Ps[s] = Cs[s];
            Pf4[s] = Cf[s][4];
#pragma unroll
            for (int q = 0; q < 5; ++q) Cf[s][q] = Nf[s][q];
        }
        decode_row<P>(Qr, k, Nf);
#pragma unroll
        for (int q = 0; q < 4; ++q) Cu[q] = Nu[q];
    }
    return bad;
}

// Rows per group of a side strip, and the rows of a side task of the batch
// (groups of 8 lanes).
constexpr int kSideRows = 8;
static_assert(kSideTaskRows == 4 * kSideRows, "a side task is one warp");

// ------------------------------------------------- two steps per sweep

constexpr int kPairCols = 28;  // output columns of a warp in the two-step kernel
constexpr int kDeep = 3;       // the two-step kernel writes points at least this far from every edge

// Two time steps of the deep interior of a rectangle (no periodic axis, no
// void points) in one sweep: the warp marches its strip's rows computing step
// n + 1 from copy A (state n) exactly as bulk_strip does, rounds it to its
// stored form as a store and reload would, and from those values step n + 2,
// which it writes to copy B.  Lanes are columns xs - 2 .. xs + 29: step n + 1
// is valid in lanes 1..30, step n + 2 in lanes 2..29 (output columns xs ..
// xs + 27).  Rows [j0, j1) need step n + 1 at rows j0 - 1 .. j1 and state n
// at rows j0 - 2 .. j1 + 1.  A point at least kDeep from every edge depends
// at step n + 2 only on interior points at step n + 1 that are at least 2
// from the edges, which the boundary reset of step n does not touch, so
// nothing here needs the boundary passes.
// WRAP: a lattice periodic in both axes; every point, and u, du/dt take the
// steps one by one.
template <typename P, bool WRAP = false>
__device__ __forceinline__ bool pair_strip(const Geo& g, const Consts& c, const KCof<P>& k, const View<P>& A,
                                           const View<P>& B, int xs, int j0, int j1) {
    using V = typename P::V;
    const unsigned FULL = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    const int xl = xs - 2 + lane;
    const bool col_ok = WRAP || xl < g.nx;             // without WRAP xl >= 1 always (xs >= kDeep)
    const int col = WRAP ? wrap(xl, g.nx) : col_ok ? xl : g.nx - 1;
    const bool out_lane = lane >= 2 && lane < 2 + kPairCols && xl < (WRAP ? g.nx : g.nx - kDeep);
    const size_t PL = g.plane;
    auto at = [&](int j) { return (size_t)(WRAP ? wrap(j, g.ny) : j) * (size_t)g.px + (size_t)col; };

    // step n (state n, read): rows r - 1, r, r + 1 and r + 2 in flight
    V P0s[2], P0f4[2];
    V C0f[2][5], C0s[2], C0m[2];
    V N0f[2][5];
    typename P::Raw Qr;
    // step n + 1: rows r - 2 (moment, f^4), r - 1 (all); filled by the first
    // two iterations, which write nothing
    V P1s[2] = {}, P1f4[2] = {};
    V C1f[2][5] = {}, C1s[2] = {}, C1m[2] = {};
    double C1u[4] = {};   // u, du/dt of row r - 1 at step n (loaded one iteration ahead)
    V C1a[2] = {};        // the accelerations of row r - 1 at step n

    {
        V t[2][5];
        P::load_raw(A.f, PL, at(j0 - 2), col_ok, Qr);
        decode_row<P>(Qr, k, t);
#pragma unroll
        for (int s = 0; s < 2; ++s) {
            P0s[s] = sum5(t[s][0], t[s][1], t[s][2], t[s][3], t[s][4]);
            P0f4[s] = t[s][4];
        }
    }
    P::load_raw(A.f, PL, at(j0 - 1), col_ok, Qr);
    decode_row<P>(Qr, k, C0f);
    P::load_raw(A.f, PL, at(j0), col_ok, Qr);
    decode_row<P>(Qr, k, N0f);
#pragma unroll
    for (int s = 0; s < 2; ++s) {
        C0m[s] = add_rn(add_rn(C0f[s][1], C0f[s][2]), add_rn(C0f[s][3], C0f[s][4]));
        C0s[s] = add_rn(C0f[s][0], C0m[s]);
    }
    bool bad = false;
    // r: the row of step n + 1 computed this iteration; step n + 2 at r - 1
    for (int r = j0 - 1; r <= j1; ++r) {
        P::load_raw(A.f, PL, at(r + 2), col_ok && r + 2 <= j1 + 1, Qr);
        // u, du/dt only where a point is written: row r, used by the next
        // iteration's second stage
        double Nu[4];
        load_uv(A.u, PL, at(r), out_lane && r >= j0 && r < j1, Nu);
        V N0m[2], N0s[2];
#pragma unroll
        for (int s = 0; s < 2; ++s) {
            N0m[s] = add_rn(add_rn(N0f[s][1], N0f[s][2]), add_rn(N0f[s][3], N0f[s][4]));
            N0s[s] = add_rn(N0f[s][0], N0m[s]);
        }
        // step n + 1 at row r (bulk_strip's arithmetic)
        V N1f[2][5], N1a[2];
        {
            V sW[2], sE[2], out[2][5];
#pragma unroll
            for (int s = 0; s < 2; ++s) {
                sW[s] = __shfl_up_sync(FULL, C0s[s], 1);
                sE[s] = __shfl_down_sync(FULL, C0s[s], 1);
                V f3W = __shfl_up_sync(FULL, C0f[s][3], 1);
                V f1E = __shfl_down_sync(FULL, C0f[s][1], 1);
                out[s][0] = add_rn(C0f[s][0], fma_rn(k.two_a0[s], C0m[s], -mul_rn(k.eight_a[s], C0f[s][0])));
                out[s][1] = fma_rn(k.two_a[s], sW[s], -f3W);
                out[s][3] = fma_rn(k.two_a[s], sE[s], -f1E);
                out[s][2] = fma_rn(k.two_a[s], P0s[s], -P0f4[s]);
                out[s][4] = fma_rn(k.two_a[s], N0s[s], -N0f[s][2]);
            }
            // the accelerations at step n, for the second stage, which
            // integrates both steps at once
            accel_interior_v<V>(sW[0], sE[0], P0s[0], N0s[0], sW[1], sE[1], P0s[1], N0s[1], k, N1a[0], N1a[1]);
            // as stored at row r and read back
            typename P::Raw q;
            P::pack(at(r), out, k, q);
            decode_row<P>(q, k, N1f);
        }
        V N1m[2], N1s[2];
#pragma unroll
        for (int s = 0; s < 2; ++s) {
            N1m[s] = add_rn(add_rn(N1f[s][1], N1f[s][2]), add_rn(N1f[s][3], N1f[s][4]));
            N1s[s] = add_rn(N1f[s][0], N1m[s]);
        }
        // step n + 2 at row r - 1
        if (r - 1 >= j0) {  // warp-uniform
            V sW[2], sE[2], out[2][5];
#pragma unroll
            for (int s = 0; s < 2; ++s) {
                sW[s] = __shfl_up_sync(FULL, C1s[s], 1);
                sE[s] = __shfl_down_sync(FULL, C1s[s], 1);
                V f3W = __shfl_up_sync(FULL, C1f[s][3], 1);
                V f1E = __shfl_down_sync(FULL, C1f[s][1], 1);
                out[s][0] = add_rn(C1f[s][0], fma_rn(k.two_a0[s], C1m[s], -mul_rn(k.eight_a[s], C1f[s][0])));
                out[s][1] = fma_rn(k.two_a[s], sW[s], -f3W);
                out[s][3] = fma_rn(k.two_a[s], sE[s], -f1E);
                out[s][2] = fma_rn(k.two_a[s], P1s[s], -P1f4[s]);
                out[s][4] = fma_rn(k.two_a[s], N1s[s], -N1f[s][2]);
            }
            if (out_lane) {
                const size_t p = at(r - 1);
                V ax, ay;
                accel_interior_v<V>(sW[0], sE[0], P1s[0], N1s[0], sW[1], sE[1], P1s[1], N1s[1], k, ax, ay);
                double u2[4];
                if constexpr (WRAP) {
                    double u1[4];
                    newmark(C1u[0], C1u[2], widen(C1a[0]), c, u1[0], u1[2]);
                    newmark(C1u[1], C1u[3], widen(C1a[1]), c, u1[1], u1[3]);
                    newmark(u1[0], u1[2], widen(ax), c, u2[0], u2[2]);
                    newmark(u1[1], u1[3], widen(ay), c, u2[1], u2[3]);
                } else {
                    newmark2(C1u[0], C1u[2], C1a[0], ax, c, u2[0], u2[2]);
                    newmark2(C1u[1], C1u[3], C1a[1], ay, c, u2[1], u2[3]);
                }
                P::store_point(B.f, PL, p, out, k);
#pragma unroll
                for (int q = 0; q < 4; ++q) LBPS_ST(&B.u[(size_t)q * PL + p], u2[q]);
                bad |= !isfinite(out[0][0] + out[1][0]);
            }
        }
        // shift both windows
#pragma unroll
        for (int s = 0; s < 2; ++s) {
            P1s[s] = C1s[s];
            P1f4[s] = C1f[s][4];
            C1s[s] = N1s[s];
            C1m[s] = N1m[s];
#pragma unroll
            for (int q = 0; q < 5; ++q) C1f[s][q] = N1f[s][q];
            P0s[s] = C0s[s];
            P0f4[s] = C0f[s][4];
            C0s[s] = N0s[s];
            C0m[s] = N0m[s];
#pragma unroll
            for (int q = 0; q < 5; ++q) C0f[s][q] = N0f[s][q];
        }
#pragma unroll
        for (int q = 0; q < 4; ++q) C1u[q] = Nu[q];
        C1a[0] = N1a[0];
        C1a[1] = N1a[1];
        decode_row<P>(Qr, k, N0f);
    }
    return bad;
}

}  // namespace

}  // namespace lbps
