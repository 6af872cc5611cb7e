// CUDA kernels of the plane-strain lattice Boltzmann time loop
// (arXiv:2301.00228, algorithm summary of Fig. 3), sm_103a.
//
// One time step is three launches on one stream:
//   boundary newmark  acceleration of each boundary point (Eq. acc_neumann,
//                     from the stresses kept with the state copy, or Eq.
//                     acc_dirichlet) and u, du/dt at t + dt (Eq.
//                     integration);
//   bulk              every interior point: acceleration (Eq. navier),
//                     Newmark, and the pull form of the LBE (Eq. LBE).
//                     Memory-bound stencil: reads copy A once, writes copy B
//                     once;
//   boundary reset    phi, psi at boundary points from differences of the new
//                     u (Eq. psi_phi_at_bound), their populations by Eq.
//                     correction-f, the value each streams into its
//                     interior neighbour (Eq. LBE_mod), and the stresses of
//                     the new u (Eq. strain, Eq. hooke) for the next step.
// Copies A (time t) and B (time t + dt) swap after each step.  Every kernel is
// a template over the population storage policy (lbps_device.cuh): FP32 or
// FP64 planes, or FP32 moments (f^0, J) with the non-equilibrium pair sums in
// 16 bits.
#include <algorithm>
#include <type_traits>

#include "lbps_steps.cuh"
#ifdef LBPS_CHECKED
#include <utility>
#include <vector>
#endif

namespace lbps {

namespace {

enum {
    FLD_UX = 0, FLD_UY = 1, FLD_VX = 2, FLD_VY = 3, FLD_PHI = 4, FLD_PSI = 5,
    FLD_FPHI = 6, FLD_FPSI = 7, FLD_CONS = 8, FLD_KIN = 9, FLD_STRAIN = 10
};

// ------------------------------------------------------------------ init

// Fig. 3 initialisation: phi = div u, psi = curl u by finite differences of
// u(x, 0) (already copied into copy A), populations at equilibrium (Eq. feq).
template <typename P>
__global__ void init_kernel(Geo g, Consts c, KCof<P> k, View<P> A) {
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    int j = blockIdx.y * blockDim.y + threadIdx.y;
    if (i >= g.nx || j >= g.ny) return;
    const double* ux = A.u;
    const double* uy = A.u + g.plane;
    size_t p = (size_t)j * g.px + i;
    if (!body_at(g, i, j)) {  // void points hold no state: all zero
        for (int q = 0; q < 4; ++q) LBPS_ST(&A.u[(size_t)q * g.plane + p], 0.0);
        const double z[2] = {0.0, 0.0};
        P::store_eq_point(A.f, g.plane, p, c, z, z, z, k);
        return;
    }
    double phi = ddx(ux, g.px, i, j, g, c.inv2h) + ddy(uy, g.px, i, j, g, c.inv2h);
    double psi = ddx(uy, g.px, i, j, g, c.inv2h) - ddy(ux, g.px, i, j, g, c.inv2h);
    double vx = LBPS_LD(&A.u[2 * g.plane + p]), vy = LBPS_LD(&A.u[3 * g.plane + p]);
    // First moments from du/dt (J_phi = -v, J_psi = (-v_y, v_x)), in lattice
    // units Jbar = J dt / dh (c cancels: c^alpha . J / (2 c^2) = e_alpha . Jbar / 2).
    // At rest (both +0) the products are known; skipping them and their
    // conversions leaves 12 of 22 FP64 instructions (the kernel is bound by them).
    const double sv[2] = {phi, psi};
    if ((__double_as_longlong(vx) | __double_as_longlong(vy)) == 0) {
        const typename P::V jx[2] = {-(typename P::V)0, -(typename P::V)0}, jy[2] = {-(typename P::V)0, (typename P::V)0};
        P::store_eq_point(A.f, g.plane, p, c, sv, jx, jy, k);
        return;
    }
    double q = c.dt / c.dh;
    const double jx[2] = {-vx * q, -vy * q}, jy[2] = {-vy * q, vx * q};
    P::store_eq_point(A.f, g.plane, p, c, sv, jx, jy, k);
}

// Sets *bad if any of the first `planes` FP64 planes of u holds a
// non-finite value at a lattice point (the input check of the host
// initialisation; the pitch padding is not looked at).
__global__ void finite_check_kernel(Geo g, const double* __restrict__ u, int planes, unsigned* bad) {
    const size_t n = (size_t)g.nx * (size_t)g.ny;
    const size_t total = n * (size_t)planes;
    for (size_t t = (size_t)blockIdx.x * blockDim.x + threadIdx.x; t < total; t += (size_t)gridDim.x * blockDim.x) {
        const size_t q = t / n, r = t - q * n;
        const size_t j = r / (size_t)g.nx, i = r - j * (size_t)g.nx;
        if (!isfinite(LBPS_LDG(&u[q * g.plane + j * (size_t)g.px + i]))) atomicOr(bad, 1u);
    }
}

// Size of the lattice first moment J that the initial state implies, for the
// choice of the 16-bit storage scale (the stored non-equilibrium sums are
// smaller): per
// point sqrt(2 a_phi) max(|phi|, |psi|) + (|v_x| + |v_y|) dt / dh (a plane
// wave has |Jbar| = sqrt(2 a_phi) |phi| for the dilatation; the shear part is
// smaller by c_s / c_d).  Maximum over the lattice into *out (FP32 bits of a
// non-negative value, which order like unsigned integers).
__global__ void scale_probe_kernel(Geo g, Consts c, const double* __restrict__ u, double sq, unsigned* out) {
    __shared__ unsigned sh[8];
    const int lane = threadIdx.x;   // a block is 8 warps
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    int j = blockIdx.y * blockDim.y + threadIdx.y;
    float est = 0.0f;
    if (i < g.nx && j < g.ny && body_at(g, i, j)) {
        const double* ux = u;
        const double* uy = u + g.plane;
        size_t p = (size_t)j * g.px + i;
        double phi = ddx(ux, g.px, i, j, g, c.inv2h) + ddy(uy, g.px, i, j, g, c.inv2h);
        double psi = ddx(uy, g.px, i, j, g, c.inv2h) - ddy(ux, g.px, i, j, g, c.inv2h);
        const double vx = LBPS_LD(&u[2 * g.plane + p]), vy = LBPS_LD(&u[3 * g.plane + p]);
        double e = sq * fmax(fabs(phi), fabs(psi));
        // at rest there is nothing to add (and no FP64 division)
        if (((__double_as_longlong(vx) | __double_as_longlong(vy)) << 1) != 0)
            e += (fabs(vx) + fabs(vy)) * c.dt / c.dh;
        est = isfinite(e) ? (float)e : 3.0e38f;
    }
    const unsigned m = __reduce_max_sync(0xffffffffu, __float_as_uint(est));
    if (lane == 0) sh[threadIdx.y] = m;
    __syncthreads();
    if (lane == 0 && threadIdx.y == 0) {
        unsigned best = 0;
        for (int q = 0; q < 8; ++q) best = max(best, sh[q]);
        atomicMax(out, best);
    }
}

// ------------------------------------------------------------- boundary

template <typename P>
__global__ void __launch_bounds__(128) boundary_stress_kernel(Geo g, Consts c, View<P> A,
                                                              const BNode* __restrict__ bn, int nb) {
    int b = blockIdx.x * blockDim.x + threadIdx.x;
    if (b < nb) boundary_stress(g, c, A.u, A.u + g.plane, bn, nb, A.s, b);
}

template <typename P>
__global__ void __launch_bounds__(128, 8) boundary_newmark_kernel(Geo g, Consts c, View<P> A, View<P> B,
                                                               const BNode* __restrict__ bn, int nb,
                                                               const unsigned long long* __restrict__ tstep) {
    int b = blockIdx.x * blockDim.x + threadIdx.x;
    if (b >= nb) return;
    const double n = (double)LBPS_LD(tstep);
    for (int part = blockIdx.y; part < 2; part += gridDim.y) boundary_newmark(g, c, A, B, bn, nb, A.s, n, b, part);
}

// The last pass of a step also advances the step counter (one thread; no
// other thread of the pass reads it).
template <typename P>
__global__ void __launch_bounds__(128, 6) boundary_reset_kernel(Geo g, Consts c, KCof<P> k, View<P> A, View<P> B,
                                                             const BNode* __restrict__ bn, int nb, unsigned* flag,
                                                             unsigned long long* tstep) {
    int b = blockIdx.x * blockDim.x + threadIdx.x;
    if (blockIdx.y == 1) {
        if (b < nb) neighbour_stresses(g, c, B.u, B.u + g.plane, bn, nb, B.s, b);
        return;
    }
    bool bad = false;
    if (b < nb)
        bad = gridDim.y == 2 ? boundary_reset<P>(g, c, k, A, B, bn, nb, b)
                             : boundary_reset<P, true>(g, c, k, A, B, bn, nb, b);
    if (bad) atomicOr(flag, 1u);
    if (b == 0) LBPS_ST(tstep, LBPS_LD(tstep) + 1ull);
}

template <typename P>
__global__ void __launch_bounds__(128) boundary_stream_y_kernel(Geo g, Consts c, KCof<P> k, View<P> A, View<P> B,
                                                                const BNode* __restrict__ bn, int nb) {
    int b = blockIdx.x * blockDim.x + threadIdx.x;
    if (b < nb) boundary_stream_y(g, c, k, A, B, bn, b);
}

// Copies the populations of every boundary point of copy A into A's boundary
// mirror.  Run after the kernels that write them in place (initialisation,
// synchronisation); the reset pass keeps the mirror current otherwise.
template <typename P>
__global__ void __launch_bounds__(128) boundary_mirror_kernel(Geo g, View<P> A, const BNode* __restrict__ bn,
                                                              int nb) {
    int b = blockIdx.x * blockDim.x + threadIdx.x;
    if (b >= nb) return;
    const int i = LBPS_LD(&bn[b].i), j = LBPS_LD(&bn[b].j);
    typename P::Raw r;
    P::load_raw(A.f, g.plane, (size_t)j * g.px + i, true, r);
    P::store_raw(A.m, g.mplane, (size_t)b, r);
}

// ---------------------------------------------------------------- bulk

template <typename P, int MINB, int UVD>
__global__ void __launch_bounds__(128, MINB) bulk_kernel(Geo g, Consts c, KCof<P> k, View<P> A, View<P> B,
                                                         unsigned* flag, int rows_per_warp) {
    const int warp = blockIdx.x * kWarpsPerBlock + (threadIdx.x >> 5);
    const int xs = warp * kStripCols;
    if (xs >= g.nx) return;  // whole warp
    const int j0 = blockIdx.y * rows_per_warp;
    const int j1 = min(j0 + rows_per_warp, g.ny);
    // General geometry: a warp whose rows all lie in its strip's run of rows
    // without interior points (inside a hole) has nothing to write, and no
    // interior point reads those rows: it returns before loading them.
    if (g.gap && j0 >= LBPS_LD(&g.gap[2 * warp]) && j1 <= LBPS_LD(&g.gap[2 * warp + 1])) return;
    const bool bad = bulk_strip<P, UVD>(g, c, k, A, B, xs, j0, j1);
    if (__any_sync(0xffffffffu, bad) && (threadIdx.x & 31) == 0) atomicOr(flag, 1u);
}

// ------------------------------------------------- two steps per sweep

// The interior kernel on the points 1 .. fw from the edges only (the frame
// passes of sweeps of several steps).  Blocks 0 .. bands - 1: the bottom and the
// top band, strips of rows; then the left and right bands between them, a side
// strip a warp, groups of W lanes (W >= fw + 2).
template <typename P, int UVD, int W>
__device__ __forceinline__ void frame(const Geo& g, const Consts& c, const KCof<P>& k, const View<P>& A,
                                      const View<P>& B, unsigned* flag, int fw, int bands) {
    bool bad;
    const int wid = threadIdx.x >> 5;
    if (blockIdx.x < (unsigned)bands) {
        const int per = bands / 2, top = blockIdx.x >= (unsigned)per;
        const int xs = ((blockIdx.x - top * per) * kWarpsPerBlock + wid) * kStripCols;
        if (xs >= g.nx) return;  // whole warp
        const int j0 = top ? g.ny - 1 - fw : 1;
        bad = bulk_strip<P, UVD, true>(g, c, k, A, B, xs, j0, j0 + fw, Win{1, g.nx - 1, j0, j0 + fw});
    } else {
        const int t = (blockIdx.x - bands) * kWarpsPerBlock + wid;
        const int j0 = 1 + fw + (t >> 1) * (32 / W * kSideRows), je = g.ny - 1 - fw;
        if (j0 >= je) return;  // whole warp
        const bool right = t & 1;
        bad = side_strip<P, W>(g, c, k, A, B, right ? g.nx - W : 0, right ? g.nx - 1 - fw : 1, right ? g.nx - 1 : 1 + fw,
                               j0, je, kSideRows);
    }
    if (__any_sync(0xffffffffu, bad) && (threadIdx.x & 31) == 0) atomicOr(flag, 1u);
}

template <typename P, int MINB, int UVD>
__global__ void __launch_bounds__(128, MINB) frame_kernel(Geo g, Consts c, KCof<P> k, View<P> A, View<P> B,
                                                          unsigned* flag, int fw, int bands) {
    frame<P, UVD, 8>(g, c, k, A, B, flag, fw, bands);
}
template <typename P, int MINB, int UVD>
__global__ void __launch_bounds__(128, MINB) frame_wide_kernel(Geo g, Consts c, KCof<P> k, View<P> A, View<P> B,
                                                               unsigned* flag, int fw, int bands) {
    frame<P, UVD, 16>(g, c, k, A, B, flag, fw, bands);
}

template <typename P, int MINB>
__global__ void __launch_bounds__(128, MINB) pair_kernel(Geo g, Consts c, KCof<P> k, View<P> A, View<P> B,
                                                         unsigned* flag, int rows_per_warp) {
    const int warp = blockIdx.x * kWarpsPerBlock + (threadIdx.x >> 5);
    const int xs = kDeep + warp * kPairCols;
    if (xs >= g.nx - kDeep) return;  // whole warp
    const int j0 = kDeep + blockIdx.y * rows_per_warp;
    const int j1 = min(j0 + rows_per_warp, g.ny - kDeep);
    if (j0 >= j1) return;
    const bool bad = pair_strip<P>(g, c, k, A, B, xs, j0, j1);
    if (__any_sync(0xffffffffu, bad) && (threadIdx.x & 31) == 0) atomicOr(flag, 1u);
}

// --------------------------------------------------------------- batches

// The boundary passes of a step (1 Newmark, 2 reset, 3 the y streams of the
// reset where P::kSplitStream) over the boundary points of every lattice in
// the batch (one thread per point and part, the parts in blockIdx.y).
template <typename P>
__global__ void __launch_bounds__(128) boundary_batch_kernel(const DomDesc<P>* __restrict__ dd,
                                                             const BndTask* __restrict__ tasks, int ntasks,
                                                             int parity, int pass, int stage) {
    int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= ntasks) return;
    const BndTask tk = tasks[t];
    const DomDesc<P>& d = dd[tk.dom];
    const int a = d.cur ^ parity;
    // the copies the pass reads and writes (stage: see launch_boundary_batch)
    const View<P>& S = stage == 2 ? d.x : d.v[a];
    const View<P>& D = stage == 1 ? d.x : d.v[a ^ 1];
    if (pass == 1)
        for (int part = blockIdx.y; part < 2; part += gridDim.y)
            boundary_newmark(d.g, d.c, S, D, d.bn, d.nb, S.s, (double)LBPS_LD(d.tstep), tk.b, part);
    else if (pass == 3)
        boundary_stream_y(d.g, d.c, d.k, S, D, d.bn, tk.b);
    else {
        if (blockIdx.y == 1) {
            neighbour_stresses(d.g, d.c, D.u, D.u + d.g.plane, d.bn, d.nb, D.s, tk.b);
            return;
        }
        const bool bad = gridDim.y == 2 ? boundary_reset<P>(d.g, d.c, d.k, S, D, d.bn, d.nb, tk.b)
                                        : boundary_reset<P, true>(d.g, d.c, d.k, S, D, d.bn, d.nb, tk.b);
        if (bad) atomicOr(d.flag, 1u);
        if (tk.b == 0) LBPS_ST(d.tstep, LBPS_LD(d.tstep) + 1ull);
    }
}

// The interior of every lattice in the batch: a persistent grid (as many
// blocks as fit on the GPU at once) whose warps take strip tasks from the
// work list through the counter *next (zero before the launch) until none is
// left, so no wave of short tasks leaves the GPU half idle at the end.  Each
// warp keeps the descriptor of the lattice it works on in shared memory and
// copies a new one only when the next task belongs to another lattice.
template <typename P, int MINB, int UVD>
__global__ void __launch_bounds__(128, MINB) bulk_batch_kernel(const DomDesc<P>* __restrict__ dd,
                                                               const BulkTask* __restrict__ tasks, int ntasks,
                                                               const BndTask* __restrict__ btasks, int parity,
                                                               unsigned* next) {
    __shared__ DomDesc<P> sd[kWarpsPerBlock];
    const unsigned FULL = 0xffffffffu;
    const int wid = threadIdx.x >> 5, lane = threadIdx.x & 31;
    int cached = -1;
    for (;;) {
        unsigned t = 0;
        if (lane == 0) t = atomicAdd(next, 1u);
        t = __shfl_sync(FULL, t, 0);
        if (t >= (unsigned)ntasks) break;  // whole warp
        const BulkTask tk = tasks[t];
        if (tk.j0 < 0) {
            // Newmark task (warp-uniform): boundary points tk.xs .. tk.xs +
            // tk.j1 - 1 of the boundary work list, one per lane.  It reads
            // copy A and writes only boundary u, du/dt of copy B, which no
            // strip task touches; the reset pass after this kernel reads them.
            if (lane < tk.j1) {
                const BndTask bt = btasks[tk.xs + lane];
                const DomDesc<P>& d = dd[bt.dom];
                const int a = d.cur ^ parity;
                const double n = (double)LBPS_LD(d.tstep);
                boundary_newmark(d.g, d.c, d.v[a], d.v[a ^ 1], d.bn, d.nb, d.v[a].s, n, bt.b, 0);
                boundary_newmark(d.g, d.c, d.v[a], d.v[a ^ 1], d.bn, d.nb, d.v[a].s, n, bt.b, 1);
            }
            continue;
        }
        if (tk.dom != cached) {
            __syncwarp();  // every lane is done with the previous descriptor
            const unsigned* src = reinterpret_cast<const unsigned*>(dd + tk.dom);
            unsigned* dst = reinterpret_cast<unsigned*>(sd + wid);
            for (int q = lane; q < (int)(sizeof(DomDesc<P>) / 4); q += 32) dst[q] = src[q];
            __syncwarp();
            cached = tk.dom;
        }
        const DomDesc<P>& d = sd[wid];
        const int a = d.cur ^ parity;
        bool bad = bulk_strip<P, UVD>(d.g, d.c, d.k, d.v[a], d.v[a ^ 1], tk.xs, tk.j0, tk.j1);
        if (__any_sync(FULL, bad) && lane == 0) atomicOr(d.flag, 1u);
    }
}

// Two steps per sweep for every lattice of a batch: stage 1 of a pair (see
// launch_pair_batch) with the strips' rows loaded through registers (FP64
// storage; the others take them by TMA, lbps_sweep.cu).  The tasks are those of pair_kernel, frame_kernel and
// boundary_newmark_kernel on each lattice, so each lattice gets the same bits
// as run on its own with two steps per sweep.  Frame strips take the shape
// that loads u one row ahead (the results do not depend on it).
template <typename P, int MINB>
__global__ void __launch_bounds__(128, MINB) pair_batch_kernel(const DomDesc<P>* __restrict__ dd,
                                                               const PairTask* __restrict__ tasks, int ntasks,
                                                               const BndTask* __restrict__ btasks, int parity,
                                                               unsigned* next) {
    __shared__ DomDesc<P> sd[kWarpsPerBlock];
    const unsigned FULL = 0xffffffffu;
    const int wid = threadIdx.x >> 5, lane = threadIdx.x & 31;
    int cached = -1;
    for (;;) {
        unsigned t = 0;
        if (lane == 0) t = atomicAdd(next, 1u);
        t = __shfl_sync(FULL, t, 0);
        if (t >= (unsigned)ntasks) break;  // whole warp
        const PairTask tk = tasks[t];
        if (tk.kind == kNewmarkTask) {
            if (lane < tk.j1) {
                const BndTask bt = btasks[tk.xs + lane];
                const DomDesc<P>& d = dd[bt.dom];
                const int a = d.cur ^ parity;
                const double n = (double)LBPS_LD(d.tstep);
                boundary_newmark(d.g, d.c, d.v[a], d.x, d.bn, d.nb, d.v[a].s, n, bt.b, 0);
                boundary_newmark(d.g, d.c, d.v[a], d.x, d.bn, d.nb, d.v[a].s, n, bt.b, 1);
            }
            continue;
        }
        if (tk.dom != cached) {
            __syncwarp();  // every lane is done with the previous descriptor
            const unsigned* src = reinterpret_cast<const unsigned*>(dd + tk.dom);
            unsigned* dst = reinterpret_cast<unsigned*>(sd + wid);
            for (int q = lane; q < (int)(sizeof(DomDesc<P>) / 4); q += 32) dst[q] = src[q];
            __syncwarp();
            cached = tk.dom;
        }
        const DomDesc<P>& d = sd[wid];
        const int a = d.cur ^ parity;
        bool bad;
        if (tk.kind == kPairStrip) {
            bad = pair_strip<P>(d.g, d.c, d.k, d.v[a], d.v[a ^ 1], tk.xs, tk.j0, tk.j1);
        } else if (tk.kind == kSideStrip) {
            bad = side_strip<P, 8>(d.g, d.c, d.k, d.v[a], d.x, tk.xs, tk.x0, tk.x1, tk.j0, tk.j1, kSideRows);
        } else {
            bad = bulk_strip<P, 1, true>(d.g, d.c, d.k, d.v[a], d.x, tk.xs, tk.j0, tk.j1, Win{tk.x0, tk.x1, tk.y0, tk.y1});
        }
        if (__any_sync(FULL, bad) && lane == 0) atomicOr(d.flag, 1u);
    }
}

// Stage 2 of a pair, one task a warp: the frame strips and Newmark tasks only,
// so 5 blocks fit on an SM.  Every task is a chain of scattered loads; what
// counts is how many run at once (256 lattices: as a persistent grid of the
// stage-1 kernel's 4 blocks per SM 156 us).
template <typename P>
__global__ void __launch_bounds__(128, sizeof(typename P::V) == 8 ? 3 : 5)
    edge_batch_kernel(const DomDesc<P>* __restrict__ dd, const PairTask* __restrict__ tasks, int ntasks,
                      const BndTask* __restrict__ btasks, int parity) {
    __shared__ DomDesc<P> sd[kWarpsPerBlock];
    const int wid = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int t = blockIdx.x * kWarpsPerBlock + wid;
    if (t >= ntasks) return;  // whole warp
    const PairTask tk = tasks[t];
    if (tk.kind == kNewmarkTask) {
        if (lane < tk.j1) {
            const BndTask bt = btasks[tk.xs + lane];
            const DomDesc<P>& d = dd[bt.dom];
            const View<P>& D = d.v[d.cur ^ parity ^ 1];
            const double n = (double)LBPS_LD(d.tstep);
            boundary_newmark(d.g, d.c, d.x, D, d.bn, d.nb, d.x.s, n, bt.b, 0);
            boundary_newmark(d.g, d.c, d.x, D, d.bn, d.nb, d.x.s, n, bt.b, 1);
        }
        return;
    }
    const unsigned* src = reinterpret_cast<const unsigned*>(dd + tk.dom);
    unsigned* dst = reinterpret_cast<unsigned*>(sd + wid);
    for (int q = lane; q < (int)(sizeof(DomDesc<P>) / 4); q += 32) dst[q] = src[q];
    __syncwarp();
    const DomDesc<P>& d = sd[wid];
    const View<P>& D = d.v[d.cur ^ parity ^ 1];
    const bool bad = tk.kind == kSideStrip
                         ? side_strip<P, 8>(d.g, d.c, d.k, d.x, D, tk.xs, tk.x0, tk.x1, tk.j0, tk.j1, kSideRows)
                         : bulk_strip<P, 1, true>(d.g, d.c, d.k, d.x, D, tk.xs, tk.j0, tk.j1,
                                                  Win{tk.x0, tk.x1, tk.y0, tk.y1});
    if (__any_sync(0xffffffffu, bad) && lane == 0) atomicOr(d.flag, 1u);
}

// ------------------------------------------------------------------ sync

// Sec. 3.2: phi, psi from differences of u at every point, populations by
// Eq. correction-f with the current first moments.  In place.
template <typename P>
__global__ void sync_kernel(Geo g, Consts c, KCof<P> k, View<P> A) {
    using V = typename P::V;
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    int j = blockIdx.y * blockDim.y + threadIdx.y;
    if (i >= g.nx || j >= g.ny || !body_at(g, i, j)) return;
    const double* ux = A.u;
    const double* uy = A.u + g.plane;
    size_t p = (size_t)j * g.px + i;
    double s[2];
    s[0] = ddx(ux, g.px, i, j, g, c.inv2h) + ddy(uy, g.px, i, j, g, c.inv2h);
    s[1] = ddx(uy, g.px, i, j, g, c.inv2h) - ddy(ux, g.px, i, j, g, c.inv2h);
    V jx[2], jy[2];   // first moments in the arithmetic type of the storage
    for (int set = 0; set < 2; ++set) {
        V f[5];
        P::load5(A.f, g.plane, p, set, k, f);
        jx[set] = sub_rn(f[1], f[3]);
        jy[set] = sub_rn(f[2], f[4]);
    }
    P::store_eq_point(A.f, g.plane, p, c, s, jx, jy, k);
}

// ---------------------------------------------------------------- fields

template <typename P>
__device__ inline double moment0_fp64(const View<P>& A, size_t plane, size_t p, int set, const KCof<P>& k) {
    double b[5];
    P::load5d(A.f, plane, p, set, k, b);
    return b[0] + ((b[1] + b[2]) + (b[3] + b[4]));
}

// Scalar field value at (i, j).
template <typename P>
__device__ inline double field_value(const Geo& g, const Consts& c, const KCof<P>& k, const View<P>& A, int field,
                                     int i, int j) {
    size_t p = (size_t)j * g.px + i;
    switch (field) {
    case FLD_UX: case FLD_UY: case FLD_VX: case FLD_VY: return A.u[(size_t)field * g.plane + p];
    case FLD_PHI: return moment0_fp64(A, g.plane, p, 0, k);
    case FLD_PSI: return moment0_fp64(A, g.plane, p, 1, k);
    case FLD_KIN: {
        // kinetic energy density rho |du/dt|^2 / 2 (0 at void points)
        if (!body_at(g, i, j)) return 0.0;
        const double vx = A.u[2 * g.plane + p], vy = A.u[3 * g.plane + p];
        return 0.5 * c.rho * (vx * vx + vy * vy);
    }
    case FLD_STRAIN: {
        // strain energy density sigma : eps / 2 = lambda tr(eps)^2 / 2 + mu eps : eps
        // (Eq. hooke with eps of Eq. strain by the finite differences of Sec. 3.1.2)
        if (!body_at(g, i, j)) return 0.0;
        const double* ux = A.u;
        const double* uy = A.u + g.plane;
        const double exx = ddx(ux, g.px, i, j, g, c.inv2h);
        const double eyy = ddy(uy, g.px, i, j, g, c.inv2h);
        const double exy = 0.5 * (ddy(ux, g.px, i, j, g, c.inv2h) + ddx(uy, g.px, i, j, g, c.inv2h));
        const double tr = exx + eyy;
        return 0.5 * c.lam * tr * tr + c.mu * (exx * exx + eyy * eyy + 2.0 * exy * exy);
    }
    default: {
        // consistency error e(x, t) of Sec. 4 (0 at void points)
        if (!body_at(g, i, j)) return 0.0;
        const double* ux = A.u;
        const double* uy = A.u + g.plane;
        double div = ddx(ux, g.px, i, j, g, c.inv2h) + ddy(uy, g.px, i, j, g, c.inv2h);
        double curl = ddx(uy, g.px, i, j, g, c.inv2h) - ddy(ux, g.px, i, j, g, c.inv2h);
        double e1 = moment0_fp64(A, g.plane, p, 1, k) - curl;
        double e0 = moment0_fp64(A, g.plane, p, 0, k) - div;
        return sqrt(e1 * e1 + e0 * e0);
    }
    }
}

// Dense FP64 copy of rows [j0, j0 + rows) of a field.  Population fields
// write 5 consecutive [rows][nx] blocks.
template <typename P>
__global__ void extract_kernel(Geo g, Consts c, KCof<P> k, View<P> A, int field, int j0, int rows, double* dst) {
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    int jr = blockIdx.y * blockDim.y + threadIdx.y;
    if (i >= g.nx || jr >= rows) return;
    int j = j0 + jr;
    size_t d = (size_t)jr * g.nx + i;
    if (field == FLD_FPHI || field == FLD_FPSI) {
        int set = field == FLD_FPHI ? 0 : 1;
        size_t p = (size_t)j * g.px + i;
        size_t blk = (size_t)rows * g.nx;
        double f[5];
        P::load5d(A.f, g.plane, p, set, k, f);
        for (int q = 0; q < 5; ++q) dst[q * blk + d] = f[q];
        return;
    }
    dst[d] = field_value<P>(g, c, k, A, field, i, j);
}

// --------------------------------------------------------------- norms

constexpr int kNormThreads = 256;

template <typename P>
__global__ void __launch_bounds__(kNormThreads) norms_partial_kernel(Geo g, Consts c, KCof<P> k, View<P> A,
                                                                     int field,
                                                                     const double* __restrict__ ref,
                                                                     double* partials) {
    __shared__ double sh[4][kNormThreads];
    double s0 = 0.0, s1 = 0.0, s2 = 0.0, mx = 0.0;
    size_t n = (size_t)g.nx * g.ny;
    for (size_t d = (size_t)blockIdx.x * blockDim.x + threadIdx.x; d < n; d += (size_t)gridDim.x * blockDim.x) {
        int i = (int)(d % g.nx), j = (int)(d / g.nx);
        double x = field_value<P>(g, c, k, A, field, i, j);
        double r = ref ? ref[d] : 0.0;
        double e = x - r;
        s0 += e * e;
        s1 += r * r;
        s2 += x;
        mx = fmax(mx, fabs(x));
    }
    sh[0][threadIdx.x] = s0;
    sh[1][threadIdx.x] = s1;
    sh[2][threadIdx.x] = s2;
    sh[3][threadIdx.x] = mx;
    __syncthreads();
    for (int w = kNormThreads / 2; w > 0; w >>= 1) {
        if (threadIdx.x < w) {
            sh[0][threadIdx.x] += sh[0][threadIdx.x + w];
            sh[1][threadIdx.x] += sh[1][threadIdx.x + w];
            sh[2][threadIdx.x] += sh[2][threadIdx.x + w];
            sh[3][threadIdx.x] = fmax(sh[3][threadIdx.x], sh[3][threadIdx.x + w]);
        }
        __syncthreads();
    }
    if (threadIdx.x == 0)
        for (int q = 0; q < 4; ++q) partials[(size_t)blockIdx.x * 4 + q] = sh[q][0];
}

__global__ void __launch_bounds__(kNormThreads) norms_final_kernel(const double* partials, int nblk, double* out) {
    __shared__ double sh[4][kNormThreads];
    double s[4] = {0.0, 0.0, 0.0, 0.0};
    for (int b = threadIdx.x; b < nblk; b += kNormThreads) {
        s[0] += partials[(size_t)b * 4];
        s[1] += partials[(size_t)b * 4 + 1];
        s[2] += partials[(size_t)b * 4 + 2];
        s[3] = fmax(s[3], partials[(size_t)b * 4 + 3]);
    }
    for (int q = 0; q < 4; ++q) sh[q][threadIdx.x] = s[q];
    __syncthreads();
    for (int w = kNormThreads / 2; w > 0; w >>= 1) {
        if (threadIdx.x < w) {
            sh[0][threadIdx.x] += sh[0][threadIdx.x + w];
            sh[1][threadIdx.x] += sh[1][threadIdx.x + w];
            sh[2][threadIdx.x] += sh[2][threadIdx.x + w];
            sh[3][threadIdx.x] = fmax(sh[3][threadIdx.x], sh[3][threadIdx.x + w]);
        }
        __syncthreads();
    }
    if (threadIdx.x == 0)
        for (int q = 0; q < 4; ++q) out[q] = sh[q][0];
}

// Both energies in one pass: per block the sums over body points of |du/dt|^2,
// tr(d)^2, d_xx^2 + d_yy^2 and (d_xy + d_yx)^2 with the unscaled differences d
// of u; the constants come in at the end (13 FP64 instructions a point instead
// of 32 for the two densities; bound by them).
template <typename P>
__global__ void __launch_bounds__(kNormThreads) energy_partial_kernel(Geo g, View<P> A, double* partials) {
    __shared__ double sh[4][kNormThreads];
    const double* ux = A.u;
    const double* uy = A.u + g.plane;
    double s[4] = {0.0, 0.0, 0.0, 0.0};
    for (int j = blockIdx.y; j < g.ny; j += gridDim.y)
        for (int i = blockIdx.x * kNormThreads + threadIdx.x; i < g.nx; i += gridDim.x * kNormThreads) {
            if (!body_at(g, i, j)) continue;
            const size_t p = (size_t)j * g.px + i;
            const double vx = LBPS_LD(&A.u[2 * g.plane + p]), vy = LBPS_LD(&A.u[3 * g.plane + p]);
            const int kx = diff_kind(g, i, j, 1, 0), ky = diff_kind(g, i, j, 0, 1);
            const double exx = diff3(ux + p, kx, i, g.nx, 1), eyx = diff3(uy + p, kx, i, g.nx, 1);
            const double exy = diff3(ux + p, ky, j, g.ny, g.px), eyy = diff3(uy + p, ky, j, g.ny, g.px);
            const double tr = add_rn(exx, eyy), sh2 = add_rn(exy, eyx);
            s[0] = fma_rn(vx, vx, fma_rn(vy, vy, s[0]));
            s[1] = fma_rn(tr, tr, s[1]);
            s[2] = fma_rn(exx, exx, fma_rn(eyy, eyy, s[2]));
            s[3] = fma_rn(sh2, sh2, s[3]);
        }
#pragma unroll
    for (int q = 0; q < 4; ++q) sh[q][threadIdx.x] = s[q];
    __syncthreads();
    for (int w = kNormThreads / 2; w > 0; w >>= 1) {
        if (threadIdx.x < w)
            for (int q = 0; q < 4; ++q) sh[q][threadIdx.x] += sh[q][threadIdx.x + w];
        __syncthreads();
    }
    if (threadIdx.x < 4)
        partials[((size_t)blockIdx.y * gridDim.x + blockIdx.x) * 4 + threadIdx.x] = sh[threadIdx.x][0];
}

// out = kinetic and strain energy per dh^2 (sums of the densities).
__global__ void __launch_bounds__(kNormThreads) energy_final_kernel(Consts c, const double* partials, int nblk,
                                                                    double* out) {
    __shared__ double sh[4][kNormThreads];
    double s[4] = {0.0, 0.0, 0.0, 0.0};
    for (int b = threadIdx.x; b < nblk; b += kNormThreads)
#pragma unroll
        for (int q = 0; q < 4; ++q) s[q] += partials[(size_t)b * 4 + q];
#pragma unroll
    for (int q = 0; q < 4; ++q) sh[q][threadIdx.x] = s[q];
    __syncthreads();
    for (int w = kNormThreads / 2; w > 0; w >>= 1) {
        if (threadIdx.x < w)
            for (int q = 0; q < 4; ++q) sh[q][threadIdx.x] += sh[q][threadIdx.x + w];
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        out[0] = 0.5 * c.rho * sh[0][0];
        out[1] = (0.5 * c.lam * sh[1][0] + c.mu * (sh[2][0] + 0.5 * sh[3][0])) * (c.inv2h * c.inv2h);
    }
}

// Rows of a state copy to or from a caller buffer, 16 bytes per thread and
// step; segment blockIdx.y.  The lattice side of each copy goes through the
// checked accessors, the caller's buffer is not part of a lattice block.
__global__ void copy_segments_kernel(CopySegs s) {
    const int q = blockIdx.y;
    if (q >= s.n) return;
    const uint4* a = reinterpret_cast<const uint4*>(s.src[q]);
    uint4* b = reinterpret_cast<uint4*>(s.dst[q]);
    const size_t n16 = s.bytes[q] / 16;
    for (size_t t = (size_t)blockIdx.x * blockDim.x + threadIdx.x; t < n16; t += (size_t)gridDim.x * blockDim.x) {
#ifdef LBPS_CHECKED
        if (!chk_ok(s.pack ? &a[t] : &b[t], __LINE__)) continue;
#endif
        b[t] = a[t];
    }
}

dim3 grid2d(int nx, int ny, dim3 blk) { return dim3((nx + blk.x - 1) / blk.x, (ny + blk.y - 1) / blk.y); }

}  // namespace

// ------------------------------------------------------------- launchers

// Threads per boundary point of the Newmark and reset passes.  Few points are
// bound by the FP64 instructions of each warp, so two warps share a point's
// parts; many points are bound by the sectors they gather, which one thread
// fetches once for both parts (256 lattices, 297 000 points: the reset 84 us
// with one thread, 94 us with two).
int boundary_parts(int points) { return points <= 32768 ? 2 : 1; }

template <typename P>
cudaError_t launch_boundary_batch(const DomDesc<P>* dd, const BndTask* tasks, int ntasks, int parity, int pass_lo,
                                  int pass_hi, cudaStream_t st, int stage) {
    if (ntasks > 0)
        for (int pass = pass_lo; pass < pass_hi; ++pass) {
            boundary_batch_kernel<P>
                <<<dim3((ntasks + 127) / 128, pass == 3 ? 1 : boundary_parts(ntasks)), 128, 0, st>>>(dd, tasks, ntasks, parity, pass, stage);
            if (pass == 2 && P::kSplitStream)
                boundary_batch_kernel<P><<<(ntasks + 127) / 128, 128, 0, st>>>(dd, tasks, ntasks, parity, 3, stage);
        }
    return cudaGetLastError();
}

// Blocks of the persistent batch kernel: those resident on all SMs at once.
template <typename K>
int resident_blocks(K kernel) {
    int dev = 0, sms = 0, per_sm = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return -1;
    if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) return -1;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, 32 * kWarpsPerBlock, 0) != cudaSuccess)
        return -1;
    return sms * (per_sm > 0 ? per_sm : 1);
}

template <typename P, int MINB, int UVD>
cudaError_t launch_bulk_batch_v(const DomDesc<P>* dd, const BulkTask* tasks, int ntasks, const BndTask* btasks,
                                int parity, unsigned* next, cudaStream_t st) {
    auto kern = bulk_batch_kernel<P, MINB, UVD>;
    int blocks = resident_blocks(kern);
    if (blocks < 0) return cudaGetLastError();
    blocks = min(blocks, (ntasks + kWarpsPerBlock - 1) / kWarpsPerBlock);
    cudaError_t e = cudaMemsetAsync(next, 0, sizeof(unsigned), st);
    if (e != cudaSuccess) return e;
    kern<<<blocks, 32 * kWarpsPerBlock, 0, st>>>(dd, tasks, ntasks, btasks, parity, next);
    return cudaGetLastError();
}

template <typename P>
cudaError_t launch_pair_batch(const DomDesc<P>* dd, const PairTask* tasks, int ntasks, const BndTask* btasks,
                              int parity, int stage, unsigned* next, cudaStream_t st) {
    if (ntasks <= 0) return cudaGetLastError();
    if (stage == 2) {
        edge_batch_kernel<P><<<(ntasks + kWarpsPerBlock - 1) / kWarpsPerBlock, 32 * kWarpsPerBlock, 0, st>>>(
            dd, tasks, ntasks, btasks, parity);
        return cudaGetLastError();
    }
    // 4 blocks per SM (at 5 the two kinds of strips together spill)
    auto kern = pair_batch_kernel<P, sizeof(typename P::V) == 8 ? 2 : 4>;
    int blocks = resident_blocks(kern);
    if (blocks < 0) return cudaGetLastError();
    blocks = min(blocks, (ntasks + kWarpsPerBlock - 1) / kWarpsPerBlock);
    kern<<<blocks, 32 * kWarpsPerBlock, 0, st>>>(dd, tasks, ntasks, btasks, parity, next);
    return cudaGetLastError();
}

template <typename P>
cudaError_t launch_bulk_batch(const DomDesc<P>* dd, const BulkTask* tasks, int ntasks, const BndTask* btasks,
                              int parity, int variant, unsigned* next, cudaStream_t st) {
    if (ntasks <= 0) return cudaGetLastError();
    switch (variant) {
    case 0: return launch_bulk_batch_v<P, 6, 2>(dd, tasks, ntasks, btasks, parity, next, st);
    case 1: return launch_bulk_batch_v<P, 5, 2>(dd, tasks, ntasks, btasks, parity, next, st);
    case 2: return launch_bulk_batch_v<P, 4, 2>(dd, tasks, ntasks, btasks, parity, next, st);
    case 3: return launch_bulk_batch_v<P, 8, 2>(dd, tasks, ntasks, btasks, parity, next, st);
    case 4: return launch_bulk_batch_v<P, 6, 1>(dd, tasks, ntasks, btasks, parity, next, st);
    case 5: return launch_bulk_batch_v<P, 5, 1>(dd, tasks, ntasks, btasks, parity, next, st);
    case 6: return launch_bulk_batch_v<P, 4, 1>(dd, tasks, ntasks, btasks, parity, next, st);
    default: return launch_bulk_batch_v<P, 8, 1>(dd, tasks, ntasks, btasks, parity, next, st);
    }
}

cudaError_t launch_copy_segments(const CopySegs& s, cudaStream_t st) {
    if (s.n <= 0) return cudaSuccess;
    size_t most = 0;
    for (int q = 0; q < s.n; ++q) most = std::max(most, s.bytes[q] / 16);
    const int bx = (int)std::min<size_t>((most + 255) / 256, 1024);
    copy_segments_kernel<<<dim3(std::max(bx, 1), s.n), 256, 0, st>>>(s);
    return cudaGetLastError();
}

#ifdef LBPS_CHECKED
namespace {
// the table of live blocks, mirrored on the host and uploaded whole
std::vector<std::pair<const char*, const char*>> ranges;
}  // namespace

bool check_live(const void* p, size_t bytes) {
    const char* lo = static_cast<const char*>(p);
    return std::any_of(ranges.begin(), ranges.end(),
                       [&](const auto& r) { return lo >= r.first && lo + bytes <= r.second; });
}
#endif

cudaError_t set_check_range(const void* base, size_t bytes, cudaStream_t st) {
#ifdef LBPS_CHECKED
    const char* lo = static_cast<const char*>(base);
    ranges.erase(std::remove_if(ranges.begin(), ranges.end(), [&](const auto& r) { return r.first == lo; }),
                 ranges.end());
    if (bytes > 0) {
        if (ranges.size() >= (size_t)kChkRanges) return cudaErrorInvalidValue;
        ranges.emplace_back(lo, lo + bytes);
    }
    std::vector<const char*> los, his;
    for (const auto& r : ranges) {
        los.push_back(r.first);
        his.push_back(r.second);
    }
    const int n = (int)ranges.size();
    cudaError_t e = cudaStreamSynchronize(st);  // no kernel in flight sees a half-written table
    if (e == cudaSuccess) e = upload_check_table(los.data(), his.data(), n);
    if (e == cudaSuccess) e = fused_check_table(los.data(), his.data(), n);
    if (e == cudaSuccess) e = sweep_check_table(los.data(), his.data(), n);
    return e;
#else
    (void)base;
    (void)bytes;
    (void)st;
    return cudaSuccess;
#endif
}

int check_report(unsigned long long out[2]) {
#ifdef LBPS_CHECKED
    if (cudaDeviceSynchronize() != cudaSuccess) return -1;
    int rc = read_check_report(out);
    if (rc > 0 && out[0] == 0) rc = fused_check_report(out);
    if (rc > 0 && out[0] == 0) rc = sweep_check_report(out);
    return rc;
#else
    out[0] = out[1] = 0;
    return 0;
#endif
}

cudaError_t launch_finite_check(const Geo& g, const double* u, int planes, unsigned* bad, cudaStream_t st) {
    int dev = 0, sms = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) !=
                                                  cudaSuccess)
        return cudaGetLastError();
    const size_t total = (size_t)g.nx * (size_t)g.ny * (size_t)planes;
    const size_t want = (total + 255) / 256;
    const int blocks = (int)std::min<size_t>(want, (size_t)sms * 8);
    finite_check_kernel<<<blocks, 256, 0, st>>>(g, u, planes, bad);
    return cudaGetLastError();
}

cudaError_t launch_scale_probe(const Geo& g, const Consts& c, const double* u, double sq, unsigned* out,
                               cudaStream_t st) {
    dim3 blk(32, 8);
    scale_probe_kernel<<<grid2d(g.nx, g.ny, blk), blk, 0, st>>>(g, c, u, sq, out);
    return cudaGetLastError();
}

template <typename P>
cudaError_t launch_init(const Geo& g, const Consts& c, const KCof<P>& k, View<P> A, cudaStream_t st) {
    dim3 blk(32, 8);
    init_kernel<P><<<grid2d(g.nx, g.ny, blk), blk, 0, st>>>(g, c, k, A);
    return cudaGetLastError();
}

template <typename P>
cudaError_t launch_mirror(const Geo& g, View<P> A, const BNode* bn, int nb, cudaStream_t st) {
    if (nb > 0) boundary_mirror_kernel<P><<<(nb + 127) / 128, 128, 0, st>>>(g, A, bn, nb);
    return cudaGetLastError();
}

template <typename P>
cudaError_t launch_boundary(const Geo& g, const Consts& c, const KCof<P>& k, View<P> A, View<P> B, const BNode* bn,
                            int nb, unsigned* flag, unsigned long long* tstep, cudaStream_t st,
                            int pass_lo, int pass_hi) {
    if (nb > 0) {
        const int blocks = (nb + 127) / 128, parts = boundary_parts(nb);
        for (int pass = pass_lo; pass < pass_hi; ++pass) {
            if (pass == 0) boundary_stress_kernel<P><<<blocks, 128, 0, st>>>(g, c, A, bn, nb);
            if (pass == 1) boundary_newmark_kernel<P><<<dim3(blocks, parts), 128, 0, st>>>(g, c, A, B, bn, nb, tstep);
            if (pass == 2) boundary_reset_kernel<P><<<dim3(blocks, parts), 128, 0, st>>>(g, c, k, A, B, bn, nb, flag, tstep);
            if (pass == 2 && P::kSplitStream)
                boundary_stream_y_kernel<P><<<blocks, 128, 0, st>>>(g, c, k, A, B, bn, nb);
        }
    }
    return cudaGetLastError();
}

template <typename P>
cudaError_t launch_bulk(const Geo& g, const Consts& c, const KCof<P>& k, View<P> A, View<P> B, unsigned* flag,
                        cudaStream_t st, const Tuning& tu) {
    int warps = (g.nx + kStripCols - 1) / kStripCols;
    dim3 grid((warps + kWarpsPerBlock - 1) / kWarpsPerBlock, (g.ny + tu.rows_per_warp - 1) / tu.rows_per_warp);
    dim3 blk(32 * kWarpsPerBlock);
    switch (tu.variant) {
    case 0: bulk_kernel<P, 6, 2><<<grid, blk, 0, st>>>(g, c, k, A, B, flag, tu.rows_per_warp); break;
    case 1: bulk_kernel<P, 5, 2><<<grid, blk, 0, st>>>(g, c, k, A, B, flag, tu.rows_per_warp); break;
    case 2: bulk_kernel<P, 4, 2><<<grid, blk, 0, st>>>(g, c, k, A, B, flag, tu.rows_per_warp); break;
    case 3: bulk_kernel<P, 8, 2><<<grid, blk, 0, st>>>(g, c, k, A, B, flag, tu.rows_per_warp); break;
    case 4: bulk_kernel<P, 6, 1><<<grid, blk, 0, st>>>(g, c, k, A, B, flag, tu.rows_per_warp); break;
    case 5: bulk_kernel<P, 5, 1><<<grid, blk, 0, st>>>(g, c, k, A, B, flag, tu.rows_per_warp); break;
    case 6: bulk_kernel<P, 4, 1><<<grid, blk, 0, st>>>(g, c, k, A, B, flag, tu.rows_per_warp); break;
    default: bulk_kernel<P, 8, 1><<<grid, blk, 0, st>>>(g, c, k, A, B, flag, tu.rows_per_warp); break;
    }
    return cudaGetLastError();
}

template <typename P>
cudaError_t launch_frame(const Geo& g, const Consts& c, const KCof<P>& k, View<P> A, View<P> B, unsigned* flag,
                         cudaStream_t st, int fw) {
    // FP64 populations need the 4-blocks shape (the others spill there);
    // BFP13 fits 6 blocks with u prefetched one row ahead, not two
    constexpr int minb = sizeof(typename P::V) == 8 ? 4 : 6;
    constexpr int uvd = std::is_same<P, PopBfp13>::value ? 1 : 2;
    const int strips = (g.nx + kStripCols - 1) / kStripCols;
    const int bands = 2 * ((strips + kWarpsPerBlock - 1) / kWarpsPerBlock);
    auto run = [&](auto kern, int W) {
        const int task = 32 / W * kSideRows, sides = 2 * ((g.ny - 2 - 2 * fw + task - 1) / task);
        kern<<<bands + (sides + kWarpsPerBlock - 1) / kWarpsPerBlock, 32 * kWarpsPerBlock, 0, st>>>(g, c, k, A, B, flag,
                                                                                                   fw, bands);
    };
    if (fw + 2 <= 8)
        run(frame_kernel<P, minb, uvd>, 8);
    else
        run(frame_wide_kernel<P, minb, uvd>, 16);
    return cudaGetLastError();
}

template <typename P>
cudaError_t launch_pair(const Geo& g, const Consts& c, const KCof<P>& k, View<P> A, View<P> B, unsigned* flag,
                        cudaStream_t st, int rows) {
    const int warps = (g.nx - 2 * kDeep + kPairCols - 1) / kPairCols;
    const dim3 grid((warps + kWarpsPerBlock - 1) / kWarpsPerBlock, (g.ny - 2 * kDeep + rows - 1) / rows);
    // blocks per SM that fit without spilling: 5 for FP32 and the 16-bit
    // formats (96 registers; 8192^2 FP32: 70.2 against 67.1 GLUPS at 4),
    // 2 for FP64
    constexpr int minb = sizeof(typename P::V) == 8 ? 2 : 5;
    pair_kernel<P, minb><<<grid, 32 * kWarpsPerBlock, 0, st>>>(g, c, k, A, B, flag, rows);
    return cudaGetLastError();
}

template <typename P>
cudaError_t launch_sync(const Geo& g, const Consts& c, const KCof<P>& k, View<P> A, cudaStream_t st) {
    dim3 blk(32, 8);
    sync_kernel<P><<<grid2d(g.nx, g.ny, blk), blk, 0, st>>>(g, c, k, A);
    return cudaGetLastError();
}

template <typename P>
cudaError_t launch_extract_rows(const Geo& g, const Consts& c, const KCof<P>& k, View<P> A, int field, int j0,
                                int rows, double* dst, cudaStream_t st) {
    dim3 blk(32, 8);
    extract_kernel<P><<<grid2d(g.nx, rows, blk), blk, 0, st>>>(g, c, k, A, field, j0, rows, dst);
    return cudaGetLastError();
}

template <typename P>
cudaError_t launch_norms(const Geo& g, const Consts& c, const KCof<P>& k, View<P> A, int field, const double* ref,
                         double* partials, double* out4, cudaStream_t st) {
    size_t n = (size_t)g.nx * g.ny;
    int nblk = (int)((n + kNormThreads - 1) / kNormThreads);
    if (nblk > kNormBlocks) nblk = kNormBlocks;
    norms_partial_kernel<P><<<nblk, kNormThreads, 0, st>>>(g, c, k, A, field, ref, partials);
    norms_final_kernel<<<1, kNormThreads, 0, st>>>(partials, nblk, out4);
    return cudaGetLastError();
}

template <typename P>
cudaError_t launch_energy(const Geo& g, const Consts& c, View<P> A, double* partials, double* out2, cudaStream_t st) {
    // a block per row; flat lattices split their rows too, a thread keeping at
    // least 4 columns (a block per row only: 20000 x 20 156 us, 300000 x 16 2064)
    const int rows = std::min(g.ny, kNormBlocks);
    const int cols = std::max(1, std::min(kNormBlocks / rows, g.nx / (4 * kNormThreads)));
    energy_partial_kernel<P><<<dim3(cols, rows), kNormThreads, 0, st>>>(g, A, partials);
    energy_final_kernel<<<1, kNormThreads, 0, st>>>(c, partials, cols * rows, out2);
    return cudaGetLastError();
}

#define LBPS_INSTANTIATE(P)                                                                                   \
    template cudaError_t launch_energy<P>(const Geo&, const Consts&, View<P>, double*, double*, cudaStream_t);   \
    template cudaError_t launch_init<P>(const Geo&, const Consts&, const KCof<P>&, View<P>, cudaStream_t);  \
    template cudaError_t launch_frame<P>(const Geo&, const Consts&, const KCof<P>&, View<P>, View<P>, unsigned*,  \
                                         cudaStream_t, int);                                                  \
    template cudaError_t launch_pair<P>(const Geo&, const Consts&, const KCof<P>&, View<P>, View<P>, unsigned*,   \
                                        cudaStream_t, int);                                                   \
    template cudaError_t launch_mirror<P>(const Geo&, View<P>, const BNode*, int, cudaStream_t);            \
    template cudaError_t launch_boundary<P>(const Geo&, const Consts&, const KCof<P>&, View<P>, View<P>,      \
                                            const BNode*, int, unsigned*, unsigned long long*,                \
                                            cudaStream_t, int, int);                                          \
    template cudaError_t launch_bulk<P>(const Geo&, const Consts&, const KCof<P>&, View<P>, View<P>,          \
                                        unsigned*, cudaStream_t, const Tuning&);                              \
    template cudaError_t launch_sync<P>(const Geo&, const Consts&, const KCof<P>&, View<P>, cudaStream_t);  \
    template cudaError_t launch_extract_rows<P>(const Geo&, const Consts&, const KCof<P>&, View<P>, int, int, \
                                                int, double*, cudaStream_t);                                  \
    template cudaError_t launch_norms<P>(const Geo&, const Consts&, const KCof<P>&, View<P>, int,            \
                                         const double*, double*, double*, cudaStream_t);                     \
    template cudaError_t launch_boundary_batch<P>(const DomDesc<P>*, const BndTask*, int, int, int, int,      \
                                                  cudaStream_t, int);                                         \
    template cudaError_t launch_pair_batch<P>(const DomDesc<P>*, const PairTask*, int, const BndTask*, int, int, \
                                              unsigned*, cudaStream_t);                                       \
    template cudaError_t launch_bulk_batch<P>(const DomDesc<P>*, const BulkTask*, int, const BndTask*, int, int, \
                                              unsigned*, cudaStream_t);

LBPS_INSTANTIATE(PopDirect<float>)
LBPS_INSTANTIATE(PopDirect<double>)
LBPS_INSTANTIATE(PopNeq16<__nv_bfloat16>)
LBPS_INSTANTIATE(PopNeq16<__half>)
LBPS_INSTANTIATE(PopBfp13)

}  // namespace lbps
