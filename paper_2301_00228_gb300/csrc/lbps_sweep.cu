// Several time steps of the deep interior of a rectangle in one sweep.
//
// A point at least K + 1 from every edge depends, K steps later, only on
// interior points that the boundary reset of the steps between leaves alone
// (the reset of a step changes the points at most 1 from an edge, and that
// reaches one point further each step).  So a sweep that reads the state once
// and writes it once advances those points by K steps; the boundary rules and
// the points up to K from the edges run step by step beside it.
//
// Each warp marches down a strip of 32 columns, K pipeline stages deep: a row
// enters as state n, each iteration moves every stage one row on, and the row
// K - 1 above leaves as state n + K.  A stage keeps the row before (moment,
// f^4) and its own row; x neighbours come by shuffles, so each step costs a
// column on both sides (32 - 2 K columns come out).  Every step rounds to the
// stored form, so the populations are the bits of single steps.  u, du/dt wait
// in shared memory until their row leaves and then take two steps at a time
// (newmark2).
#include <algorithm>
#include <cstring>

#include <cuda.h>

#include "lbps_steps.cuh"

namespace lbps {

namespace {

// Polls of an mbarrier before a warp gives up (a second or more).
#ifndef LBPS_SWEEP_POLLS
#define LBPS_SWEEP_POLLS (1 << 22)
#endif
constexpr int kMaxWaits = LBPS_SWEEP_POLLS;
constexpr int kDrainWaits = 1 << 22;   // for each copy still under way then

__device__ __forceinline__ unsigned smem_addr(const void* p) { return (unsigned)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(unsigned long long* bar) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_addr(bar)) : "memory");
}

__device__ __forceinline__ void mbar_expect(unsigned long long* bar, unsigned bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_addr(bar)), "r"(bytes) : "memory");
}

// The same answer in every lane of the warp.
__device__ __forceinline__ bool mbar_wait(unsigned long long* bar, unsigned parity, int polls) {
#pragma unroll 1
    for (int n = 0; n < polls; ++n) {
        unsigned ok;
        asm volatile(
            "{\n.reg .pred p;\n"
            "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
            "selp.u32 %0, 1, 0, p;\n}\n"
            : "=r"(ok)
            : "r"(smem_addr(bar)), "r"(parity)
            : "memory");
        if (__all_sync(0xffffffffu, ok)) return true;
    }
    return false;
}

__device__ __forceinline__ void tma_load(void* dst, const CUtensorMap* map, int x, int y, unsigned long long* bar) {
    asm volatile(
        "cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], "
        "[%5];" ::"r"(smem_addr(dst)),
        "l"(map), "r"(x), "r"(y), "r"(0), "r"(smem_addr(bar))
        : "memory");
}

// Before the first use of a tensor map that lies in global memory (written by
// the host): what was copied there is seen by the copies issued from here on,
// not a map that an earlier launch used at the same address.
__device__ __forceinline__ void acquire_map(const CUtensorMap* map) {
    asm volatile("fence.proxy.tensormap::generic.acquire.sys [%0], 128;" ::"l"(map) : "memory");
}

template <typename P>
constexpr bool kHashed = false;
template <typename H>
constexpr bool kHashed<PopNeq16<H>> = true;

// Ends a warp's reads of a slot before a copy into it is issued: orders every
// lane's earlier shared-memory loads before later asynchronous copies (without
// it ptxas may move a load whose value is needed late past the copy's issue),
// then waits for every lane.
__device__ __forceinline__ void release_slot() {
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    __syncwarp();
}

// Shape of a sweep of K steps over 4-byte population planes.  A warp's lanes
// are 32 columns, of which the inner OUT come out K steps later.  A slot of
// the warp's ring holds two rows: the box of the populations ([plane][2][BOX]
// words, from column xs - SKIP - K, a multiple of 4) and the box of u, du/dt
// of the rows that leave the pipeline with them ([4][2][OUT] doubles).
template <typename P, int K>
struct Sweep {
    static constexpr int OUT = 32 - 2 * K;
    static constexpr int SKIP = (4 - K % 4) % 4;
    static constexpr int BOX = (32 + SKIP + 3) / 4 * 4;
    static constexpr int PLANES = P::kBytesPerPoint / 4;
    static constexpr int F_BYTES = PLANES * 2 * BOX * 4;
    static constexpr int U_OFF = (F_BYTES + 127) / 128 * 128;
    static constexpr int U_BYTES = 4 * 2 * OUT * 8;
    static constexpr int SLOT = U_OFF + (U_BYTES + 127) / 128 * 128;
    static constexpr int DEPTH = K == 4 ? 4 : 2;   // slots; 16 or 9.5 KB a warp
    // blocks per SM: FP16 and BF16 spill at 96 registers (8192^2 FP16: 743 us
    // a step at 4 blocks, 830 at 5)
    static constexpr int MINB = K == 4 ? 3 : kHashed<P> ? 4 : 5;
    static constexpr int DEEP = K + 1;   // distance from the edges of the points a sweep writes
    static constexpr size_t kSmem = (size_t)kWarpsPerBlock * DEPTH * SLOT;
};

// What a row keeps of its accelerations until its last step: the sums of each
// pair of steps that newmark2 takes, or the first acceleration of a pair.
template <typename V>
struct Acc {
    V a[2];        // the acceleration of a pair's first step
    V sa[2], sb[2];  // 3 a0 + a1 and a0 + a1 of the pair before
};

// EXACT: u, du/dt take the steps one by one (the bits of single steps), not two
// at a time.  margin: the distance from the edges of the points it writes.
template <typename P, int K, bool EXACT = false>
__device__ __forceinline__ bool sweep_strip(const Geo& g, const Consts& c, const KCof<P>& k,
                                            const CUtensorMap* mf, const CUtensorMap* mu, const View<P>& B, char* ring,
                                            unsigned long long* bars, unsigned& base, int xs, int j0, int j1,
                                            bool& timeout, int margin = K + 1) {
    using V = typename P::V;
    using S = Sweep<P, K>;
    const unsigned FULL = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    const int col = xs - K + lane;
    const bool out_lane = lane >= K && lane < 32 - K && col >= margin && col < g.nx - margin;
    const size_t PL = g.plane;
    const int nq = j1 - j0 + 2 * K, ngroups = (nq + 1) / 2;   // rows read, and pairs of them
    const int nit = nq - 2;

    // pair q of this strip is pair base + q of the warp's ring
    auto slot_of = [&](int q) { return (int)((base + (unsigned)q) % (unsigned)S::DEPTH); };
    // a warp gives up as a whole (its lanes shuffle), and only when the copies
    // it issued have landed or run out too (after the return the block's shared
    // memory may be another block's)
    auto landed = [&](int q, int polls) {
        return mbar_wait(bars + slot_of(q), ((base + (unsigned)q) / (unsigned)S::DEPTH) & 1u, polls);
    };
    auto arrived = [&](int q) {
        if (landed(q, kMaxWaits)) return true;
#pragma unroll 1
        for (int p = q; p < q + S::DEPTH && p < ngroups; ++p) landed(p, kDrainWaits);
        return false;
    };
    auto issue = [&](int q) {   // lane 0
        char* slot = ring + slot_of(q) * S::SLOT;
        unsigned long long* bar = bars + slot_of(q);
        // rows j0 - K + 2q, + 1 of the populations; the rows that leave while they enter
        mbar_expect(bar, S::F_BYTES + (q >= K ? S::U_BYTES : 0));
        tma_load(slot, mf, xs - K - S::SKIP, j0 - K + 2 * q, bar);
        if (q >= K) tma_load(slot + S::U_OFF, mu, xs, j0 + 2 * (q - K), bar);
    };
    if (lane == 0)
        for (int q = 0; q < S::DEPTH && q < ngroups; ++q) issue(q);

    auto read_row = [&](const char* slot, int half, V (&f)[2][5]) {
        const unsigned* w = reinterpret_cast<const unsigned*>(slot) + half * S::BOX + S::SKIP + lane;
        unsigned words[S::PLANES];
#pragma unroll
        for (int q = 0; q < S::PLANES; ++q) words[q] = w[q * 2 * S::BOX];
        typename P::Raw r;
        static_assert(sizeof(r) == sizeof(words), "a point's words are its planes in order");
        memcpy(&r, words, sizeof(r));
        decode_row<P>(r, k, f);
    };

    // per stage: the row before (moment, f^4) and the row itself
    V Ps[K][2] = {}, P4[K][2] = {}, Cf[K][2][5] = {}, Cm[K][2] = {};
    Acc<V> hist[K] = {};
    bool bad = false;

    auto iterate = [&](const char* slot, int half, int it) {
        V N[2][5];
        read_row(slot, half, N);
        Acc<V> from = {};   // of the row that enters this stage, from the stage before
        V out[2][5];
        V ax = 0, ay = 0;
#pragma unroll
        for (int s = 0; s < K; ++s) {
            V Nm[2], Ns[2], Cs[2], sW[2], sE[2];
#pragma unroll
            for (int q = 0; q < 2; ++q) {
                Nm[q] = add_rn(add_rn(N[q][1], N[q][2]), add_rn(N[q][3], N[q][4]));
                Ns[q] = add_rn(N[q][0], Nm[q]);
                Cs[q] = add_rn(Cf[s][q][0], Cm[s][q]);
                sW[q] = __shfl_up_sync(FULL, Cs[q], 1);
                sE[q] = __shfl_down_sync(FULL, Cs[q], 1);
                const V f3W = __shfl_up_sync(FULL, Cf[s][q][3], 1);
                const V f1E = __shfl_down_sync(FULL, Cf[s][q][1], 1);
                out[q][0] = add_rn(Cf[s][q][0], fma_rn(k.two_a0[q], Cm[s][q], -mul_rn(k.eight_a[q], Cf[s][q][0])));
                out[q][1] = fma_rn(k.two_a[q], sW[q], -f3W);
                out[q][3] = fma_rn(k.two_a[q], sE[q], -f1E);
                out[q][2] = fma_rn(k.two_a[q], Ps[s][q], -P4[s][q]);
                out[q][4] = fma_rn(k.two_a[q], Ns[q], -N[q][2]);
            }
            accel_interior_v<V>(sW[0], sE[0], Ps[s][0], Ns[0], sW[1], sE[1], Ps[s][1], Ns[1], k, ax, ay);
#pragma unroll
            for (int q = 0; q < 2; ++q) {
                Ps[s][q] = Cs[q];
                P4[s][q] = Cf[s][q][4];
                Cm[s][q] = Nm[q];
#pragma unroll
                for (int d = 0; d < 5; ++d) Cf[s][q][d] = N[q][d];
            }
            if (s + 1 < K) {
                const Acc<V> keep = hist[s];
                hist[s] = from;
                if (s & 1) {   // the second step of a pair: its sums
                    hist[s].sa[0] = fma_rn((V)3, from.a[0], ax);
                    hist[s].sa[1] = fma_rn((V)3, from.a[1], ay);
                    hist[s].sb[0] = add_rn(from.a[0], ax);
                    hist[s].sb[1] = add_rn(from.a[1], ay);
                } else {
                    hist[s].a[0] = ax;
                    hist[s].a[1] = ay;
                }
                from = keep;
                // as stored at this stage's row and read back
                typename P::Raw raw;
                P::pack((size_t)(j0 - K + 1 + it - s) * (size_t)g.px + (size_t)col, out, k, raw);
                decode_row<P>(raw, k, N);
            }
        }
        if (it >= 2 * K - 2 && out_lane) {   // the first test is uniform over the warp
            const int e = it - (2 * K - 2);
            const size_t p = (size_t)(j0 + e) * (size_t)g.px + (size_t)col;
            const double* us = reinterpret_cast<const double*>(slot + S::U_OFF) + half * S::OUT + lane - K;
            double u[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) u[q] = us[q * 2 * S::OUT];
            if constexpr (K == 4) {
#pragma unroll
                for (int q = 0; q < 2; ++q) {
                    const double sa = widen(from.sa[q]), sb = widen(from.sb[q]);
                    u[q] = fma_rn(c.half_dt2, sa, fma_rn(c.dt2, u[2 + q], u[q]));
                    u[2 + q] = fma_rn(c.dt, sb, u[2 + q]);
                }
            }
            if constexpr (EXACT) {
                static_assert(K == 2, "one acceleration is kept");
                newmark(u[0], u[2], widen(from.a[0]), c, u[0], u[2]);
                newmark(u[1], u[3], widen(from.a[1]), c, u[1], u[3]);
                newmark(u[0], u[2], widen(ax), c, u[0], u[2]);
                newmark(u[1], u[3], widen(ay), c, u[1], u[3]);
            } else {
                newmark2(u[0], u[2], from.a[0], ax, c, u[0], u[2]);
                newmark2(u[1], u[3], from.a[1], ay, c, u[1], u[3]);
            }
            P::store_point(B.f, PL, p, out, k);
#pragma unroll
            for (int q = 0; q < 4; ++q) LBPS_ST(&B.u[(size_t)q * PL + p], u[q]);
            bad |= !isfinite(out[0][0] + out[1][0]);
        }
    };

    // rows 0 and 1: the window of the first stage
    if (!arrived(0)) {
        timeout = true;
        return false;
    }
    {
        const char* slot = ring + slot_of(0) * S::SLOT;
        V t[2][5];
        read_row(slot, 0, t);
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            Ps[0][q] = sum5(t[q][0], t[q][1], t[q][2], t[q][3], t[q][4]);
            P4[0][q] = t[q][4];
        }
        read_row(slot, 1, Cf[0]);
#pragma unroll
        for (int q = 0; q < 2; ++q)
            Cm[0][q] = add_rn(add_rn(Cf[0][q][1], Cf[0][q][2]), add_rn(Cf[0][q][3], Cf[0][q][4]));
    }
    release_slot();
    if (lane == 0 && S::DEPTH < ngroups) issue(S::DEPTH);
    for (int q = 1; q < ngroups; ++q) {
        char* slot = ring + slot_of(q) * S::SLOT;
        if (!arrived(q)) {
            timeout = true;
            return bad;
        }
        iterate(slot, 0, 2 * q - 2);
        if (2 * q - 1 < nit) iterate(slot, 1, 2 * q - 1);
        release_slot();
        if (lane == 0 && q + S::DEPTH < ngroups) issue(q + S::DEPTH);
    }
    base += (unsigned)ngroups;
    return bad;
}

// The barriers of a warp's ring, before its first strip.
template <typename S>
__device__ __forceinline__ void init_ring(unsigned long long* bars) {
    if ((threadIdx.x & 31) == 0) {
        for (int q = 0; q < S::DEPTH; ++q) mbar_init(bars + q);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    __syncwarp();
}

// What bounds it: K = 4 in FP32, the FP64 pipe (12 instructions of 64 cycles a
// row and warp; 75 % busy on 3072^2, issue 49 %, DRAM 46 %, 363 us for 4 steps);
// K = 2 in the 16-bit formats, the issue slots their codec takes (BFP13 77 %,
// FP64 52 %, DRAM 73 %, 208 us for 2 steps; K = 4 takes 556 us for 4).  The
// rows come by TMA, two at a time and DEPTH pairs ahead, so no registers hold
// rows in flight: the kernel this replaced loaded them through registers, one
// row ahead, and waited on them (8192^2, two steps: FP32 1784 us, FP16 1632;
// now FP32 two steps 1626, four steps 2214; FP16 1398).  Blocks per SM: what
// the registers allow without spilling in earnest (K = 4 at 128 registers
// spills 314 bytes and takes 3340 us).
template <typename P, int K, int MINB, bool EXACT>
__global__ void __launch_bounds__(128, MINB) sweep_kernel(Geo g, Consts c, KCof<P> k,
                                                          const __grid_constant__ CUtensorMap mf,
                                                          const __grid_constant__ CUtensorMap mu, View<P> B,
                                                          unsigned* flag, int rows) {
    using S = Sweep<P, K>;
    extern __shared__ __align__(128) char smem[];
    __shared__ unsigned long long bars[kWarpsPerBlock * S::DEPTH];
    const int wid = threadIdx.x >> 5;
    const int xs = (blockIdx.x * kWarpsPerBlock + wid) * S::OUT;
    const int j0 = S::DEEP + blockIdx.y * rows, j1 = min(j0 + rows, g.ny - S::DEEP);
    if (xs >= g.nx - S::DEEP || j0 >= j1) return;   // whole warp
    init_ring<S>(bars + wid * S::DEPTH);
    bool timeout = false;
    unsigned base = 0;
    const bool bad = sweep_strip<P, K, EXACT>(g, c, k, &mf, &mu, B, smem + wid * (S::DEPTH * S::SLOT),
                                       bars + wid * S::DEPTH, base, xs, j0, j1, timeout);
    if (timeout) atomicOr(flag, kFlagTimeout);
    if (__any_sync(0xffffffffu, bad) && (threadIdx.x & 31) == 0) atomicOr(flag, kFlagNonfinite);
}

// Two exact steps of a lattice periodic in both axes, every point: the strips
// and chunks whose reads stay inside the planes by TMA, those across a seam
// (a box does not wrap) with loads through registers.
template <typename P, int MINB>
__global__ void __launch_bounds__(128, MINB) sweep_periodic_kernel(Geo g, Consts c, KCof<P> k,
                                                                   const __grid_constant__ CUtensorMap mf,
                                                                   const __grid_constant__ CUtensorMap mu, View<P> A,
                                                                   View<P> B, unsigned* flag, int rows) {
    using S = Sweep<P, 2>;
    extern __shared__ __align__(128) char smem[];
    __shared__ unsigned long long bars[kWarpsPerBlock * S::DEPTH];
    const int wid = threadIdx.x >> 5;
    const int xs = (blockIdx.x * kWarpsPerBlock + wid) * S::OUT;
    const int j0 = blockIdx.y * rows, j1 = min(j0 + rows, g.ny);
    if (xs >= g.nx || j0 >= j1) return;   // whole warp
    bool bad, timeout = false;
    if (xs >= 2 && xs + 30 <= g.nx && j0 >= 2 && j1 + 3 <= g.ny) {
        init_ring<S>(bars + wid * S::DEPTH);
        unsigned base = 0;
        bad = sweep_strip<P, 2, true>(g, c, k, &mf, &mu, B, smem + wid * (S::DEPTH * S::SLOT), bars + wid * S::DEPTH,
                                      base, xs, j0, j1, timeout, 0);
    } else {
        bad = pair_strip<P, true>(g, c, k, A, B, xs, j0, j1);
    }
    if (timeout) atomicOr(flag, kFlagTimeout);
    if (__any_sync(0xffffffffu, bad) && (threadIdx.x & 31) == 0) atomicOr(flag, kFlagNonfinite);
}

// Stage 1 of a pair of steps of every lattice of a batch (launch_pair_batch):
// the two-step strips as sweeps of K = 2 fed by TMA, the frame strips and
// Newmark tasks as in pair_batch_kernel.  The tensor maps of each lattice's
// two copies lie in device memory.
template <typename P>
__global__ void __launch_bounds__(128, 4) sweep_batch_kernel(const DomDesc<P>* __restrict__ dd,
                                                             const SweepMaps* __restrict__ maps,
                                                             const PairTask* __restrict__ tasks, int ntasks,
                                                             const BndTask* __restrict__ btasks, int parity,
                                                             unsigned* next) {
    using S = Sweep<P, 2>;
    extern __shared__ __align__(128) char smem[];
    __shared__ unsigned long long bars[kWarpsPerBlock * S::DEPTH];
    __shared__ DomDesc<P> sd[kWarpsPerBlock];
    const unsigned FULL = 0xffffffffu;
    const int wid = threadIdx.x >> 5, lane = threadIdx.x & 31;
    init_ring<S>(bars + wid * S::DEPTH);
    unsigned base = 0;
    int cached = -1, mapped = -1;   // the lattice of the descriptor, of the maps acquired last
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
        bool bad, timeout = false;
        if (tk.kind == kPairStrip) {
            const CUtensorMap* m = reinterpret_cast<const CUtensorMap*>(maps + tk.dom) + 2 * a;
            if (tk.dom != mapped) {
                if (lane == 0) {   // the lane that issues the copies
                    acquire_map(m);
                    acquire_map(m + 1);
                }
                mapped = tk.dom;
            }
            bad = sweep_strip<P, 2>(d.g, d.c, d.k, m, m + 1, d.v[a ^ 1], smem + wid * (S::DEPTH * S::SLOT),
                                    bars + wid * S::DEPTH, base, tk.xs, tk.j0, tk.j1, timeout);
        } else if (tk.kind == kSideStrip) {
            bad = side_strip<P, 8>(d.g, d.c, d.k, d.v[a], d.x, tk.xs, tk.x0, tk.x1, tk.j0, tk.j1, kSideRows);
        } else {
            bad = bulk_strip<P, 1, true>(d.g, d.c, d.k, d.v[a], d.x, tk.xs, tk.j0, tk.j1,
                                         Win{tk.x0, tk.x1, tk.y0, tk.y1});
        }
        if (timeout) {
            atomicOr(d.flag, kFlagTimeout);
            break;
        }
        if (__any_sync(FULL, bad) && lane == 0) atomicOr(d.flag, kFlagNonfinite);
    }
}

using EncodeFn = CUresult (*)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                              const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                              CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

// cuTensorMapEncodeTiled of the driver, null where it has none.
EncodeFn encode_fn() {
#ifdef LBPS_NO_TENSOR_MAPS
    return nullptr;
#else
    void* fn = nullptr;
    cudaDriverEntryPointQueryResult found;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &fn, 12000, cudaEnableDefault, &found) !=
        cudaSuccess) {
        cudaGetLastError();
        return nullptr;
    }
    return found == cudaDriverEntryPointSuccess ? reinterpret_cast<EncodeFn>(fn) : nullptr;
#endif
}

cudaError_t encode(CUtensorMap* m, CUtensorMapDataType type, int elem, void* base, const Geo& g, int planes, int box_x) {
    const EncodeFn fn = encode_fn();
    if (!fn) return cudaErrorNotSupported;
#ifdef LBPS_CHECKED
    // the copies read only inside the map (and zeros beyond it), the map only inside a live block
    if (!check_live(base, (size_t)planes * g.plane * elem)) return cudaErrorInvalidValue;
#endif
    const cuuint64_t dims[3] = {(cuuint64_t)g.px, (cuuint64_t)g.ny, (cuuint64_t)planes};
    const cuuint64_t strides[2] = {(cuuint64_t)g.px * elem, (cuuint64_t)g.plane * elem};
    const cuuint32_t box[3] = {(cuuint32_t)box_x, 2, (cuuint32_t)planes}, one[3] = {1, 1, 1};
    const CUresult r = fn(m, type, 3, base, dims, strides, box, one, CU_TENSOR_MAP_INTERLEAVE_NONE,
                          CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                          CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS ? cudaSuccess : cudaErrorInvalidValue;
}

// Rows per chunk.  Tall chunks recompute fewer rows around them; short ones
// end more often, so that the boundary launches beside the sweep find room
// on the SMs, and fill the last wave.  Measured, us a step: K = 4 FP32 8192^2
// 601 / 578 / 576 / 578 with 32 / 64 / 96 / 128 rows: any height from 64 on, so 96,
// which fills the last wave of 2047 x 1533 (41.8 / 43.0 / 35.6 / 46.1) but not of
// every size (2048^2 58 us, 1.2 times the time a point); K = 2 FP16 2047 x 1533
// 48.1 / 49.2 / 71.1 with 16 / 32 / 64 rows, 4096^2 204 / 201 / -, BFP13 4096^2
// 206 / 201 / 211.
// Below 6 M points a K = 2 launch is a few waves of blocks: the height of 16 .. 32
// rows whose waves cost least, a chunk costing its rows and 8 around them
// (1024^2 BF16: 16 rows are 640 blocks on 608 places). free: places left to the
// boundary launches beside the sweep, in tenths.
int sweep2_rows(const Geo& g, int blocks_x, int height, int per_sm, int free) {
    if ((long long)g.nx * g.ny >= (6ll << 20)) return 32;
    int dev = 0, sms = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) {
        cudaGetLastError();
        return 16;
    }
    const long long places = std::max(1, sms * per_sm * (10 - free) / 10);
    int rows = 16;
    long long best = 0;
    for (int r = 16; r <= 32; r += 2) {
        const long long blocks = (long long)blocks_x * ((height + r - 1) / r);
        const long long cost = (blocks + places - 1) / places * (r + 8);
        if (best == 0 || cost < best) {
            best = cost;
            rows = r;
        }
    }
    return rows;
}

}  // namespace

bool tensor_maps() { return encode_fn() != nullptr; }

template <typename P, int K, bool EXACT>
cudaError_t launch_sweep(const Geo& g, const Consts& c, const KCof<P>& k, View<P> A, View<P> B, unsigned* flag,
                         cudaStream_t st) {
    using S = Sweep<P, K>;
    CUtensorMap mf, mu;
    cudaError_t e = encode(&mf, CU_TENSOR_MAP_DATA_TYPE_UINT32, 4, A.f, g, S::PLANES, S::BOX);
    if (e == cudaSuccess) e = encode(&mu, CU_TENSOR_MAP_DATA_TYPE_UINT64, 8, A.u, g, 4, S::OUT);
    if (e != cudaSuccess) return e;
    auto kern = sweep_kernel<P, K, S::MINB, EXACT>;
    e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)S::kSmem);
    if (e != cudaSuccess) return e;
    const int strips = (g.nx - S::DEEP + S::OUT - 1) / S::OUT;
    const int height = g.ny - 2 * S::DEEP, blocks_x = (strips + kWarpsPerBlock - 1) / kWarpsPerBlock;
    const int rows = K == 4 ? 96 : sweep2_rows(g, blocks_x, height, S::MINB, 1);
    const dim3 grid(blocks_x, (height + rows - 1) / rows);
    kern<<<grid, 32 * kWarpsPerBlock, S::kSmem, st>>>(g, c, k, mf, mu, B, flag, rows);
    return cudaGetLastError();
}

template <typename P>
cudaError_t launch_sweep_periodic(const Geo& g, const Consts& c, const KCof<P>& k, View<P> A, View<P> B, unsigned* flag,
                                  cudaStream_t st) {
    using S = Sweep<P, 2>;
    CUtensorMap mf, mu;
    cudaError_t e = encode(&mf, CU_TENSOR_MAP_DATA_TYPE_UINT32, 4, A.f, g, S::PLANES, S::BOX);
    if (e == cudaSuccess) e = encode(&mu, CU_TENSOR_MAP_DATA_TYPE_UINT64, 8, A.u, g, 4, S::OUT);
    if (e != cudaSuccess) return e;
    auto kern = sweep_periodic_kernel<P, 4>;
    e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)S::kSmem);
    if (e != cudaSuccess) return e;
    const int strips = (g.nx + S::OUT - 1) / S::OUT, blocks_x = (strips + kWarpsPerBlock - 1) / kWarpsPerBlock;
    const int rows = sweep2_rows(g, blocks_x, g.ny, 4, 0);
    const dim3 grid(blocks_x, (g.ny + rows - 1) / rows);
    kern<<<grid, 32 * kWarpsPerBlock, S::kSmem, st>>>(g, c, k, mf, mu, A, B, flag, rows);
    return cudaGetLastError();
}

static_assert(sizeof(SweepMaps) == 4 * sizeof(CUtensorMap), "four tensor maps");

template <typename P>
cudaError_t make_sweep_maps(const Geo& g, View<P> v0, View<P> v1, SweepMaps* out) {
    using S = Sweep<P, 2>;
    CUtensorMap m[4];
    const View<P> v[2] = {v0, v1};
    cudaError_t e = cudaSuccess;
    for (int q = 0; q < 2 && e == cudaSuccess; ++q) {
        e = encode(&m[2 * q], CU_TENSOR_MAP_DATA_TYPE_UINT32, 4, v[q].f, g, S::PLANES, S::BOX);
        if (e == cudaSuccess) e = encode(&m[2 * q + 1], CU_TENSOR_MAP_DATA_TYPE_UINT64, 8, v[q].u, g, 4, S::OUT);
    }
    if (e == cudaSuccess) memcpy(out, m, sizeof(m));
    return e;
}

template <typename P>
cudaError_t launch_sweep_batch(const DomDesc<P>* dd, const SweepMaps* maps, const PairTask* tasks, int ntasks,
                               const BndTask* btasks, int parity, unsigned* next, cudaStream_t st) {
    using S = Sweep<P, 2>;
    if (ntasks <= 0) return cudaSuccess;
    auto kern = sweep_batch_kernel<P>;
    int dev = 0, sms = 0, per_sm = 0;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)S::kSmem);
    if (e == cudaSuccess) e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e == cudaSuccess)
        e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, 32 * kWarpsPerBlock, S::kSmem);
    if (e != cudaSuccess) return e;
    const int blocks = min(sms * max(per_sm, 1), (ntasks + kWarpsPerBlock - 1) / kWarpsPerBlock);
    kern<<<blocks, 32 * kWarpsPerBlock, S::kSmem, st>>>(dd, maps, tasks, ntasks, btasks, parity, next);
    return cudaGetLastError();
}

#ifdef LBPS_CHECKED
cudaError_t sweep_check_table(const char* const* los, const char* const* his, int n) {
    return upload_check_table(los, his, n);
}
int sweep_check_report(unsigned long long out[2]) { return read_check_report(out); }
#endif

#define LBPS_INSTANTIATE(P)                                                                                       \
    template cudaError_t launch_sweep<P, 2, false>(const Geo&, const Consts&, const KCof<P>&, View<P>, View<P>,   \
                                                   unsigned*, cudaStream_t);                                      \
    template cudaError_t launch_sweep<P, 2, true>(const Geo&, const Consts&, const KCof<P>&, View<P>, View<P>,    \
                                                  unsigned*, cudaStream_t);                                       \
    template cudaError_t launch_sweep_periodic<P>(const Geo&, const Consts&, const KCof<P>&, View<P>, View<P>,    \
                                                  unsigned*, cudaStream_t);                                       \
    template cudaError_t make_sweep_maps<P>(const Geo&, View<P>, View<P>, SweepMaps*);                            \
    template cudaError_t launch_sweep_batch<P>(const DomDesc<P>*, const SweepMaps*, const PairTask*, int,         \
                                               const BndTask*, int, unsigned*, cudaStream_t);

LBPS_INSTANTIATE(PopDirect<float>)
LBPS_INSTANTIATE(PopNeq16<__nv_bfloat16>)
LBPS_INSTANTIATE(PopNeq16<__half>)
LBPS_INSTANTIATE(PopBfp13)
template cudaError_t launch_sweep<PopDirect<float>, 4, false>(const Geo&, const Consts&, const KC<float>&,
                                                              View<PopDirect<float>>, View<PopDirect<float>>,
                                                              unsigned*, cudaStream_t);

}  // namespace lbps
