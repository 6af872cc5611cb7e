// Many time steps of one lattice in one cooperative launch.
//
// What bounds a small lattice's step is latency: the interior kernel and the
// boundary reset of a step depend on each other, and as separate launches each
// costs its start and its drain besides its chain of loads.  Here the grid
// stays on the SMs and meets at a barrier instead (about 2300 cycles, up to
// 5000 where every thread has stores on the way).  Every block keeps its tasks
// and its boundary table for all steps, and one warp takes one strip of a few
// rows, so that a phase is one wave.  Against graphs of 32 steps (three
// launches a step): 64^2 FP64 storage 10.6 us a step against 15.7, 300^2 FP32
// 8.9 against 10.3, 389 x 1171 15.6 against 20.0, 1024^2 with a hole 39.4
// against 45.7; a single step through lbps_step on 128 x 96 19.8 us against
// 32.1.
#include <algorithm>

#include "lbps_steps.cuh"

namespace lbps {

namespace {

// Polls of a barrier before it gives up (about a second or more); the wait
// then ends with kFlagTimeout set instead of hanging the GPU.
constexpr int kMaxPolls = 1 << 21;

// Boundary tasks (32 points each) whose table entries a block keeps in shared
// memory.
constexpr int kTableTasks = 8;

__device__ __forceinline__ unsigned poll_acquire(const unsigned* p) {
    unsigned v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}

__device__ __forceinline__ void add_release(unsigned* p, unsigned x) {
    asm volatile("red.release.gpu.global.add.u32 [%0], %1;" ::"l"(p), "r"(x) : "memory");
}

// Barrier over the grid (every block resident: a cooperative launch).  Block 0
// adds 2^31 - (blocks - 1) and every other block 1, so the top bit flips when
// the last block arrives and the low bits are as before.  phase: the top bit
// before the barrier, flipped here.  Returns false in every thread of a block
// whose wait ran out.
__device__ __forceinline__ bool grid_barrier(unsigned* bar, unsigned& phase, unsigned* flag, unsigned* host,
                                             int* alive) {
    __syncthreads();
    if (threadIdx.x == 0) {
        add_release(bar, blockIdx.x == 0 ? 0x80000000u - (gridDim.x - 1u) : 1u);
        int polls = 0;
        while (((poll_acquire(bar) ^ phase) & 0x80000000u) == 0u && ++polls < kMaxPolls) {}
        if (polls >= kMaxPolls) {
            atomicOr(flag, kFlagTimeout);
            if (host) *(volatile unsigned*)(host + 1) = 1u;
            *alive = 0;
        }
    }
    phase ^= 0x80000000u;
    __syncthreads();
    return *alive != 0;
}

// GEN: general geometry (a template so that the code of rectangles does not
// carry it).
template <typename P, int THREADS, int UVD, bool GEN>
__global__ void __launch_bounds__(THREADS, 1) fused_kernel(Geo g, Consts c, KCof<P> k, View<P> A0, View<P> B0,
                                                           const BNode* __restrict__ bn, int nb, unsigned* flag,
                                                           unsigned long long* tstep, unsigned* bar,
                                                           unsigned* host, int steps, int rows) {
    __shared__ int alive;
    const int wid = threadIdx.x >> 5, lane = threadIdx.x & 31, warps = blockDim.x >> 5;
    const int G = gridDim.x, cta = blockIdx.x;
    const int strips = (g.nx + kStripCols - 1) / kStripCols, chunks = (g.ny + rows - 1) / rows;
    const int nst = strips * chunks;                       // strip tasks
    const int nbt = (nb + 31) / 32;                        // boundary tasks
    // this block's tasks: consecutive ones, down a strip, so that the warps of
    // a block share their halo rows in its L1
    const int s0 = (int)((long long)nst * cta / G), s1 = (int)((long long)nst * (cta + 1) / G);
    const int b0 = (int)((long long)nbt * cta / G), b1 = (int)((long long)nbt * (cta + 1) / G);
    const int nbp = 2 * (b1 - b0);                         // two parts of each boundary task
#ifdef LBPS_CHECKED
    const BNode* table = bn;
#else
    // the boundary table entries of this block, constant over the steps
    __shared__ BNode sbn[kTableTasks * 32];
    const BNode* table = bn;
    if (b1 - b0 <= kTableTasks) {
        const int words = (min(32 * b1, nb) - 32 * b0) * (int)(sizeof(BNode) / 4);
        const unsigned* src = reinterpret_cast<const unsigned*>(bn + 32 * b0);
        for (int q = threadIdx.x; q < words; q += blockDim.x) reinterpret_cast<unsigned*>(sbn)[q] = src[q];
        table = sbn - 32 * b0;
    }
#endif
    // after a launch that timed out the barrier word holds arrivals of blocks
    // that are gone: nothing runs until the next state clears it
    if (threadIdx.x == 0) alive = (LBPS_LD(flag) & kFlagTimeout) == 0u;
    const unsigned long long n0 = LBPS_LD(tstep);
    unsigned phase = poll_acquire(bar);   // before this block's first arrival, so the top bit is the old one
    __syncthreads();
    if (!alive) return;
    bool bad = false;
    for (int s = 0; s < steps; ++s) {
        const View<P> A = (s & 1) ? B0 : A0, B = (s & 1) ? A0 : B0;
        for (int t = wid; t < nbp + (s1 - s0); t += warps) {
            if (t < nbp) {
                const int b = 32 * (b0 + (t >> 1)) + lane;
                if (b < nb) boundary_newmark(g, c, A, B, table, nb, A.s, (double)(n0 + (unsigned)s), b, t & 1);
            } else {
                const int q = s0 + t - nbp, strip = q / chunks;
                const int j0 = (q - strip * chunks) * rows, j1 = min(j0 + rows, g.ny);
                // rows of a hole: nothing to write, nothing an interior point reads
                if (GEN && g.gap && j0 >= LBPS_LD(&g.gap[2 * strip]) && j1 <= LBPS_LD(&g.gap[2 * strip + 1])) continue;
                bad |= bulk_strip<P, UVD, false, false, GEN>(g, c, k, A, B, strip * kStripCols, j0, j1);
            }
        }
        if (nb > 0) {
            if (!grid_barrier(bar, phase, flag, host, &alive)) return;
            for (int t = wid; t < nbp; t += warps) {
                const int b = 32 * (b0 + (t >> 1)) + lane;
                if (b >= nb) continue;
                if (t & 1)
                    neighbour_stresses(g, c, B.u, B.u + g.plane, table, nb, B.s, b);
                else
                    bad |= boundary_reset<P>(g, c, k, A, B, table, nb, b);
            }
            if (P::kSplitStream) {
                if (!grid_barrier(bar, phase, flag, host, &alive)) return;
                for (int t = b0 + wid; t < b1; t += warps) {
                    const int b = 32 * t + lane;
                    if (b < nb) boundary_stream_y(g, c, k, A, B, table, b);
                }
            }
        }
        if (s + 1 < steps && !grid_barrier(bar, phase, flag, host, &alive)) return;
    }
    if (bad) {
        atomicOr(flag, kFlagNonfinite);
        if (host) *(volatile unsigned*)host = 1u;
    }
    // every block has read the counter before its first barrier
    if (nb > 0 && cta == 0 && threadIdx.x == 0) LBPS_ST(tstep, n0 + (unsigned)steps);
}

}  // namespace

template <typename P>
cudaError_t launch_fused(const Geo& g, const Consts& c, const KCof<P>& k, View<P> A, View<P> B, const BNode* bn,
                         int nb, unsigned* flag, unsigned long long* tstep, unsigned* bar, unsigned* host, int steps,
                         cudaStream_t st) {
    // FP64 storage needs 128 registers a thread.  The others: 16 warps per SM
    // up to 2^19 points, where the phases are short (389 x 1171: 15.7 us a step
    // against 16.3 with 20), 20 above, where more rows in flight pay (1024^2
    // BF16: 33.7 against 39.6).
    constexpr bool wide = sizeof(typename P::V) == 8;
    const int threads_max = wide || (long long)g.nx * g.ny <= (1ll << 19) ? 512 : 640;
    int dev = 0, sms = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return e;
    const int strips = (g.nx + kStripCols - 1) / kStripCols, nbt = (nb + 31) / 32;
    // the lowest strips whose tasks, with the boundary tasks, are one per
    // warp of the grid (at most 16 rows; then the warps take several)
    const int warps_max = threads_max / 32;
    auto per_block = [&](int rows) {
        const long long nst = (long long)strips * ((g.ny + rows - 1) / rows);
        return (nst + sms - 1) / sms + 2 * ((nbt + sms - 1) / sms);
    };
    int rows = 1;
    while (rows < 16 && per_block(rows) > warps_max) ++rows;
    const long long nst = (long long)strips * ((g.ny + rows - 1) / rows);
    int blocks = (int)std::min<long long>(sms, std::max<long long>(nst, 2 * nbt));
    const int warps = (int)std::min<long long>(
        warps_max, (nst + blocks - 1) / blocks + 2 * ((nbt + blocks - 1) / blocks));
    const void* kern = reinterpret_cast<const void*>(g.general ? fused_kernel<P, 512, 1, true>
                                                               : fused_kernel<P, 512, 1, false>);
    if constexpr (!wide)
        if (threads_max == 640)
            kern = reinterpret_cast<const void*>(g.general ? fused_kernel<P, 640, 1, true>
                                                           : fused_kernel<P, 640, 1, false>);
    Geo ga = g;
    Consts ca = c;
    KCof<P> ka = k;
    void* args[] = {&ga, &ca, &ka, &A, &B, &bn, &nb, &flag, &tstep, &bar, &host, &steps, &rows};
    return cudaLaunchCooperativeKernel(kern, dim3(blocks), dim3(32 * warps), args, 0, st);
}

#ifdef LBPS_CHECKED
cudaError_t fused_check_table(const char* const* los, const char* const* his, int n) {
    return upload_check_table(los, his, n);
}
int fused_check_report(unsigned long long out[2]) { return read_check_report(out); }
#endif

#define LBPS_INSTANTIATE(P)                                                                                      \
    template cudaError_t launch_fused<P>(const Geo&, const Consts&, const KCof<P>&, View<P>, View<P>, const BNode*, \
                                         int, unsigned*, unsigned long long*, unsigned*, unsigned*, int, cudaStream_t);

LBPS_INSTANTIATE(PopDirect<float>)
LBPS_INSTANTIATE(PopDirect<double>)
LBPS_INSTANTIATE(PopNeq16<__nv_bfloat16>)
LBPS_INSTANTIATE(PopNeq16<__half>)
LBPS_INSTANTIATE(PopBfp13)

}  // namespace lbps
