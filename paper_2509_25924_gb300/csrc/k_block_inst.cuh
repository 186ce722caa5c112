// The iteration kernels and their host launchers, for window radii 1..10.
// Each k_block_*.cu translation unit instantiates some kinds for one level
// storage type, so the instantiations compile in parallel.
#pragma once
#include "k_block.cuh"
#include "k_walk.cuh"

namespace ofv {

// Launch shape of one kind of iteration kernel.
template <typename T, int KS, int KIND> struct IterShape {
    using WS = WalkShape<ks_radius(KS), ks_shape(KS)>;
    static constexpr int TX = WS::TX, TY = WS::TY, NT = WS::NT, MINB = WS::MINB;
    static constexpr size_t smem = walk_smem_bytes<T, WS>();
};
template <typename T, int KS> struct IterShape<T, KS, ITER_VAR> {
    using BS = BlockShape<KS>;
    static constexpr int TX = BS::TS, TY = BS::TS, NT = BS::NT, MINB = BS::MINB;
    static constexpr size_t smem = block_smem_bytes<T, KS>();
};

// One tile per CTA; blockIdx.z selects the pair.
//
// ITER_BOX, 8 pairs of 1 Mp, level 0, FP32, KR 4, V0 from the previous
// iteration (ncu): 17.1 M shared-memory wavefronts, 60.5 M warp instructions
// (231 thread instructions per output), LSU data pipe 63 % of peak over the
// launch and issue 49 %, 105 us; the one-pixel-per-thread form before it:
// 23.2 M wavefronts, 99.6 M instructions, 121 us.  Shared-memory wavefronts
// bound it: 24 taps and 5 stores a pixel of the halo tile became 11 + 5, and
// the window sums 13 + 11 words per output instead of 35.  64 fields of a
// 1 Mp stream 4025 -> 3300 us, one 21 Mp pair 1236 -> 1024 us, KR 10 with
// NR 2 (24 fields of 1 Mp) 2184 -> 2006 us.
template <typename T, int KS, int KIND>
__global__ void __launch_bounds__(IterShape<T, KS, KIND>::NT, IterShape<T, KS, KIND>::MINB)
    k_iter_block(const __grid_constant__ BlockParams prm)
{
    extern __shared__ __align__(128) float4 smem_f4[];
    __shared__ __align__(8) uint64_t s_bar[4];
    const int z = blockIdx.z;
    const CUtensorMap *tm1 = prm.use_tma ? &prm.tm[z][0] : nullptr, *tm2 = prm.use_tma ? &prm.tm[z][1] : nullptr;
    if constexpr (KIND == ITER_VAR) {
        block_tile<T, KS, LD_READ_ONLY>(prm.a[z], prm.mode, blockIdx.x,
                                        prm.row0 / IterShape<T, KS, KIND>::TY + blockIdx.y, smem_f4, tm1, tm2, prm.err,
                                        s_bar);
    } else {
        walk_tile<T, typename IterShape<T, KS, KIND>::WS, KIND == ITER_BOX ? LD_READ_ONLY : LD_AFTER_WAIT,
                  KIND == ITER_KEEP, KIND != ITER_BOX>(
            prm.a[z], prm.mode, blockIdx.x, blockIdx.y, prm.row0, prm.row1, smem_f4, tm1, tm2, prm.err, s_bar,
            prm.overlap == 2);
    }
}

__device__ __forceinline__ int ld_acquire(const int *p)
{
    int v;
    asm volatile("ld.acquire.gpu.global.s32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}

// What a work unit's tile needs, in shared memory (held in registers the
// arguments made the walk spill).
struct UnitArgs {
    IterArgs a;
    int mode, bx, by;
    int key;                // stage * npairs + pair
    const int *cnt;         // the unit's dependency counter, or null
    int need;               //   and the count that completes it
    const CUtensorMap *tm;  // tensor maps of the two level images, or null
};

template <bool VAR, int TX>
__device__ __forceinline__ void fill_unit(const QueueParams &q, int unit, UnitArgs &o)
{
    const int4 d = __ldg(q.unit_desc + unit);
    const int s = d.x, p = d.y, tile = d.z;
    const BatchPair &bp = q.pairs[p];
    const int l = q.L - 1 - s / q.IT, t = s % q.IT;
    IterArgs &a = o.a;
    o.key = s * q.npairs + p;
    o.cnt = s > 0 ? q.done + (s - 1) * q.npairs + p : nullptr;
    o.need = d.w;
    a.P1 = bp.P1[l];
    a.P2 = bp.P2[l];
    a.H = bp.H[l];
    a.W = bp.W[l];
    a.pitch = bp.pitch[l];
    a.vpitch = bp.vpitch;
    a.vcpitch = bp.vpitch;
    a.kr = q.kr;
    a.eps_rel = q.eps_rel;
    a.eps_abs = q.eps_abs;
    a.mask = nullptr;
    a.inc = a.gauss = 0;
    if (VAR) {
        a.inc = q.inc;
        a.gauss = q.gauss;
        for (int k = 0; k <= kBlockMaxKR; ++k) a.wg[k] = q.wg[k];
    }
    o.mode = s == 0 ? V0_ZERO : t == 0 ? V0_UP : V0_SAME;
    a.V0 = a.Vc = s > 0 ? bp.vb[(s - 1) & 1] : nullptr;
    if (o.mode == V0_UP) {
        a.Hc = bp.H[l + 1];
        a.Wc = bp.W[l + 1];
    }
    const bool last = s == q.L * q.IT - 1;
    a.u_out = last ? bp.u : nullptr;
    a.v_out = last ? bp.v : nullptr;
    a.Vout = last ? nullptr : bp.vb[s & 1];
    const int ntx = (a.W + TX - 1) / TX;
    o.by = tile / ntx;
    o.bx = tile - o.by * ntx;
    o.tm = q.tmaps ? q.tmaps + ((size_t)p * 16 + l) * 2 : nullptr;
}

// One work unit per CTA, claimed in schedule order when the CTA starts.
template <typename T, int KS, int KIND>
__global__ void __launch_bounds__(IterShape<T, KS, KIND>::NT, IterShape<T, KS, KIND>::MINB)
    k_iter_queue(const __grid_constant__ QueueParams q)
{
    constexpr bool VAR = KIND == ITER_VAR;
    constexpr int TX = IterShape<T, KS, KIND>::TX;
    extern __shared__ __align__(128) float4 smem_f4[];
    __shared__ UnitArgs o;
    __shared__ int s_fail;
    __shared__ __align__(8) uint64_t s_bar[4];
    if (threadIdx.x == 0) {
        const int unit = atomicAdd(q.head, 1);
        int fail = unit >= q.total_units;  // never, with a grid of total_units CTAs
        if (!fail) {
            fill_unit<VAR, TX>(q, unit, o);
            if (o.cnt && ld_acquire(o.cnt) < o.need) {
                const long long t0 = global_ns();
                int spins = 0;
                while (ld_acquire(o.cnt) < o.need) {
                    if (++spins > q.spin_limit || global_ns() - t0 > q.timeout_ns) {
                        atomicCAS(q.error, 0, 1 + unit);
                        if (q.host_err) *reinterpret_cast<volatile int *>(q.host_err) = 1 + unit;
                        fail = 1;
                        break;
                    }
                    __nanosleep(128);
                }
            }
        }
        s_fail = fail;
    }
    __syncthreads();
    if (s_fail) return;
    const CUtensorMap *tm1 = o.tm, *tm2 = o.tm ? o.tm + 1 : nullptr;
    if constexpr (VAR) {
        block_tile<T, KS, LD_SAME_LAUNCH>(o.a, o.mode, o.bx, o.by, smem_f4, tm1, tm2, q.tma_err, s_bar);
    } else {
        walk_tile<T, typename IterShape<T, KS, KIND>::WS, LD_SAME_LAUNCH, false, false>(
            o.a, o.mode, o.bx, o.by, 0, o.a.H, smem_f4, tm1, tm2, q.tma_err, s_bar, false);
    }
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) atomicAdd(q.done + o.key, 1);
}

template <typename T, int KS, int KIND>
cudaError_t run_block(const BlockParams &p, dim3 grid, int dev, cudaStream_t s)
{
    static size_t granted[64] = {};  // dynamic shared memory raised per device
    constexpr size_t smem = IterShape<T, KS, KIND>::smem;
    auto kern = k_iter_block<T, KS, KIND>;
    if (dev < 0 || dev >= 64 || granted[dev] < smem) {
        cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
        if (dev >= 0 && dev < 64) granted[dev] = smem;
    }
    return launch_after(KIND == ITER_CHAIN || KIND == ITER_KEEP, kern, grid, dim3(IterShape<T, KS, KIND>::NT), smem, s, p);
}

// KS = kr + 16 shape for the radii and shapes instantiated here: every
// radius with its default shape; the alternative shapes without the
// estimator variants (keeping the window sums, of radii 3 and 4, whose small
// levels take them).  Box windows of radii 1 and 2, whose two shapes are one
// tile, run the default for both.  0 when not instantiated.
template <int KIND>
constexpr bool has_alt(int kr)
{
    return walk_has_alt(kr) &&
           (KIND == ITER_BOX || KIND == ITER_CHAIN || (KIND == ITER_KEEP && (kr == 3 || kr == 4)));
}
template <int KIND>
constexpr int ks_of(int kr, int shape)
{
    if (kr < 1 || kr > kBlockMaxKR || shape < 0 || shape > 1) return 0;
    if (KIND != ITER_VAR && !walk_has_alt(kr)) shape = 0;
    return shape != 0 && !has_alt<KIND>(kr) ? 0 : kr + 16 * shape;
}

#define OFV_KS_CASES(X)                                                                                    \
    X(1) X(2) X(3) X(4) X(5) X(6) X(7) X(8) X(9) X(10)                                                      \
    OFV_KS_ALT(X, 17) OFV_KS_ALT(X, 18) OFV_KS_ALT(X, 19) OFV_KS_ALT(X, 20) OFV_KS_ALT(X, 21)                \
    OFV_KS_ALT(X, 22) OFV_KS_ALT(X, 23) OFV_KS_ALT(X, 24) OFV_KS_ALT(X, 25) OFV_KS_ALT(X, 26)

template <typename T, int KIND>
cudaError_t launch_block_t(const BlockParams &p, int kr, int npairs, cudaStream_t s, int shape)
{
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    const IterArgs &a = p.a[0];
    switch (ks_of<KIND>(kr, shape)) {
#define OFV_KS_ALT(X, K) \
    case K:              \
        if constexpr (has_alt<KIND>((K) - 16)) { X##_BODY(K) } else { break; }
#define OFV_BLOCK_CASE(K) case K: OFV_BLOCK_CASE_BODY(K)
#define OFV_BLOCK_CASE_BODY(K)                                                                             \
    {                                                                                                      \
        using IS = IterShape<T, K, KIND>;                                                                  \
        const dim3 grid((a.W + IS::TX - 1) / IS::TX, (p.row1 - p.row0 + IS::TY - 1) / IS::TY, npairs);     \
        return run_block<T, K, KIND>(p, grid, dev, s);                                                     \
    }
    OFV_KS_CASES(OFV_BLOCK_CASE)
#undef OFV_BLOCK_CASE
#undef OFV_BLOCK_CASE_BODY
#undef OFV_KS_ALT
    default: break;
    }
    return cudaErrorInvalidValue;
}

template <typename T, int KS, int KIND>
cudaError_t run_queue(const QueueParams &q, int dev, cudaStream_t s)
{
    static size_t granted[64] = {};
    constexpr size_t smem = IterShape<T, KS, KIND>::smem;
    auto kern = k_iter_queue<T, KS, KIND>;
    if (dev < 0 || dev >= 64 || granted[dev] < smem) {
        cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
        if (dev >= 0 && dev < 64) granted[dev] = smem;
    }
    kern<<<q.total_units, IterShape<T, KS, KIND>::NT, smem, s>>>(q);
    return cudaGetLastError();
}

template <typename T, int KS, int KIND>
int queue_occupancy_kr()
{
    constexpr size_t smem = IterShape<T, KS, KIND>::smem;
    cudaFuncSetAttribute(k_iter_queue<T, KS, KIND>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    int n = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k_iter_queue<T, KS, KIND>, IterShape<T, KS, KIND>::NT, smem) !=
        cudaSuccess)
        return 0;
    return n;
}

// The variants' batched kernel has its own thread count: KS | 32 (see
// BlockShape).
#define QKS(K) (KIND == ITER_VAR ? ((K) | 32) : (K))

// Batched launch: one CTA per work unit.
template <typename T, int KIND>
cudaError_t launch_queue_t(const QueueParams &q, int kr, cudaStream_t s, int shape)
{
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    switch (ks_of<KIND>(kr, shape)) {
#define OFV_KS_ALT(X, K) \
    case K:              \
        if constexpr (has_alt<KIND>((K) - 16)) { X##_BODY(K) } else { break; }
#define OFV_QUEUE_CASE(K) case K: OFV_QUEUE_CASE_BODY(K)
#define OFV_QUEUE_CASE_BODY(K) return run_queue<T, QKS(K), KIND>(q, dev, s);
    OFV_KS_CASES(OFV_QUEUE_CASE)
#undef OFV_QUEUE_CASE
#undef OFV_QUEUE_CASE_BODY
#undef OFV_KS_ALT
    default: break;
    }
    return cudaErrorInvalidValue;
}

// Resident CTAs per SM of the batched launch.
template <typename T, int KIND>
int queue_occupancy_t(int kr, int shape)
{
    switch (ks_of<KIND>(kr, shape)) {
#define OFV_KS_ALT(X, K) \
    case K:              \
        if constexpr (has_alt<KIND>((K) - 16)) { X##_BODY(K) } else { break; }
#define OFV_OCC_CASE(K) case K: OFV_OCC_CASE_BODY(K)
#define OFV_OCC_CASE_BODY(K) return queue_occupancy_kr<T, QKS(K), KIND>();
    OFV_KS_CASES(OFV_OCC_CASE)
#undef OFV_OCC_CASE
#undef OFV_OCC_CASE_BODY
#undef OFV_KS_ALT
    default: break;
    }
    return 0;
}

#define OFV_INSTANTIATE_BLOCK(T, KIND) \
    template cudaError_t launch_block_t<T, KIND>(const BlockParams &, int, int, cudaStream_t, int);
#define OFV_INSTANTIATE_QUEUE(T, KIND)                                                             \
    template cudaError_t launch_queue_t<T, KIND>(const QueueParams &, int, cudaStream_t, int); \
    template int queue_occupancy_t<T, KIND>(int, int);

}  // namespace ofv
