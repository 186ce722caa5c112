// Host launcher of the block-tiled iteration kernel.
#include <cstring>

#include "k_block.cuh"
#include "k_walk.cuh"

namespace ofv {

extern template cudaError_t launch_block_t<float, ITER_BOX>(const BlockParams &, int, int, cudaStream_t, int);
extern template cudaError_t launch_block_t<float, ITER_CHAIN>(const BlockParams &, int, int, cudaStream_t, int);
extern template cudaError_t launch_block_t<__half, ITER_CHAIN>(const BlockParams &, int, int, cudaStream_t, int);
extern template cudaError_t launch_block_t<__nv_bfloat16, ITER_CHAIN>(const BlockParams &, int, int, cudaStream_t, int);
extern template cudaError_t launch_block_t<float, ITER_KEEP>(const BlockParams &, int, int, cudaStream_t, int);
extern template cudaError_t launch_block_t<float, ITER_VAR>(const BlockParams &, int, int, cudaStream_t, int);
extern template cudaError_t launch_block_t<__half, ITER_BOX>(const BlockParams &, int, int, cudaStream_t, int);
extern template cudaError_t launch_block_t<__half, ITER_KEEP>(const BlockParams &, int, int, cudaStream_t, int);
extern template cudaError_t launch_block_t<__half, ITER_VAR>(const BlockParams &, int, int, cudaStream_t, int);
extern template cudaError_t launch_block_t<__nv_bfloat16, ITER_BOX>(const BlockParams &, int, int, cudaStream_t, int);
extern template cudaError_t launch_block_t<__nv_bfloat16, ITER_KEEP>(const BlockParams &, int, int, cudaStream_t, int);
extern template cudaError_t launch_block_t<__nv_bfloat16, ITER_VAR>(const BlockParams &, int, int, cudaStream_t, int);

bool block_supports(int kr) { return kr >= 1 && kr <= kBlockMaxKR; }

// The solve's reciprocal on its own, for its error test.
__global__ void k_recip(const float *x, float *y, int n)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) y[i] = recip_newton(x[i]);
}

cudaError_t launch_recip(const float *x, float *y, int n, cudaStream_t s)
{
    if (n < 0) return cudaErrorInvalidValue;
    if (n == 0) return cudaSuccess;
    k_recip<<<(n + 255) / 256, 256, 0, s>>>(x, y, n);
    return cudaGetLastError();
}

namespace {
// Whether a launch of one pair takes the smaller tiles (56 x 24, three CTAs
// per SM) of radii 3 and 4, whose tensor maps and fields are the same: below
// 2.5 waves of the default tiles on the 152 SMs (two CTAs each) the shorter
// tile leaves less of the last wave empty.  Measured, us per pair at KR 4,
// PSL 2, IT 3, default / smaller: 256 x 256 100.3 / 88.1, 1024 x 1024 (level 0
// 1.6 waves) 135.4 / 128.9; with smaller tiles everywhere a stream of 8 pairs
// per launch, whose groups overlap, takes 3412 instead of 3292 us for 64
// fields of 1 Mp.
bool walk_small_tiles(int kr, int W, int rows)
{
    if (kr < 3 || kr > 4) return false;
    const long long tiles = (long long)((W + walk_tile_w(kr, 0) - 1) / walk_tile_w(kr, 0)) *
                            ((rows + walk_tile_h(kr, 0) - 1) / walk_tile_h(kr, 0));
    return 2 * tiles < 5 * 2 * 152;
}

template <typename T>
cudaError_t launch_kind(const BlockParams &p, int kind, int kr, int npairs, cudaStream_t s, int shape)
{
    switch (kind) {
    case ITER_VAR: return launch_block_t<T, ITER_VAR>(p, kr, npairs, s, shape);
    case ITER_CHAIN: return launch_block_t<T, ITER_CHAIN>(p, kr, npairs, s, shape);
    case ITER_KEEP: return launch_block_t<T, ITER_KEEP>(p, kr, npairs, s, shape);
    default: return launch_block_t<T, ITER_BOX>(p, kr, npairs, s, shape);
    }
}
}  // namespace

cudaError_t launch_iter_block(const IterArgs *a, int npairs, int store, int mode, cudaStream_t s,
                              const CUtensorMap *const *tm, int *err, int row0, int nrows, int shape, int overlap)
{
    if (npairs < 1 || npairs > kBlockMaxBatch || !block_supports(a[0].kr)) return cudaErrorInvalidValue;
    BlockParams p;
    memset(&p, 0, sizeof p);
    for (int k = 0; k < npairs; ++k) p.a[k] = a[k];
    p.mode = mode;
    p.err = err;
    p.row0 = row0;
    p.overlap = overlap;
    p.row1 = nrows > 0 ? row0 + nrows : a[0].H;
    p.use_tma = 0;
    if (tm) {
        p.use_tma = 1;
        for (int k = 0; k < npairs; ++k) {
            if (!tm[2 * k] || !tm[2 * k + 1]) {
                p.use_tma = 0;
                break;
            }
            p.tm[k][0] = *tm[2 * k];
            p.tm[k][1] = *tm[2 * k + 1];
        }
    }
    // the kernels with variant code only when a variant is on, and those that
    // keep the window sums only for the reverse mode (uniform per launch)
    const bool var = a[0].inc || a[0].gauss || a[0].mask;
    const int kind = var ? ITER_VAR : a[0].s_out ? ITER_KEEP : overlap ? ITER_CHAIN : ITER_BOX;
    if (kind == ITER_VAR) shape = 0;  // its only shape, and that of its tensor maps' box
    if (kind == ITER_KEEP && shape != 0 && a[0].kr > 4) {
        // the default shape only, whose box tensor maps made for the other one
        // would not match; up to radius 4 the shapes share the box
        p.use_tma = 0;
        shape = 0;
    }
    if (kind != ITER_VAR && shape == 0 && npairs == 1 && walk_small_tiles(a[0].kr, a[0].W, p.row1 - row0)) shape = 1;
    switch (store) {
    case ST_F16: return launch_kind<__half>(p, kind, a[0].kr, npairs, s, shape);
    case ST_BF16: return launch_kind<__nv_bfloat16>(p, kind, a[0].kr, npairs, s, shape);
    default: return launch_kind<float>(p, kind, a[0].kr, npairs, s, shape);
    }
}

namespace {
template <typename T, int KS>
void box_ks(int *cols, int *rows, bool var)
{
    using SS = WalkStage<T, WalkShape<ks_radius(KS), ks_shape(KS)>>;
    *cols = var ? StageShape<T, KS>::SP : SS::SP;
    *rows = var ? StageShape<T, KS>::SHB : SS::SHB;
}

template <typename T>
void box_of(int kr, int shape, int *cols, int *rows, bool var)
{
    *cols = *rows = 0;
    if (kr < 1 || kr > kBlockMaxKR || shape < 0 || shape > 1) return;
    switch (kr + 16 * shape) {
#define OFV_BOX_CASE(K) \
    case K: box_ks<T, K>(cols, rows, var); return;
    OFV_BOX_CASE(1) OFV_BOX_CASE(2) OFV_BOX_CASE(3) OFV_BOX_CASE(4) OFV_BOX_CASE(5)
    OFV_BOX_CASE(6) OFV_BOX_CASE(7) OFV_BOX_CASE(8) OFV_BOX_CASE(9) OFV_BOX_CASE(10)
    OFV_BOX_CASE(17) OFV_BOX_CASE(18) OFV_BOX_CASE(19) OFV_BOX_CASE(20) OFV_BOX_CASE(21)
    OFV_BOX_CASE(22) OFV_BOX_CASE(23) OFV_BOX_CASE(24) OFV_BOX_CASE(25) OFV_BOX_CASE(26)
#undef OFV_BOX_CASE
    default: return;
    }
}
}  // namespace

void block_stage_box(int store, int kr, int *cols, int *rows, int shape, bool var)
{
    switch (store) {
    case ST_F16: box_of<__half>(kr, shape, cols, rows, var); break;
    case ST_BF16: box_of<__nv_bfloat16>(kr, shape, cols, rows, var); break;
    default: box_of<float>(kr, shape, cols, rows, var); break;
    }
}

}  // namespace ofv
