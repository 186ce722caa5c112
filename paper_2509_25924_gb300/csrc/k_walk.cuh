// Column-walk form of the fused Gauss-Newton iteration (Sec. 2 step 3,
// Eq. 2): the tile body behind OFV_PATH_FUSED for the box window.
//
// One CTA owns a TX x TY tile of output pixels and works on chip:
//   0. stage both level images over the tile, its window halo, a REACH px
//      warp margin and the gradient stencil (TMA in row bands, each
//      waited for by the warps that read it; 16-byte cp.async rows where the
//      caller has no tensor maps); a box that overhangs the image has its
//      border replicated in shared memory;
//   1. a thread walks NROW consecutive rows of one column and forms the five
//      products of each pixel;
//   2. vertical window sums of a column per thread (of two in packed FP32 where
//      the threads are too few), over the products;
//   3. horizontal window sums of eight adjacent outputs per thread for all
//      five channels, the guarded solve and the store, without another pass
//      through shared memory.
//
// Products from differences of mirrored taps.  The symmetric warp samples
// frame 2 at k + h and frame 1 at k - h, so tap s of frame 2's stencil and
// tap -s of frame 1's carry the same weight.  With E(s) = P2(k + s) -
// P1(k - s) the residual and the summed gradient are one stencil over E:
//   It = sum_s w(s) E(s),  2 Gx = sum_s w(s) (E(s + ex) - E(s - ex)) / 2,
// so 12 differences replace one of the two bilinear evaluations.
//
// Window-sum order.  Vertical sums are formed per unit of eight rows and
// horizontal sums per group of eight columns, both counted from the image's
// corner (tiles start at multiples of them), so the order of
// additions depends on the pixel's position alone and tiles of any size give
// the same field bit for bit.  Sums are additions only (a core shared by the
// outputs of a group, extended by running sums outwards), as ill-conditioned
// solves need.
#pragma once
#include <type_traits>

#include "k_block.cuh"

namespace ofv {

// Tile of window radius R: TX x TY output pixels (SHAPE 0 the default, 1 a
// smaller one).
//
// COLS: a warp walks 32 adjacent columns, and the staged images have a pitch
// of a whole number of 128-byte lines, so a tap's bank depends on its column
// alone: lanes that sample at different rows never conflict, which is what
// turbulent fields need (walk loads per 32 outputs, 1 Mp, counted on the
// analytic fields: 48 wavefronts against 80 with a pitch of 72 words and
// 8 x 4 lanes; a smooth vortex 18 either way).
// Not COLS (the default tiles of radii 5..10, whose halo would leave an
// eighth of the lanes or more idle): consecutive lanes take consecutive
// columns and go on in the next segment.
template <int R_, int SHAPE_> struct WalkShape {
    static constexpr int R = R_, SHAPE = SHAPE_;
    static constexpr bool COLS = R <= 4 || SHAPE == 1;
    static constexpr int TX = walk_tile_w(R, SHAPE), TY = walk_tile_h(R, SHAPE);
    static constexpr int RW = TX + 2 * R, RH = TY + 2 * R;   // product region
    static constexpr int NW = (RW + 31) / 32;                // COLS: warps across the region
    // Segments of a column: as many as the threads hold.  (64-px tiles of radii
    // 6 and 7 with 12 segments walked 84 rows for 76 and 78: a stream of 32
    // fields of 1 Mp at R 6 2385 instead of 2265 us, FP16 levels 2363 / 2274.)
    static constexpr int NSEG = R <= 4 ? (TY == 40 ? 6 : 4) : SHAPE == 1 ? 6 : R == 5 ? 8 : R <= 7 ? 13 : 12;
    static constexpr int NROW = (RH + NSEG - 1) / NSEG;      // rows a thread walks
    static constexpr int NT = COLS ? 32 * NW * NSEG : R == 5 ? 480 : 1024;
    // resident CTAs per SM (the launch bound keeps radii 9 and 10 of the smaller
    // shape at 80 registers: with 85 only one of the two CTAs fits, 32 fields of
    // 1 Mp at R 10 4.55 instead of 3.08 ms)
    static constexpr int MINB = R <= 4 ? (TY == 40 ? 2 : 3) : SHAPE == 0 && R > 5 ? 1 : 2;
    static constexpr bool ALL = COLS && RW % 32 == 0 && RH == NSEG * NROW;  // every thread stores NROW pixels
    // row pitch of the product planes: an odd multiple of 4, so that octets
    // of lanes on two rows, eight columns apart, read distinct banks in phase 3
    static constexpr int P = (RW + (R & 1) * 2 + 3) / 8 * 8 + 4;
    static constexpr int PLANE = RH * P;
    static constexpr int PROD = (5 * PLANE + 31) / 32 * 32;  // floats; the staged images follow 128-byte aligned
    // Vertical sums, in order units of VG rows: a thread runs down a whole
    // column (VW 1) or column pair (VW 2) in place.
    static constexpr int VG = 8, VW = 5 * RW <= NT ? 1 : 2;
    static constexpr int VITEMS = 5 * RW / VW;
    static constexpr int G = 8;                              // pixels of an output group
    static constexpr int GQ = (TX / G + 3) / 4;              // octets of lanes of a row pair
    static constexpr int GITEMS = TY / 2 * GQ * 8;
    static constexpr int SH = RH + 2 * kBlockReach + 3;      // staged rows
    static_assert(NT <= 1024 && VITEMS <= NT && NROW <= 16, "one item per thread");
    static_assert(P >= RW + (R & 1) * 2 && P % 8 == 4 && RW % 2 == 0, "column pairs and 16-byte rows");
    static_assert(TX % 8 == 0 && TY % VG == 0, "order units");

    // Column rx of the region, first row ry0 and first stored row i0 of a
    // thread's walk.  A segment that would run past the region starts early
    // enough to lie inside it; rows before i0 belong to the segment above.
    __host__ __device__ static void item(int tid, int &rx, int &ry0, int &i0)
    {
        int seg;
        bool on;
        if (COLS) {
            const int w = tid >> 5;
            seg = w / NW;
            rx = (w - seg * NW) * 32 + (tid & 31);
            on = RW % 32 == 0 || rx < RW;
        } else {
            seg = tid / RW;
            rx = tid - seg * RW;
            on = seg < NSEG;
            seg = on ? seg : NSEG - 1;
        }
        rx = on || !COLS ? rx : RW - 1;
        ry0 = RH == NSEG * NROW || seg * NROW < RH - NROW ? seg * NROW : RH - NROW;
        i0 = on ? seg * NROW - ry0 : NROW;
    }
    // First and last staged row that warp w reads (warps up to REACH px).
    __host__ __device__ static void rows_of_warp(int w, int &lo, int &hi)
    {
        int rx, i0;
        item(32 * w, rx, lo, i0);
        item(32 * w + 31, rx, hi, i0);
        hi += NROW - 1 + 2 * kBlockReach + 3;
    }
    // Row and first column of output group t (eight pixels); false: none.
    // An octet of lanes takes four groups of one row and the same four of the
    // next, which P puts on the other halves of the banks' octets.
    __host__ __device__ static bool group(int t, int &oy, int &ox)
    {
        const int l = t & 7, o = t >> 3, g = o % GQ * 4 + (l & 3);
        oy = o / GQ * 2 + (l >> 2);
        ox = G * g;
        return TX / G % 4 == 0 || g < TX / G;
    }
};

// Staged box: SHT rows (NBAND TMA bands of SHB rows) of SP elements per frame.
template <typename T, typename WS> struct WalkStage {
    static constexpr int VEC = 16 / (int)sizeof(T), LINE = 128 / (int)sizeof(T);
    static constexpr int SPN = WS::RW + 2 * kBlockReach + 3 + VEC - 1;  // columns needed, with the alignment slack
    static constexpr int SP = WS::COLS ? (SPN + LINE - 1) / LINE * LINE : (SPN + VEC - 1) / VEC * VEC;
    static constexpr int NV = SP / VEC;
    // the two shapes of radii up to 4 share the box of a band (and the
    // tensor maps): a quarter of the rows of the 40-row tile
    static constexpr int SHB = WS::R <= 4 ? (40 + 2 * WS::R + 2 * kBlockReach + 3 + 3) / 4
                                          : band_rows(WS::SH, SP * (int)sizeof(T));
    static constexpr int NBAND = WS::R <= 4 ? (WS::SH + SHB - 1) / SHB : 3;
    static constexpr int SHT = SP * sizeof(T) % 128 == 0 ? WS::SH : NBAND * SHB;  // bands start 128-byte aligned
    static constexpr int STG = (SHT * SP * (int)sizeof(T) + 127) / 128 * 128 / (int)sizeof(T);
    // first row of band b; the last band ends with the box and repeats some
    // rows of the one before
    __host__ __device__ static constexpr int band_row(int b) { return b * SHB < SHT - SHB ? b * SHB : SHT - SHB; }
};

template <typename T, typename WS>
constexpr size_t walk_smem_bytes()
{
    return sizeof(float) * WS::PROD + sizeof(T) * 2 * WalkStage<T, WS>::STG;
}

// floor(v / 2) and the fraction by one rounded-down add of 1.5 * 2^23: the
// sum's low mantissa bits are the integer.  |v / 2| < 2^22; beyond, and for
// NaN, the integer read from the bits lies outside any reach test.
constexpr float kFloorMagic = 12582912.f;  // 1.5 * 2^23 = 0x4B400000
__device__ __forceinline__ void half_floor(float v, int &i, float &f)
{
    const float t = __fmaf_rd(v, 0.5f, kFloorMagic);
    i = __float_as_int(t) - 0x4B400000;
    f = fmaf(0.5f, v, -(t - kFloorMagic));
}

// Products of a pixel whose warp leaves the staged margin (from global
// memory) or whose taps are clamped at the image border (from the staged
// tile): the general sampler.  st1, st2: staged frames with origin (sx0, sy0).
template <typename T, int SP>
__device__ __noinline__ void products_general(const T *P1, const T *P2, int H, int W, int pitch, const T *st1,
                                              const T *st2, int sx0, int sy0, int x, int y, float2 V0, float *q,
                                              int plane)
{
    const float hx = 0.5f * V0.x, hy = 0.5f * V0.y;
    Sample s1, s2;
    if (hx >= -kBlockReach && hx < kBlockReach && hy >= -kBlockReach && hy < kBlockReach) {
        s1 = sample_staged<T, SP>(st1, sx0, sy0, P1, H, W, pitch, x, y, -hx, -hy);
        s2 = sample_staged<T, SP>(st2, sx0, sy0, P2, H, W, pitch, x, y, hx, hy);
    } else {
        s1 = sample_global(P1, H, W, pitch, x, y, -hx, -hy);
        s2 = sample_global(P2, H, W, pitch, x, y, hx, hy);
    }
    const float Gx = 0.5f * (s1.gx + s2.gx), Gy = 0.5f * (s1.gy + s2.gy);
    const float r = Gx * V0.x + Gy * V0.y - (s2.val - s1.val);
    q[0] = Gx * Gx;
    q[plane] = Gx * Gy;
    q[2 * plane] = Gy * Gy;
    q[3 * plane] = Gx * r;
    q[4 * plane] = Gy * r;
}

// f(lane, bit) for every bit set in the lanes' masks, 32 at a time over the
// warp (all lanes call).  What the lanes wrote before is visible in f.
template <typename F>
__device__ __forceinline__ void warp_compact(unsigned mask, const F &f)
{
    if (!__any_sync(0xffffffffu, mask != 0)) return;
    __syncwarp();
    const int lane = threadIdx.x & 31, cnt = __popc(mask);
    int incl = cnt;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const int t = __shfl_up_sync(0xffffffffu, incl, d);
        if (lane >= d) incl += t;
    }
    const int total = __shfl_sync(0xffffffffu, incl, 31);
    for (int base = 0; base < total; base += 32) {
        const int j = base + lane;
        int own = 0;  // lanes whose inclusive count is <= j
#pragma unroll
        for (int d = 16; d > 0; d >>= 1) {
            const int t = __shfl_sync(0xffffffffu, incl, own + d - 1);
            if (t <= j) own += d;
        }
        unsigned m = __shfl_sync(0xffffffffu, mask, own);
        int k = j - (__shfl_sync(0xffffffffu, incl, own) - __shfl_sync(0xffffffffu, cnt, own));
        if (j < total) {
            for (; k > 0; --k) m &= m - 1;
            f(own, __ffs(m) - 1);
        }
        __syncwarp();
    }
}

// Phase 1: the thread walks NROW rows of its column.  Each frame's 4 x 4
// taps stay in registers and one new row is loaded per step (8 shared loads
// for a pixel instead of 24), a step ahead at the offset in use; when the
// integer offset changes anywhere in the warp, the warp loads all four rows.
// EDGE: the tile's box overhangs the image, so pixels outside it get zero
// products and pixels whose taps would be clamped go to the general sampler,
// as do warps beyond the staged margin; those are gathered over the warp and
// done together at the end.
template <typename T, typename WS, int COH, int MODE, bool EDGE>
__device__ __forceinline__ void walk_products(const IterArgs &a, int mode, const T *__restrict__ st1,
                                              const T *__restrict__ st2, int sx0, int sy0, int px0, int py0,
                                              float *prod, uint64_t *bars, int *err)
{
    using SS = WalkStage<T, WS>;
    constexpr int P = WS::P, PLANE = WS::PLANE, NROW = WS::NROW, SP = SS::SP;
    const int tid = threadIdx.x;
    int rx, ry0, i0;
    WS::item(tid, rx, ry0, i0);
    const int x = px0 + rx, y0 = py0 + ry0;
    const int H = a.H, W = a.W;
    const int xc = EDGE ? min(max(x, 0), W - 1) : x;
    const float lx = EDGE ? (float)min(x, W - 1 - x) : 0.f;

    // V0 of row i of the column, loaded PF rows ahead
    const float2 *v0p = nullptr;
    if (MODE == V0_SAME && !EDGE) v0p = a.V0 + (int64_t)y0 * a.vpitch + x;
    // V0_UP inside the image: horizontally interpolated coarse rows y >> 1
    // and (y >> 1) + 1, kept while the walk stays between them
    float2 hA = make_float2(0.f, 0.f), hB = hA;
    auto coarse = [&](int cy) {
        const int cx = x >> 1;
        const float fx = (x & 1) ? 0.5f : 0.f, wx = 1.f - fx;
        const float2 *row = a.Vc + (int64_t)min(cy, a.Hc - 1) * a.vcpitch;
        const float2 c0 = ld_field<COH>(row + min(cx, a.Wc - 1)), c1 = ld_field<COH>(row + min(cx + 1, a.Wc - 1));
        return make_float2(fmaf(fx, c1.x, wx * c0.x), fmaf(fx, c1.y, wx * c0.y));
    };
    auto fetch = [&](int i) {
        if (MODE == V0_ZERO) return make_float2(0.f, 0.f);
        if (EDGE) return fetch_v0_rt<COH>(a, mode, xc, min(max(y0 + i, 0), H - 1));
        if (MODE == V0_SAME) return ld_field<COH>(v0p + (int64_t)i * a.vpitch);
        const int y = y0 + i;
        if (i == 0) {
            hA = coarse(y >> 1);
            hB = coarse((y >> 1) + 1);
        } else if (!(y & 1)) {
            hA = hB;
            hB = coarse((y >> 1) + 1);
        }
        const float fy = (y & 1) ? 0.5f : 0.f, wy = 1.f - fy;
        return make_float2(2.f * fmaf(fy, hB.x, wy * hA.x), 2.f * fmaf(fy, hB.y, wy * hA.y));
    };
    constexpr int PF = 3 < NROW ? 3 : NROW;
    float2 V0q[NROW];
#pragma unroll
    for (int i = 0; i < PF; ++i) V0q[i] = fetch(i);

    if (bars) {
        __syncthreads();  // barriers initialised before anyone waits on them
        // the bands this warp's rows reach
        int r_lo, r_hi;
        WS::rows_of_warp(tid >> 5, r_lo, r_hi);
        for (int b = 0; b < SS::NBAND; ++b)
            if (SS::band_row(b) <= r_hi && SS::band_row(b) + SS::SHB > r_lo &&
                !mbar_wait_bounded(bars + b, 0u, 2000000000LL)) {
                if (err) atomicExch(err, 1);  // report; the tile's results are then undefined
                mbar_wait_bounded(bars + b, 0u, 1000000000LL);
            }
    }

    // staged origins of the two stencils at row 0, offset (-REACH, -REACH)
    // (see `off`): frame 2 one left of and above the pixel, frame 1 two
    const int b0 = (y0 - sy0) * SP + (x - sx0);
    const T *const o2 = st2 + (b0 - (kBlockReach + 1) * (SP + 1));
    const T *const o1 = st1 + (b0 + (kBlockReach - 2) * (SP + 1));
    const T *p1 = o1, *p2 = o2;
    int off = -1;
    float2 A1[5], A2[5], B1[5], B2[5];  // rows of taps: (1, 2) of each frame in A, (0, 3) in B; frame 1 mirrored
    float *q = prod + ry0 * P + rx;
    unsigned slow = 0;
    auto load_row = [&](int n) {  // the taps' row n of the walk (stencil row r of pixel i: n = i + r)
        const T *t2 = p2 + n * SP, *t1 = p1 + n * SP;
        const int s = n % 5;
        A2[s] = make_float2(to_f(t2[1]), to_f(t2[2]));
        B2[s] = make_float2(to_f(t2[0]), to_f(t2[3]));
        A1[s] = make_float2(to_f(t1[2]), to_f(t1[1]));
        B1[s] = make_float2(to_f(t1[3]), to_f(t1[0]));
    };
#pragma unroll
    for (int i = 0; i < NROW; ++i) {
        const float2 V0 = V0q[i];
        if (i + PF < NROW) V0q[i + PF] = fetch(i + PF);
        int ix, iy;
        float fx, fy;
        half_floor(V0.x, ix, fx);
        half_floor(V0.y, iy, fy);
        const bool near =
            ((unsigned)(ix + kBlockReach) | (unsigned)(iy + kBlockReach)) < (unsigned)(2 * kBlockReach);
        bool general = !near;
        if (EDGE) {
            const int y = y0 + i;
            general = general || !(0.5f * fabsf(V0.x) <= lx) || !(0.5f * fabsf(V0.y) <= (float)min(y, H - 1 - y));
        }
        // a pixel that goes to the general sampler takes the taps of offset 0
        // here, which are always staged; its products are replaced below
        const int noff = near ? (iy + kBlockReach) * SP + (ix + kBlockReach) : kBlockReach * (SP + 1);
        if (__any_sync(0xffffffffu, noff != off)) {
            off = noff;
            p2 = o2 + off;
            p1 = o1 - off;
#pragma unroll
            for (int r = 0; r < 4; ++r) load_row(i + r);
        }
        if (i + 1 < NROW) load_row(i + 4);  // for the next pixel, if its offset is the same
        // E over the 12 taps: P0..P3 columns (1, 2) of the rows, Q1, Q2 columns (0, 3) of rows 1 and 2
        const int s0 = i % 5, s1 = (i + 1) % 5, s2 = (i + 2) % 5, s3 = (i + 3) % 5;
        const float2 P0 = sub2(A2[s0], A1[s3]), P1 = sub2(A2[s1], A1[s2]), P2 = sub2(A2[s2], A1[s1]),
                     P3 = sub2(A2[s3], A1[s0]);
        const float2 Q1 = sub2(B2[s1], B1[s2]), Q2 = sub2(B2[s2], B1[s1]);
        const float2 fyy = make_float2(fy, fy);
        const float2 Pv = fma2(fyy, sub2(P2, P1), P1), Qv = fma2(fyy, sub2(Q2, Q1), Q1);
        const float2 D0 = sub2(P2, P0), D1 = sub2(P3, P1);
        const float2 Dv = fma2(fyy, sub2(D1, D0), D0);
        const float It = fmaf(fx, Pv.y - Pv.x, Pv.x);
        const float g0 = Pv.y - Qv.x, g1 = Qv.y - Pv.x;
        // G = (g1 + g2) / 2 of halved differences
        const float Gx = 0.25f * fmaf(fx, g1 - g0, g0);
        const float Gy = 0.25f * fmaf(fx, Dv.y - Dv.x, Dv.x);
        const float r = fmaf(Gx, V0.x, fmaf(Gy, V0.y, -It));
        float p[5] = {Gx * Gx, Gx * Gy, Gy * Gy, Gx * r, Gy * r};
        if (EDGE) {
            const int y = y0 + i;
            if ((unsigned)x >= (unsigned)W || (unsigned)y >= (unsigned)H) {
                general = false;
                p[0] = p[1] = p[2] = p[3] = p[4] = 0.f;
            }
        }
        if (WS::ALL || i >= i0) {
            if (general) slow |= 1u << i;
#pragma unroll
            for (int c = 0; c < 5; ++c) q[c * PLANE + i * P] = p[c];
        }
    }
    // the warp's pixels for the general sampler
    warp_compact(slow, [&](int own, int row) {
        int cx, cr, i0o;
        WS::item((tid & ~31) + own, cx, cr, i0o);
        cr += row;
        const int gx = px0 + cx, gy = py0 + cr;
        products_general<T, SP>(static_cast<const T *>(a.P1), static_cast<const T *>(a.P2), H, W, a.pitch, st1, st2, sx0,
                                sy0, gx, gy, fetch_v0_rt<COH>(a, mode, gx, gy), prod + cr * P + cx, PLANE);
    });
}

__host__ __device__ __forceinline__ float add_v(float a, float b) { return a + b; }
__device__ __forceinline__ float2 add_v(float2 a, float2 b) { return __fadd2_rn(a, b); }

// Window sums of G consecutive outputs from the G + 2R values load(0) ..
// load(G + 2R - 1), in registers: blocks of up to 2R+1 outputs share a core
// of values, which running sums extend downwards in index (into o[]) and
// upwards (pre).  Additions only; each value is loaded once.  A core of four
// values or more is summed in halves: in one chain a sum of 21 values rounds 20
// times in a row, which left the fields of R 8 .. 10 up to 4 % further off the
// 64-bit ones than the block decomposition (R 10: 1.06e-7 relative against
// 1.03e-7; in halves 0.98e-7), at the same speed.
template <int R, int G, typename V, typename Load>
__host__ __device__ __forceinline__ void window_group(const Load &load, V (&o)[G])
{
    constexpr int WIN = 2 * R + 1;
    V v[G + 2 * R];
#pragma unroll
    for (int b = 0; b < G; b += WIN) {
        const int m = G - b < WIN ? G - b : WIN;  // outputs b .. b + m - 1
        const int old = b > 0 ? b + 2 * R : 0;    // values below it were loaded by the block before
        auto val = [&](int r) {
            if (r >= old) v[r] = load(r);
            return v[r];
        };
        const int n = WIN + 1 - m, half = n >= 4 ? (n + 1) / 2 : n;  // values of the core, of its first part
        V s = val(b + m - 1);
#pragma unroll
        for (int r = 1; r < half; ++r) s = add_v(s, val(b + m - 1 + r));
        if (n > half) {
            V t = val(b + m - 1 + half);
#pragma unroll
            for (int r = half + 1; r < n; ++r) t = add_v(t, val(b + m - 1 + r));
            s = add_v(s, t);
        }
        o[b + m - 1] = s;
#pragma unroll
        for (int k = m - 2; k >= 0; --k) {
            s = add_v(s, val(b + k));
            o[b + k] = s;
        }
        if (m > 1) {
            V pre = val(b + WIN);
            o[b + 1] = add_v(o[b + 1], pre);
#pragma unroll
            for (int k = 2; k < m; ++k) {
                pre = add_v(pre, val(b + k + 2 * R));
                o[b + k] = add_v(o[b + k], pre);
            }
        }
    }
}

// Vertical window sums of a whole column (V float) or column pair (float2) in
// place: N outputs in order units of VG rows.  A unit's rows are read before
// any is overwritten by it, the 2R rows it shares with the next stay in
// registers.
template <int R, int N, int VG, int P, typename V>
__device__ __forceinline__ void walk_vcolumn(float *col)
{
    V v[N + 2 * R];
#pragma unroll
    for (int r = 0; r < 2 * R; ++r) v[r] = *reinterpret_cast<const V *>(col + r * P);
#pragma unroll
    for (int g = 0; g < N; g += VG) {
#pragma unroll
        for (int r = g + 2 * R; r < g + VG + 2 * R; ++r) v[r] = *reinterpret_cast<const V *>(col + r * P);
        V o[VG];
        window_group<R>([&](int r) { return v[g + r]; }, o);
#pragma unroll
        for (int k = 0; k < VG; ++k) *reinterpret_cast<V *>(col + (g + k) * P) = o[k];
    }
}

// The guarded solve of G adjacent pixels and their store (gx a multiple of
// G).  KEEP: the window sums go to a.s_out too (reverse mode).
template <int COH, bool KEEP, int G>
__device__ __forceinline__ void walk_solve(const IterArgs &a, int mode, int gx, int gy, const float (&S)[5][G])
{
    float2 V[G];
    unsigned keep = 0;  // pixels whose guard keeps V0
#pragma unroll
    for (int k = 0; k < G; ++k) {
        const float sxx = S[0][k], sxy = S[1][k], syy = S[2][k], sxr = S[3][k], syr = S[4][k];
        const float tr = sxx + syy, det = sxx * syy - sxy * sxy;
        const float inv = recip_newton(det);
        V[k] = make_float2((syy * sxr - sxy * syr) * inv, (sxx * syr - sxy * sxr) * inv);
        if (!(tr > a.eps_abs) || det <= a.eps_rel * tr * tr) keep |= 1u << k;
    }
    if (keep) {
#pragma unroll
        for (int k = 0; k < G; ++k)
            if ((keep >> k & 1u) && gx + k < a.W) V[k] = fetch_v0_rt<COH>(a, mode, gx + k, gy);
    }
    const bool full = gx + G <= a.W;
    if (KEEP) {
#pragma unroll
        for (int c = 0; c < 5; ++c) {
            float *d = a.s_out + c * a.s_plane + (size_t)gy * a.s_pitch + gx;
            if (full) {
#pragma unroll
                for (int k = 0; k < G; k += 4)
                    *reinterpret_cast<float4 *>(d + k) = make_float4(S[c][k], S[c][k + 1], S[c][k + 2], S[c][k + 3]);
            } else {
#pragma unroll
                for (int k = 0; k < G; ++k)
                    if (gx + k < a.W) d[k] = S[c][k];
            }
        }
    }
    if (a.u_out) {
        float *u = a.u_out + (int64_t)gy * a.W + gx, *v = a.v_out + (int64_t)gy * a.W + gx;
        if (full && ((reinterpret_cast<uintptr_t>(u) | reinterpret_cast<uintptr_t>(v)) & 15u) == 0) {
#pragma unroll
            for (int k = 0; k < G; k += 4) {
                *reinterpret_cast<float4 *>(u + k) = make_float4(V[k].x, V[k + 1].x, V[k + 2].x, V[k + 3].x);
                *reinterpret_cast<float4 *>(v + k) = make_float4(V[k].y, V[k + 1].y, V[k + 2].y, V[k + 3].y);
            }
        } else {
#pragma unroll
            for (int k = 0; k < G; ++k)
                if (gx + k < a.W) {
                    u[k] = V[k].x;
                    v[k] = V[k].y;
                }
        }
    } else {
        float2 *d = a.Vout + (int64_t)gy * a.vpitch + gx;  // rows and gx are multiples of 16 bytes
        if (full) {
#pragma unroll
            for (int k = 0; k < G; k += 2)
                *reinterpret_cast<float4 *>(d + k) = make_float4(V[k].x, V[k].y, V[k + 1].x, V[k + 1].y);
        } else {
#pragma unroll
            for (int k = 0; k < G; ++k)
                if (gx + k < a.W) d[k] = V[k];
        }
    }
}

// Replicates the border rows and columns of a staged box two pixels beyond
// the image: all that samples inside the image reach (the rest of the box
// outside it is never used).
template <typename T, typename WS>
__device__ __forceinline__ void walk_fill_border(T *stage, int sx0, int sy0, int H, int W)
{
    using SS = WalkStage<T, WS>;
    constexpr int SP = SS::SP, STG = SS::STG, SHT = SS::SHT, NT = WS::NT;
    const int tid = threadIdx.x;
    const int ya = max(sy0, -2), yb = min(sy0 + SHT - 1, H + 1);  // rows and columns to make valid
    const int xa = max(sx0, -2), xb = min(sx0 + SP - 1, W + 1);
    auto cell = [&](int f, int y, int x) -> T & { return stage[f * STG + (y - sy0) * SP + (x - sx0)]; };
    const int nrow = yb - ya + 1;
    for (int t = tid; t < 8 * nrow; t += NT) {  // columns -2, -1, W, W + 1 of both frames
        const int f = (t >> 2) & 1, k = t & 3, y = ya + (t >> 3);
        const int x = k < 2 ? k - 2 : W + k - 2;
        if (x >= xa && x <= xb) cell(f, y, x) = cell(f, min(max(y, 0), H - 1), k < 2 ? 0 : W - 1);
    }
    const int x0 = max(xa, 0), ncol = min(xb, W - 1) - x0 + 1;
    for (int t = tid; t < ncol; t += NT)  // rows -2, -1, H, H + 1
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            const int f = k >> 2, y = (k & 3) < 2 ? (k & 3) - 2 : H + (k & 3) - 2;
            if (y >= ya && y <= yb) cell(f, y, x0 + t) = cell(f, (k & 3) < 2 ? 0 : H - 1, x0 + t);
        }
}

// One tile (the CTA's only one): the output pixels from (bx TX, row0 + by TY)
// on, rows below row1 and the level's end.  TMA staging needs tensor maps
// tm1, tm2 (box SP x SHB), or null, and NBAND mbarriers in shared memory.
// COH: how fields are read (FieldLoad).  CHAIN: the
// launch may have started before the one ahead of it ended; its images are
// staged ahead of the wait for that launch if early.
template <typename T, typename WS, int COH, bool KEEP, bool CHAIN>
__device__ __forceinline__ void walk_tile(const IterArgs &a, int mode, int bx, int by, int row0, int row1,
                                          float4 *smem_f4, const CUtensorMap *tm1, const CUtensorMap *tm2, int *err,
                                          uint64_t *tma_bars, bool early)
{
    static_assert(COH != LD_READ_ONLY || !CHAIN, "the launch ahead writes V0 while a chained one is resident");
    using SS = WalkStage<T, WS>;
    constexpr int TX = WS::TX, TY = WS::TY, R = WS::R, RW = WS::RW, P = WS::P, PLANE = WS::PLANE, NT = WS::NT;
    constexpr int SP = SS::SP, NV = SS::NV, VEC = SS::VEC, STG = SS::STG, SHT = SS::SHT, SHB = SS::SHB;
    constexpr int NBAND = SS::NBAND;
    const int tid = threadIdx.x;
    float *prod = reinterpret_cast<float *>(smem_f4);
    T *stage = reinterpret_cast<T *>(prod + WS::PROD);
    const int H = a.H, W = a.W, pitch = a.pitch;
    const int tx0 = bx * TX, ty0 = row0 + by * TY, px0 = tx0 - R, py0 = ty0 - R;
    const int sy0 = py0 - kBlockReach - 1;
    const int sxn = px0 - kBlockReach - 1;
    const int sx0 = (sxn >= 0 ? sxn / VEC : -((-sxn + VEC - 1) / VEC)) * VEC;  // floor to a VEC multiple
    const bool interior = sx0 >= 0 && sx0 + SS::SPN <= W && sy0 >= 0 && sy0 + WS::SH <= H;
    uint64_t *bars = nullptr;

    // phase 0
    if (CHAIN && !early) pdl_wait();
    if (tm1 != nullptr) {
        if (tid == 0) {
            mbar_init_n<NBAND>(tma_bars);
            for (int b = 0; b < NBAND; ++b) {  // elements outside the image arrive as zero
                mbar_expect_tx(&tma_bars[b], (unsigned)(2 * SHB * SP * sizeof(T)));
                const int r = SS::band_row(b);
                tma_load_2d(stage + r * SP, tm1, sx0, sy0 + r, &tma_bars[b]);
                tma_load_2d(stage + STG + r * SP, tm2, sx0, sy0 + r, &tma_bars[b]);
            }
        }
        if (interior) {
            bars = tma_bars;  // waited for band by band in phase 1
        } else {
            __syncthreads();
            for (int b = 0; b < NBAND; ++b)
                if (!mbar_wait_bounded(&tma_bars[b], 0u, 2000000000LL)) {
                    if (err) atomicExch(err, 1);
                    mbar_wait_bounded(&tma_bars[b], 0u, 1000000000LL);
                }
        }
    } else {
        // rows clamped as a whole; chunks that begin inside the image as they
        // are (columns W .. pitch - 1 of a row are allocated)
        const T *P1 = static_cast<const T *>(a.P1), *P2 = static_cast<const T *>(a.P2);
        for (int t = tid; t < 2 * SHT * NV; t += NT) {
            const int f = t >= SHT * NV ? 1 : 0;
            const int r = t - f * SHT * NV;
            const int row = r / NV, v = r - row * NV;
            const int gx0 = sx0 + v * VEC;
            if (gx0 >= 0 && gx0 < W)
                cp_async16(stage + f * STG + row * SP + v * VEC,
                           (f ? P2 : P1) + (int64_t)min(max(sy0 + row, 0), H - 1) * pitch + gx0);
        }
        cp_async_wait_all();
        __syncthreads();
    }
    if (!interior) {
        walk_fill_border<T, WS>(stage, sx0, sy0, H, W);
        __syncthreads();
    }

    if (CHAIN) {
        if (early) pdl_wait();
        pdl_trigger();
    }

    // phase 1
    const T *st2 = stage + STG;
#define OFV_WALK(MODE, EDGE) walk_products<T, WS, COH, MODE, EDGE>(a, mode, stage, st2, sx0, sy0, px0, py0, prod, bars, err)
    if (interior) {
        if (mode == V0_SAME) OFV_WALK(V0_SAME, false);
        else if (mode == V0_UP) OFV_WALK(V0_UP, false);
        else OFV_WALK(V0_ZERO, false);
    } else {
        OFV_WALK(V0_SAME, true);  // V0 by the run-time mode
    }
#undef OFV_WALK
    // every band has landed before the CTA can finish (no copy in flight at exit)
    if (bars && tid == 0)
        for (int b = 0; b < NBAND; ++b) mbar_wait_bounded(&bars[b], 0u, 1000000000LL);
    __syncthreads();

    // phase 2: vertical sums over the products
    if (tid < WS::VITEMS) {
        constexpr int NP = RW / WS::VW;
        const int c = tid / NP, k = tid - c * NP;
        walk_vcolumn<R, TY, WS::VG, P, std::conditional_t<WS::VW == 2, float2, float>>(prod + c * PLANE + WS::VW * k);
    }
    __syncthreads();

    // phase 3: horizontal sums, solve and store, G pixels per item
    constexpr int G = WS::G;
    const int ylim = min(H, row1);
    for (int t = tid; t < WS::GITEMS; t += NT) {
        int oy, ox;
        const bool on = WS::group(t, oy, ox);
        const int gy = ty0 + oy, gx = tx0 + ox;
        if (!on || gy >= ylim || gx >= W) continue;
        float S[5][G];
#pragma unroll
        for (int c = 0; c < 5; ++c) {
            const float4 *row = reinterpret_cast<const float4 *>(prod + c * PLANE + oy * P + ox);
            constexpr int NV4 = (G + 2 * R + 3) / 4;
            float v[4 * NV4];
#pragma unroll
            for (int k = 0; k < NV4; ++k) *reinterpret_cast<float4 *>(v + 4 * k) = row[k];
            window_group<R>([&](int r) { return v[r]; }, S[c]);
        }
        walk_solve<COH, KEEP>(a, mode, gx, gy, S);
    }
}

}  // namespace ofv
