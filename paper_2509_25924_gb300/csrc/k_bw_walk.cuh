// Adjoint of one stage's samples (reverse mode, window radii 1..10): from
// the gradients of the five products to the image gradients and the gradient
// of V0, in the mirrored-difference form of the forward walk (k_walk.cuh).
//
// With E(s) = P2(k + s) - P1(k - s) the residual and the averaged gradient of
// a pixel are one stencil over 12 values E, so their adjoint is 12 values
// gE(s), added to the gradient of frame 2 at tap s and subtracted from that
// of frame 1 at tap -s.  A warp walks 32 adjacent columns down NROW rows with
// the taps and the gradients of each frame's 4 x 4 stencil in registers: a
// step loads one row of taps and retires one row of gradients.  Where the
// whole warp samples at one integer offset, a retired row is summed across
// the lanes first and reaches memory as one add per column instead of twelve
// per pixel and frame.  Pixels whose stencil leaves the image, and samples
// exactly on a cell boundary (whose one-sided slopes differ between the
// frames), are gathered over the warp and take the general form of
// samples_adjoint_pixel at the end.
//
// The per-tile form it replaces accumulated 20 terms a pixel and frame in
// shared memory, where a float add is a compare-and-swap loop.
#pragma once
#include "k_bw_block.cuh"
#include "k_walk.cuh"

namespace ofv {

// Rows a warp walks: 8, or 4 where the 8-row warps of a level would all be
// resident at once (152 SMs x 16 warps), so that only the length of a walk
// counts.
constexpr int kBwRows = 8, kBwRowsSmall = 4;
inline int bw_rows(int H, int W)
{
    return (long long)((W + 31) / 32) * ((H + kBwRows - 1) / kBwRows) <= 152 * 16 ? kBwRowsSmall : kBwRows;
}

// GV0: the gradient of V0 is wanted (not at the first stage).
template <typename T, bool GV0, int NROW, typename General>
__device__ __forceinline__ void bw_samples_walk(const IterArgs &a, int mode, const Planes5 &gq, float2 *gV0, float *gP1,
                                                float *gP2, int gpitch, const General &general)
{
    const int lane = threadIdx.x & 31;
    const int x = blockIdx.x * 32 + lane;
    const int y0 = (blockIdx.y * (blockDim.x / 32) + (threadIdx.x >> 5)) * NROW;
    const int H = a.H, W = a.W, pitch = a.pitch;
    if (y0 >= H) return;
    const T *P1 = static_cast<const T *>(a.P1), *P2 = static_cast<const T *>(a.P2);
    const T *p1 = P1, *p2 = P2;   // first row of the stencil's taps at the step's row
    float *g1 = gP1, *g2 = gP2;   // gradients there
    int kx = 0, ky = 0;           // integer offset in use
    bool live = false;            // the lane has one
    bool uni = false;             // all lanes have the same
    float2 A1[4], A2[4], B1[4], B2[4];  // taps by row: columns (1, 2) in A, (0, 3) in B; frame 1 mirrored
    float2 dA1[4], dA2[4], dB1[4], dB2[4];  // gradients of them
#pragma unroll
    for (int s = 0; s < 4; ++s) dA1[s] = dA2[s] = dB1[s] = dB2[s] = make_float2(0.f, 0.f);

    auto red = [](float *p, float v) {
        if (v != 0.f) atomicAdd(p, v);
    };
    // one row of gradients of a frame, columns c0 .. c3, to memory at p
    auto retire4 = [&](float *p, float c0, float c1, float c2, float c3) {
        if (uni) {
            const float t1 = __shfl_sync(0xffffffffu, c1, (lane - 1) & 31);
            const float t2 = __shfl_sync(0xffffffffu, c2, (lane - 2) & 31);
            const float t3 = __shfl_sync(0xffffffffu, c3, (lane - 3) & 31);
            // lane l holds column l of the row; the wrapped terms are columns 32, 33, 34
            red(p, c0 + (lane >= 1 ? t1 : 0.f) + (lane >= 2 ? t2 : 0.f) + (lane >= 3 ? t3 : 0.f));
            if (lane < 3) red(p + 32, (lane < 1 ? t1 : 0.f) + (lane < 2 ? t2 : 0.f) + t3);
        } else if (live) {
            red(p, c0);
            red(p + 1, c1);
            red(p + 2, c2);
            red(p + 3, c3);
        }
    };
    // Row n of the walk lives in slot n mod 4, passed as a constant; k rows
    // below the step's own (the pointers follow the walk).
    auto retire = [&](int s, int k) {
        retire4(g2 + k * gpitch, dB2[s].x, dA2[s].x, dA2[s].y, dB2[s].y);
        retire4(g1 + k * gpitch, dB1[s].y, dA1[s].y, dA1[s].x, dB1[s].x);
        dA1[s] = dA2[s] = dB1[s] = dB2[s] = make_float2(0.f, 0.f);
    };
    auto load_row = [&](int s, int k) {
        const T *t2 = p2 + k * pitch, *t1 = p1 + k * pitch;
        A2[s] = make_float2(ld_store(t2 + 1), ld_store(t2 + 2));
        B2[s] = make_float2(ld_store(t2), ld_store(t2 + 3));
        A1[s] = make_float2(ld_store(t1 + 2), ld_store(t1 + 1));
        B1[s] = make_float2(ld_store(t1 + 3), ld_store(t1));
    };
    // V0 and the products' gradients of a row, loaded a step ahead
    struct In {
        float2 V0, gV0;
        float q[5];
    };
    const int xc = min(x, W - 1);
    auto fetch = [&](int y) {  // rows below the image repeat its last (and are not used)
        const int yc = min(y, H - 1);
        In in;
        in.V0 = fetch_v0_rt<LD_READ_ONLY>(a, mode, xc, yc);
        if (GV0) in.gV0 = gV0[(int64_t)yc * a.vpitch + xc];
        const int64_t o = (int64_t)yc * gq.pitch + xc;
#pragma unroll
        for (int c = 0; c < 5; ++c) in.q[c] = gq.p[c][o];  // written by the launch ahead
        return in;
    };
    unsigned rest = 0;  // rows whose pixel needs the general form
    In nxt = fetch(y0);
#pragma unroll 1
    for (int ib = 0; ib < NROW; ib += 4) {
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            // a step past the image's last row has no pixel: what is left of
            // the walk is retired
            const int y = y0 + ib + j;
            const int s0 = j, s1 = (j + 1) & 3, s2 = (j + 2) & 3, s3 = (j + 3) & 3;
            const In cur = nxt;
            if (ib + j + 1 < NROW) nxt = fetch(y + 1);
            const float2 V0 = cur.V0;
            const float q0 = cur.q[0], q1 = cur.q[1], q2 = cur.q[2], q3 = cur.q[3], q4 = cur.q[4];
            int ix, iy;
            float fx, fy;
            half_floor(V0.x, ix, fx);
            half_floor(V0.y, iy, fy);
            constexpr int kFar = 1 << 21;  // offsets half_floor resolves
            const bool in = x < W && y < H && (unsigned)(ix + kFar) < 2u * kFar && (unsigned)(iy + kFar) < 2u * kFar &&
                            x + ix >= 1 && x + ix <= W - 3 && x - ix >= 2 && x - ix <= W - 2 && y + iy >= 1 &&
                            y + iy <= H - 3 && y - iy >= 2 && y - iy <= H - 2;
            const bool fast = in && (!GV0 || (fx != 0.f && fy != 0.f));
            const bool change = fast != live || (fast && (ix != kx || iy != ky));
            if (__any_sync(0xffffffffu, change)) {
                // three rows hold gradients at the old offset
                retire(s0, 0);
                retire(s1, 1);
                retire(s2, 2);
                live = fast;
                if (fast) {
                    kx = ix;
                    ky = iy;
                    const int64_t r2 = y + iy - 1, r1 = y - iy - 2;
                    p2 = P2 + (r2 * pitch + x + ix - 1);
                    p1 = P1 + (r1 * pitch + x - ix - 2);
                    g2 = gP2 + (r2 * gpitch + x + ix - 1);
                    g1 = gP1 + (r1 * gpitch + x - ix - 2);
                    load_row(s0, 0);
                    load_row(s1, 1);
                    load_row(s2, 2);
                }
                const int fx0 = __shfl_sync(0xffffffffu, kx, 0), fy0 = __shfl_sync(0xffffffffu, ky, 0);
                uni = __all_sync(0xffffffffu, live && kx == fx0 && ky == fy0);
            }
            if (fast) {
                load_row(s3, 3);
                const float2 E0 = sub2(A2[s0], A1[s3]), E1 = sub2(A2[s1], A1[s2]), E2 = sub2(A2[s2], A1[s1]),
                             E3 = sub2(A2[s3], A1[s0]);
                const float2 F1 = sub2(B2[s1], B1[s2]), F2 = sub2(B2[s2], B1[s1]);
                const float wx = 1.f - fx, wy = 1.f - fy;
                const float2 dP = sub2(E2, E1), dF = sub2(F2, F1), D0 = sub2(E2, E0), D1 = sub2(E3, E1);
                const float2 fyy = make_float2(fy, fy);
                const float2 Pv = fma2(fyy, dP, E1), Fv = fma2(fyy, dF, F1), dD = sub2(D1, D0), Dv = fma2(fyy, dD, D0);
                const float It = fmaf(fx, Pv.y - Pv.x, Pv.x);
                const float u0 = Pv.y - Fv.x, u1 = Fv.y - Pv.x;
                const float Gx = 0.25f * fmaf(fx, u1 - u0, u0), Gy = 0.25f * fmaf(fx, Dv.y - Dv.x, Dv.x);
                const float r = fmaf(Gx, V0.x, fmaf(Gy, V0.y, -It));
                // products -> Gx, Gy, It
                const float gr = Gx * q3 + Gy * q4;
                const float gGx = 0.25f * (2.f * Gx * q0 + Gy * q1 + r * q3 + V0.x * gr);
                const float gGy = 0.25f * (Gx * q1 + 2.f * Gy * q2 + r * q4 + V0.y * gr);
                if (GV0) {
                    const float hx = gGx * (u1 - u0) + gGy * (Dv.y - Dv.x) - gr * (Pv.y - Pv.x);
                    const float hy = gGx * (wx * (dP.y - dF.x) + fx * (dF.y - dP.x)) + gGy * (wx * dD.x + fx * dD.y) -
                                     gr * (wx * dP.x + fx * dP.y);
                    float2 g = cur.gV0;
                    g.x += Gx * gr + 0.5f * hx;
                    g.y += Gy * gr + 0.5f * hy;
                    gV0[(int64_t)y * a.vpitch + x] = g;
                }
                // Gx, Gy, It -> the rows' interpolations -> E
                const float2 gPv = make_float2(-wx * gr - fx * gGx, -fx * gr + wx * gGx);
                const float2 gFv = make_float2(-wx * gGx, fx * gGx);
                const float2 gDv = make_float2(wx * gGy, fx * gGy);
                const float2 wyy = make_float2(wy, wy);
                const float2 gD0 = __fmul2_rn(wyy, gDv), gD1 = __fmul2_rn(fyy, gDv);
                const float2 gE1 = sub2(__fmul2_rn(wyy, gPv), gD1), gE2 = fma2(fyy, gPv, gD0);
                const float2 gF1 = __fmul2_rn(wyy, gFv), gF2 = __fmul2_rn(fyy, gFv);
                dA2[s0] = sub2(dA2[s0], gD0);
                dA2[s1] = __fadd2_rn(dA2[s1], gE1);
                dA2[s2] = __fadd2_rn(dA2[s2], gE2);
                dA2[s3] = __fadd2_rn(dA2[s3], gD1);
                dB2[s1] = __fadd2_rn(dB2[s1], gF1);
                dB2[s2] = __fadd2_rn(dB2[s2], gF2);
                dA1[s3] = __fadd2_rn(dA1[s3], gD0);
                dA1[s2] = sub2(dA1[s2], gE1);
                dA1[s1] = sub2(dA1[s1], gE2);
                dA1[s0] = sub2(dA1[s0], gD1);
                dB1[s2] = sub2(dB1[s2], gF1);
                dB1[s1] = sub2(dB1[s1], gF2);
            } else if (x < W && y < H) {
                rest |= 1u << (ib + j);
            }
            retire(s0, 0);
            p1 += pitch;
            p2 += pitch;
            g1 += gpitch;
            g2 += gpitch;
        }
    }
    retire(0, 0);
    retire(1, 1);
    retire(2, 2);
    // the pixels left over, gathered over the warp
    warp_compact(rest, [&](int own, int row) { general(blockIdx.x * 32 + own, y0 + row); });
}

}  // namespace ofv
