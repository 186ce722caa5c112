// Host-side check of the column walk's index arithmetic (built and run by
// test_walk_schedule.py; no GPU needed).  For every storage type, window
// radius and tile edge it goes through the items of each phase and checks that
//   * every pixel of the product region is stored by exactly one thread;
//   * the taps of every pixel a thread forms, at every integer offset the
//     fast path takes, lie inside the staged box and in TMA bands its warp
//     waits for;
//   * the vertical items cover every column pair and row once and read rows
//     of the region, and the output groups cover the tile once, with loads
//     inside a plane's row and octets of lanes on distinct banks;
//   * the staged box is one TMA can copy and the tile fits its share of
//     shared memory;
//   * the smaller shape is another tile where walk_has_alt says so;
//   * no further segment of a column that would shorten the walks fits the
//     threads.
// Prints one line per case and "FAIL" on any violation.
#include <cstdio>
#include <cstring>
#include <vector>
#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include "k_walk.cuh"

using namespace ofv;

template <typename T, int R, int SHAPE>
static int check(const char *tname)
{
    using WS = WalkShape<R, SHAPE>;
    using SS = WalkStage<T, WS>;
    constexpr int RW = WS::RW, RH = WS::RH, P = WS::P, NROW = WS::NROW, SP = SS::SP, VEC = SS::VEC, D = kBlockReach;
    int bad = 0;
    std::vector<int> stored(RW * RH, 0);
    for (int tid = 0; tid < WS::NT; ++tid) {
        int rx, ry0, i0;
        WS::item(tid, rx, ry0, i0);
        if (rx < 0 || rx >= RW || ry0 < 0 || ry0 + NROW > RH) ++bad;
        int lo, hi;
        WS::rows_of_warp(tid >> 5, lo, hi);
        if (lo < 0 || hi >= SS::SHT) ++bad;
        for (int slack = 0; slack < VEC; ++slack)  // columns by which the box starts left of the margin
            for (int i = 0; i < NROW; ++i) {
                const int b0 = (ry0 + D + 1) * SP + rx + D + 1 + slack;
                for (int oy = 0; oy < 2 * D; oy += 2 * D - 1)  // the extreme offsets in each direction
                    for (int ox = 0; ox < 2 * D; ox += 2 * D - 1) {
                        const int off = oy * SP + ox;
                        const int o2 = b0 - (D + 1) * (SP + 1) + off, o1 = b0 + (D - 2) * (SP + 1) - off;
                        for (int r = 0; r < 4; ++r)
                            for (int c = 0; c < 4; ++c)
                                for (int f = 0; f < 2; ++f) {
                                    const int t = (f ? o2 : o1) + (i + r) * SP + c;
                                    const int row = t / SP, col = t % SP;
                                    // expected position of the tap
                                    const int er = f ? ry0 + i + oy + r : ry0 + i + 2 * D - 1 - oy + r;
                                    const int ec = f ? rx + slack + ox + c : rx + slack + 2 * D - 1 - ox + c;
                                    if (t < 0 || row != er || col != ec || row < lo || row > hi || col >= SS::SPN) ++bad;
                                }
                    }
                if (slack == 0 && i >= i0) ++stored[(ry0 + i) * RW + rx];
            }
    }
    for (int v : stored) bad += v != 1;
    std::vector<int> summed(5 * RW, 0);
    for (int tid = 0; tid < WS::VITEMS; ++tid) {
        constexpr int NP = RW / WS::VW;
        const int c = tid / NP, k = tid % NP;
        if (c >= 5 || WS::VW * k + WS::VW > P) {
            ++bad;
            continue;
        }
        for (int j = 0; j < WS::VW; ++j) ++summed[c * RW + WS::VW * k + j];
    }
    for (int v : summed) bad += v != 1;
    // output groups: each once, octets of lanes on distinct banks, loads inside the plane's rows
    constexpr int G = WS::G;
    std::vector<int> group(WS::TX / G * WS::TY, 0);
    for (int t = 0; t < WS::GITEMS; ++t) {
        int oy, ox;
        if (!WS::group(t, oy, ox)) continue;
        if (oy < 0 || oy >= WS::TY || ox < 0 || ox % G || ox + G > WS::TX || ox + (G + 2 * R + 3) / 4 * 4 > P) {
            ++bad;
            continue;
        }
        ++group[oy * (WS::TX / G) + ox / G];
        for (int k = t & ~7; k < t; ++k) {
            int y, x;
            if (WS::group(k, y, x)) bad += ((y * P + x) & 31) == ((oy * P + ox) & 31);  // 16-byte loads
        }
    }
    for (int v : group) bad += v != 1;
    if (P % 4 || WS::PLANE % 4 || WS::PROD % 32) ++bad;
    // the TMA box: 16-byte multiple wide, at most 256 elements, bands 128-byte aligned
    if (SP * sizeof(T) % 16 || SP > 256 || SS::SHB > 256 || SP < SS::SPN || SS::SHT < WS::SH) ++bad;
    for (int b = 0; b < SS::NBAND; ++b)
        if (SS::band_row(b) * SP * sizeof(T) % 128 || SS::band_row(b) > b * SS::SHB) ++bad;
    if (SS::band_row(SS::NBAND - 1) + SS::SHB != SS::SHT || SS::STG < SS::SHT * SP) ++bad;
    const size_t smem = walk_smem_bytes<T, WS>();
    if (WS::MINB * (smem + 1024 + 32) > 228 * 1024 || smem > 227 * 1024 - 512) ++bad;
    if (SHAPE == 1) {
        using W0 = WalkShape<R, 0>;
        const bool same = W0::TX == WS::TX && W0::TY == WS::TY && W0::NT == WS::NT;
        if (same == walk_has_alt(R)) ++bad;
    }
    if (!WS::COLS && (WS::NSEG + 1) * RW <= WS::NT && (RH + WS::NSEG) / (WS::NSEG + 1) < NROW) ++bad;
    if (WS::TX != walk_tile_w(R, SHAPE) || WS::TY != walk_tile_h(R, SHAPE)) ++bad;
    printf("%s KR %2d tile %2dx%2d NT %4d rows %d SP %d P %d smem %zu bad %d%s\n", tname, R, WS::TX, WS::TY, WS::NT,
           NROW, SP, P, smem, bad, bad ? " FAIL" : "");
    return bad != 0;
}

template <typename T, int SHAPE>
static int shape(const char *n)
{
    return check<T, 1, SHAPE>(n) + check<T, 2, SHAPE>(n) + check<T, 3, SHAPE>(n) + check<T, 4, SHAPE>(n) +
           check<T, 5, SHAPE>(n) + check<T, 6, SHAPE>(n) + check<T, 7, SHAPE>(n) + check<T, 8, SHAPE>(n) +
           check<T, 9, SHAPE>(n) + check<T, 10, SHAPE>(n);
}

template <typename T>
static int all(const char *n)
{
    return shape<T, 0>(n) + shape<T, 1>(n);
}

int main()
{
    const int fails = all<float>("f32 ") + all<__half>("f16 ") + all<__nv_bfloat16>("bf16");
    printf("%d failing cases\n", fails);
    return fails != 0;
}
