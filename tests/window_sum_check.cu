// Rounding of the window sums, on the host (built and run by
// test_walk_schedule.py; no GPU needed): (2R+1)^2 sums of random products,
// formed as the column walk forms them (units of eight rows, then groups of
// eight columns, window_group) and as the variants' tiles do (blocks of 2R+1
// values, window_sums_inplace), against sums in double.  Prints the two
// relative errors (root mean square) per radius and "FAIL" where the walk's is
// more than 1 % above the other: what the samples leave open (R 1, where both
// forms add the same values pairwise, reads 0.7 %).
#include <cmath>
#include <cstdio>
#include <random>
#include <vector>
#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include "k_walk.cuh"

using namespace ofv;

struct Strided {
    const float *p;
    int stride;
    __host__ __device__ float operator()(int r) const { return p[r * stride]; }
};

// tiles: how many tiles of TS x TS outputs are summed
template <int R>
static int check(int tiles)
{
    constexpr int TS = 48, N = TS + 2 * R;
    std::mt19937 rng(100 + R);
    std::normal_distribution<float> nd;
    double err[2] = {0, 0}, ref = 0;
    for (int t = 0; t < tiles; ++t) {
        std::vector<float> x(N * N), blk, w;
        for (float &v : x) {
            const float g = nd(rng);
            v = g * g;  // a squared gradient
        }
        blk = w = x;
        for (int r = 0; r < N; ++r) window_sums_inplace<R, TS>(blk.data() + r * N, 1);
        for (int c = 0; c < TS; ++c) window_sums_inplace<R, TS>(blk.data() + c, N);
        for (int c = 0; c < N; ++c)
            for (int g = 0; g < TS; g += 8) {
                float o[8];
                window_group<R>(Strided{x.data() + g * N + c, N}, o);
                for (int k = 0; k < 8; ++k) w[(g + k) * N + c] = o[k];
            }
        for (int r = 0; r < TS; ++r)
            for (int g = 0; g < TS; g += 8) {
                float o[8];
                window_group<R>(Strided{w.data() + r * N + g, 1}, o);
                for (int k = 0; k < 8; ++k) {
                    double s = 0;
                    for (int a = 0; a <= 2 * R; ++a)
                        for (int b = 0; b <= 2 * R; ++b) s += x[(r + a) * N + g + k + b];
                    err[0] += (o[k] - s) * (o[k] - s);
                    err[1] += (blk[r * N + g + k] - s) * (blk[r * N + g + k] - s);
                    ref += s * s;
                }
            }
    }
    const double walk = std::sqrt(err[0] / ref), block = std::sqrt(err[1] / ref);
    const bool bad = walk > 1.01 * block;
    printf("R %2d walk %.3e blocks %.3e%s\n", R, walk, block, bad ? " FAIL" : "");
    return bad;
}

int main()
{
    const int fails = check<1>(60) + check<2>(60) + check<3>(60) + check<4>(60) + check<5>(60) + check<6>(60) +
                      check<7>(60) + check<8>(60) + check<9>(60) + check<10>(60);
    printf("%d failing radii\n", fails);
    return fails != 0;
}
