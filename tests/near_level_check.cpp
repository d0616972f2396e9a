// Host check of near_level (walk_levels.cuh): within 2^-17 of every power of 16 in range on both sides, and no further.
#define __host__
#define __device__
#define __forceinline__ inline
#include <cmath>
#include <cstdio>
#include <initializer_list>
#include "walk_levels.cuh"
int main() {
    int bad = 0;
    for (int k = -31; k <= 31; k++) {
        const double t = std::ldexp(1.0, 4 * k);
        for (int s = -1; s <= 1; s += 2)
            for (double d : {0.0, 0x1p-24, 0x1p-23, 0x1p-20, 0x1p-18, 0x1.8p-18, 0x1.fp-18, 0x1p-17, 0x1.1p-17, 0x1.8p-17,
                             0x1p-16, 0x1p-10, 0.3, 0.9}) {
                const float x = (float)(t * (1.0 + s * d));
                const bool want = std::fabs((double)x / t - 1.0) <= 0x1p-17;
                if (near_level(x) != want && bad++ < 10) printf("16^%d %+a: %d\n", k, s * d, !want);
            }
        for (int q = 1; q < 4; q++)  // powers of two between
            if (near_level((float)std::ldexp(t, q)) && bad++ < 10) printf("16^%d 2^%d\n", k, q);
    }
    for (float x : {0.0f, -0.0f, INFINITY, NAN, 1e-42f}) bad += near_level(x) ? 1 : 0;
    printf("bad %d\n", bad);
    return bad != 0;
}
