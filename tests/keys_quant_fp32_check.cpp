// Host check of the key quantisation's FP32 evaluation (keys_quant.cuh) against floor(((double)x - (double)xmin) *
// scale): wherever it says that it decided, the value must be the same.  Operands: boxes of many sizes and offsets,
// positions at random, one ulp apart, and aimed at the grid's planes.  Prints the counts, non-zero on a mismatch.
#define __host__
#define __device__
#define __forceinline__ inline
#include <cmath>
#include <cstdio>
#include <cstdint>
#include <cstring>
#include <random>
#include "keys_quant.cuh"
int main() {
    std::mt19937_64 g(777);
    auto uni = [&]() { return (double)(g() >> 11) * 0x1p-53; };
    const double QMAX = (double)((1 << 21) - 1);
    long long n = 0, decided = 0, bad = 0;
    for (int box = 0; box < 60000; box++) {
        // lower corner and side: from boxes far off the origin to ones around it, from tiny to huge
        const double side0 = std::ldexp(1.0 + uni(), (int)(g() % (box % 10 == 0 ? 200 : 40)) - (box % 10 == 0 ? 100 : 20));
        const float xmin = (float)((uni() * 2.0 - 1.0) * side0 * std::ldexp(1.0, (int)(g() % 12) - 6));
        const float xmax = (float)(xmin + side0);
        const double side = ((double)xmax - (double)xmin) * (box % 3 ? 1.0 : 1.0 + 3.0 * uni());
        if (!(side > 0.0) || !std::isfinite(side)) continue;
        const double scale = 2097152.0 / side;
        float sh, sl;
        if (!gtq_fp32_scale(scale, &sh, &sl)) continue;
        for (int k = 0; k < 100; k++) {
            float x;
            if (k % 3 == 0) x = (float)(xmin + uni() * ((double)xmax - xmin));
            else {  // near a plane of the grid
                x = (float)(xmin + std::floor(uni() * 2097152.0) / scale);
                for (int j = (int)(g() % 5); j > 0; j--) x = std::nextafterf(x, (g() & 1) ? INFINITY : -INFINITY);
            }
            if (!(x >= xmin) || !(x <= xmax)) continue;
            uint32_t q = 0;
            n++;
            if (!quantise_fp32(x, xmin, sh, sl, &q)) continue;
            decided++;
            volatile double d = (double)x - (double)xmin;
            volatile double t = d * scale;
            const double f = std::fmin(std::floor(t), QMAX);
            if ((double)q != f) {
                if (bad++ < 10) printf("MISMATCH x=%a xmin=%a scale=%a q=%u ref=%.0f\n", x, xmin, scale, q, f);
            }
        }
    }
    uint32_t q;
    const float odd[] = {INFINITY, -INFINITY, NAN, 3e38f};
    for (float a : odd)
        for (float b : odd) {
            const bool ok = quantise_fp32(a, b, 1.0f, 0.0f, &q);
            if (ok && !(a - b < 4194304.0f)) bad++;
        }
    printf("cases %lld decided %lld mismatches %lld\n", n, decided, bad);
    return bad != 0;
}
