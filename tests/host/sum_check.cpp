// Host-side check of the Build epilogue's sums (no GPU): 128 kernel entries and
// their squares, added in chunks of 16, are as exact as FP64 sums in the order of
// the entries (to the final rounding to FP64, 2^-53).  Over any range the small
// terms of a chunk, at most 2^-22 of its sum, meet FP32 roundings: 2^-48 at most.
// Prints "ok" and exits 0 on success.
#include <cmath>
#include <cstdint>
#include <cstdio>

#include "krr_internal.h"

namespace {

uint64_t g_state = 2024;
double uniform() {  // (0, 1)
    g_state = g_state * 6364136223846793005ull + 1442695040888963407ull;
    return ((double)(g_state >> 11) + 0.5) * 0x1p-53;
}

float entry(int kind) {
    switch (kind) {
        case 0: return (float)std::exp(-0.74 + 0.1 * (uniform() - 0.5));               // gamma = 1 / M
        case 1: return uniform() < 0.02 ? 1.f : (float)std::exp(-6.0 + uniform());      // gamma = 8 / M
        case 2: return (float)(uniform() < 0.15 ? 0.02 * uniform() : std::exp(-9.0 - uniform()));  // cohorts
        case 3: return (float)((2000.0 - std::floor(600.0 + 300.0 * uniform())) / 1000.0);         // IBS
        case 4: return (float)std::floor(20000.0 + 40000.0 * uniform());                // Gram
        case 5: return (float)std::exp(-25.0 * uniform());                              // any range
        default: return 0.f;
    }
}

}  // namespace

int main() {
    for (int kind = 0; kind < 7; ++kind) {
        double e1 = 0.0, e2 = 0.0, f1 = 0.0, f2 = 0.0;
        for (int run = 0; run < 2000; ++run) {
            krr::WideSum w1, w2;
            double d1 = 0.0, d2 = 0.0;
            long double x1 = 0.0L, x2 = 0.0L;  // 64 bits or more
            for (int ch = 0; ch < 8; ++ch) {
                krr::ChunkSum c1, c2;
                for (int e = 0; e < 16; e += 4) {
                    const float v[4] = {entry(kind), entry(kind), entry(kind), entry(kind)};
                    c1.add4(v[0], v[1], v[2], v[3]);
                    c2.add_squares4(v[0], v[1], v[2], v[3]);
                    for (float u : v) {
                        d1 += (double)u;
                        d2 += (double)u * (double)u;
                        x1 += (long double)u;
                        x2 += (long double)u * (long double)u;
                    }
                }
                w1.add(c1);
                w2.add(c2);
            }
            if (x2 == 0.0L) {
                if (w1.value() != 0.0 || w2.value() != 0.0) return 1;
                continue;
            }
            const double r1 = (double)((w1.value() - x1) / x1), r2 = (double)((w2.value() - x2) / x2);
            const double s1 = (double)((d1 - x1) / x1), s2 = (double)((d2 - x2) / x2);
            e1 += r1 * r1, e2 += r2 * r2, f1 += s1 * s1, f2 += s2 * s2;
        }
        e1 = std::sqrt(e1 / 2000), e2 = std::sqrt(e2 / 2000), f1 = std::sqrt(f1 / 2000), f2 = std::sqrt(f2 / 2000);
        std::printf("kind %d: sum %.2e (FP64 %.2e), squares %.2e (FP64 %.2e)\n", kind, e1, f1, e2, f2);
        const double any = kind == 5 ? 0x1p-48 : 0x1p-53;
        if (!(e1 <= f1 + any) || !(e2 <= f2 + any)) return 2;
    }
    std::printf("ok\n");
    return 0;
}
