// Host-side check of the addition that carries its rounding errors on (no
// GPU): every entry stays within its own rounding whatever its neighbours'
// magnitudes, and the errors of a run nearly cancel.  Prints "ok" and exits 0.
#include <cmath>
#include <cstdint>
#include <cstdio>

#include "krr_internal.h"

namespace {

uint64_t g_state = 12345;
double uniform() {  // (0, 1)
    g_state = g_state * 6364136223846793005ull + 1442695040888963407ull;
    return ((double)(g_state >> 11) + 0.5) * 0x1p-53;
}

}  // namespace

int main() {
    // magnitudes of neighbouring entries: equal, 1e5 apart in turn, spread over seven decades
    for (int kind = 0; kind < 3; ++kind) {
        double sum2 = 0.0, plain2 = 0.0;
        for (int run = 0; run < 4000; ++run) {
            float carry = 0.f;
            double sum = 0.0, plain = 0.0;
            for (int k = 0; k < 32; ++k) {
                const double scale = kind == 0 ? 1.0
                                   : kind == 1 ? ((k & 1) ? 1e-4 : 10.0)
                                               : std::pow(10.0, -5.0 + 7.0 * uniform());
                const float s = (float)((uniform() < 0.5 ? -1.0 : 1.0) * (0.5 + uniform()) * scale);
                const float x = (float)((2.0 * uniform() - 1.0) * 1e-3 * scale);
                const double exact = (double)s + (double)x;
                const float f = krr::add_carry(s, x, carry);
                // half an ulp of rounding and at most half an ulp taken in
                if (!(std::fabs((double)f - exact) <= 1.51 * 0x1p-24 * std::fabs(exact))) {
                    std::printf("entry: kind %d, %g for %g\n", kind, (double)f, exact);
                    return 1;
                }
                sum += (double)f - exact;
                plain += (double)(float)(s + x) - exact;
            }
            sum2 += sum * sum;
            plain2 += plain * plain;
        }
        // entries of one magnitude: a third of the sum of independent roundings; never above it
        if (!(sum2 <= (kind == 0 ? 1.0 / 9.0 : 1.0) * plain2)) {
            std::printf("sum: kind %d, %g against %g\n", kind, std::sqrt(sum2), std::sqrt(plain2));
            return 2;
        }
    }
    // zeros take nothing, and a sum that is not finite leaves the carry alone
    float carry = 1e-3f;
    if (krr::add_carry(0.f, 0.f, carry) != 0.f || carry != 1e-3f) return 3;
    if (!(krr::add_carry(INFINITY, 1.f, carry) == INFINITY) || carry != 1e-3f) return 4;
    if (krr::add_carry(NAN, 1.f, carry) == 0.f || carry != 1e-3f) return 5;
    std::printf("ok\n");
    return 0;
}
