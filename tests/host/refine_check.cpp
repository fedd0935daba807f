// Host-side check of the refinement's stopping decision on synthetic residual
// histories (no GPU).  Prints "ok" and exits 0 on success, else the failing case.
#include <cmath>
#include <cstdio>
#include <vector>

#include "krr_internal.h"

namespace {

// One error component per mode or phenotype: a stationary step multiplies it
// by its own factor; `floor` is the residual that no step removes.
struct Mode {
    double weight, factor;
};

// Runs the decision as the solve does; returns the step it stops at, the
// residual there in *rel.
int run(const std::vector<Mode> &modes, double floor, double level, double tol, double *rel) {
    krr::RefineStall stall;
    double best = INFINITY;
    for (int it = 0; it < 30; ++it) {
        double s = floor * floor;
        for (const Mode &m : modes) {
            const double v = m.weight * std::pow(m.factor, it + 1);
            s += v * v;
        }
        *rel = std::sqrt(s);
        if (*rel <= tol || stall(it, *rel, best, level)) return it;
        best = std::fmin(best, *rel);
    }
    return 30;
}

}  // namespace

int main() {
    const double tol = 1e-7;
    double rel = 0.0;
    // The gain of a step falls when the fast components are gone.  Above the
    // level of FP32 rounding refinement goes on and reaches the tolerance.
    const std::vector<std::vector<Mode>> slow = {
        {{1.0, 0.005}, {0.01, 0.12}},               // two contraction rates
        {{1.0, 1e-3}, {1.0, 1e-3}, {1e-3, 0.3}},    // one slow column among fast ones
        {{1.0, 2e-3}, {1e-2, 0.05}, {1e-4, 0.4}},   // three rates
    };
    for (size_t i = 0; i < slow.size(); ++i)
        for (double level : {0.0, 1e-9, 5e-8, (double)NAN})
            if (run(slow[i], 1e-9, level, tol, &rel) >= 30 || !(rel <= tol)) {
                std::printf("history %d, level %g: stopped at %g\n", (int)i, level, rel);
                return 1;
            }
    // A gain that collapses below that level ends it (3.3e-4, 4.6e-7, 1.2e-7), above it does not.
    const std::vector<Mode> collapse = {{1.0, 3.3e-4}, {7.4e-6, 0.25}};
    if (run(collapse, 0.0, 2.7e-6, tol, &rel) != 2 || run(collapse, 0.0, 2e-8, tol, &rel) != 3 || !(rel <= tol)) {
        std::printf("collapse: %g\n", rel);
        return 2;
    }
    // A step that does not halve the residual ends it at any level.
    if (run({{1.0, 0.01}}, 1e-3, 1e-9, tol, &rel) != 2) {
        std::printf("not halved: %g\n", rel);
        return 3;
    }
    std::printf("ok\n");
    return 0;
}
