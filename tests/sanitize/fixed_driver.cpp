/* Runs the host construction of the fixed-point step's constants over lattice
 * speeds inside and outside the range of the kernels, and relaxation times up
 * to both limits; inside the range every constant is its value to 2^-60.  Built
 * with UndefinedBehaviorSanitizer by tests/test_fixed_constants.py.          */
#include <cstdio>

#include "rlb_fixed.cuh"

static int bad = 0;

static void check(const rlb::FxConst& k, long double want, int s) {
    const long double got = ldexpl((long double)k.h, 32 - s) + ldexpl((long double)k.l, 1 - s);
    if (fabsl(got - want) > 4 * ldexpl(1.0L, -60)) ++bad;
}

int main() {
    const double taus[] = {0.5000000000000001, 0.51, 0.8, 1.0, 30.0, 1e6, 1e12};
    const double speeds[] = {1e-150, 0.01, 0.3, 0.57, 0.99, 1.0, 1.1, 1.3, 1.5, 1.7320508, 2.0, 2.1, 10.0, 1e6, 1e150};
    const long double w = 1.0L - ldexpl(1.0L, -54);  // the binary64 weights
    for (double tau : taus)
        for (double c : speeds) {
            const double om = 1.0 / tau;
            const rlb::FxRun k = rlb::make_fx_run(om, c);
            const long double c2 = (long double)c * c;
            if (k.c_l != (float)c || k.three_cl != 3.0 * c || k.m3cl2 != -3.0 * c * c || k.omw != 1.0 - om) ++bad;
            if (!rlb::fx_covers(c)) {
                if (k.kE.h | k.kE1.h | k.k0.h | k.kE0.h) ++bad;
                continue;
            }
            check(k.kE, w * om / (36 * c2), 65);
            check(k.kU, w * om / 12, 65);
            check(k.kS, w * om / 36, 65);
            check(k.k0, w * om * (1 - 2 / (3 * c2)), 62);
            check(k.kE1, w / (36 * c2), 65);
            check(k.kE0, w * (3 - 2 / c2) / 3, 62);
            check(k.kQ, 5.0L / 9, 63);
            check(k.kG, 1.0L / 6, 63);
        }
    printf("%s\n", bad ? "wrong constants" : "ok");
    return bad != 0;
}
