// The integer Matern evaluation (csrc/matern_int.cuh) at large distances, on the CPU against long
// double: the polynomials of a general nu reach to x = 1,280 (their last octave), here those of the
// factor 1 + x + x^2 / 3, which cubic monomials hold exactly up to rounding.  Prints the largest
// relative error (less the conditioning of e^-x), the calls taken and those left to FP64.
#include <cmath>
#include <cstdio>
#include <vector>

#include "matern_int.cuh"

using namespace egs;
typedef long double ld;

int main()
{
    std::vector<double> tab(EGS_MT_DOUBLES, 0.0);
    std::vector<int64_t> itab(EGS_MT_INTS);
    for (int iv = 0; iv < EGS_MT_OCT * EGS_MT_SUB; ++iv) {
        // x = c + h s on the sub-interval
        const ld sc = ldexpl(1.25L, iv / EGS_MT_SUB + EGS_MT_E0);
        const ld c = sc * (1.0L + (iv % EGS_MT_SUB + 0.5L) / EGS_MT_SUB), h = sc * 0.5L / EGS_MT_SUB;
        double *a = &tab[iv * EGS_MT_NC];
        a[0] = (double)(1.0L + c + c * c / 3.0L);
        a[1] = (double)(h + 2.0L * c * h / 3.0L);
        a[2] = (double)(h * h / 3.0L);
        mi::scale_interval(a, &itab[iv * (EGS_MT_NC + 1)]);
    }
    const double theta[3] = {1.7, 0.001, 0.8};
    egs_matern_params P;
    if (egs_matern_params_init(theta, &P)) return 1;
    double worst = 0.0;
    long taken = 0, left = 0, far = 0;
    for (double x = 500.0; x < 1290.0; x += 0.37) {
        const double r = x * theta[1], q = r * r;
        double v;
        if (!mi::matern_int(&P, itab.data(), q, &v)) {
            if (x < 1279.0) ++left;
            continue;
        }
        ++taken;
        const ld xx = sqrtl((ld)q) / (ld)theta[1];
        const ld want = (ld)theta[0] * expl(-xx) * (1.0L + xx + xx * xx / 3.0L);
        if (want < 0x1p-1021L) {
            far += v == 0.0 || v <= 0x1p-1020;
            continue;
        }
        ++far;
        const double err = (double)(fabsl((ld)v - want) / want) - (double)(xx * 0x1p-60L);
        if (err > worst) worst = err;
    }
    std::printf("worst=%.3g taken=%ld left=%ld wrong_far=%ld\n", worst, taken, left, taken - far);
    return 0;
}
