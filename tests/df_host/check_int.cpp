// CPU check of the integer Matern evaluation (csrc/matern_int.cuh, which compiles for the host)
// against long double: the closed forms, and the general-nu branch with polynomials of a known
// factor (g = 1 + x + x^2 / 3, interpolated at Chebyshev points in long double and rounded to
// double as the device's builder stores them).  Prints the largest relative errors.
#include <cmath>
#include <cstdio>
#include <random>
#include <vector>

#include "matern_int.cuh"

using namespace egs;
typedef long double ld;

static ld factor(int kind, ld x)
{
    return kind == EGS_MATERN_HALF ? 1.0L : (kind == EGS_MATERN_3HALF ? 1.0L + x : 1.0L + x + x * x / 3.0L);
}

int main()
{
    std::mt19937_64 g(11);
    std::uniform_real_distribution<double> U(0.0, 1.0);
    std::vector<double> tab(EGS_MT_DOUBLES);
    std::vector<int64_t> itab(EGS_MT_INTS);
    const ld pi = acosl(-1.0L);
    for (int iv = 0; iv < EGS_MT_OCT * EGS_MT_SUB; ++iv) {
        constexpr int N = EGS_MT_NC;
        ld val[N], c[N], a[N] = {}, tm[N] = {}, t[N] = {}, tn[N];
        for (int i = 0; i < N; ++i) {
            const ld s = cosl(pi * (i + 0.5L) / N);
            const ld y = ldexpl(1.0L + (iv % EGS_MT_SUB + 0.5L * (1.0L + s)) / EGS_MT_SUB, iv / EGS_MT_SUB + EGS_MT_E0);
            val[i] = factor(EGS_MATERN_5HALF, 1.25L * y);
        }
        for (int k = 0; k < N; ++k) {
            c[k] = 0;
            for (int i = 0; i < N; ++i) c[k] += val[i] * cosl(pi * k * (i + 0.5L) / N);
            c[k] *= (k ? 2.0L : 1.0L) / N;
        }
        tm[0] = 1, t[1] = 1, a[0] = c[0], a[1] = c[1];
        for (int k = 1; k + 1 < N; ++k) {
            for (int j = 0; j < N; ++j) tn[j] = (j ? 2 * t[j - 1] : 0) - tm[j];
            for (int j = 0; j < N; ++j) a[j] += c[k + 1] * tn[j], tm[j] = t[j], t[j] = tn[j];
        }
        for (int j = 0; j < N; ++j) tab[iv * N + j] = (double)a[j];
        mi::scale_interval(&tab[iv * N], &itab[iv * (N + 1)]);
    }
    double worst[4] = {0, 0, 0, 0};
    long taken[4] = {0, 0, 0, 0}, edge = 0;
    const double nus[4] = {0.8, 0.5, 1.5, 2.5};
    for (int kind = 0; kind < 4; ++kind) {
        for (int rep = 0; rep < 40; ++rep) {
            const double theta[3] = {std::exp2(20 * U(g) - 10), std::exp2(16 * U(g) - 10), nus[kind]};
            egs_matern_params P;
            if (egs_matern_params_init(theta, &P)) return 1;
            for (int i = 0; i < 20000; ++i) {
                // x over 2^-14 .. 2^9, some q at the edges of a binade
                double r = theta[1] * std::exp2(23 * U(g) - 14), q = r * r;
                if (i % 50 == 0) q = std::exp2(std::floor(std::log2(q)));
                if (i % 50 == 1) q = std::nextafter(std::exp2(std::floor(std::log2(q))), 0.0);
                double v;
                if (!mi::matern_int(&P, itab.data(), q, &v)) continue;
                ++taken[kind];
                const ld x = sqrtl((ld)q) / (ld)theta[1];
                const ld want = (ld)theta[0] * expl(-x) * factor(kind == 0 ? EGS_MATERN_5HALF : kind, x);
                // the conditioning of e^-x: x is formed to 2^-60 (three truncations at 2^-62)
                const double err = (double)(fabsl((ld)v - want) / want) - (double)(x * 0x1p-60L);
                if (err > worst[kind]) worst[kind] = err;
            }
            double v;
            const double bad[6] = {0.0, 0x1p-1074, 0x1p-1030, INFINITY, NAN, 1e300 * theta[1]};
            for (double q : bad) edge += mi::matern_int(&P, itab.data(), q, &v) ? 1 : 0;
        }
    }
    std::printf("general=%.3g half=%.3g threehalf=%.3g fivehalf=%.3g taken=%ld edge=%ld\n", worst[0], worst[1], worst[2],
                worst[3], taken[0] + taken[1] + taken[2] + taken[3], edge);
    return 0;
}
