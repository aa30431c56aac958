// The Matern covariance of two locations in the plane (Eq. 2) by 64-bit integer arithmetic.
//
// Why: a warp-wide FP64 instruction holds its SM sub-partition for 64 clocks on GB300, an
// integer one for 1 or 2.  The FP64 evaluation (matern.cuh) costs about 28 of them with a closed
// form and 45 with the local polynomials of a general nu; here the squared distance takes four
// (its cancellation needs them) and the rest, from the bits of dx^2 + dy^2 on, is fixed-point
// arithmetic on normalised 64-bit mantissas, about 250 instructions:
//   r = sqrt(q)     s = m y, y the hardware's approximation of 1 / sqrt(m) (24 bits), corrected
//                   by the binomial series of (1 - e)^-1/2, e = 1 - m y^2 formed exactly
//   y = r 0.8 / theta2                      one product (the constant from the host, 64 bits)
//   theta1 e^-x     x = 1.25 y; x log2(e) = n + j / 256 + t: 2^-n in the exponent, theta1 2^(-j/256)
//                   from a table of 64-bit mantissas, e^-(t ln 2) by its Taylor polynomial of
//                   degree 5 (Tang, ACM TOMS 15, 1989, in fixed point; t ln 2 < 2^-8.5)
//   the factor      1 + x, 1 + x + x^2 / 3, or the local polynomial of a general nu by Horner's
//                   rule with its coefficients scaled to a common power of two per interval
// and one rounding to double at the end.  Every intermediate keeps 57 bits or more, so the
// result is closer to exact than the FP64 evaluation's.  The functions compile for the host too.
#pragma once
#include <cstdint>
#include <cstring>

#include "matern_params.h"

#ifdef __CUDACC__
#define EGS_HD __host__ __device__ __forceinline__
#else
#define EGS_HD inline
#endif

namespace egs {
namespace mi {

EGS_HD uint64_t wide(uint32_t a, uint32_t b) { return (uint64_t)a * b; }
EGS_HD int64_t wide_s(int32_t a, int32_t b) { return (int64_t)a * b; }

// The upper 64 bits of a b.
EGS_HD uint64_t mulhi_exact(uint64_t a, uint64_t b)
{
#ifdef __CUDA_ARCH__
    return __umul64hi(a, b);
#else
    return (uint64_t)(((unsigned __int128)a * b) >> 64);
#endif
}

EGS_HD int64_t mulhi_s(int64_t a, int64_t b)
{
#ifdef __CUDA_ARCH__
    return __mul64hi(a, b);
#else
    return (int64_t)(((__int128)a * b) >> 64);
#endif
}

// The first, up to 2 units too small: without the product of the lower halves
// and its carries (an exact one takes about twice the instructions).
EGS_HD uint64_t mulhi(uint64_t a, uint64_t b)
{
    const uint32_t ah = (uint32_t)(a >> 32), al = (uint32_t)a, bh = (uint32_t)(b >> 32), bl = (uint32_t)b;
    return wide(ah, bh) + (wide(ah, bl) >> 32) + (wide(al, bh) >> 32);
}

// a b 2^-64 + add for signed numbers, within 3 units; |a| < 2^62.  b = bh 2^32 + bl with both
// halves signed (split_s).
EGS_HD void split_s(int64_t b, int32_t *bh, int32_t *bl)
{
    *bl = (int32_t)(uint32_t)b;
    *bh = (int32_t)((b - *bl) >> 32);
}
EGS_HD int64_t mulhi_add(int64_t a, int32_t bh, int32_t bl, int64_t add)
{
    const int32_t ah = (int32_t)(a >> 32), al = (int32_t)((uint32_t)a >> 1);
    return add + wide_s(ah, bh) + wide_s((int32_t)(wide_s(al, bh) >> 32), 2) + (int32_t)(wide_s(ah, bl) >> 32);
}

EGS_HD int clz64(uint64_t x)
{
#ifdef __CUDA_ARCH__
    return __clzll((long long)x);
#else
    return __builtin_clzll(x);
#endif
}

EGS_HD uint64_t f64_bits(double x)
{
#ifdef __CUDA_ARCH__
    return (uint64_t)__double_as_longlong(x);
#else
    uint64_t u;
    std::memcpy(&u, &x, 8);
    return u;
#endif
}

EGS_HD double bits_f64(uint64_t u)
{
#ifdef __CUDA_ARCH__
    return __longlong_as_double((long long)u);
#else
    double x;
    std::memcpy(&x, &u, 8);
    return x;
#endif
}

// 1 / sqrt(m), m in [1, 4), to about 22 bits, as an integer in units of 2^-24, 2^23 .. 2^24 - 1.
// mb: the bits of m as a float.
EGS_HD uint32_t rsqrt24(uint32_t mb)
{
#ifdef __CUDA_ARCH__
    float y;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(__uint_as_float(mb)));
    y = fminf(fmaxf(y, 0.5f), 0x1.fffffep-1f);
    return (__float_as_uint(y) & 0x7FFFFFu) | 0x800000u;
#else
    float m;
    std::memcpy(&m, &mb, 4);
    float y = (float)(1.0 / __builtin_sqrt((double)m)) * (1.0f + 0x1p-23f);
    y = y < 0.5f ? 0.5f : (y > 0x1.fffffep-1f ? 0x1.fffffep-1f : y);
    uint32_t u;
    std::memcpy(&u, &y, 4);
    return (u & 0x7FFFFFu) | 0x800000u;
#endif
}

// h 2^e (h > 0) rounded to a double; results below the smallest normal number are 0.
EGS_HD double pack(uint64_t h, int e)
{
    const int lz = clz64(h);
    h <<= lz;
    const int be = e + 63 - lz + 1023;
    if (be <= 0) return 0.0;
    if (be >= 2047) return bits_f64(0x7FF0000000000000ull);
    return bits_f64(((uint64_t)(be - 1) << 52) + (h >> 11) + ((h >> 10) & 1));
}

EGS_HD uint64_t shr(uint64_t x, int s) { return s < 64 ? x >> s : 0; }

// The local polynomials (EGS_MT_NC coefficients a_j per interval, in s in [-1, 1)) as integers:
// coefficient j of an interval is round(a_j 4^j 2^(62 - E)), for Horner's rule in s / 4, with E
// such that no partial value reaches 2^62; E after them.
EGS_HD void scale_interval(const double *a, int64_t *out)
{
    double bound = 0.0, tail = 0.0;
    for (int j = EGS_MT_NC - 1; j >= 0; --j) {
        const double m = (a[j] < 0.0 ? -a[j] : a[j]) * (double)(1 << (2 * j));
        tail = m + 0.25 * tail;
        bound = tail > bound ? tail : bound;
    }
    const int be = (int)((f64_bits(bound) >> 52) & 0x7FF);
    const bool ok = be > 0 && be < 0x7FF;
    const int E = be - 1022;  // bound < 2^E
    for (int j = 0; j < EGS_MT_NC; ++j) {
        const uint64_t b = f64_bits(a[j]);
        const int ex = (int)((b >> 52) & 0x7FF);
        const uint64_t m = ex ? (b & 0xFFFFFFFFFFFFFull) | 0x10000000000000ull : 0;
        const int sh = ex - 1075 + 2 * j + 62 - E;  // a_j 4^j 2^(62 - E) = m 2^sh, sh <= 9
        uint64_t v = sh >= 0 ? m << (sh & 63) : (sh > -64 ? (m + (1ull << (-sh - 1))) >> (-sh) : 0);
        out[j] = ok ? ((b >> 63) ? -(int64_t)v : (int64_t)v) : 0;
    }
    out[EGS_MT_NC] = E;
}

// C for a squared distance q = dx^2 + dy^2.  False if q or the parameters are outside this
// arithmetic's range (q = 0, subnormal or not finite; x beyond e^-x's or the polynomials' range):
// the caller then takes the FP64 evaluation.  itab: the integer polynomials of a general nu.
EGS_HD bool matern_int(const egs_matern_params *P, const int64_t *itab, double q, double *out)
{
    const uint64_t qb = f64_bits(q);
    const int eq = (int)(qb >> 52);
    if ((unsigned)(eq - 1) >= 0x7FEu) return false;
    // sqrt(q) = R 2^(k - 62), R in [2^62, 2^63)
    const int E = eq - 1023, k = E >> 1, odd = E & 1;
    const uint64_t mant = (qb & 0xFFFFFFFFFFFFFull) | 0x10000000000000ull;
    const uint64_t M = mant << (10 + odd);
    const uint32_t Yi = rsqrt24(((uint32_t)(127 + odd) << 23) | ((uint32_t)(mant >> 29) & 0x7FFFFFu));
    const int64_t e = (int64_t)(1ull << 62) - (int64_t)mulhi_exact(M, ((uint64_t)Yi * Yi) << 16);
    const uint64_t S0 = wide((uint32_t)(M >> 32), Yi << 8) + (wide((uint32_t)M, Yi << 8) >> 32);  // M Yi 2^-24, floor
    const int64_t eh = e >> 20;
    const int64_t c = (e >> 1) + ((3 * (eh * eh)) >> 25);
    uint64_t R = S0 + (uint64_t)mulhi_s((int64_t)(S0 >> 1), c * 8);
    R = R < (1ull << 62) ? 1ull << 62 : (R >> 63 ? (1ull << 63) - 1 : R);  // a rounding beyond [1, 2)
    // y = r 0.8 / theta2 = Y 2^(ey - 63), Y in [2^63, 2^64)
    uint64_t Y = mulhi_exact(R << 1, P->iy_m);
    int ey = k + P->iy_e;
    if (Y >> 63) ++ey;
    else Y <<= 1;
    const bool general = P->kind == EGS_MATERN_GENERAL;
    if (ey > (general ? EGS_MT_E0 + EGS_MT_OCT - 1 : 8) || ey < (general ? EGS_MT_E0 : -60)) return false;
    // theta1 e^-x = Er 2^(th1_e - n - 63)
    const uint64_t Z = mulhi_exact(Y, 0xE6D4C9F3B31DECEBull);  // 1.25 / ln 2 in units of 2^-63
    const int sh = ey + 2;
    const uint64_t frac = sh >= 0 ? Z << sh : shr(Z, -sh);
    const int n = sh > 0 ? (int)(Z >> (64 - sh)) : 0;
    const uint64_t V = mulhi(frac << 8, 0xB17217F7D1CF79ACull) >> 8;  // v = t ln 2, units of 2^-64
    const uint64_t V2 = mulhi(V << 8, V << 8);                        // v^2, units of 2^-80
    const uint32_t vh = (uint32_t)(V >> 24), v2h = (uint32_t)(V2 >> 32);
    const uint32_t w = 0x2AAAAAABu - (uint32_t)(((uint64_t)vh * 0x0AAAAAABu) >> 40) +
                       (uint32_t)(((uint64_t)v2h * 0x02222222u) >> 48);  // 1/6 - v/24 + v^2/120
    const uint64_t v3 = (uint64_t)vh * v2h;                              // v^3, units of 2^-88
    const uint64_t Q = V - (V2 >> 17) + (((v3 >> 31) * w) >> 25);        // 1 - e^-v
    const uint64_t Tj = P->exp2_tab[frac >> 56];
    const uint64_t Er = Tj - mulhi(Tj, Q);
    const int ee = P->th1_e - n;
    switch (P->kind) {
    case EGS_MATERN_HALF:
        *out = pack(Er, ee - 63);
        return true;
    case EGS_MATERN_3HALF:
    case EGS_MATERN_5HALF: {
        const uint64_t X = (Y >> 1) + (Y >> 3);  // x = X 2^(ey - 62)
        const int up = ey > 0 ? ey : 0, dn = ey < 0 ? -ey : 0;
        uint64_t A;  // the factor in units of 2^(exA)
        int exA;
        if (P->kind == EGS_MATERN_3HALF) {
            A = ((1ull << 61) >> up) + shr(X, 1 + dn);
            exA = up - 61;
        } else {
            const uint64_t T3 = mulhi(mulhi(X, X), 0x5555555555555555ull);  // x^2 / 3, 2^(2 ey - 60)
            A = ((1ull << 60) >> (2 * up)) + shr(X, 2 + (ey > 0 ? up : dn)) + shr(T3, 2 * dn);
            exA = 2 * up - 60;
        }
        *out = pack(mulhi(A << 1, Er), exA + ee);
        return true;
    }
    default: {
        const int iv = (ey - EGS_MT_E0) * EGS_MT_SUB + ((int)(Y >> 60) & 7);
        const int64_t u = (int64_t)((Y << 4) ^ (1ull << 63)) >> 1;  // s / 4, units of 2^-64
        const int64_t *a = itab + iv * (EGS_MT_NC + 1);
        int32_t uh, ul;
        split_s(u, &uh, &ul);
        int64_t p = a[EGS_MT_NC - 1];
#ifdef __CUDA_ARCH__
#pragma unroll
#endif
        for (int j = EGS_MT_NC - 2; j >= 0; --j) p = mulhi_add(p, uh, ul, a[j]);
        if (p <= 0) return false;
        *out = pack(mulhi((uint64_t)p << 2, Er), (int)a[EGS_MT_NC] + ee - 63);
        return true;
    }
    }
}

}  // namespace mi
}  // namespace egs
