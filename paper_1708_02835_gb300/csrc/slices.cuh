// Exact BF16 slicing of operand rows for the FP64-accurate tensor-core
// products of ozaki.cu (error-free splitting after Ozaki, Ogita, Oishi and
// Rump, Numer. Algorithms 59 (2012)).  A row x of length K <= 1024 with
// |x| < 2^e gets the scale s = 2^(e-7) and five slices q_1..q_5: the balanced
// base-128 digits of x / s rounded to a multiple of 2^-28, every q_i an integer
// of at most 8 bits times 2^{-7(i-1)} (exact in BF16), so that
// x = s (q_1 + ... + q_5) up to s 2^-29.  Slice i of a row goes to
// dst[i * slice_stride + c].  One warp per row.
#pragma once
#include <cuda_bf16.h>

namespace egs {

constexpr int kSlices = 5;

// Returns e (|x| < 2^e for every entry of the row; 0 for a zero row).  A row
// with an infinity or a NaN becomes NaN slices.
// Integer arithmetic throughout: |x| < 2^e, f = x 2^(35 - e) rounded, its five balanced digits in
// base 128 (the conversions and rounding of an FP64 version run on the FP64 pipe, 64 clocks a
// warp and sub-partition each: 100 us for a 512 x 512 tile, 12 us so).  Lanes take two
// consecutive columns; K is a multiple of 64.
__device__ __forceinline__ void mant_exp(double x, unsigned long long &m, int &ex, bool &neg)
{
    const unsigned long long u = (unsigned long long)__double_as_longlong(x);
    ex = (int)((u >> 52) & 0x7FF);
    m = (u & 0xFFFFFFFFFFFFFull) | (ex ? 0x10000000000000ull : 0ull);
    ex = (ex ? ex : 1) - 1075;
    neg = (u >> 63) != 0;
}
__device__ __forceinline__ void mant_exp(float x, unsigned long long &m, int &ex, bool &neg)
{
    const unsigned u = __float_as_uint(x);
    ex = (int)((u >> 23) & 0xFF);
    m = (u & 0x7FFFFFu) | (ex ? 0x800000u : 0u);
    ex = (ex ? ex : 1) - 150;
    neg = (u >> 31) != 0;
}

// The biased exponent of |x| (0: zero or subnormal), and from a row's largest one the e with
// |x| < 2^e (a row of zeros: 0).
__device__ __forceinline__ unsigned exp_bits(double x) { return ((unsigned)__double2hiint(x) >> 20) & 0x7FF; }
__device__ __forceinline__ unsigned exp_bits(float x) { return (__float_as_uint(x) >> 23) & 0xFF; }
template <typename E>
__device__ __forceinline__ int slice_exp(unsigned mh)
{
    return mh == 0 ? 0 : (int)mh - (sizeof(E) == 8 ? 1022 : 126);
}

// The BF16 bits of the five slices of x.
template <typename E>
__device__ __forceinline__ void digits5(E x, int e, unsigned (&d)[kSlices])
{
    unsigned long long m;
    int ex;
    bool neg;
    mant_exp(x, m, ex, neg);
    const int sh = e - 35 - ex;  // f = m 2^-sh
    long long f = sh <= 0 ? (long long)(m << (-sh & 63)) : (sh < 60 ? (long long)((m + (1ull << (sh - 1))) >> sh) : 0);
    if (neg) f = -f;
#pragma unroll
    for (int i = kSlices - 1; i >= 0; --i) {
        int q;
        if (i > 0) {
            q = (int)((f + 64) & 127) - 64;
            f = (f - q) >> 7;
        } else {
            q = (int)f;
        }
        const float v = __int_as_float(0x4B400000 + q) - 12582912.0f;  // (float)q, |q| <= 128
        d[i] = __float_as_uint(v * __int_as_float((127 - 7 * i) << 23)) >> 16;  // exact: 8 significant bits
    }
}

template <typename E>
__device__ __forceinline__ int slice_row(const E *src, int K, __nv_bfloat16 *__restrict__ dst, size_t slice_stride,
                                         double *scale)
{
    const int lane = threadIdx.x & 31;
    E x[32];
    unsigned mh = 0;  // largest biased exponent
#pragma unroll
    for (int j = 0; j < 16; ++j) {
        const int c = 2 * lane + 64 * j;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            x[2 * j + h] = c < K ? src[c + h] : (E)0;
            mh = max(mh, exp_bits(x[2 * j + h]));
        }
    }
    mh = __reduce_max_sync(0xffffffffu, mh);
    const int e = slice_exp<E>(mh);  // |x| < 2^e
    const bool bad = mh == (sizeof(E) == 8 ? 0x7FFu : 0xFFu);
    if (lane == 0) *scale = ldexp(1.0, e - 7);
#pragma unroll
    for (int j = 0; j < 16; ++j) {
        const int c = 2 * lane + 64 * j;
        if (c < K) {
            unsigned d0[kSlices], d1[kSlices];
            digits5(x[2 * j], e, d0);
            digits5(x[2 * j + 1], e, d1);
#pragma unroll
            for (int i = 0; i < kSlices; ++i)
                *reinterpret_cast<unsigned *>(dst + (size_t)i * slice_stride + c) = bad ? 0x7FC07FC0u : d0[i] | (d1[i] << 16);
        }
    }
    return e;
}

}  // namespace egs
