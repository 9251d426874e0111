// Fixed-point pair arithmetic for the FP64-accurate operator: an FP64-class
// dot product on the integer and FP32 pipes.
//
// GB300's FP64 pipe issues 1.7 instructions per clock and SM, its integer
// multiply-add (32 x 32 + 64 -> 64 bits) about 50 and its FP32 FMA 121
// (measured).  A value is a pair (h, l): the 32-bit integer h and the float l
// stand for (h + l) 2^s, with the scale s known to the caller and |l| of the
// order of one unit of h, so a pair holds 30 + 24 bits.  In a product sum
//
//   sum_j (ah_j + al_j)(xh_j + xl_j)
//     = sum_j ah_j xh_j                       one 64-bit integer sum, exact
//     + sum_j (ah_j xl_j + al_j xh_j)         about 2^-31 of it: plain FP32
//     + sum_j al_j xl_j                       below 2^-60 of it: dropped
//
// a term costs one integer multiply-add and two FP32 FMAs; the same term in
// double-float arithmetic (compensated Dot2 on float pairs) costs 12 FP32
// instructions, because every addition of the leading parts needs its
// rounding error, which the integer sum does not have.
//
// The leading sum A is in units of 2^-32 of the result's h (the callers scale
// the constants a so that |A| < 2^62), the FP32 sum B in units of h itself:
// the constants' float parts al and af = (float)ah carry the factor 2^-32.
// Integer additions wrap, so only the results have to be in range, not the
// intermediate sums.
#pragma once

#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>
#include <string.h>

namespace nekgb {
namespace fx {

struct Pair {
    int h;
    float l;
};

struct Acc {
    long long A;
    float B;
};

__host__ __device__ __forceinline__ float bits_f(int b) {
#ifdef __CUDA_ARCH__
    return __int_as_float(b);
#else
    float f;
    memcpy(&f, &b, 4);
    return f;
#endif
}
__host__ __device__ __forceinline__ double bits_d(long long b) {
#ifdef __CUDA_ARCH__
    return __longlong_as_double(b);
#else
    double d;
    memcpy(&d, &b, 8);
    return d;
#endif
}
__host__ __device__ __forceinline__ long long d_bits(double d) {
#ifdef __CUDA_ARCH__
    return __double_as_longlong(d);
#else
    long long b;
    memcpy(&b, &d, 8);
    return b;
#endif
}

__host__ __device__ __forceinline__ long long wrap_add(long long a, long long b) {
    return (long long)((unsigned long long)a + (unsigned long long)b);
}
__host__ __device__ __forceinline__ long long wrap_sub(long long a, long long b) {
    return (long long)((unsigned long long)a - (unsigned long long)b);
}

// acc = (ah + al)(xh + xl) and acc += (ah + al)(xh + xl); xf = (float)xh,
// af = (float)ah 2^-32, al already times 2^-32.
__host__ __device__ __forceinline__ Acc first(int ah, float al, float af, int xh, float xl, float xf) {
    Acc c;
    c.A = (long long)ah * xh;
    c.B = fmaf(af, xl, al * xf);
    return c;
}
__host__ __device__ __forceinline__ void add(Acc &c, int ah, float al, float af, int xh, float xl, float xf) {
    c.A = wrap_add(c.A, (long long)ah * xh);
    c.B = fmaf(af, xl, fmaf(al, xf, c.B));
}

// The accumulated value as a pair.  A carries an offset of half a unit
// (kHalf), so its top word is h rounded to nearest and the low word, less the
// offset, is a fraction in [-1/2, 1/2): a small |l| keeps the rounding
// errors of the FP32 sums of the next product small.
constexpr long long kHalf = 0x80000000ll;
__host__ __device__ __forceinline__ Pair pair_of(long long A, float B) {
    Pair p;
    p.h = (int)(A >> 32);
    p.l = fmaf((float)(int)((unsigned)A ^ 0x80000000u), 0x1p-32f, B);
    return p;
}

// Pair of v with |v| < 2^(emax - 1022) (emax: biased exponent), in units of
// 2^(emax - 1052): |h| < 2^30.  Integer operations only; bits below 2^-32 of
// a unit are dropped.  Values more than 2^62 below the scale become 0.  The
// caller's emax is at least kMinExp, so a subnormal v (whose mantissa has no
// implicit bit) is shifted out.
constexpr int kMinExp = 64;
// An exponent that stands for "not finite" (a NaN or an Inf in an element's input
// or factors), far above every exponent of finite data (below 2^12, as sums of
// them): its values become 0, and Scale makes the results NaN.
constexpr int kNotFinite = 1 << 14;
__host__ __device__ __forceinline__ Pair from_double(double v, int emax) {
    const unsigned long long b = (unsigned long long)d_bits(v);
    const unsigned hi = (unsigned)(b >> 32);
    const unsigned m = (unsigned)((int)hi >> 31);                                 // all ones if negative
    const unsigned long long M = ((((unsigned long long)((hi & 0xfffffu) | 0x100000u)) << 32) | (unsigned)b) << 9;
    int sh = emax - (int)((hi >> 20) & 0x7ffu);
    sh = sh < 63 ? sh : 63;
    const unsigned long long f = M >> sh;                                         // h in the top word
    Pair p;
    p.h = (int)(((unsigned)(f >> 32) ^ m) - m);
    p.l = (float)(unsigned)f * bits_f((int)(0x2f800000u | (m & 0x80000000u)));    // +- 2^-32
    return p;
}

// 2^k as a double, -1022 <= k <= 1023
__host__ __device__ __forceinline__ double pow2(int k) { return bits_d((long long)(k + 1023) << 52); }

// x 2^k (two exact power-of-two factors)
__host__ __device__ __forceinline__ double scale2(double x, int k) {
    k = k < -2040 ? -2040 : (k > 2040 ? 2040 : k);
    const int k1 = k / 2;
    return x * pow2(k1) * pow2(k - k1);
}

// (h + l) 2^so in FP64, rounded once: 2^52 + 2^31 + h and the same for
// rint(l 2^25) are doubles by construction (|l| < 64; worst case 33 for the
// sum of the three partials at n = 16), and two FP64 FMAs scale them, add
// them and take their offsets off: every step but the last is exact.
// Outside +-900 (rest) the caller multiplies the results by a second factor,
// post, which brings the exponent to where it belongs (they then overflow or
// underflow as FP64 does).  The same factor makes the results of an element with
// non-finite data NaN.
struct Scale {
    double f, f2, c;
    int rest;            // what +-900 leaves of so
    __host__ __device__ __forceinline__ void set(int so) {
        const int s = so < -900 ? -900 : (so > 900 ? 900 : so);
        f = pow2(s);
        f2 = pow2(s - 25);
        c = -(4503599627370496.0 + 2147483648.0 + 134217728.0 + 64.0) * f;
        rest = so - s;
    }
    __host__ __device__ __forceinline__ double post() const {
        if (rest > kNotFinite / 4) return bits_d(0x7ff8000000000000ll);
        return pow2(rest < -1022 ? -1022 : (rest > 1023 ? 1023 : rest));
    }
    __host__ __device__ __forceinline__ double operator()(Pair p) const {
#ifdef __CUDA_ARCH__
        const int li = __float2int_rn(p.l * 0x1p25f);
#else
        const int li = (int)rintf(p.l * 0x1p25f);
#endif
        const double mh = bits_d((long long)(0x4330000000000000ull | (unsigned)(p.h ^ 0x80000000)));
        const double ml = bits_d((long long)(0x4330000000000000ull | (unsigned)(li ^ 0x80000000)));
        return fma(ml, f2, fma(mh, f, c));
    }
};

}  // namespace fx
}  // namespace nekgb
