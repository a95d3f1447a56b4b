// dg_fixed.h -- fixed-point linear maps on the integer units for the FP64 path.
//
// GB300's FP64 pipe takes one warp instruction per 76 cycles and sub-partition (measured; a
// conversion between FP64 and FP32 or an integer costs 64), a 32 x 32 + 64 bit multiply-add
// (IMAD.WIDE) 2.4.  The constant linear maps of the scheme (volume term, traces, lift, cell
// average) therefore run in fixed point: the values of one component of one cell share an
// exponent, and a product of a value and a coefficient is three IMAD.WIDE.
//
// A value is x = v 2^(E - 1081), E the largest biased FP64 exponent of the values that share
// it, |v| < 2^59, held as v = h 2^28 + l (0 <= l < 2^28); a coefficient is c = C 2^-k, C = H 2^28
// + L (-2^27 <= L < 2^27).  Sums of products keep the high and the cross products,
//     sum v C = 2^56 (sum h H + 2^-28 sum (h L + l H)) + O(2^55 sqrt(terms)),
// so a map's result carries an absolute error of about 2^-60 of its largest value times the sum
// of its coefficients' magnitudes, where the FP64 chain of fused multiply-adds it replaces has
// 2^-53 of its partial sums.  Every accumulator fits 64 bits for sum |C| <= 2^58 and at most 16
// terms: |sum h H| <= 2^31 2^30, |sum h L| <= 16 2^31 2^27, |sum l H| <= 2^28 2^30.
//
// Host and device compile the same functions (the host form is what the accuracy tests run).
#pragma once

#include <math.h>
#include <stdint.h>
#include <string.h>

namespace crkdg {

// limbs of a fixed-point value or coefficient
struct alignas(8) Fx {
    int h, l;
};

#ifdef __CUDACC__
#define CRKDG_HD __host__ __device__ __forceinline__
#else
#define CRKDG_HD inline
#endif

CRKDG_HD unsigned long long fx_bits(double x) {
#ifdef __CUDA_ARCH__
    return (unsigned long long)__double_as_longlong(x);
#else
    unsigned long long u;
    memcpy(&u, &x, 8);
    return u;
#endif
}
CRKDG_HD double fx_from_bits(unsigned long long u) {
#ifdef __CUDA_ARCH__
    return __longlong_as_double((long long)u);
#else
    double x;
    memcpy(&x, &u, 8);
    return x;
#endif
}

// biased exponent of x (0 for zero and subnormal numbers)
CRKDG_HD int fx_exp(double x) { return (int)(fx_bits(x) >> 52) & 0x7ff; }

// x in units of 2^(E - 1081), E >= fx_exp(x); rounded down, zero exactly zero
CRKDG_HD Fx fx_of(double x, int E) {
    const unsigned long long b = fx_bits(x);
    const int e = (int)(b >> 52) & 0x7ff;
    long long m = (long long)(((b & 0xfffffffffffffull) | 0x10000000000000ull) << 6);
    if ((long long)b < 0) m = -m;
    if (e == 0) m = 0;
    const int d = E - e;
    m >>= d > 63 ? 63 : d;
    Fx r;
    r.h = (int)(m >> 28);
    r.l = (int)m & 0xfffffff;
    return r;
}

// sums of products
struct FxSum {
    long long hh, mid;
};
CRKDG_HD void fx_mac(FxSum &s, const Fx &v, const Fx &c) {
    s.hh += (long long)v.h * c.h;
    s.mid += (long long)v.h * c.l;
    s.mid += (long long)v.l * c.h;
}
// the sum in units of 2^56 2^(E - 1081) 2^-k
CRKDG_HD long long fx_sum(const FxSum &s) { return s.hh + (s.mid >> 28); }

// x 2^sh as FP64, rounded to nearest.  The result's exponent must be in the normal range.
CRKDG_HD double fx_double(long long x, int sh) {
#ifdef __CUDA_ARCH__
    const double r = __ll2double_rn(x);
#else
    const double r = (double)x;
#endif
    return x == 0 ? 0.0 : fx_from_bits(fx_bits(r) + ((unsigned long long)(long long)sh << 52));
}
// the shift of a sum of values with exponent E and coefficients scaled by 2^k
CRKDG_HD int fx_shift(int E, int k) { return E - 1025 - k; }

// coefficient c scaled by 2^k, |c| 2^k < 2^58 (host)
inline Fx fx_coef(double c, int k) {
    const long long C = llrint(ldexp(c, k));
    Fx r;
    r.h = (int)((C + (1ll << 27)) >> 28);
    r.l = (int)(C - ((long long)r.h << 28));
    return r;
}

}  // namespace crkdg
