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

// x 2^sh as FP64, rounded to nearest (below 2^-1022 zero).  The result must not overflow.
CRKDG_HD double fx_double(long long x, int sh) {
#ifdef __CUDA_ARCH__
    const double r = __ll2double_rn(x);
    const int hi = __double2hiint(r), e = (hi >> 20) & 0x7ff;
    const bool z = e == 0 || e + sh <= 0;
    return __hiloint2double(z ? 0 : hi + sh * 0x100000, z ? 0 : __double2loint(r));
#else
    const double r = (double)x;
    const int e = fx_exp(r);
    return e == 0 || e + sh <= 0 ? 0.0 : fx_from_bits(fx_bits(r) + ((unsigned long long)(long long)sh << 52));
#endif
}
// the shift of a sum of values with exponent E and coefficients scaled by 2^k
CRKDG_HD int fx_shift(int E, int k) { return E - 1025 - k; }

// ----------------------------------------------------------------------- Euler fluxes
//
// The nonlinear part on the integer units: a value is m 2^(x - 61), m a signed 64-bit mantissa
// (62 bits from an FP64 number), so a product is three IMAD.WIDE and a shift where FP64 takes
// its pipe 76 cycles, and keeps about 60 bits.

// 31-bit limbs of a mantissa |m| < 2^62
struct Limb {
    int h, l;
};
CRKDG_HD Limb fx_limb(long long m) { return Limb{(int)(m >> 31), (int)m & 0x7fffffff}; }
// a b 2^-62 (value exponents: x_a + x_b + 1), within 2 units
CRKDG_HD long long fx_mul(const Limb &a, const Limb &b) {
    long long t = (long long)a.h * b.l;
    t += (long long)a.l * b.h;
    return (long long)a.h * b.h + (t >> 31);
}
// a b 2^-61 (value exponents: x_a + x_b), for |a b| < 2^124: up to 63 bits
CRKDG_HD long long fx_mul_wide(const Limb &a, const Limb &b) {
    long long t = (long long)a.h * b.l;
    t += (long long)a.l * b.h;
    return 2 * ((long long)a.h * b.h) + (t >> 30);
}
// m 2^-s, s >= 0 (rounded down)
CRKDG_HD long long fx_shr(long long m, int s) { return m >> (s > 63 ? 63 : s); }

// mantissa of x (exponent fx_exp(x) - 1023); zero and subnormal numbers give zero
CRKDG_HD long long fx_mant(double x) {
    const unsigned long long b = fx_bits(x);
    long long m = (long long)(((b & 0xfffffffffffffull) | 0x10000000000000ull) << 9);
    if ((long long)b < 0) m = -m;
    if (((b >> 52) & 0x7ff) == 0) m = 0;
    return m;
}

// 2^122 / M for M in [2^61, 2^62): the FP32 reciprocal of M's leading bits (2^-22), then
// r (1 + e + e^2) with e = 1 - M r to 2^-60.
CRKDG_HD long long fx_recip(long long M) {
    const unsigned fb = 0x3f800000u | ((unsigned)(M >> 38) & 0x7fffffu);
#ifdef __CUDA_ARCH__
    float y;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(__uint_as_float(fb)));
    const int r0 = __float2int_rn(y * 1073741824.0f);
#else
    float f;
    memcpy(&f, &fb, 4);
    const int r0 = (int)lrintf((1.0f / f) * 1073741824.0f);
#endif
    const Limb m = fx_limb(M);
    long long e = (1ll << 60) - (long long)m.h * r0;
    e -= ((long long)m.l * r0) >> 31;
    const int eh = (int)(e >> 8);  // |e| < 2^38
    e += ((long long)eh * eh) >> 44;
    const long long w = (long long)r0 * (int)(e >> 8) + (((long long)r0 * ((int)e & 255)) >> 8);
    return ((long long)r0 << 31) + (w >> 21);
}

// Mantissa and exponent (m 2^(xr - 61), 2^60 <= m <= 2^61) of the root of v 2^(x - 61), v >= 0: with f the
// value over an even power of two in [1, 4), y the FP32 reciprocal root of its leading bits (e = 1 - f y^2
// below 2^-21) and t = f y, t (1 + e/2 + 3 e^2 / 8), within about 2^-57.  Eight IMAD.WIDE, where FP64's root
// holds its pipe for about 690 cycles.
CRKDG_HD long long fx_root(long long v, int x, int &xr) {
    if (v <= 0) {
        xr = -4000;
        return 0;
    }
#ifdef __CUDA_ARCH__
    const int z = __clzll(v);
#else
    const int z = __builtin_clzll((unsigned long long)v);
#endif
    const long long M = v << (z - 1);    // [2^62, 2^63)
    const int e2 = x - 61 - z + 1 + 62;  // the value is (M 2^-62) 2^e2
    const int odd = e2 & 1, h = (e2 - odd) >> 1;
    const unsigned fb = (0x3f800000u + ((unsigned)odd << 23)) | ((unsigned)(M >> 39) & 0x7fffffu);
#ifdef __CUDA_ARCH__
    float y;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(__uint_as_float(fb)));
    const int y0 = __float2int_rn(y * 1073741824.0f);
#else
    float f;
    memcpy(&f, &fb, 4);
    const int y0 = (int)lrintf((1.0f / sqrtf(f)) * 1073741824.0f);
#endif
    const long long a = M >> (2 - odd);  // f 2^60
    const int ah = (int)(a >> 31), al = (int)a & 0x7fffffff;
    const long long t = (((long long)ah * y0) << 1) + (((long long)al * y0) >> 30);
    const int th = (int)(t >> 31), tl = (int)t & 0x7fffffff;
    const long long e = (1ll << 60) - ((((long long)th * y0) << 1) + (((long long)tl * y0) >> 30));
    const int eh = (int)(e >> 8);
    const long long c = (e >> 1) + ((3 * (((long long)eh * eh) >> 44)) >> 3);
    const int ch = (int)(c >> 8), cl = (int)c & 255;
    xr = h + 1;
    return t + (((long long)th * ch) >> 21) + (((long long)th * cl) >> 29) + (((long long)tl * ch) >> 52);
}

// gamma - 1 and gamma as mantissas: g1 2^-62 and g 2^(-61)
struct FxGas {
    Limb g1, g;
};

// Everything the fluxes of one state share.  Exponents are those of the values (m 2^(x - 61));
// q[d] = m_d w_d, c = m_x w_y, p and H = E + p share the exponent X (H halved: X + 1).
template <int DIM>
struct FxPoint {
    long long m[DIM], w[DIM], q[DIM], c, p, hh, r;
    int xm[DIM], xw[DIM], xr, X;
};
constexpr int kFxNone = -4000;  // exponent of a zero

// For rho > 0, E > 0, exponents below the overflow bounds (fx_state) and gamma < 2.
template <int DIM>
CRKDG_HD void fx_point(const double *u, const FxGas &gas, FxPoint<DIM> &o) {
    o.xr = fx_exp(u[0]) - 1023;
    o.r = fx_recip(fx_mant(u[0]));
    const Limb R = fx_limb(o.r);
    const int xe = fx_exp(u[DIM + 1]) - 1023;
    o.X = xe;
    Limb lm[DIM], lw[DIM];
    int xq[DIM];
#pragma unroll
    for (int d = 0; d < DIM; ++d) {
        const int e = fx_exp(u[1 + d]);
        o.xm[d] = e == 0 ? kFxNone : e - 1023;
        o.m[d] = fx_mant(u[1 + d]);
        lm[d] = fx_limb(o.m[d]);
        o.w[d] = fx_mul_wide(lm[d], R);  // R <= 2^61: below 2^62
        o.xw[d] = o.xm[d] - o.xr;
        lw[d] = fx_limb(o.w[d]);
        xq[d] = o.xm[d] + o.xw[d] + 1;
        o.X = o.X > xq[d] ? o.X : xq[d];
    }
    long long k = 0;
#pragma unroll
    for (int d = 0; d < DIM; ++d) {
        o.q[d] = fx_shr(fx_mul(lm[d], lw[d]), o.X - xq[d]);
        k += o.q[d];
    }
    o.c = 0;
    if (DIM == 2) o.c = fx_shr(fx_mul(lm[0], lw[DIM - 1]), o.X - (o.xm[0] + o.xw[DIM - 1] + 1));
    const long long E = fx_shr(fx_mant(u[DIM + 1]), o.X - xe);
    o.p = fx_mul(fx_limb(E - (k >> 1)), gas.g1);
    o.hh = (E + o.p) >> 1;
}

// (E + p) w_d, exponent X + xw[d] + 1, up to 63 bits
template <int DIM>
CRKDG_HD long long fx_energy_flux(const FxPoint<DIM> &o, int d) {
    return fx_mul_wide(fx_limb(o.hh), fx_limb(DIM == 2 && d == 1 ? o.w[DIM - 1] : o.w[0]));
}

// limbs (dg_fixed's 59 bits) of m 2^(x - 61) in units of 2^(E - 1081), E - 1023 >= x (and one more
// for |m| >= 2^62)
CRKDG_HD Fx fx_limbs(long long m, int x, int E) {
    const long long v = fx_shr(m, E - 1023 - x + 3);
    Fx r;
    r.h = (int)(v >> 28);
    r.l = (int)v & 0xfffffff;
    return r;
}
// m 2^(x - 61) as FP64
CRKDG_HD double fx_value(long long m, int x) { return fx_double(m, x - 61); }

// coefficient c scaled by 2^k, |c| 2^k < 2^58 (host)
inline Fx fx_coef(double c, int k) {
    const long long C = llrint(ldexp(c, k));
    Fx r;
    r.h = (int)((C + (1ll << 27)) >> 28);
    r.l = (int)(C - ((long long)r.h << 28));
    return r;
}

}  // namespace crkdg
