// dg_core.cuh -- device code of the FP64 cRKDG path (arXiv 2412.16002).
//
// Included by exactly one translation unit per dimension (dg_1d.cu, dg_2d.cu),
// each of which owns its copy of the constant tables.
//
// Work decomposition: one thread per (cell, node), whole cells per warp (CfgW), so that
// every exchange inside a cell is warp-synchronous.  The line operators (volume term,
// traces, lift, S_K interpolation) exchange node data through shared memory.  Per-cell
// reductions (min/max over S_K) are taken by one leader thread per cell in a fixed
// order, so every result is deterministic.
//
// Nodal Q^k form of the operators (collocation at the Gauss points, exact
// diagonal mass matrix), per x-line of a cell with traces u_L = sum_a l_a(-1) u_a,
// u_R = sum_a l_a(+1) u_a:
//   G_a = (2/h) [ sum_q Dhat[a][q] f_q - l_a(+1)/w_a f(u_R) + l_a(-1)/w_a f(u_L) ]
// (Sec. 2.1 with the (k+1)-point Gauss rule); in 2D the y-lines add the same
// term.  F replaces f(u_R), f(u_L) by the Lax--Friedrichs flux (eq. dxDG), so
// F = G + lift(fhat - f(u_int)); the final kernel adds exactly that correction.
#pragma once

#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include "dg_fixed.h"
#include "dg_types.h"

namespace crkdg {

static __constant__ NodalTables c_tab[3];  // n = 2, 3, 4

// ----------------------------------------------------------------------------- helpers

__device__ __forceinline__ unsigned long long dbits(double x) { return (unsigned long long)__double_as_longlong(x); }
__device__ __forceinline__ double bitsd(unsigned long long u) { return __longlong_as_double((long long)u); }
// order-preserving map of a double onto uint64 (for atomicMin over signed values)
__device__ __forceinline__ unsigned long long ordbits(double x) {
    unsigned long long u = dbits(x);
    return (u >> 63) ? ~u : (u | 0x8000000000000000ull);
}

// Comparisons and min/max that need no FP64 arithmetic run on the integer units: the
// FP64 pipe of this part takes one warp instruction per 64 cycles whatever the number
// of active lanes, while a 64-bit integer compare-and-select costs a few ALU issues.
// Keys of +inf and -inf under ordbits.
constexpr unsigned long long kKeyPosInf = 0xfff0000000000000ull;
constexpr unsigned long long kKeyNegInf = 0x000fffffffffffffull;
// inverse of ordbits
__device__ __forceinline__ double ordbits_inv(unsigned long long k) {
    return bitsd((k >> 63) ? (k & 0x7fffffffffffffffull) : ~k);
}
// x != 0.0 on the integer units (NaN counts as non-zero, as for the comparison)
__device__ __forceinline__ bool nonzero_bits(double x) { return (dbits(x) << 1) != 0ull; }
__device__ __forceinline__ bool isnan_bits(double x) {
    return (dbits(x) & 0x7fffffffffffffffull) > 0x7ff0000000000000ull;
}
__device__ __forceinline__ unsigned long long umin64(unsigned long long a, unsigned long long b) { return a < b ? a : b; }
__device__ __forceinline__ unsigned long long umax64(unsigned long long a, unsigned long long b) { return a > b ? a : b; }
// x > 0.0 (false for NaN)
__device__ __forceinline__ bool positive_bits(double x) {
    long long b = (long long)dbits(x);
    return b > 0ll && b <= 0x7ff0000000000000ll;
}
// x >= y for y > 0 (false when x is NaN)
__device__ __forceinline__ bool ge_pos_bits(double x, double y) {
    long long b = (long long)dbits(x);
    return b >= (long long)dbits(y) && b <= 0x7ff0000000000000ll;
}
// t < 1.0 for t in [0, 1] (a limiter's scaling factor)
__device__ __forceinline__ bool below_one(double t) { return (dbits(t) & 0x7fffffffffffffffull) < 0x3ff0000000000000ull; }
// fmax of two non-negative doubles (a NaN operand is ignored, as by fmax)
__device__ __forceinline__ double fmax_nonneg(double a, double b) {
    if (isnan_bits(a)) return b;
    if (isnan_bits(b)) return a;
    return bitsd(umax64(dbits(a), dbits(b)));
}

// x / 2 on the integer units
__device__ __forceinline__ double half_of(double x) {
    const unsigned e = (unsigned)(dbits(x) >> 52) & 0x7ffu;
    return e > 1u && e < 0x7ffu ? bitsd(dbits(x) - (1ull << 52)) : 0.5 * x;
}

// x truncated towards zero to FP32 on the integer units (a conversion instruction takes the FP64
// pipe 64 cycles): below 2^-126 it is zero, beyond the FP32 range infinite (NaN included).
__device__ __forceinline__ float trunc_f(double x) {
    const unsigned hi = (unsigned)__double2hiint(x), lo = (unsigned)__double2loint(x);
    const unsigned mag = hi & 0x7fffffffu;
    unsigned f = __funnelshift_l(lo, mag - (896u << 20), 3);
    if (mag < (897u << 20)) f = 0u;
    if (mag >= (1151u << 20)) f = 0x7f800000u;
    return __uint_as_float(f | (hi & 0x80000000u));
}

// 1/x by the Newton-Raphson iteration r <- r + r (1 - x r) (quadratic convergence) from
// the hardware's approximate reciprocal (rcp.approx.ftz.f64); two steps reach double
// precision (within an ulp of the rounded quotient).  Arguments outside [2^-1000,
// 2^1001) in magnitude (zero, subnormal, huge, inf, NaN) take the IEEE division.  On this
// part a dependent FP64 operation costs 64 cycles and the IEEE reciprocal about seven.
__device__ __forceinline__ double recip_nr(double x) {
    const unsigned e = (unsigned)(dbits(x) >> 52) & 0x7ffu;
    if (e < 1023u - 1000u || e > 1023u + 1000u) return 1.0 / x;
    double r;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(x));
    double t = fma(-x, r, 1.0);
    r = fma(r, t, r);
    t = fma(-x, r, 1.0);
    return fma(r, t, r);
}

// theta = num/den clamped to [0, 1]; a non-positive denominator gives 0
__device__ __forceinline__ double ratio01(double num, double den) {
    if (!(den > 0.0)) return 0.0;
    double t = num * recip_nr(den);
    if (!(t >= 0.0)) t = 0.0;
    return t > 1.0 ? 1.0 : t;
}

// ----------------------------------------------------------------------------- physics


// Euler flux . e_dir and spectral radius given ri = 1/rho, written with explicit
// roundings (fma, __dmul_rn, __dadd_rn): the compiler cannot contract them
// differently where they are inlined, so a trace's flux stored by the inner kernel
// equals, bit for bit, the same flux recomputed by the final kernel.
template <int DIM>
__device__ __forceinline__ void euler_flux_ri(const Params &P, const double *u, int dir, double ri, double *f) {
    const double gm1 = P.gamma - 1.0;
    if constexpr (DIM == 1) {
        double w = __dmul_rn(u[1], ri);
        double p = __dmul_rn(gm1, fma(-0.5 * u[1], w, u[2]));
        f[0] = u[1];
        f[1] = fma(u[1], w, p);
        f[2] = __dmul_rn(__dadd_rn(u[2], p), w);
    } else {
        double wx = __dmul_rn(u[1], ri), wy = __dmul_rn(u[2], ri);
        double p = __dmul_rn(gm1, fma(-0.5, fma(u[1], wx, __dmul_rn(u[2], wy)), u[3]));
        double wd = dir == 0 ? wx : wy;
        f[0] = u[1 + dir];
        f[1] = dir == 0 ? fma(u[1], wd, p) : __dmul_rn(u[1], wd);
        f[2] = dir == 1 ? fma(u[2], wd, p) : __dmul_rn(u[2], wd);
        f[3] = __dmul_rn(__dadd_rn(u[3], p), wd);
    }
}
template <int DIM>
__device__ __forceinline__ double euler_speed_ri(const Params &P, const double *u, int dir, double ri) {
    double kin = DIM == 1 ? __dmul_rn(u[1], u[1]) : fma(u[1], u[1], __dmul_rn(u[2], u[2]));
    double p = __dmul_rn(P.gamma - 1.0, fma(-0.5 * kin, ri, u[DIM + 1]));
    double c2 = __dmul_rn(__dmul_rn(P.gamma, p), ri);
    double c = positive_bits(c2) ? sqrt(c2) : 0.0;
    return __dadd_rn(fabs(__dmul_rn(u[1 + dir], ri)), c);
}

// flux f(u) . e_dir  (eq. claws; Euler eq. Euler, Euler-2)
template <int PHYS, int DIM>
__device__ __forceinline__ void flux_dir(const Params &P, const double *u, int dir, double *f) {
    if constexpr (PHYS == PH_ADV) {
        f[0] = (dir == 0 ? P.velx : P.vely) * u[0];
    } else if constexpr (PHYS == PH_BURG) {
        f[0] = 0.5 * u[0] * u[0];
    } else {
        euler_flux_ri<DIM>(P, u, dir, recip_nr(u[0]), f);
    }
}

// both directions with one reciprocal (2D)
template <int PHYS>
__device__ __forceinline__ void flux_xy(const Params &P, const double *u, double *fx, double *fy) {
    if constexpr (PHYS == PH_ADV) {
        fx[0] = P.velx * u[0];
        fy[0] = P.vely * u[0];
    } else if constexpr (PHYS == PH_BURG) {
        fx[0] = fy[0] = 0.5 * u[0] * u[0];
    } else {
        const double ri = recip_nr(u[0]);
        const double wx = __dmul_rn(u[1], ri), wy = __dmul_rn(u[2], ri);
        const double p = __dmul_rn(P.gamma - 1.0, fma(-0.5, fma(u[1], wx, __dmul_rn(u[2], wy)), u[3]));
        const double ep = __dadd_rn(u[3], p);
        fx[0] = u[1];
        fx[1] = fma(u[1], wx, p);
        fx[2] = __dmul_rn(u[2], wx);
        fx[3] = __dmul_rn(ep, wx);
        fy[0] = u[2];
        fy[1] = __dmul_rn(u[1], wy);
        fy[2] = fma(u[2], wy, p);
        fy[3] = __dmul_rn(ep, wy);
    }
}

// spectral radius of df/du . e_dir (alpha of the LF flux, a0 of Sec. 2.1)
template <int PHYS, int DIM>
__device__ __forceinline__ double speed_dir(const Params &P, const double *u, int dir) {
    if constexpr (PHYS == PH_ADV) {
        return fabs(dir == 0 ? P.velx : P.vely);
    } else if constexpr (PHYS == PH_BURG) {
        return fabs(u[0]);
    } else {
        return euler_speed_ri<DIM>(P, u, dir, recip_nr(u[0]));
    }
}

// flux_dir and speed_dir given the reciprocal ri = 1/rho of the state (Euler; other
// fluxes ignore it): the same values as flux_dir and speed_dir, one division fewer
// when a state needs both.
template <int PHYS, int DIM>
__device__ __forceinline__ void flux_dir_ri(const Params &P, const double *u, int dir, double ri, double *f) {
    if constexpr (PHYS != PH_EULER) {
        flux_dir<PHYS, DIM>(P, u, dir, f);
    } else {
        euler_flux_ri<DIM>(P, u, dir, ri, f);
    }
}
template <int PHYS, int DIM>
__device__ __forceinline__ double speed_dir_ri(const Params &P, const double *u, int dir, double ri) {
    if constexpr (PHYS != PH_EULER) {
        return speed_dir<PHYS, DIM>(P, u, dir);
    } else {
        return euler_speed_ri<DIM>(P, u, dir, ri);
    }
}
template <int PHYS>
__device__ __forceinline__ double recip_rho(const double *u) {
    if constexpr (PHYS == PH_EULER) return recip_nr(u[0]);
    return 0.0;
}
// both for one state; returns the spectral radius
template <int PHYS, int DIM>
__device__ __forceinline__ double flux_speed_dir(const Params &P, const double *u, int dir, double *f) {
    double ri = recip_rho<PHYS>(u);
    flux_dir_ri<PHYS, DIM>(P, u, dir, ri, f);
    return speed_dir_ri<PHYS, DIM>(P, u, dir, ri);
}

// Largest exponent of a state's components (and smallest of the density) that the integer forms
// take: products of three such values and their differences stay far from overflow.  Small
// momenta and energies need no bound; results below 2^-1022 become zero.
constexpr int kFxExpLo = 1023 - 150, kFxExpHi = 1023 + 150;
// Binades below a cell's largest value to which sums of values with its exponent (59 bits, six roundings of 2^-58)
// are as accurate as FP64's (2^-53): the errors are 0.8 units at 3, 2.4 at 4, 6.1 at 5, FP64's 0.8 (Euler Q^2).
constexpr int kFxKeep = 3;
// an Euler state that fx_point takes
template <int DIM>
__device__ __forceinline__ bool fx_state(const double *u) {
    bool ok = positive_bits(u[0]) && positive_bits(u[DIM + 1]) && fx_exp(u[0]) >= kFxExpLo;
#pragma unroll
    for (int c = 0; c < DIM + 2; ++c) ok = ok && fx_exp(u[c]) <= kFxExpHi;
    return ok;
}

// Normal flux (FP64) of direction dir from the shared parts of a state, and its spectral radius.
template <int DIM>
__device__ __forceinline__ void fx_face_flux(const FxPoint<DIM> &o, const double *u, int dir, double *f) {
    f[0] = u[1 + dir];
    if constexpr (DIM == 1) {
        f[1] = fx_value(o.q[0] + o.p, o.X);
        f[2] = fx_value(fx_energy_flux<DIM>(o, 0), o.X + o.xw[0] + 1);
    } else {
        const double n = fx_value((dir ? o.q[1] : o.q[0]) + o.p, o.X), t = fx_value(o.c, o.X);
        f[1] = dir ? t : n;
        f[2] = dir ? n : t;
        f[3] = fx_value(fx_energy_flux<DIM>(o, dir), o.X + (dir ? o.xw[1] : o.xw[0]) + 1);
    }
}
template <int DIM>
__device__ __forceinline__ double fx_face_speed(const FxGas &gas, const FxPoint<DIM> &o, int dir) {
    const int d = DIM == 2 ? dir : 0;
    const long long w = DIM == 2 && d ? o.w[DIM - 1] : o.w[0];
    const int xw = DIM == 2 && d ? o.xw[DIM - 1] : o.xw[0];
    const long long a = w < 0 ? -w : w;
    if (o.p <= 0) return fx_value(a, xw);
    // sound speed: c^2 = gamma p / rho
    int xc;
    const long long c = fx_root(fx_mul(fx_limb(fx_mul(fx_limb(o.p), fx_limb(o.r))), gas.g), o.X - o.xr + 2, xc);
    const int x = xw > xc ? xw : xc;
    return fx_value(fx_shr(a, x - xw) + fx_shr(c, x - xc), x);
}

// Normal flux f and spectral radius (returned) of one state at a face point: on the integer
// units (dg_fixed.h: about 2^-60 where FP64 rounds at 2^-53 per operation, and no FP64 pipe but for
// the conversions and the root) where the state allows it, a rule of the state alone, so that every
// kernel gets the same bits for the same state.
template <int PHYS, int DIM>
__device__ __forceinline__ double face_flux(const Params &P, const double *u, int dir, bool want_speed, double *f) {
    if constexpr (PHYS == PH_EULER) {
        if (P.fx.on && fx_state<DIM>(u)) {
            FxPoint<DIM> o;
            fx_point<DIM>(u, P.fx.gas, o);
            fx_face_flux<DIM>(o, u, dir, f);
            return want_speed ? fx_face_speed<DIM>(P.fx.gas, o, dir) : 0.0;
        }
    }
    return flux_speed_dir<PHYS, DIM>(P, u, dir, f);
}

// Trial-step rate at one point: sum over directions of lambda_d / h_d, so that
// dt = CFL / max rate (eq. numerical_experiment:CFL, directional radii summed in 2D).
// The Euler form shares the reciprocal and the sound speed between the directions.
// Explicit roundings, as in euler_flux_ri: every kernel that takes a rate gets the same bits.
template <int PHYS, int DIM>
__device__ __forceinline__ double sk_rate(const Params &P, const double *u) {
    if constexpr (PHYS == PH_EULER) {
        const double ri = recip_nr(u[0]);
        const double kin = DIM == 1 ? __dmul_rn(u[1], u[1]) : fma(u[1], u[1], __dmul_rn(u[2], u[2]));
        const double p = __dmul_rn(P.gamma - 1.0, fma(-0.5 * kin, ri, u[DIM + 1]));
        const double c2 = __dmul_rn(__dmul_rn(P.gamma, p), ri);
        const double c = positive_bits(c2) ? sqrt(c2) : 0.0;
        double r = __dmul_rn(__dadd_rn(fabs(__dmul_rn(u[1], ri)), c), 0.5 * P.rhx);
        if constexpr (DIM == 2) r = fma(__dadd_rn(fabs(__dmul_rn(u[2], ri)), c), 0.5 * P.rhy, r);
        return r;
    } else {
        double r = speed_dir<PHYS, DIM>(P, u, 0) * (0.5 * P.rhx);
        if constexpr (DIM == 2) r = fma(speed_dir<PHYS, DIM>(P, u, 1), 0.5 * P.rhy, r);
        return r;
    }
}

// rho e = E - |m|^2 / (2 rho)   (eq. Euler-limiter2)
template <int DIM>
__device__ __forceinline__ double rho_e(const double *u) {
    const double kin = DIM == 1 ? __dmul_rn(u[1], u[1]) : fma(u[1], u[1], __dmul_rn(u[2], u[2]));
    return fma(-0.5 * kin, recip_nr(u[0]), u[DIM + 1]);
}

// The exact theta_2 of one S_K point (the alternative to eq. Euler-limiter2's concavity ratio):
// along u(t) = ub + t (u - ub) the density, momentum and energy are linear in t, so with
// rho(t) > 0, rho e(u(t)) >= eps <=> h(t) = (E(t) - eps) rho(t) - |m(t)|^2 / 2 >= 0, a quadratic
// a t^2 + b t + c.  h(0) = rho_bar (rho e(ub) - eps) > 0 for an admissible average and h(1) < 0
// at a violating point: one root in (0, 1), taken in the cancellation-free form
// q = -(b + sign(b) sqrt(b^2 - 4ac)) / 2, roots q / a and c / q.  1 when h(1) >= 0, 0 when the
// average is not strictly inside.  FP64, IEEE division and square root (rare: limited cells).
template <int DIM>
__device__ double theta2_point(const double *ub, const double *u, double eps) {
    const double dr = u[0] - ub[0], dE = u[DIM + 1] - ub[DIM + 1];
    double mm = 0.0, md = 0.0, dd = 0.0;
#pragma unroll
    for (int d = 1; d <= DIM; ++d) {
        const double dm = u[d] - ub[d];
        mm += ub[d] * ub[d];
        md += ub[d] * dm;
        dd += dm * dm;
    }
    const double c = (ub[DIM + 1] - eps) * ub[0] - 0.5 * mm;
    const double b = (ub[DIM + 1] - eps) * dr + dE * ub[0] - md;
    const double a = dE * dr - 0.5 * dd;
    if (!(c > 0.0)) return 0.0;
    if (a + b + c >= 0.0) return 1.0;
    double disc = b * b - 4.0 * a * c;
    if (disc < 0.0) disc = 0.0;
    const double q = -0.5 * (b + (b >= 0.0 ? sqrt(disc) : -sqrt(disc)));
    double best = 2.0;
    if (a != 0.0) {
        const double r = q / a;
        if (r > 0.0 && r < 1.0 && r < best) best = r;
    }
    if (q != 0.0) {
        const double r = c / q;
        if (r > 0.0 && r < 1.0 && r < best) best = r;
    }
    return best <= 1.0 ? best : 0.0;
}

// averages in B (scalar) or B^eps (Euler, rho >= eps and rho e >= eps); NaN fails
template <int PHYS, int DIM>
__device__ __forceinline__ bool admissible(const Params &P, const double *ub) {
    if constexpr (PHYS == PH_EULER) {
        return ub[0] >= P.eps && rho_e<DIM>(ub) >= P.eps;
    } else {
        return ub[0] >= P.lo && ub[0] <= P.hi;
    }
}

// exterior trace on a boundary side (final stage only)
template <int PHYS, int DIM>
__device__ __forceinline__ void boundary_state(const Params &P, int side, const double *ui, double *ue) {
    constexpr int M = ncomp(PHYS, DIM);
    int bc = P.bc[side];
    if (bc == BC_DIRICHLET) {
#pragma unroll
        for (int c = 0; c < M; ++c) ue[c] = P.bcs[side][c];
    } else {
#pragma unroll
        for (int c = 0; c < M; ++c) ue[c] = ui[c];
        if constexpr (PHYS == PH_EULER) {
            if (bc == BC_REFLECT) ue[1 + side / 2] = -ui[1 + side / 2];
        }
    }
}

// Exterior trace of a boundary face point in the final stage: Dirichlet the side's
// state, reflect the interior trace with the normal momentum negated, outflow the
// cell average of the same stage value (avg; a constant state is kept exactly, and
// the Lax--Friedrichs flux keeps its dissipation on outflow faces).
template <int PHYS, int DIM>
__device__ __forceinline__ void exterior_state(const Params &P, int side, const double *ui, const double *avg,
                                               double *ue) {
    constexpr int M = ncomp(PHYS, DIM);
    if (P.bc[side] == BC_OUTFLOW) {
#pragma unroll
        for (int c = 0; c < M; ++c) ue[c] = avg[c];
    } else {
        boundary_state<PHYS, DIM>(P, side, ui, ue);
    }
}

// neighbour across side (0 L, 1 R, 2 B, 3 T), or -1 on a non-periodic boundary
__device__ __forceinline__ int neighbour(const Params &P, int cell, int side) {
    int cx = cell % P.nx, cy = cell / P.nx;
    switch (side) {
    case 0: return cx > 0 ? cell - 1 : (P.bc[0] == BC_PERIODIC ? cell + P.nx - 1 : -1);
    case 1: return cx < P.nx - 1 ? cell + 1 : (P.bc[1] == BC_PERIODIC ? cell - P.nx + 1 : -1);
    case 2: return cy > 0 ? cell - P.nx : (P.bc[2] == BC_PERIODIC ? cell + (P.ny - 1) * P.nx : -1);
    default: return cy < P.ny - 1 ? cell + P.nx : (P.bc[3] == BC_PERIODIC ? cell - (P.ny - 1) * P.nx : -1);
    }
}

// The same, and -1 on a side that a non-rectangular domain's geometry word gives a boundary
// kind (the FP64 final stage; the kernels that reject a geometry keep the plain rule)
__device__ __forceinline__ int neighbour_geo(const Params &P, int cell, int side) {
    if (P.geo != nullptr && ((P.geo[cell] >> (4 * side)) & 15u) != GEO_MESH) return -1;
    return neighbour(P, cell, side);
}

// Exterior trace of a boundary face point of a non-rectangular domain (Examples 4.8, 4.9) in
// the final stage: the side's kind in the cell's geometry word decides.  pos is the face
// point's index along the face, stage the traced stage (its time t0 + c_i dt moves the
// shock line); kind GEO_MESH falls back to the rectangle side's condition.
template <int PHYS, int DIM, int N>
__device__ __forceinline__ void geo_exterior(const Params &P, int cell, int side, int pos, int stage,
                                             const double *ui, const double *avg, double *ue) {
    constexpr int M = ncomp(PHYS, DIM);
    const unsigned kind = (P.geo[cell] >> (4 * side)) & 15u;
    if (kind == GEO_STATE_A || kind == GEO_STATE_B || kind == GEO_SHOCK) {
        int which = kind == GEO_STATE_B ? 1 : 0;
        if (kind == GEO_SHOCK) {
            const NodalTables &T = c_tab[N - 2];
            const int cx = cell % P.nx;
            const double xi = side == 0 ? -1.0 : side == 1 ? 1.0 : T.xg[pos];
            const double x = P.x0 + (cx + 0.5 * (xi + 1.0)) * (2.0 / P.rhx);
            double ci = 0.0;
            for (int j = 0; j < stage; ++j) ci += P.A[stage][j];
            which = x < P.shock_x0 + P.shock_speed * (P.t0 + ci * P.dt) ? 0 : 1;
        }
#pragma unroll
        for (int c = 0; c < M; ++c) ue[c] = P.gstate[which][c];
    } else if (kind == GEO_WALL) {
#pragma unroll
        for (int c = 0; c < M; ++c) ue[c] = ui[c];
        if constexpr (PHYS == PH_EULER) ue[1 + side / 2] = -ui[1 + side / 2];
    } else if (kind == GEO_OUTFLOW) {
#pragma unroll
        for (int c = 0; c < M; ++c) ue[c] = avg[c];
    } else {
        exterior_state<PHYS, DIM>(P, side, ui, avg, ue);
    }
}

// ----------------------------------------------------------------------------- block layout

template <int DIM, int N, int PHYS>
struct Cfg {
    static constexpr int D = DIM;
    static constexpr int NP = N;
    static constexpr int PH = PHYS;
    static constexpr int M = ncomp(PHYS, DIM);
    static constexpr int NN = DIM == 2 ? N * N : N;       // nodes per cell
    static constexpr int NF = DIM == 2 ? N : 1;           // quadrature points per face
    static constexpr int NTR = 2 * DIM * NF;              // face points per cell
    static constexpr int L = nlob(N);                     // Gauss--Lobatto points
    static constexpr int NSK = DIM == 2 ? 2 * N * L : L;  // |S_K|
    static constexpr int NCB = cells_per_block(DIM, N);  // cells per block
    static constexpr int NT = NCB * NN;                   // threads per block (multiple of 32)
    static constexpr int PPT = (NSK + NN - 1) / NN;       // S_K points per thread
    static constexpr int FPT = (NTR + NN - 1) / NN;       // face points per thread
    static constexpr bool WARP = false;                   // cells may straddle warps
};

// The same with whole cells per warp: 32 / NN cells on a warp's first lanes, the remaining lanes
// (Q^2: 5 of 32) shadowing the last one (same cell, node and values).  A cell's exchanges then
// need a warp barrier instead of a block barrier, and a warp whose cells need the limiter's or
// the operator's slow path does not hold up the others.
template <int DIM, int N, int PHYS>
struct CfgW : Cfg<DIM, N, PHYS> {
    static constexpr int CPW = 32 / Cfg<DIM, N, PHYS>::NN;  // cells per warp
    static constexpr int NT = kWarpThreads;
    static constexpr int NCB = CPW * (NT / 32);
    static constexpr bool WARP = true;
};

// this thread's cell within the block and node within the cell
template <class C>
__device__ __forceinline__ void place(int &lc, int &node) {
    if constexpr (C::WARP) {
        int l = threadIdx.x & 31;
        if (l >= C::CPW * C::NN) l = C::CPW * C::NN - 1;
        const int w = l / C::NN;
        lc = (threadIdx.x >> 5) * C::CPW + w;
        node = l - w * C::NN;
    } else {
        lc = threadIdx.x / C::NN;
        node = threadIdx.x - lc * C::NN;
    }
}

// whether this lane shadows a cell's last node: what a thread reads and rewrites in shared memory is for
// the node's own lane alone, a shadow's turn would count it again
template <class C>
__device__ __forceinline__ bool shadow_lane() {
    return C::WARP && (int)(threadIdx.x & 31) >= (32 / C::NN) * C::NN;
}

// barrier (with a vote) over the threads that share a cell's data
template <class C>
__device__ __forceinline__ void cell_sync() {
    if constexpr (C::WARP)
        __syncwarp();
    else
        __syncthreads();
}
template <class C>
__device__ __forceinline__ bool cell_sync_or(bool x) {
    if constexpr (C::WARP) {
        const bool r = __any_sync(0xffffffffu, x);
        __syncwarp();
        return r;
    } else
        return __syncthreads_or(x);
}

// Shared memory of one cell.  Warps run ahead of one another, so nothing of a cell overlaps
// another cell's part; the size is 48 bytes modulo 128, which puts the same element of a warp's
// cells on different banks.
template <class C>
struct CellData {
    double u[C::M][C::NN];
    union {  // fluxes live inside eval_G only; the FP32 node copies inside the limiter only
        double f[C::D][C::M][C::NN];
        float uf[C::M][C::NN];
    };
    double tf[C::NTR][C::M];
    double avg[C::M];
    union {  // the limiter's reductions and the final kernel's edge speeds never overlap
        unsigned long long red[C::NN][2];  // ordbits keys
        double ts[C::NTR];  // spectral radii of the traces (eval_G of a traced stage)
        double al[C::NTR];
    };
    double th[2];
    int bad;
};
template <class C>
struct alignas(16) PadCell : CellData<C> {
    static constexpr int kPad = (128 + 48 - (int)sizeof(CellData<C>) % 128) % 128;
    char pad[kPad ? kPad : 128];
};
template <class C>
struct Smem {
    PadCell<C> c[C::NCB];
};

// value of every component at S_K point p of the cell whose nodes are su
template <int DIM, int N, int M, int NN>
__device__ __forceinline__ void sk_eval(const double (&su)[M][NN], int p, double *v) {
    const NodalTables &T = c_tab[N - 2];
    constexpr int L = nlob(N);
    if constexpr (DIM == 1) {
#pragma unroll
        for (int c = 0; c < M; ++c) {
            double s = 0.0;
#pragma unroll
            for (int a = 0; a < N; ++a) s = fma(T.Igl[p][a], su[c][a], s);
            v[c] = s;
        }
    } else {
        if (p < N * L) {  // (x^GL_alpha, y^G_beta): interpolate along row beta
            int beta = p / L, al = p - beta * L;
#pragma unroll
            for (int c = 0; c < M; ++c) {
                double s = 0.0;
#pragma unroll
                for (int a = 0; a < N; ++a) s = fma(T.Igl[al][a], su[c][beta * N + a], s);
                v[c] = s;
            }
        } else {  // (x^G_beta, y^GL_alpha): interpolate along column beta
            int q = p - N * L;
            int beta = q / L, al = q - beta * L;
#pragma unroll
            for (int c = 0; c < M; ++c) {
                double s = 0.0;
#pragma unroll
                for (int b = 0; b < N; ++b) s = fma(T.Igl[al][b], su[c][b * N + beta], s);
                v[c] = s;
            }
        }
    }
}

// FP32 screen of the limiter.  v: the FP32 interpolation to S_K point p of the FP32
// copies uf of the cell's FP64 node values; e: a bound on |FP64 interpolation - v| per
// component, 4 (n + 3) 2^-24 sum_a |l_a| |uf_a| (the roundings of the nodes and the
// weights to FP32, of the n FP32 and the n FP64 fused multiply-adds: (n + 3) 2^-24 of
// that sum, taken 4 times).
template <int DIM, int N, int M, int NN>
__device__ __forceinline__ void sk_eval_screen(const float (&su)[M][NN], int p, float *v, float *e) {
    const NodalTables &T = c_tab[N - 2];
    constexpr int L = nlob(N);
    constexpr float K = 4.0f * (N + 3) * 5.9604644775390625e-08f;
    int beta = 0, al = p, stride = 1, off = 0;
    if constexpr (DIM == 2) {
        if (p < N * L) {
            beta = p / L;
            al = p - beta * L;
            stride = 1;
            off = beta * N;
        } else {
            const int q = p - N * L;
            beta = q / L;
            al = q - beta * L;
            stride = N;
            off = beta;
        }
    }
#pragma unroll
    for (int c = 0; c < M; ++c) {
        float s = 0.0f, a = 0.0f;
#pragma unroll
        for (int k = 0; k < N; ++k) {
            const float w = T.Iglf[al][k], x = su[c][off + k * stride];
            s = fmaf(w, x, s);
            a = fmaf(fabsf(w), fabsf(x), a);
        }
        v[c] = s;
        e[c] = K * a;
    }
}

// True when the FP32 value v (bound e per component on its distance to the FP64 value)
// proves that the FP64 value lies in the bounds: scalar lo <= v <= hi; Euler rho >= eps
// and rho e = E - |m|^2 / (2 rho) >= eps, with rho e bounded below by
// (E - e_E) - (|m| + e_m)^2 / (2 (rho - e_rho)) less 2^-20 of its magnitudes (the FP32
// rounding of this bound and the FP64 rounding of rho e).  NaN and inf never pass.
template <int PHYS, int DIM>
__device__ __forceinline__ bool screen_point(const Params &P, const float *v, const float *e) {
    if (!P.scr_on) return false;
    if constexpr (PHYS == PH_EULER) {
        constexpr int M = DIM + 2;
        const float rlo = v[0] - e[0];
        if (!(rlo >= P.scr_eps && rlo <= 3.0e38f)) return false;
        float m2 = 0.0f;
#pragma unroll
        for (int d = 0; d < DIM; ++d) {
            const float ma = fabsf(v[1 + d]) + e[1 + d];
            m2 = fmaf(ma, ma, m2);
        }
        const float kin = 0.5f * m2 / rlo;
        const float elo = v[M - 1] - e[M - 1];
        const float lb = (elo - kin) - 9.5367431640625e-07f * (fabsf(elo) + kin);
        return lb >= P.scr_eps && lb <= 3.0e38f;
    } else {
        return v[0] - e[0] >= P.scr_lo && v[0] + e[0] <= P.scr_hi;
    }
}

// An upper bound of sk_rate's FP64 value at a point whose FP64 components lie within e of v and
// that screen_point has cleared (Euler): the density from below, momenta, and pressure from above,
// and 2^-18 for the roundings of this bound and of the FP64 form.  Infinity or NaN where the
// bound fails; the callers then evaluate the point.
template <int PHYS, int DIM>
__device__ __forceinline__ float rate_bound(const Params &P, const float *v, const float *e) {
    if constexpr (PHYS == PH_EULER) {
        const float up = 1.0f + 3.814697265625e-06f;
        const float ri = __frcp_rn(v[0] - e[0]), rj = __frcp_rn(v[0] + e[0]);
        float kin = 0.0f, adv = 0.0f;
        const float hr[2] = {0.5f * P.scr_rh[0], 0.5f * P.scr_rh[1]};
#pragma unroll
        for (int d = 0; d < DIM; ++d) {
            const float lo = fmaxf(fabsf(v[1 + d]) - e[1 + d], 0.0f);
            kin = fmaf(lo, lo, kin);
            adv = fmaf(fabsf(v[1 + d]) + e[1 + d], hr[d], adv);
        }
        const float el = v[DIM + 1] + e[DIM + 1];
        // el - kin rj / 2 with its own rounding covered by 2^-20 of both terms
        const float re = fmaxf((el - 0.5f * kin * rj) + 9.5367431640625e-07f * (el + 0.5f * kin * rj), 0.0f);
        const float c = sqrtf(P.scr_gg * re * ri);
        return fmaf(adv, ri, c * (DIM == 2 ? hr[0] + hr[1] : hr[0])) * up;
    } else {
        return INFINITY;
    }
}

// S_K bound predicate used by the limiter's verification and by the margins
template <int PHYS, int DIM>
__device__ __forceinline__ bool point_ok(const Params &P, const double *v) {
    if constexpr (PHYS == PH_EULER) {
        return v[0] >= P.eps && rho_e<DIM>(v) >= P.eps;
    } else {
        return v[0] >= P.lo && v[0] <= P.hi;
    }
}

// Cell averages of all components (Gauss weights; the mass matrix is exact), block
// collective without a barrier: fn(c, avg_c) is called once per component by one
// thread of the cell.  2D Q^3 Euler (16 nodes, a cell on one half-warp): each
// component is split over 4 lanes of 4 terms and summed by two xor shuffles, 6 FP64
// instructions instead of a 16-term chain on 4 of the 16 lanes.  Otherwise one
// thread per component sums the nodes in order.  All threads of the block must call it.
template <class C, class Fn>
__device__ __forceinline__ void cell_averages(const double (&su)[C::M][C::NN], int node, Fn fn) {
    constexpr int DIM = C::D, N = C::NP, M = C::M, NN = C::NN;
    const NodalTables &T = c_tab[N - 2];
    if constexpr (DIM == 2 && NN == 16 && M == 4) {
        const int c = node >> 2, r = node & 3;
        double s = 0.0;
#pragma unroll
        for (int q = 4 * r; q < 4 * r + 4; ++q) s = fma(T.w2[q], su[c][q], s);
        s += __shfl_xor_sync(0xffffffffu, s, 1);
        s += __shfl_xor_sync(0xffffffffu, s, 2);
        if (r == 0) fn(c, s);
    } else {
        for (int c = node; c < M; c += NN) {
            double s = 0.0;
#pragma unroll
            for (int q = 0; q < NN; ++q) s = fma(DIM == 2 ? T.w2[q] : T.w1[q], su[c][q], s);
            fn(c, s);
        }
    }
}

// ----------------------------------------------------------------------------- limiter

// Rounding safety of the limiter: every theta below 1 is multiplied by
// (1-2^-40) so the rescaled polynomial lands strictly inside the bound; if the
// re-evaluation on S_K still finds a point outside, the final scaling towards
// the average is multiplied by the retry factors 1-2^-30, 1-2^-20, 1-2^-10, 0.
constexpr double kMargin = 1.0 - 9.094947017729282e-13;
__device__ __forceinline__ double retry_factor(int attempt) {
    switch (attempt) {
    case 1: return 1.0 - 9.313225746154785e-10;
    case 2: return 1.0 - 9.5367431640625e-07;
    case 3: return 1.0 - 0.0009765625;
    default: return 0.0;
    }
}

// Scaling limiter of one stage (Prop. 2.4 scalar, eq. Euler-limiter1/2), block
// collective.  u: this thread's node values (in/out).  pts (with need_pts): on return
// the values at this thread's S_K points of the limited polynomial.  With check_avg the
// admissibility of the cell average sets *B.flag (Sec. 4.1 restart test).
//
// Most cells need no limiting.  An FP32 screen (screen_point, with a bound on its
// distance to the FP64 values) first tests every S_K point; when it clears every cell of
// the block (or warp), the FP64 limiter would leave all of them unchanged (theta = 1) and
// it is skipped: the results are those of the FP64 path.  The averages need no test of
// their own then: an average is a convex combination of the S_K values (Prop. 2.2), rho e is
// concave, and the screen leaves 2^-20 of |E| and |m|^2 / 2 rho (and 2^-22 of the nodes'
// magnitudes), far above the FP64 rounding of the average.  Returns true when it was
// skipped; pts is then not set, and with want_rate rhi bounds this thread's point rates.
template <class C>
__device__ bool limit_block(const Params &P, const Bufs &B, Smem<C> &S, int lc, int node, bool active,
                            double *u, double (&pts)[C::PPT][C::M], bool check_avg, bool stats, bool want_rate,
                            float &rhi) {
    constexpr int DIM = C::D, N = C::NP, PHYS = C::PH;
    constexpr int M = C::M, NN = C::NN, NSK = C::NSK, PPT = C::PPT;

    // 1. publish node values (and FP32 copies for the screen: truncated, 2^-23 of the value,
    //    which the bound of sk_eval_screen covers)
    cell_sync<C>();  // earlier readers of the cell's arrays are done
#pragma unroll
    for (int c = 0; c < M; ++c) {
        S.c[lc].u[c][node] = u[c];
        S.c[lc].uf[c][node] = PHYS == PH_EULER ? trunc_f(u[c]) : (float)u[c];
    }
    cell_sync<C>();
    // 2. FP32 screen of this thread's S_K points
    bool unsafe = false;
    rhi = 0.0f;
#pragma unroll
    for (int j = 0; j < PPT; ++j) {
        int p = node + j * NN;
        if (p < NSK) {
            float v[M], e[M];
            sk_eval_screen<DIM, N, M, NN>(S.c[lc].uf, p, v, e);
            if (!screen_point<PHYS, DIM>(P, v, e)) unsafe = true;
            if (want_rate) {
                const float r = rate_bound<PHYS, DIM>(P, v, e);
                rhi = fmaxf(rhi, r == r ? r : INFINITY);  // a bound that fails bounds nothing
            }
        }
    }
    if (!cell_sync_or<C>(unsafe)) return true;  // every cell cleared
    cell_averages<C>(S.c[lc].u, node, [&](int c, double s) { S.c[lc].avg[c] = s; });
    cell_sync<C>();
    // 3. values at S_K and this thread's extremes (order-preserving integer keys)
    unsigned long long kmin = kKeyPosInf, kmax = kKeyNegInf;
#pragma unroll
    for (int j = 0; j < PPT; ++j) {
        int p = node + j * NN;
        if (p < NSK) {
            sk_eval<DIM, N, M, NN>(S.c[lc].u, p, pts[j]);
            if (isnan_bits(pts[j][0])) {
                kmin = kKeyNegInf;  // NaN counts as a violation
            } else {
                unsigned long long k = ordbits(pts[j][0]);
                kmin = umin64(kmin, k);
                kmax = umax64(kmax, k);
            }
        }
    }
    S.c[lc].red[node][0] = kmin;
    S.c[lc].red[node][1] = kmax;
    double ub[M];
#pragma unroll
    for (int c = 0; c < M; ++c) ub[c] = S.c[lc].avg[c];
    cell_sync<C>();
    // 4. leader: admissibility of the average and theta (theta_1 for Euler)
    double reb = 0.0;  // leader: rho e of the average (Euler)
    if (node == 0) {
        unsigned long long kmn = kKeyPosInf, kmx = kKeyNegInf;
        for (int q = 0; q < NN; ++q) {
            kmn = umin64(kmn, S.c[lc].red[q][0]);
            kmx = umax64(kmx, S.c[lc].red[q][1]);
        }
        const double mn = ordbits_inv(kmn), mx = ordbits_inv(kmx);
        if constexpr (PHYS == PH_EULER) {
            reb = rho_e<DIM>(ub);
            if (check_avg && active && !(ge_pos_bits(ub[0], P.eps) && ge_pos_bits(reb, P.eps))) atomicOr(B.flag, 1);
        } else {
            if (check_avg && active && !admissible<PHYS, DIM>(P, ub)) atomicOr(B.flag, 1);
        }
        double th = 1.0;
        if constexpr (PHYS == PH_EULER) {
            if (!ge_pos_bits(mn, P.eps)) th = ratio01(ub[0] - P.eps, ub[0] - mn);
        } else {
            if (mx > P.hi) th = fmin(th, ratio01(P.hi - ub[0], mx - ub[0]));
            if (mn < P.lo) th = fmin(th, ratio01(ub[0] - P.lo, ub[0] - mn));
        }
        S.c[lc].th[0] = below_one(th) ? th * kMargin : th;
        S.c[lc].th[1] = 1.0;
        S.c[lc].bad = 0;
    }
    cell_sync<C>();
    double th1 = S.c[lc].th[0];
    double th2 = 1.0;
    if constexpr (PHYS == PH_EULER) {
        // 5. rho e at S_K with the density already scaled by theta_1
        unsigned long long km = kKeyPosInf, kt = ordbits(1.0);
#pragma unroll
        for (int j = 0; j < PPT; ++j) {
            int p = node + j * NN;
            if (p < NSK) {
                double v[M];
#pragma unroll
                for (int c = 0; c < M; ++c) v[c] = pts[j][c];
                if (below_one(th1)) v[0] = th1 * (v[0] - ub[0]) + ub[0];
                double re = rho_e<DIM>(v);
                km = isnan_bits(re) ? kKeyNegInf : umin64(km, ordbits(re));  // NaN counts as a violation
                // the exact solve: the smallest per-point theta over the violating points
                if (P.theta2_exact && !ge_pos_bits(re, P.eps))
                    kt = umin64(kt, ordbits(isnan_bits(re) ? 0.0 : theta2_point<DIM>(ub, v, P.eps)));
            }
        }
        S.c[lc].red[node][1] = km;
        S.c[lc].red[node][0] = kt;
        cell_sync<C>();
        if (node == 0) {
            unsigned long long kmn = kKeyPosInf, ktn = ordbits(1.0);
            for (int q = 0; q < NN; ++q) {
                kmn = umin64(kmn, S.c[lc].red[q][1]);
                ktn = umin64(ktn, S.c[lc].red[q][0]);
            }
            const double mn = ordbits_inv(kmn);
            S.c[lc].th[1] = ge_pos_bits(mn, P.eps) ? 1.0
                          : P.theta2_exact        ? ordbits_inv(ktn) * kMargin
                                                  : ratio01(reb - P.eps, reb - mn) * kMargin;
        }
        cell_sync<C>();
        th2 = S.c[lc].th[1];
    }
    // 6. rescale towards the average
    bool limited = below_one(th1) || below_one(th2);
    double uo[M];
#pragma unroll
    for (int c = 0; c < M; ++c) uo[c] = u[c];
    auto apply = [&](double t2) {
        if constexpr (PHYS == PH_EULER) {
            double r = below_one(th1) ? th1 * (uo[0] - ub[0]) + ub[0] : uo[0];
            u[0] = below_one(t2) ? t2 * (r - ub[0]) + ub[0] : r;
#pragma unroll
            for (int c = 1; c < M; ++c) u[c] = below_one(t2) ? t2 * (uo[c] - ub[c]) + ub[c] : uo[c];
        } else {
            double t = th1 * t2;
            u[0] = t < 1.0 ? t * (uo[0] - ub[0]) + ub[0] : uo[0];
        }
    };
    double tfin = th2;
    if (limited) apply(th2);
    // 7. verify the limited cells on S_K with the same interpolation; shrink on a
    //    rounding violation (the final scaling factor towards the average)
    bool any_limited = cell_sync_or<C>(limited);
    if (any_limited) {
        for (int attempt = 0; attempt <= 4; ++attempt) {
#pragma unroll
            for (int c = 0; c < M; ++c) S.c[lc].u[c][node] = u[c];
            cell_sync<C>();
            bool viol = false;
            if (limited) {
#pragma unroll
                for (int j = 0; j < PPT; ++j) {
                    int p = node + j * NN;
                    if (p < NSK) {
                        sk_eval<DIM, N, M, NN>(S.c[lc].u, p, pts[j]);
                        if (!point_ok<PHYS, DIM>(P, pts[j])) viol = true;
                    }
                }
            }
            if (viol) S.c[lc].bad = 1;
            bool again = cell_sync_or<C>(viol);
            if (!again || attempt == 4) break;
            bool mine = S.c[lc].bad != 0;
            cell_sync<C>();
            if (node == 0) S.c[lc].bad = 0;
            if (mine) {
                // Euler: theta_2 (all components); scalars: th2 == 1 so the factor multiplies theta
                tfin = th2 * retry_factor(attempt + 1);
                apply(tfin);
            }
        }
    }
    if (stats && active && node == 0 && limited) {
        double tr = PHYS == PH_EULER ? fmin(th1, tfin) : th1 * tfin;
        atomicAdd(B.nlim, 1ull);
        atomicMin(B.thmin, dbits(tr > 0.0 ? tr : 0.0));
    }
    cell_sync<C>();
    return false;
}

// Posts the largest trial-step rate over the S_K points of the limited state (limit_block's
// cleared, rhi and pts).  A warp whose FP32 bounds stay at or below the rate already posted by
// others cannot raise the maximum and skips the FP64 interpolation and rates (114 FP64
// instructions per warp in Q^3): the posted maximum is the same.
template <class C>
__device__ __forceinline__ void post_rate(const Params &P, const Bufs &B, const Smem<C> &S, int lc, int node, bool own,
                                          bool cleared, float rhi, double (&pts)[C::PPT][C::M]) {
    constexpr int DIM = C::D, N = C::NP, PHYS = C::PH;
    constexpr int M = C::M, NN = C::NN;
    bool need = own;
    if constexpr (PHYS == PH_EULER) {
        if (cleared) {
            const double now = bitsd(*(const volatile unsigned long long *)B.a0);
            need = own && !(rhi <= fminf(trunc_f(now), 3.0e38f));
        }
    }
    if (__any_sync(0xffffffffu, need)) {
        double amax = 0.0;
#pragma unroll
        for (int j = 0; j < C::PPT; ++j) {
            int p = node + j * NN;
            if (p < C::NSK && own) {
                if (cleared) sk_eval<DIM, N, M, NN>(S.c[lc].u, p, pts[j]);
                amax = fmax_nonneg(amax, sk_rate<PHYS, DIM>(P, pts[j]));
            }
        }
        __syncwarp();
        unsigned long long abits = dbits(amax);  // non-negative: the bits order as the values
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) abits = umax64(abits, __shfl_xor_sync(0xffffffffu, abits, o));
        if ((threadIdx.x & 31) == 0 && abits > 0ull) atomicMax(B.a0, abits);
    }
}

// ----------------------------------------------------------------------------- G

// G(u) at this thread's node (block collective).  trs receives the interior
// trace states of this thread's face points; their normal fluxes stay in S.tf and,
// with want_speed, their spectral radii go to S.ts (both read back by the thread
// that computed them, for the final stage's Lax--Friedrichs flux of traced stages).
template <class C>
__device__ void eval_G(const Params &P, Smem<C> &S, int lc, int node, const double *u, double *g,
                       double (&trs)[C::FPT][C::M], bool want_speed = false) {
    constexpr int DIM = C::D, N = C::NP, PHYS = C::PH;
    constexpr int M = C::M, NN = C::NN, NF = C::NF, NTR = C::NTR, FPT = C::FPT;
    const NodalTables &T = c_tab[N - 2];
    const int a = node % N, b = DIM == 2 ? node / N : 0;
    // 1. flux at the node
    {
        double fx[M], fy[M];
        if constexpr (DIM == 2) {
            flux_xy<PHYS>(P, u, fx, fy);
        } else {
            flux_dir<PHYS, DIM>(P, u, 0, fx);
        }
#pragma unroll
        for (int c = 0; c < M; ++c) {
            S.c[lc].u[c][node] = u[c];
            S.c[lc].f[0][c][node] = fx[c];
            if constexpr (DIM == 2) S.c[lc].f[1][c][node] = fy[c];
        }
    }
    cell_sync<C>();
    // 2. volume term and interior traces
    double vx[M], vy[M];
#pragma unroll
    for (int c = 0; c < M; ++c) {
        double s = 0.0;
#pragma unroll
        for (int q = 0; q < N; ++q) s = fma(T.Dhat[a][q], S.c[lc].f[0][c][b * N + q], s);
        vx[c] = s;
        if constexpr (DIM == 2) {
            double t = 0.0;
#pragma unroll
            for (int r = 0; r < N; ++r) t = fma(T.Dhat[b][r], S.c[lc].f[1][c][r * N + a], t);
            vy[c] = t;
        }
    }
#pragma unroll
    for (int j = 0; j < FPT; ++j) {
        int fp = node + j * NN;
        if (fp < NTR) {
            int face = fp / NF, pos = fp - face * NF;
            const double *l = (face & 1) ? T.lp : T.lm;
#pragma unroll
            for (int c = 0; c < M; ++c) {
                double s = 0.0;
                if (DIM == 1 || face < 2) {
#pragma unroll
                    for (int q = 0; q < N; ++q) s = fma(l[q], S.c[lc].u[c][pos * N + q], s);
                } else {
#pragma unroll
                    for (int q = 0; q < N; ++q) s = fma(l[q], S.c[lc].u[c][q * N + pos], s);
                }
                trs[j][c] = s;
            }
            double f[M];
            const double sp = face_flux<PHYS, DIM>(P, trs[j], face >> 1, want_speed, f);
#pragma unroll
            for (int c = 0; c < M; ++c) S.c[lc].tf[fp][c] = f[c];
            if (want_speed) S.c[lc].ts[fp] = sp;
        }
    }
    cell_sync<C>();
    // 3. lift the interior-trace edge terms
#pragma unroll
    for (int c = 0; c < M; ++c) {
        double gx = vx[c] - T.liftp[a] * S.c[lc].tf[NF + b][c] + T.liftm[a] * S.c[lc].tf[b][c];
        double gv = P.rhx * gx;
        if constexpr (DIM == 2) {
            double gy = vy[c] - T.liftp[b] * S.c[lc].tf[3 * NF + a][c] + T.liftm[b] * S.c[lc].tf[2 * NF + a][c];
            gv = fma(P.rhy, gy, gv);
        }
        g[c] = gv;
    }
}

// G at a warp's nodes with the FP64 form's arithmetic (eval_G), for the warps that the
// fixed-point form below refuses.  Out of line: it is rare.
template <class C>
__device__ __noinline__ void eval_G_slow(const Params &P, Smem<C> &S, int lc, int node, const double *u, double *g,
                                         double (&trs)[C::FPT][C::M], bool want_speed) {
    cell_sync<C>();
    eval_G<C>(P, S, lc, node, u, g, trs, want_speed);
}

// The same with eval_G_fx's results, for the cells with `mine`.
template <class C, class Put, class Fn>
__device__ __forceinline__ void eval_G_64(const Params &P, Smem<C> &S, int lc, int node, const double *u, double *g,
                                          bool mine, bool want_speed, bool want_avg, Put put, Fn avg) {
    constexpr int M = C::M, NN = C::NN, NF = C::NF, NTR = C::NTR, FPT = C::FPT;
    CellData<C> &D = S.c[lc];
    double uu[M], gg[M], tt[FPT][M];
#pragma unroll
    for (int c = 0; c < M; ++c) uu[c] = u[c];
    eval_G_slow<C>(P, S, lc, node, uu, gg, tt, want_speed);
    cell_sync<C>();
    if (mine) {
#pragma unroll
        for (int c = 0; c < M; ++c) g[c] = gg[c];
#pragma unroll
        for (int j = 0; j < FPT; ++j) {
            const int fp = node + j * NN;
            if ((j + 1) * NN <= NTR || fp < NTR) {
                double sp = 0.0;
                if (want_speed)
                    for (int q = 0; q < NF; ++q) sp = fmax_nonneg(sp, D.ts[fp / NF * NF + q]);
                put(j, tt[j], D.tf[fp], sp);
            }
        }
    }
    if (want_avg)
        cell_averages<C>(D.u, node, [&](int c, double v) {
            if (mine) avg(c, v);
        });
    cell_sync<C>();
}

// Fixed-point coefficients and the tableau's products with dt, in shared memory.
template <class C>
struct alignas(16) BlockTab {
    Fx cx[C::NP][C::NP], cy[C::NP][C::NP], lx[C::NP][2], ly[C::NP][2];
    Fx tl[2][C::NP], w[C::NN];
    double dtA[MAXS][MAXS], dtb[MAXS];
};
// Filled by the whole block (the caller's barrier follows).
template <class C>
__device__ __forceinline__ void fill_tab(const Params &P, BlockTab<C> &B) {
    constexpr int N = C::NP;
    const NodalTables &T = c_tab[N - 2];
    for (int t = threadIdx.x; t < N * N; t += C::NT) {
        B.cx[t / N][t % N] = P.fx.cx[t / N][t % N];
        if constexpr (C::D == 2) B.cy[t / N][t % N] = P.fx.cy[t / N][t % N];
        if (t < 2 * N) {
            B.lx[t / 2][t & 1] = P.fx.lx[t / 2][t & 1];
            if constexpr (C::D == 2) B.ly[t / 2][t & 1] = P.fx.ly[t / 2][t & 1];
            B.tl[t / N][t % N] = T.tlx[t / N][t % N];
        }
        if (t < C::NN) B.w[t] = C::D == 2 ? T.w2x[t] : T.w1x[t];
    }
    for (int t = (int)threadIdx.x - 64; t >= 0 && t < MAXS * MAXS + MAXS; t += C::NT) {  // the third warp
        if (t < MAXS * MAXS)
            B.dtA[t / MAXS][t % MAXS] = P.dt * P.A[t / MAXS][t % MAXS];
        else
            B.dtb[t - MAXS * MAXS] = P.dt * P.b[t - MAXS * MAXS];
    }
}

// n consecutive limbs from shared memory (16-byte accesses where the rows are aligned)
template <int N>
__device__ __forceinline__ void load_fx(const Fx *p, Fx (&v)[N]) {
    if constexpr (N % 2 == 0) {
#pragma unroll
        for (int q = 0; q < N; q += 2) {
            const int4 r = *reinterpret_cast<const int4 *>(p + q);
            v[q] = Fx{r.x, r.y};
            v[q + 1] = Fx{r.z, r.w};
        }
    } else {
#pragma unroll
        for (int q = 0; q < N; ++q) v[q] = p[q];
    }
}

// Largest of each 16-bit half over the threads of a cell.
__device__ __forceinline__ unsigned vmax_u16x2(unsigned a, unsigned b) {
    unsigned r;
    asm("max.u16x2 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(b));
    return r;
}
template <class C>
__device__ __forceinline__ unsigned cell_max_halves(unsigned w, int node) {
    constexpr int NN = C::NN;
    if constexpr ((NN & (NN - 1)) == 0) {
#pragma unroll
        for (int o = 1; o < NN; o <<= 1) w = vmax_u16x2(w, __shfl_xor_sync(0xffffffffu, w, o));
    } else {  // rotations within the cell's lanes: windows of 2, 4, ... nodes until all are covered
        int l = threadIdx.x & 31;
        if (l >= C::CPW * NN) l = C::CPW * NN - 1;
        const int base = l - node;
        int have = 1;
#pragma unroll
        for (int o = 1; o < NN; o <<= 1) {
            const int k = have + o <= NN && o == have ? o : NN - have;
            int src = node + k;
            if (src >= NN) src -= NN;
            w = vmax_u16x2(w, __shfl_sync(0xffffffffu, w, base + src));
            have += k;
            if (have >= NN) break;
        }
    }
    return w;
}

// Largest x (non-negative) over the threads of a face's points (NF consecutive nodes).
template <class C>
__device__ __forceinline__ double face_max(double x, int node) {
    constexpr int NF = C::NF;
    unsigned long long k = dbits(x);
    if constexpr (NF == 3) {
        int l = threadIdx.x & 31;
        if (l >= C::CPW * C::NN) l = C::CPW * C::NN - 1;
        const int r = node % 3, base = l - r;
        const unsigned long long k1 = __shfl_sync(0xffffffffu, k, base + (r == 2 ? 0 : r + 1));
        const unsigned long long k2 = __shfl_sync(0xffffffffu, k, base + (r == 0 ? 2 : r - 1));
        k = umax64(k, umax64(k1, k2));
    } else {
#pragma unroll
        for (int o = 1; o < NF; o <<= 1) k = umax64(k, __shfl_xor_sync(0xffffffffu, k, o));
    }
    return bitsd(k);
}

// The smaller of the largest x over a node's row and over its column (2D).
template <class C>
__device__ __forceinline__ int line_max(int x, int node) {
    constexpr int N = C::NP;
    int l = threadIdx.x & 31;
    if (l >= C::CPW * C::NN) l = C::CPW * C::NN - 1;
    const int base = l - node, a = node % N;
    int r = x, c = x;
#pragma unroll
    for (int q = 0; q < N; ++q) {
        r = max(r, __shfl_sync(0xffffffffu, x, base + node - a + q));
        c = max(c, __shfl_sync(0xffffffffu, x, base + q * N + a));
    }
    return min(r, c);
}

// Whether x holds for any thread of this thread's cell.
template <class C>
__device__ __forceinline__ bool cell_any(bool x, int node) {
    int l = threadIdx.x & 31;
    if (l >= C::CPW * C::NN) l = C::CPW * C::NN - 1;
    return ((__ballot_sync(0xffffffffu, x) >> (l - node)) & ((1u << C::NN) - 1u)) != 0u;
}

// A cell's exponents of G's fluxes: comp 0, the momentum components, the last one (scalar laws: the
// first only), two 16-bit fields per word.
struct FluxExp {
    unsigned w0, w1;
};
__device__ __forceinline__ unsigned biased_exp(int x) { return (unsigned)max(x + 1023, 0); }

// G(u) with its linear maps in fixed point (dg_fixed.h): the stage's node values, then the
// node and trace fluxes, share one exponent per cell and component, and the volume term, both
// lifts and their sum are one sum of 2 n + 4 products (2D) per node and component on the integer
// units, as are the traces and the cell average.  Euler fluxes are evaluated there too (fx_point):
// the FP64 pipe keeps the conversions to FP64, the root of the sound speed and the stage sums.
// put(j, trace, flux, radius) is called once for every face point of this thread (the radius the
// largest of its face), avg(c, value) once per cell and component with want_avg.  Warp collective.
//
// Near vacuum (a density at a node or a trace 2^-20 below the cell's largest, or not positive),
// for an energy that is not positive and for values outside the exponent range the cell takes the
// FP64 form: a rule of the cell's own values, so a cell's result does not depend on the cells it
// shares a warp with.  So does a 2D cell in which a node's density or energy is 2^-3 below the largest (kFxKeep;
// scalar laws: a row or a column of nodes): FP64 rounds a sum by its own row and column, which only in 1D always
// hold the cell's largest value.  At nodes whose row and column are small the error of G, in units of 2^-53
// of the magnitudes of a node's own terms, is the FP64 form's: 0.8 (Euler Q^2), 0.9 (Burgers Q^2) and 1.4
// (advection Q^3); without the rule it grew with the contrast (at 2^-9 to 77, 4e3 and 17).
//
// Why: with FP64 maps and fluxes a warp issues about 145 FP64 instructions per Q^3 stage, 76 cycles
// each; this form about 30, with 2000 instructions on the other pipes beside them: bound by issue and the
// FP64 pipe together.  Set state, steps, get state: 513^2 Q^3, 2 RK4 steps 15.9 ms with FP64 forms throughout,
// 4.20 with the integer ones here and in the final stage; 1024^2 Q^2, 3 Heun steps 49.6 and 17.0 ms.
template <class C, class Put, class Fn>
__device__ __forceinline__ void eval_G_fx(const Params &P, Smem<C> &S, const BlockTab<C> &Tb, int lc, int node,
                                          const double *u, double *g, bool want_speed, bool want_avg, Put put,
                                          Fn avg) {
    constexpr int DIM = C::D, N = C::NP, PHYS = C::PH;
    constexpr int M = C::M, NN = C::NN, NF = C::NF, NTR = C::NTR, FPT = C::FPT;
    constexpr int W = (M + 1) / 2;
    const int a = node % N, b = DIM == 2 ? node / N : 0;
    CellData<C> &D = S.c[lc];
    Fx(&fu)[M][NN] = reinterpret_cast<Fx(&)[M][NN]>(D.u);
    Fx(&ff)[C::D][M][NN] = reinterpret_cast<Fx(&)[C::D][M][NN]>(D.f);
    Fx(&ft)[M][NTR] = reinterpret_cast<Fx(&)[M][NTR]>(D.tf);
    auto field = [](const unsigned (&w)[W], int c) { return (int)((w[c >> 1] >> (16 * (c & 1))) & 0xffffu); };
    // whether round j gives this thread a face point: known at compile time but for a ragged last round
    auto is_point = [&](int j) { return (j + 1) * NN <= NTR || node + j * NN < NTR; };
    bool bad = P.fx.on == 0;
    // 1. node values in fixed point
    unsigned eu[W];
#pragma unroll
    for (int k = 0; k < W; ++k) eu[k] = 0u;
#pragma unroll
    for (int c = 0; c < M; ++c) {
        if (fx_exp(u[c]) > kFxExpHi) bad = true;
        eu[c >> 1] |= (unsigned)fx_exp(u[c]) << (16 * (c & 1));
    }
    const int e0 = eu[0] & 0xffffu;  // this node's density
#pragma unroll
    for (int k = 0; k < W; ++k) eu[k] = cell_max_halves<C>(eu[k], node);
    if constexpr (PHYS == PH_EULER) {
        if (!fx_state<DIM>(u) || e0 < field(eu, 0) - (DIM == 2 ? kFxKeep : 20)) bad = true;
        if (DIM == 2 && fx_exp(u[M - 1]) < field(eu, M - 1) - kFxKeep) bad = true;
    } else if constexpr (DIM == 2) {  // the flux of Burgers' law is a square
        if (line_max<C>(e0, node) < field(eu, 0) - (PHYS == PH_BURG ? 2 : kFxKeep)) bad = true;
    }
    cell_sync<C>();  // earlier readers of the cell's arrays are done
#pragma unroll
    for (int c = 0; c < M; ++c) fu[c][node] = fx_of(u[c], field(eu, c));
    cell_sync<C>();
    // 2. traces of this thread's face points and their fluxes
    FluxExp e{0u, 0u};
    long long tm[FPT][M];  // mantissas of the normal fluxes (Euler)
    int tx[FPT][3];        // their exponents: component 0, the momenta, the last
    double tf0[FPT];       // scalar laws: the flux itself
    double t[FPT][M];
#pragma unroll
    for (int j = 0; j < FPT; ++j) {
        const int fp = node + j * NN;
        if (is_point(j)) {
            const int face = fp / NF, pos = fp - face * NF;
            const int at = DIM == 1 || face < 2 ? pos * N : pos, step = DIM == 1 || face < 2 ? 1 : N;
            Fx l[N];
            load_fx<N>(Tb.tl[face & 1], l);
#pragma unroll
            for (int c = 0; c < M; ++c) {
                FxSum s{0, 0};
#pragma unroll
                for (int q = 0; q < N; ++q) fx_mac(s, fu[c][at + q * step], l[q]);
                t[j][c] = fx_double(fx_sum(s), fx_shift(field(eu, c), kFxTrace));
            }
            if constexpr (PHYS == PH_EULER) {
                if (!fx_state<DIM>(t[j]) || fx_exp(t[j][0]) < field(eu, 0) - 20) bad = true;
            }
        }
    }
    const bool any_bad = __any_sync(0xffffffffu, bad);
    const bool mine = any_bad && cell_any<C>(bad, node);  // this cell takes the FP64 form below
#pragma unroll
    for (int j = 0; j < FPT; ++j) {
        const int fp = node + j * NN;
        double f[M], sp = 0.0;
        if (is_point(j)) {
            const int dir = fp / NF >> 1;
            if constexpr (PHYS == PH_EULER) {
                FxPoint<DIM> o;
                fx_point<DIM>(t[j], P.fx.gas, o);
                if (want_speed) {
                    fx_face_flux<DIM>(o, t[j], dir, f);
                    sp = fx_face_speed<DIM>(P.fx.gas, o, dir);
                }
                const bool y = DIM == 2 && dir == 1;
                const long long nf = (y ? o.q[DIM - 1] : o.q[0]) + o.p;
                tm[j][0] = y ? o.m[DIM - 1] : o.m[0];
                tm[j][1] = y ? o.c : nf;
                if constexpr (DIM == 2) tm[j][2] = y ? nf : o.c;
                tm[j][M - 1] = fx_energy_flux<DIM>(o, dir);
                tx[j][0] = y ? o.xm[DIM - 1] : o.xm[0];
                tx[j][1] = o.X;
                tx[j][2] = o.X + (y ? o.xw[DIM - 1] : o.xw[0]) + 1;
                e.w0 = vmax_u16x2(e.w0, biased_exp(tx[j][0]) | biased_exp(o.X + 1) << 16);
                e.w1 = max(e.w1, biased_exp(tx[j][2] + 1));
            } else {
                sp = flux_speed_dir<PHYS, DIM>(P, t[j], dir, f);
                tf0[j] = f[0];
                e.w0 = max(e.w0, (unsigned)fx_exp(f[0]));
            }
        }
        if (want_speed) sp = face_max<C>(sp, node);
        if (is_point(j) && !mine) put(j, t[j], f, sp);
    }
    if (want_avg) {
        if constexpr (DIM == 2 && NN == 16 && M == 4) {  // four lanes of four nodes per component
            const int c = node >> 2, r = node & 3;
            FxSum s{0, 0};
            Fx v[4], w[4];
            load_fx<4>(&fu[c][4 * r], v);
            load_fx<4>(&Tb.w[4 * r], w);
#pragma unroll
            for (int q = 0; q < 4; ++q) fx_mac(s, v[q], w[q]);
            long long x = fx_sum(s);
            x += __shfl_xor_sync(0xffffffffu, x, 1);
            x += __shfl_xor_sync(0xffffffffu, x, 2);
            const double m = fx_double(x, fx_shift(field(eu, c), kFxAvg));
            if (r == 0) avg(c, m);
        } else {
            for (int c = node; c < M; c += NN) {
                FxSum s{0, 0};
#pragma unroll
                for (int q = 0; q < NN; ++q) fx_mac(s, fu[c][q], Tb.w[q]);
                avg(c, fx_double(fx_sum(s), fx_shift(field(eu, c), kFxAvg)));
            }
        }
        __syncwarp();
    }
    // 3. node fluxes; every flux of the cell in fixed point
    if constexpr (PHYS == PH_EULER) {
        FxPoint<DIM> o;
        fx_point<DIM>(u, P.fx.gas, o);
        long long h[DIM];
        int xh = kFxNone, x0 = kFxNone;
#pragma unroll
        for (int d = 0; d < DIM; ++d) {
            h[d] = fx_energy_flux<DIM>(o, d);
            xh = max(xh, o.X + o.xw[d] + 2);  // one more for 63 bits
            x0 = max(x0, o.xm[d]);
        }
        e.w0 = vmax_u16x2(e.w0, biased_exp(x0) | biased_exp(o.X + 1) << 16);
        e.w1 = max(e.w1, biased_exp(xh));
        e.w0 = cell_max_halves<C>(e.w0, node);
        e.w1 = cell_max_halves<C>(e.w1, node);
        const int E0 = e.w0 & 0xffffu, E1 = e.w0 >> 16, E2 = e.w1;
#pragma unroll
        for (int d = 0; d < DIM; ++d) {
            ff[d][0][node] = fx_limbs(o.m[d], o.xm[d], E0);
            ff[d][1 + d][node] = fx_limbs(o.q[d] + o.p, o.X, E1);
            ff[d][M - 1][node] = fx_limbs(h[d], o.X + o.xw[d] + 1, E2);
        }
        if constexpr (DIM == 2) ff[0][2][node] = ff[1][1][node] = fx_limbs(o.c, o.X, E1);
#pragma unroll
        for (int j = 0; j < FPT; ++j) {
            const int fp = node + j * NN;
            if (is_point(j)) {
                ft[0][fp] = fx_limbs(tm[j][0], tx[j][0], E0);
                ft[1][fp] = fx_limbs(tm[j][1], tx[j][1], E1);
                if constexpr (DIM == 2) ft[2][fp] = fx_limbs(tm[j][2], tx[j][1], E1);
                ft[M - 1][fp] = fx_limbs(tm[j][M - 1], tx[j][2], E2);
            }
        }
    } else {
        double fx[1], fy[1];
        if constexpr (DIM == 2) {
            flux_xy<PHYS>(P, u, fx, fy);
            e.w0 = max(e.w0, (unsigned)fx_exp(fy[0]));
        } else {
            flux_dir<PHYS, DIM>(P, u, 0, fx);
        }
        e.w0 = cell_max_halves<C>(max(e.w0, (unsigned)fx_exp(fx[0])), node);
        ff[0][0][node] = fx_of(fx[0], (int)e.w0);
        if constexpr (DIM == 2) ff[1][0][node] = fx_of(fy[0], (int)e.w0);
#pragma unroll
        for (int j = 0; j < FPT; ++j)
            if (is_point(j)) ft[0][node + j * NN] = fx_of(tf0[j], (int)e.w0);
    }
    cell_sync<C>();
    // 4. G: the row, the column and the four lifted face fluxes
    {
        Fx cx[N], cy[N], lx[2], ly[2];
        load_fx<N>(Tb.cx[a], cx);
        load_fx<2>(Tb.lx[a], lx);
        if constexpr (DIM == 2) {
            load_fx<N>(Tb.cy[b], cy);
            load_fx<2>(Tb.ly[b], ly);
        }
#pragma unroll
        for (int c = 0; c < M; ++c) {
            FxSum s{0, 0};
            Fx v[N];
            load_fx<N>(&ff[0][c][b * N], v);
#pragma unroll
            for (int q = 0; q < N; ++q) fx_mac(s, v[q], cx[q]);
            fx_mac(s, ft[c][b], lx[0]);
            fx_mac(s, ft[c][NF + b], lx[1]);
            if constexpr (DIM == 2) {
#pragma unroll
                for (int q = 0; q < N; ++q) fx_mac(s, ff[1][c][q * N + a], cy[q]);
                fx_mac(s, ft[c][2 * NF + a], ly[0]);
                fx_mac(s, ft[c][3 * NF + a], ly[1]);
            }
            const int E = (int)(c == 0 ? e.w0 & 0xffffu : c == M - 1 ? e.w1 : e.w0 >> 16);
            g[c] = fx_double(fx_sum(s), fx_shift(E, P.fx.k));
        }
    }
    if (any_bad) eval_G_64<C>(P, S, lc, node, u, g, mine, want_speed, want_avg, put, avg);
}

// ----------------------------------------------------------------------------- kernels

template <int DIM, int N, int PHYS>
__device__ __forceinline__ void load_node(const Params &P, const double *src, int cell, int node, bool active,
                                          double *u) {
    using C = Cfg<DIM, N, PHYS>;
#pragma unroll
    for (int c = 0; c < C::M; ++c) {
        if (active) {
            u[c] = src[((size_t)c * P.ncell + cell) * C::NN + node];
        } else {  // benign padding state for idle threads of the last block
            u[c] = (PHYS == PH_EULER && (c == 0 || c == C::M - 1)) ? 1.0 : (PHYS == PH_EULER ? 0.0 : 0.5 * (P.lo + P.hi));
        }
    }
}

template <int DIM, int N, int PHYS>
__device__ __forceinline__ void store_node(const Params &P, double *dst, int cell, int node, bool active,
                                           const double *u) {
    using C = Cfg<DIM, N, PHYS>;
    if (!active) return;
#pragma unroll
    for (int c = 0; c < C::M; ++c) dst[((size_t)c * P.ncell + cell) * C::NN + node] = u[c];
}

// Inner stages (cell-local, no neighbour data): for i = 1..s
//   u^(i) = u^n + dt sum_{j<i} a_ij G(u~^(j)),  u~^(i) = L(u^(i))   (eq. rkdg-lim)
// and the accumulation u* = u^n + dt sum_i b_i G(u~^(i)); the traces of every
// u~^(i) with b_i != 0 go to B.tr for the final kernel.
// The L2 projection of this thread's node values onto the total-degree space P^k (2D; a block
// collective): v at node = sum_q pk[node][q] v_q per component, through S.u.
template <class C>
__device__ __forceinline__ void project_pk(Smem<C> &S, int lc, int node, double *v) {
    if constexpr (C::D == 2) {
        constexpr int M = C::M, NN = C::NN;
        const NodalTables &T = c_tab[C::NP - 2];
        cell_sync<C>();  // earlier readers of S.u are done
#pragma unroll
        for (int c = 0; c < M; ++c) S.c[lc].u[c][node] = v[c];
        cell_sync<C>();
#pragma unroll
        for (int c = 0; c < M; ++c) {
            double s = 0.0;
#pragma unroll
            for (int q = 0; q < NN; ++q) s = fma(T.pk[node][q], S.c[lc].u[c][q], s);
            v[c] = s;
        }
        cell_sync<C>();  // S.u is free again
    }
}

// The source of Example 4.2's scenario I, S = d_t U + div F(U) of the manufactured solution
// rho = e^-t sin 2pi(x+y) + 2, w = (e^-t cos 2pi x sin 2pi y + 2, e^-t sin 2pi x cos 2pi y + 2),
// e = e^-t cos 2pi(x+y) / 2 + 1, at (x, y, t).  Each primitive q is held with its t-, x- and
// y-derivatives (q[0..3]); products by the product rule, then the four balance laws.
__device__ inline void scenario1_source(double gamma, double x, double y, double t, double *S) {
    const double w = 6.283185307179586, a = exp(-t);
    double sxy, cxy, sx, cx, sy, cy;
    sincos(w * (x + y), &sxy, &cxy);
    sincos(w * x, &sx, &cx);
    sincos(w * y, &sy, &cy);
    const double rho[4] = {a * sxy + 2.0, -a * sxy, w * a * cxy, w * a * cxy};
    const double vx[4] = {a * cx * sy + 2.0, -a * cx * sy, -w * a * sx * sy, w * a * cx * cy};
    const double vy[4] = {a * sx * cy + 2.0, -a * sx * cy, w * a * cx * cy, -w * a * sx * sy};
    const double ei[4] = {0.5 * a * cxy + 1.0, -0.5 * a * cxy, -0.5 * w * a * sxy, -0.5 * w * a * sxy};
    auto prod = [](const double *f, const double *g, double *h) {  // h = f g with its derivatives
        h[0] = f[0] * g[0];
#pragma unroll
        for (int d = 1; d < 4; ++d) h[d] = f[d] * g[0] + f[0] * g[d];
    };
    double mx[4], my[4], re[4], mxx[4], mxy[4], myy[4], kx[4], ky[4];
    prod(rho, vx, mx);   // rho w_x
    prod(rho, vy, my);   // rho w_y
    prod(rho, ei, re);   // rho e
    prod(mx, vx, mxx);   // rho w_x^2
    prod(mx, vy, mxy);   // rho w_x w_y
    prod(my, vy, myy);   // rho w_y^2
    double E[4], H[4], p[4];
#pragma unroll
    for (int d = 0; d < 4; ++d) {
        p[d] = (gamma - 1.0) * re[d];
        E[d] = re[d] + 0.5 * (mxx[d] + myy[d]);
        H[d] = E[d] + p[d];  // E + p
    }
    prod(H, vx, kx);  // (E + p) w_x
    prod(H, vy, ky);  // (E + p) w_y
    // index 1: d/dt, 2: d/dx, 3: d/dy
    S[0] = rho[1] + mx[2] + my[3];
    S[1] = mx[1] + mxx[2] + p[2] + mxy[3];
    S[2] = my[1] + mxy[2] + myy[3] + p[3];
    S[3] = E[1] + kx[2] + ky[3];
}

// G += S at this thread's node for stage i (time t0 + c_i dt, c_i the row sum of A): the
// collocated source is its projection by the (k+1)-point Gauss rule.
template <int DIM, int N, int PHYS>
__device__ __forceinline__ void add_source(const Params &P, int cell, int node, int stage, double *g) {
    if constexpr (DIM == 2 && PHYS == PH_EULER) {
        const NodalTables &T = c_tab[N - 2];
        double c = 0.0;
        for (int j = 0; j < stage; ++j) c += P.A[stage][j];
        const int cx = cell % P.nx, cy = cell / P.nx;
        const int a = node % N, b = node / N;
        const double hx = 2.0 / P.rhx, hy = 2.0 / P.rhy;
        const double x = P.x0 + (cx + 0.5 * (T.xg[a] + 1.0)) * hx;
        const double y = P.y0 + (cy + 0.5 * (T.xg[b] + 1.0)) * hy;
        double src[4];
        scenario1_source(P.gamma, x, y, P.t0 + c * P.dt, src);
#pragma unroll
        for (int k = 0; k < 4; ++k) g[k] += src[k];
    }
}

// FX: eval_G_fx; without it the FP64 form alone, for Euler problems out of the fixed-point range (gamma >= 2, cell
// sizes beyond 2^100), where eval_G_fx would evaluate both (1024^2 Q^2 with gamma = 2.2, 3 Heun steps:
// 48.0 -> 41.3 ms).  A kernel of its own: a branch inside took 2.5 to 6% of the other problems' time.
template <int DIM, int N, int PHYS, bool FX = true>
__device__ __forceinline__ void inner_body(const Params &P, const Bufs &B, int blk) {
    using C = CfgW<DIM, N, PHYS>;
    constexpr int M = C::M, NN = C::NN, NTR = C::NTR;
    __shared__ Smem<C> S;
    __shared__ BlockTab<C> Tb;
    int lc, node;
    place<C>(lc, node);
    const int cell = blk * C::NCB + lc;
    const bool active = cell < P.ncell;
    const bool own = active && owned(P, cell) && !solid_cell(P, cell);  // counts in the flag and statistics
    fill_tab<C>(P, Tb);
    double un[M], cur[M], acc[M], g[M];
    // only a tableau with entries below its sub-diagonal needs the earlier stages' G: local memory
    bool sub = true;
    for (int i = 2; i < P.s; ++i)
        for (int j = 0; j + 1 < i; ++j) sub = sub && !nonzero_bits(P.A[i][j]);
    double gh[MAXS][M];
    load_node<DIM, N, PHYS>(P, B.un, cell, node, active, un);
#pragma unroll
    for (int c = 0; c < M; ++c) cur[c] = acc[c] = un[c];
    __syncthreads();
    const size_t at = (size_t)cell * NTR + node, cstr = (size_t)P.ncell * NTR;
    double fs[C::FPT][M];  // sum_i b_i f(u_int^(i)) at this thread's face points
#pragma unroll
    for (int j = 0; j < C::FPT; ++j)
#pragma unroll
        for (int c = 0; c < M; ++c) fs[j][c] = 0.0;
    // not unrolled: four copies of a stage would not fit the instruction cache
#pragma unroll 1
    for (int i = 0; i < P.s; ++i) {
        if (i > 0) {
#pragma unroll
            for (int c = 0; c < M; ++c) cur[c] = un[c];
            if (sub) {
#pragma unroll
                for (int c = 0; c < M; ++c) cur[c] = fma(Tb.dtA[i][i - 1], g[c], cur[c]);
            } else {
#pragma unroll 1
                for (int j = 0; j < i; ++j)
                    if (nonzero_bits(P.A[i][j]))
#pragma unroll
                        for (int c = 0; c < M; ++c) cur[c] = fma(Tb.dtA[i][j], gh[j][c], cur[c]);
            }
            if (P.pk) project_pk<C>(S, lc, node, cur);
            double pts[C::PPT][M];
            float rhi;
            limit_block(P, B, S, lc, node, own, cur, pts, true, true, false, rhi);
        }
        const int slot = P.slot[i];
        const bool traced = slot >= 0 && active;
        const bool keep_faces = slot >= 0 && B.tsum != nullptr;
        double *dst = B.tr + (size_t)max(slot, 0) * M * P.ncell * NTR;
        auto put = [&](int j, const double *t, const double *f, double sp) {
            if (traced)
#pragma unroll
                for (int c = 0; c < M; ++c) dst[at + j * NN + c * cstr] = t[c];
            if (keep_faces) {
#pragma unroll
                for (int c = 0; c < M; ++c) fs[j][c] = fma(P.b[i], f[c], fs[j][c]);
                const int fp = node + j * NN;
                if (active && fp % C::NF == 0)
                    B.tsp[((size_t)slot * P.ncell + cell) * (2 * DIM) + fp / C::NF] = sp;
            }
        };
        auto avg = [&](int c, double v) {
            if (active) B.tavg[((size_t)slot * M + c) * P.ncell + cell] = v;  // outflow exterior state
        };
        if constexpr (FX)
            eval_G_fx<C>(P, S, Tb, lc, node, cur, g, keep_faces, slot >= 0, put, avg);
        else
            eval_G_64<C>(P, S, lc, node, cur, g, true, keep_faces, slot >= 0, put, avg);
        if (P.source && active) add_source<DIM, N, PHYS>(P, cell, node, i, g);
        if (!sub)
#pragma unroll
            for (int c = 0; c < M; ++c) gh[i][c] = g[c];
        if (P.mode == MODE_OP_G) {
#pragma unroll
            for (int c = 0; c < M; ++c) acc[c] = g[c];
        } else if (nonzero_bits(P.b[i])) {
#pragma unroll
            for (int c = 0; c < M; ++c) acc[c] = fma(Tb.dtb[i], g[c], acc[c]);
        }
    }
    if (B.tsum != nullptr && active)
#pragma unroll
        for (int j = 0; j < C::FPT; ++j)
            if (node + j * NN < NTR)
#pragma unroll
                for (int c = 0; c < M; ++c) B.tsum[at + j * NN + c * cstr] = fs[j][c];
    if (P.pk) project_pk<C>(S, lc, node, acc);
    if (active && solid_cell(P, cell))  // outside the domain: G = 0, u* = u^n
#pragma unroll
        for (int c = 0; c < M; ++c) acc[c] = P.mode == MODE_OP_G ? 0.0 : un[c];
    store_node<DIM, N, PHYS>(P, B.ustar, cell, node, active, acc);
}

template <int DIM, int N, int PHYS, bool FX>
__global__ void __launch_bounds__(kWarpThreads, 4) k_inner(const __grid_constant__ Params P, const __grid_constant__ Bufs B) {
    inner_body<DIM, N, PHYS, FX>(P, B, blockIdx.x);
}

// u += dt lift(dc) at this thread's node, dc the corrections of this thread's face points (a cell
// collective): the four products per component in fixed point with one exponent per cell and
// component (dg_fixed.h), as in eval_G_fx; corrections outside its range take the FP64 form.  So do the cells
// where a node's four corrections are all 2^-3 below the cell's largest, which FP64 would round by their own
// size, unless what the largest can add is below the node's own value: then 2^-55 of it (six units of 2^-58)
// does not reach the rounding of the result.
template <class C>
__device__ __forceinline__ void lift_faces(const Params &P, double dt, CellData<C> &D, int node, int a, int b,
                                           const double (&dc)[C::FPT][C::M], double *u) {
    constexpr int DIM = C::D, N = C::NP, M = C::M, NN = C::NN, NF = C::NF, NTR = C::NTR, FPT = C::FPT;
    constexpr int W = (M + 1) / 2;
    unsigned ef[W];
    bool bad = false;
#pragma unroll
    for (int k = 0; k < W; ++k) ef[k] = 0u;
#pragma unroll
    for (int c = 0; c < M; ++c) {
        int e = 0;
#pragma unroll
        for (int j = 0; j < FPT; ++j)
            if (node + j * NN < NTR) {
                const int ej = fx_exp(dc[j][c]);
                if (ej > 1023 + 800) bad = true;
                e = max(e, ej);
            }
        ef[c >> 1] |= (unsigned)e << (16 * (c & 1));
    }
    Fx(&ft)[M][NTR] = reinterpret_cast<Fx(&)[M][NTR]>(D.tf);
#pragma unroll
    for (int k = 0; k < W; ++k) ef[k] = cell_max_halves<C>(ef[k], node);
#pragma unroll
    for (int c = 0; c < M; ++c) {
        const int E = (int)((ef[c >> 1] >> (16 * (c & 1))) & 0xffffu);
#pragma unroll
        for (int j = 0; j < FPT; ++j) {
            const int fp = node + j * NN;
            if (fp < NTR) ft[c][fp] = fx_of(dc[j][c], E);
        }
    }
    const Fx x0 = P.fx.lx[a][0], x1 = P.fx.lx[a][1], y0 = P.fx.ly[b][0], y1 = P.fx.ly[b][1];
    cell_sync<C>();
    double v[M];
    const int reach = 58 - P.fx.k + fx_exp(dt) - 1023;  // exponent of dt times the sum of the coefficients
#pragma unroll
    for (int c = 0; c < M; ++c) {
        const int E = (int)((ef[c >> 1] >> (16 * (c & 1))) & 0xffffu);
        FxSum s{0, 0};
        if constexpr (DIM == 2) {
            const Fx f[4] = {ft[c][b], ft[c][NF + b], ft[c][2 * NF + a], ft[c][3 * NF + a]};
            fx_mac(s, f[0], x0);
            fx_mac(s, f[1], x1);
            fx_mac(s, f[2], y0);
            fx_mac(s, f[3], y1);
            int top = 0, any = 0;  // leading bits of the four: 2^(30 - j) for a value 2^-j of the largest
#pragma unroll
            for (int q = 0; q < 4; ++q) top |= f[q].h ^ (f[q].h >> 31), any |= f[q].h | f[q].l;
            if (top >> (30 - kFxKeep) == 0 && any != 0 && E + reach >= fx_exp(u[c])) bad = true;
        } else {
            fx_mac(s, ft[c][b], x0);
            fx_mac(s, ft[c][NF + b], x1);
        }
        v[c] = fx_double(fx_sum(s), fx_shift(E, P.fx.k));
    }
    if (P.fx.on == 0 || __any_sync(0xffffffffu, bad)) {
        const NodalTables &T = c_tab[N - 2];
        cell_sync<C>();  // the cell's corrections have been read
#pragma unroll
        for (int j = 0; j < FPT; ++j) {
            const int fp = node + j * NN;
            if (fp < NTR)
#pragma unroll
                for (int c = 0; c < M; ++c) D.tf[fp][c] = dc[j][c];
        }
        cell_sync<C>();
        bad = cell_any<C>(bad || P.fx.on == 0, node);
#pragma unroll
        for (int c = 0; c < M; ++c) {
            double cx = -T.liftp[a] * D.tf[NF + b][c] + T.liftm[a] * D.tf[b][c];
            double w = P.rhx * cx;
            if constexpr (DIM == 2) {
                double cy = -T.liftp[b] * D.tf[3 * NF + a][c] + T.liftm[b] * D.tf[2 * NF + a][c];
                w = fma(P.rhy, cy, w);
            }
            if (bad) v[c] = w;
        }
        cell_sync<C>();
    }
#pragma unroll
    for (int c = 0; c < M; ++c) u[c] = fma(dt, v[c], u[c]);
}

// Corrections of the interior faces of a 2D mesh, one thread per face point (a cell's lower faces): for the
// cells on both sides dc = sum_i b_i (fhat^(i) - f_int^(i)) = (F_ext - F_int) / 2 - sum_i b_i alpha^(i) (u_R^(i) -
// u_L^(i)) / 2, F the weighted flux sums, from what the inner kernel stored.  In the final kernel every face
// was evaluated by both of its cells, in Q^2 by two rounds of nine threads for twelve points, all on the
// FP64 pipe (84% busy).
template <int N, int PHYS>
__global__ void __launch_bounds__(128) k_faces(const __grid_constant__ Params P, const __grid_constant__ Bufs B) {
    constexpr int M = ncomp(PHYS, 2), NTR = 4 * N;
    const size_t per = (size_t)P.ncell * N, e = (size_t)blockIdx.x * 128 + threadIdx.x;  // points of a direction
    if (e >= 2 * per) return;
    const int dir = e >= per, face = 2 * dir;
    const size_t at = dir ? e - per : e;  // cell * N + pos
    const int cell = (int)(at / N), pos = (int)(at - (size_t)cell * N);
    // the cell below, whatever condition either side of the face has: the final kernel decides side by side
    const int cy = cell / P.nx, cx = cell - cy * P.nx;
    const bool wrap = P.bc[face] == BC_PERIODIC || P.bc[face + 1] == BC_PERIODIC;
    if ((dir ? cy : cx) == 0 && !wrap) return;
    const int nb = dir ? (cy > 0 ? cell - P.nx : cell + (P.ny - 1) * P.nx) : (cx > 0 ? cell - 1 : cell + P.nx - 1);
    const size_t cstr = (size_t)P.ncell * NTR, ro = (size_t)cell * NTR + face * N + pos, lo = (size_t)nb * NTR + (face + 1) * N + pos;
    double dc[M];
#pragma unroll
    for (int c = 0; c < M; ++c) dc[c] = 0.0;
    for (int i = 0; i < P.s; ++i) {
        const int q = P.slot[i];
        if (q < 0) continue;
        const double *tr = B.tr + (size_t)q * M * cstr, *sp = B.tsp + (size_t)q * P.ncell * 4;
        const double ba = half_of(P.b[i]) * fmax_nonneg(sp[(size_t)cell * 4 + face], sp[(size_t)nb * 4 + face + 1]);
#pragma unroll
        for (int c = 0; c < M; ++c) dc[c] = fma(ba, tr[c * cstr + lo] - tr[c * cstr + ro], dc[c]);
    }
#pragma unroll
    for (int c = 0; c < M; ++c) {
        const double d = B.tsum[c * cstr + lo] - B.tsum[c * cstr + ro];
        B.fc[(size_t)(2 * dir * M + c) * per + at] = fma(0.5, d, dc[c]);         // the cell above the face
        B.fc[(size_t)((2 * dir + 1) * M + c) * per + at] = fma(-0.5, d, dc[c]);  // and below
    }
}

// Final stage: u^{n+1} = u* + dt lift( sum_i b_i (fhat^(i) - f(u_int^(i))) ), then the
// limiter, the admissibility test and a0 of the new state.  Each face flux is
// evaluated from the same differences by both cells sharing the face, so the update is
// conservative to round-off.  The face corrections come from k_faces (FACES: 2D steps), boundary faces
// excepted; or from the flux sums and radii that the inner kernel stored (STORED: ensembles, 1D); or
// all of it is evaluated here (RECOMPUTED: the operators without a handle).  The lift runs in fixed
// point, and the rate is taken only by warps that can raise it.
enum FaceSource { RECOMPUTED = 0, STORED = 1, FACES = 2 };
template <int DIM, int N, int PHYS, int FROM = RECOMPUTED>
__device__ __forceinline__ void final_body(const Params &P, const Bufs &B, int blk) {
    using C = CfgW<DIM, N, PHYS>;
    constexpr int M = C::M, NN = C::NN, NF = C::NF, NTR = C::NTR, FPT = C::FPT;
    __shared__ Smem<C> S;
    int lc, node;
    place<C>(lc, node);
    const int cell = blk * C::NCB + lc;
    const bool active = cell < P.ncell;
    const bool own = active && owned(P, cell) && !solid_cell(P, cell);  // counts in the flag, statistics and rate
    const int a = node % N, b = DIM == 2 ? node / N : 0;
    double u[M];
    load_node<DIM, N, PHYS>(P, B.ustar, cell, node, active, u);

    // dc = sum_i b_i (fhat^(i) - f_int^(i)) = (F_ext - F_int) / 2 -+ sum_i b_i alpha^(i) (u_ext^(i) - u_int^(i)) / 2
    // with F = sum_i b_i f^(i), the sign of the side: both cells of a face form the same
    // differences.  The exterior state of a boundary face is always evaluated here.
    CellData<C> &D = S.c[lc];
    // running sums F of this thread's face points: the point's own lane forms them, and the lanes that shadow it
    // read them behind the warp barrier (six Q^2 lanes hold the same point)
    const bool first = !shadow_lane<C>();
    double(&sI)[NTR][M] = D.tf;
    double(&sE)[NTR][M] = reinterpret_cast<double(&)[NTR][M]>(D.f);
    const size_t cstr = (size_t)P.ncell * NTR;
    double dc[FPT][M];
    size_t noff[FPT];  // the partner point's offset within a component's block
    int nbr[FPT];
    bool here = FROM != FACES;  // a face point of this thread is evaluated here
#pragma unroll
    for (int j = 0; j < FPT; ++j) {
        const int fp = node + j * NN, face = fp / NF, pos = fp - face * NF;
        nbr[j] = -1;
        noff[j] = 0;
        if (fp < NTR && active) {
            nbr[j] = neighbour_geo(P, cell, face);
            if (nbr[j] >= 0) noff[j] = (size_t)nbr[j] * NTR + (face ^ 1) * NF + pos;
            here = here || nbr[j] < 0;
        }
#pragma unroll
        for (int c = 0; c < M; ++c) dc[j][c] = 0.0;
        if (FROM == FACES && nbr[j] >= 0) {
            const double *fc = B.fc + (size_t)face * M * P.ncell * NF + (size_t)((face & 1) ? nbr[j] : cell) * NF + pos;
#pragma unroll
            for (int c = 0; c < M; ++c) dc[j][c] = fc[(size_t)c * P.ncell * NF];
        }
    }
    if (__any_sync(0xffffffffu, here)) {
#pragma unroll
        for (int j = 0; j < FPT; ++j)
            if (node + j * NN < NTR && first)
#pragma unroll
                for (int c = 0; c < M; ++c) sE[node + j * NN][c] = sI[node + j * NN][c] = 0.0;
        for (int i = 0; i < P.s; ++i) {
            if (P.slot[i] < 0) continue;
            const double *tr = B.tr + (size_t)P.slot[i] * M * cstr;
            const double *sps = FROM != RECOMPUTED ? B.tsp + (size_t)P.slot[i] * P.ncell * (2 * DIM) : nullptr;
            const double bi = P.b[i];
#pragma unroll
            for (int j = 0; j < FPT; ++j) {
                const int fp = node + j * NN;
                const int face = fp / NF, pos = fp - face * NF, dir = face >> 1;
                const bool mine = fp < NTR && active && (FROM != FACES || nbr[j] < 0);
                double ui[M], ue[M], alpha = 0.0;
                if (mine) {
                    const int nb = nbr[j];
                    double f[M];
#pragma unroll
                    for (int c = 0; c < M; ++c) ui[c] = tr[c * cstr + (size_t)cell * NTR + fp];
                    if constexpr (FROM != RECOMPUTED) {
                        alpha = sps[(size_t)cell * (2 * DIM) + face];
                    } else {
                        alpha = fmax_nonneg(alpha, face_flux<PHYS, DIM>(P, ui, dir, true, f));
                        if (first)
#pragma unroll
                            for (int c = 0; c < M; ++c) sI[fp][c] = fma(bi, f[c], sI[fp][c]);
                    }
                    if (nb >= 0) {
#pragma unroll
                        for (int c = 0; c < M; ++c) ue[c] = tr[c * cstr + noff[j]];
                        if constexpr (FROM != RECOMPUTED)
                            alpha = fmax_nonneg(alpha, sps[(size_t)nb * (2 * DIM) + (face ^ 1)]);
                    } else {
                        double av[M];
#pragma unroll
                        for (int c = 0; c < M; ++c) av[c] = B.tavg[((size_t)P.slot[i] * M + c) * P.ncell + cell];
                        if (P.geo != nullptr)
                            geo_exterior<PHYS, DIM, N>(P, cell, face, pos, i, ui, av, ue);
                        else
                            exterior_state<PHYS, DIM>(P, face, ui, av, ue);
                    }
                    if (FROM == RECOMPUTED || nb < 0) {
                        alpha = fmax_nonneg(alpha, face_flux<PHYS, DIM>(P, ue, dir, true, f));
                        if (first)
#pragma unroll
                            for (int c = 0; c < M; ++c) sE[fp][c] = fma(bi, f[c], sE[fp][c]);
                    }
                }
                __syncwarp();
                alpha = face_max<C>(alpha, node);  // per-edge LF viscosity: max over the edge's points
                if (mine) {
                    const double h = half_of(bi);
                    const double ba = ((face & 1) ? -h : h) * alpha;
#pragma unroll
                    for (int c = 0; c < M; ++c) dc[j][c] = fma(ba, ue[c] - ui[c], dc[j][c]);
                }
            }
        }
        __syncwarp();  // the sums are complete
#pragma unroll
        for (int j = 0; j < FPT; ++j) {
            const int fp = node + j * NN;
            if (fp < NTR && active && (FROM != FACES || nbr[j] < 0))
#pragma unroll
                for (int c = 0; c < M; ++c) {
                    const double FI = FROM != RECOMPUTED ? B.tsum[c * cstr + (size_t)cell * NTR + fp] : sI[fp][c];
                    const double FE = FROM != RECOMPUTED && nbr[j] >= 0 ? B.tsum[c * cstr + noff[j]] : sE[fp][c];
                    dc[j][c] = fma(0.5, FE - FI, dc[j][c]);
                }
        }
    }
    cell_sync<C>();
    lift_faces<C>(P, P.dt, S.c[lc], node, a, b, dc, u);
    if (P.pk) project_pk<C>(S, lc, node, u);
    if (P.mode == MODE_OP_F) {
        if (active && solid_cell(P, cell))  // outside the domain: no operator
#pragma unroll
            for (int c = 0; c < M; ++c) u[c] = 0.0;
        store_node<DIM, N, PHYS>(P, B.unew, cell, node, active, u);
        return;
    }
    if (P.defer_limit) {  // averages and their admissibility here; limiters in k_trouble
#pragma unroll
        for (int c = 0; c < M; ++c) S.c[lc].u[c][node] = u[c];
        cell_sync<C>();
        cell_averages<C>(S.c[lc].u, node, [&](int c, double s) {
            S.c[lc].avg[c] = s;
            if (active) B.aux[(size_t)cell * M + c] = s;
        });
        cell_sync<C>();
        bool check = node == 0 && own;
        if (check) {  // the FP32 screen of the average (truncated: 2^-22 of it) clears most cells
            float v[M], e[M];
#pragma unroll
            for (int c = 0; c < M; ++c) {
                v[c] = PHYS == PH_EULER ? trunc_f(S.c[lc].avg[c]) : (float)S.c[lc].avg[c];
                e[c] = 2.384185791015625e-07f * fabsf(v[c]);
            }
            check = !screen_point<PHYS, DIM>(P, v, e);
        }
        if (check && !admissible<PHYS, DIM>(P, S.c[lc].avg)) atomicOr(B.flag, 1);
        store_node<DIM, N, PHYS>(P, B.unew, cell, node, active, u);
        return;
    }
    double pts[C::PPT][M];
    float rhi;
    const bool cleared = limit_block(P, B, S, lc, node, own, u, pts, true, true, true, rhi);
    // wave-speed rate of the new state over its S_K points (next trial step)
    post_rate<C>(P, B, S, lc, node, own, cleared, rhi, pts);
    if (active && solid_cell(P, cell)) load_node<DIM, N, PHYS>(P, B.un, cell, node, true, u);  // keeps u^n
    store_node<DIM, N, PHYS>(P, B.unew, cell, node, active, u);
}

// Resident blocks per SM the FP64 final kernel's register budget is sized for (96 registers).
constexpr int fp64_final_min_blocks() { return 5; }

template <int DIM, int N, int PHYS, int FROM>
__global__ void __launch_bounds__(kWarpThreads, fp64_final_min_blocks())
    k_final(Params P, Bufs B) {
    final_body<DIM, N, PHYS, FROM>(P, B, blockIdx.x);
}

// Limiter applied to a state (set-up projection, operator checks): un -> unew.  In
// MODE_RATE it also posts the wave-speed rate of the limited state to B.a0, from the
// same interpolation of the same values that the scan kernel would take.
template <int DIM, int N, int PHYS>
__global__ void __launch_bounds__(kWarpThreads) k_limit(Params P, Bufs B) {
    using C = CfgW<DIM, N, PHYS>;
    __shared__ Smem<C> S;
    int lc, node;
    place<C>(lc, node);
    const int cell = blockIdx.x * C::NCB + lc;
    const bool active = cell < P.ncell;
    const bool own = active && owned(P, cell) && !solid_cell(P, cell);
    const bool rate = P.mode == MODE_RATE || P.mode == MODE_LIMIT_FINAL;
    const bool check = P.mode == MODE_LIMIT_CHECK || P.mode == MODE_LIMIT_FINAL;  // standard RKDG stages
    double u[C::M], pts[C::PPT][C::M];
    load_node<DIM, N, PHYS>(P, B.un, cell, node, active, u);
    if (P.pk) project_pk<C>(S, lc, node, u);  // a state set in P^k: its L2 projection first
    float rhi;
    const bool cleared = limit_block(P, B, S, lc, node, own, u, pts, check, check, rate, rhi);
    if (rate) post_rate<C>(P, B, S, lc, node, own, cleared, rhi, pts);
    if (active && solid_cell(P, cell)) load_node<DIM, N, PHYS>(P, B.un, cell, node, true, u);  // not limited
    store_node<DIM, N, PHYS>(P, B.unew, cell, node, active, u);
}

// a0 over the S_K points of un, and the two smallest bound margins.
template <int DIM, int N, int PHYS>
__global__ void __launch_bounds__(kWarpThreads) k_scan(Params P, Bufs B) {
    using C = CfgW<DIM, N, PHYS>;
    constexpr int M = C::M, NN = C::NN;
    __shared__ Smem<C> S;
    int lc, node;
    place<C>(lc, node);
    const int cell = blockIdx.x * C::NCB + lc;
    const bool active = cell < P.ncell;
    const bool own = active && owned(P, cell) && !solid_cell(P, cell);
    double u[M];
    load_node<DIM, N, PHYS>(P, B.un, cell, node, active, u);
#pragma unroll
    for (int c = 0; c < M; ++c) S.c[lc].u[c][node] = u[c];
    cell_sync<C>();
    double amax = 0.0, m0 = INFINITY, m1 = INFINITY;
    const bool margins = P.mode != MODE_RATE;
#pragma unroll
    for (int j = 0; j < C::PPT; ++j) {
        int p = node + j * NN;
        if (p < C::NSK && own) {
            double v[M];
            sk_eval<DIM, N, M, NN>(S.c[lc].u, p, v);
            amax = fmax(amax, sk_rate<PHYS, DIM>(P, v));
            if (!margins) continue;
            double a0m, a1m;
            if constexpr (PHYS == PH_EULER) {
                a0m = v[0] - P.eps;
                a1m = rho_e<DIM>(v) - P.eps;
            } else {
                a0m = v[0] - P.lo;
                a1m = P.hi - v[0];
            }
            m0 = (a0m == a0m) ? fmin(m0, a0m) : -INFINITY;
            m1 = (a1m == a1m) ? fmin(m1, a1m) : -INFINITY;
        }
    }
    // extremes on the integer units: the rate is non-negative; the margins as ordbits keys
    unsigned long long ab = dbits(amax), k0 = ordbits(m0), k1 = ordbits(m1);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        ab = umax64(ab, __shfl_xor_sync(0xffffffffu, ab, o));
        if (margins) {
            k0 = umin64(k0, __shfl_xor_sync(0xffffffffu, k0, o));
            k1 = umin64(k1, __shfl_xor_sync(0xffffffffu, k1, o));
        }
    }
    if ((threadIdx.x & 31) == 0) {
        if (ab > 0ull) atomicMax(B.a0, ab);
        if (margins) {
            atomicMin(&B.ord[0], k0);
            atomicMin(&B.ord[1], k1);
        }
    }
}

// Cell averages of un -> aux[cell][m]
template <int DIM, int N, int PHYS>
__global__ void k_avg(Params P, Bufs B) {
    using C = Cfg<DIM, N, PHYS>;
    const NodalTables &T = c_tab[N - 2];
    int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= P.ncell * C::M) return;
    int cell = t / C::M, c = t - cell * C::M;
    const double *u = B.un + ((size_t)c * P.ncell + cell) * C::NN;
    double s = 0.0;
#pragma unroll
    for (int q = 0; q < C::NN; ++q) s = fma(DIM == 2 ? T.w2[q] : T.w1[q], u[q], s);
    B.aux[t] = s;
}

// x < 0.0 (false for -0 and NaN)
__device__ __forceinline__ bool negative_bits(double x) {
    const unsigned long long b = dbits(x);
    return b > 0x8000000000000000ull && b <= 0xfff0000000000000ull;
}
// minmod(a, b, c): the argument of least magnitude when all three share one sign, else 0,
// on the integer units (for values of one sign the one of least magnitude has the
// smallest bit pattern)
__device__ __forceinline__ double minmod3_bits(double a, double b, double c) {
    const bool pos = positive_bits(a) && positive_bits(b) && positive_bits(c);
    const bool neg = negative_bits(a) && negative_bits(b) && negative_bits(c);
    return (pos || neg) ? bitsd(umin64(dbits(a), umin64(dbits(b), dbits(c)))) : 0.0;
}
// The TVB-modified minmod test of one face-averaged trace deviation t against the
// neighbour differences dp, dm and the threshold thr: true when minmod changes t, i.e.
// (|t| <= thr ? t : minmod(t, dp, dm)) != t, on the integer units.  thr_ok = thr >= 0.
__device__ __forceinline__ bool tvb_changes(double t, double dp, double dm, double thr, bool thr_ok) {
    constexpr unsigned long long kAbs = 0x7fffffffffffffffull;
    if (thr_ok && (dbits(t) & kAbs) <= (dbits(thr) & kAbs)) return false;
    if (isnan_bits(t)) return true;  // a NaN deviation compares unequal to itself
    const unsigned long long m = dbits(minmod3_bits(t, dp, dm)), tb = dbits(t);
    return m != tb && ((m | tb) << 1) != 0ull;  // +0 and -0 compare equal
}

// The same decision in fixed point, all in one unit: t the deviation of the face average, dp and dm the
// neighbour differences, thr the threshold (below zero: none).
__device__ __forceinline__ bool tvb_changes_fx(long long t, long long dp, long long dm, long long thr) {
    if (thr >= 0 && (t < 0 ? -t : t) <= thr) return false;
    return t > 0 ? dp < t || dm < t : t < 0 && (dp > t || dm > t);
}
// x in units of 2^(E - 1081), E >= fx_exp(x), as one number
__device__ __forceinline__ long long fx_whole(double x, int E) {
    const Fx f = fx_of(x, E);
    return ((long long)f.h << 28) + f.l;
}
// The plain indicator's decision of one direction and component in fixed point: sR, sL the face averages in units
// of 2^(En - 1081) (sums of node values with the weights scaled by 2^kFxTrace), own, lo, hi the averages of the
// cell and its neighbours.  0 kept, 1 troubled, 2 left to FP64 (tvb_pair_64): infinities and NaN, a neighbour's
// average 2^kFxKeep above the node values (whose units would then be too coarse), and a deviation and a threshold
// that are both within FP64's own rounding (2^-52 of the largest value: constant cells without a
// threshold).  FP64 sums of the node values took 18 fused multiply-adds (76 cycles each) in Q^2: 501 x
// 397 Q^2, troubled-cell pass 186 -> 110 us, features 247 -> 164 us.
__device__ __forceinline__ int tvb_pair(long long sR, long long sL, int En, double own, double lo, double hi,
                                        double thr) {
    const int E = max(max(En, fx_exp(own)), max(fx_exp(lo), fx_exp(hi)));
    if (E == 0x7ff || E > En + kFxKeep) return 2;
    const int sh = E - En;
    const long long o = fx_whole(own, E), l = fx_whole(lo, E), h = fx_whole(hi, E);
    const int et = fx_exp(thr);
    long long th = 1ll << 62;  // larger than every deviation
    if (!(thr >= 0.0)) th = -1;
    else if (et <= E) th = fx_whole(thr, E);
    else if (et <= E + 3) th = fx_whole(thr, et) << (et - E);
    const long long tR = (sR >> sh) - o, tL = o - (sL >> sh);
    constexpr long long kNoise = 64;  // units of 2^-58
    if (th < kNoise && ((tR < 0 ? -tR : tR) < kNoise || (tL < 0 ? -tL : tL) < kNoise)) return 2;
    return tvb_changes_fx(tR, h - o, o - l, th) || tvb_changes_fx(tL, h - o, o - l, th) ? 1 : 0;
}
// The same in FP64 from the node values u of a component.  Out of line: rare.
template <int DIM, int N>
__device__ __noinline__ bool tvb_pair_64(const double *u, int d, double own, double lo, double hi, double thr) {
    const NodalTables &T = c_tab[N - 2];
    double fr = 0.0, fl = 0.0;
    for (int q = 0; q < (DIM == 2 ? N * N : N); ++q) {
        fr = fma(DIM == 2 ? T.trw2[d][0][q] : T.lp[q], u[q], fr);
        fl = fma(DIM == 2 ? T.trw2[d][1][q] : T.lm[q], u[q], fl);
    }
    const double dp = hi - own, dm = own - lo;
    return tvb_changes(fr - own, dp, dm, thr, thr >= 0.0) || tvb_changes(own - fl, dp, dm, thr, thr >= 0.0);
}

// 2^k, k in [-126, 127]
__device__ __forceinline__ float pow2f(int k) { return __int_as_float((k + 127) << 23); }

// u as a sum of two floats: its leading 24 bits and the rest, on the integer units
__device__ __forceinline__ void two_floats(double u, float &h, float &l) {
    h = trunc_f(u);
    const int e = (int)((dbits(u) >> 52) & 0x7ffu) - 1023;
    const float r = (float)(int)(dbits(u) & 0x1fffffffull) * 1.862645149230957e-09f;  // 2^-29
    l = e - 23 >= -126 && e < 128 ? copysignf(r * pow2f(e - 23), h) : 0.0f;
}
// d 2^-60 likewise
__device__ __forceinline__ void two_floats_fx(long long d, float &h, float &l) {
    const unsigned long long m = d < 0 ? 0ull - (unsigned long long)d : (unsigned long long)d;
    const int z = min(__clzll((long long)m), 63);
    const unsigned long long a = m << z;
    h = (float)(int)(a >> 40) * pow2f(-20 - z);
    l = (float)((int)(a >> 16) & 0xffffff) * pow2f(-44 - z);
    if (d < 0) h = -h, l = -l;
}

// Average of component c of the neighbour of `cell` across `side` (the averages are in
// aux, [cell][m]); across a domain boundary, the boundary condition applied to the
// cell's own average.
template <int PHYS, int DIM>
__device__ __forceinline__ double nb_average(const Params &P, const double *aux, int cell, int side, int c) {
    constexpr int M = ncomp(PHYS, DIM);
    const int nb = neighbour(P, cell, side);
    if (nb >= 0) return aux[(size_t)nb * M + c];
    double own[M], ext[M];
#pragma unroll
    for (int i = 0; i < M; ++i) own[i] = aux[(size_t)cell * M + i];
    boundary_state<PHYS, DIM>(P, side, own, ext);
    return ext[c];
}

// Plain troubled-cell indicator and shock limiter, then the scaling limiter (an
// optional anti-oscillation stage outside the paper's method, run once per step
// after the final stage so the inner stages stay compact).  Per component and
// direction: face-averaged trace deviations ut_R = avg_face(u_R) - ubar,
// ut_L = ubar - avg_face(u_L) against D+ / D- of the cell averages (neighbours
// across a boundary follow its condition); the cell is troubled if the
// TVB-modified minmod changes either deviation.  A troubled cell becomes
// ubar + minmod(c_x, D+x, D-x) xi + minmod(c_y, D+y, D-y) eta, with c_x, c_y its
// first Legendre moments.  Reads unew and the averages in aux; writes unew.
template <int DIM, int N, int PHYS>
__device__ __forceinline__ void trouble_body(const Params &P, const Bufs &B, int blk) {
    using C = CfgW<DIM, N, PHYS>;
    constexpr int M = C::M, NN = C::NN;
    __shared__ Smem<C> S;
    __shared__ double sP1[C::NCB][2][M];
    __shared__ int sTr[C::NCB];
    const NodalTables &T = c_tab[N - 2];
    int lc, node;
    place<C>(lc, node);
    const int cell = blk * C::NCB + lc;
    const bool active = cell < P.ncell;
    const int a = node % N, b = DIM == 2 ? node / N : 0;
    double u[M];
    load_node<DIM, N, PHYS>(P, B.unew, cell, node, active, u);
    // node values in fixed point with one exponent per cell and component
    Fx(&fu)[M][NN] = reinterpret_cast<Fx(&)[M][NN]>(S.c[lc].u);
    constexpr int W = (M + 1) / 2;
    unsigned eu[W];
#pragma unroll
    for (int k = 0; k < W; ++k) eu[k] = 0u;
#pragma unroll
    for (int c = 0; c < M; ++c) eu[c >> 1] |= (unsigned)fx_exp(u[c]) << (16 * (c & 1));
#pragma unroll
    for (int k = 0; k < W; ++k) eu[k] = cell_max_halves<C>(eu[k], node);
    auto field = [&](int c) { return (int)((eu[W > 1 ? c >> 1 : 0] >> (16 * (c & 1))) & 0xffffu); };
#pragma unroll
    for (int c = 0; c < M; ++c) fu[c][node] = fx_of(u[c], field(c));
    if (node == 0) sTr[lc] = 0;
    cell_sync<C>();
    // the decision, its (direction, component) pairs spread over the cell's threads
    if (P.ind_stage < 2) {
        for (int j = node; j < DIM * M && active; j += NN) {
            const int d = j / M, c = j - d * M;
            const Fx *wr = DIM == 2 ? T.trw2x[d][0] : T.tlx[1], *wl = DIM == 2 ? T.trw2x[d][1] : T.tlx[0];
            FxSum sr{0, 0}, sl{0, 0};
#pragma unroll
            for (int q = 0; q < NN; ++q) {
                const Fx v = fu[c][q];
                fx_mac(sr, v, wr[q]);
                fx_mac(sl, v, wl[q]);
            }
            const double own = B.aux[(size_t)cell * M + c], lo = nb_average<PHYS, DIM>(P, B.aux, cell, 2 * d, c),
                         hi = nb_average<PHYS, DIM>(P, B.aux, cell, 2 * d + 1, c);
            int t = tvb_pair(fx_sum(sr), fx_sum(sl), field(c), own, lo, hi, P.thr[d]);
            if (t == 2) t = tvb_pair_64<DIM, N>(B.unew + ((size_t)c * P.ncell + cell) * NN, d, own, lo, hi, P.thr[d]);
            if (t) atomicOr(&sTr[lc], 1);
        }
        cell_sync<C>();
    }
    bool troubled = active && (P.ind_stage >= 2 ? B.tflags[cell] != 0 : sTr[lc] != 0);
    if (P.ind_stage == 3 && active) {  // learned flags: p > 0.6 troubled, p < 0.4 smooth, else the plain flag
        const float pr = B.prob[cell];
        troubled = pr > 0.6f ? true : (pr < 0.4f ? false : troubled);
    }
    if (__any_sync(0xffffffffu, troubled)) {  // the limited first moments, spread likewise
        for (int j = node; j < DIM * M && troubled; j += NN) {
            const int d = j / M, c = j - d * M;
            const double *v = B.unew + ((size_t)c * P.ncell + cell) * NN;
            double p1 = 0.0;  // FP64: a moment has no part of the nodes in the middle, which may be the largest
#pragma unroll
            for (int q = 0; q < NN; ++q) p1 = fma(DIM == 2 ? T.pm2[d][q] : T.pm1[q], v[q], p1);
            const double own = B.aux[(size_t)cell * M + c];
            sP1[lc][d][c] = minmod3_bits(p1, nb_average<PHYS, DIM>(P, B.aux, cell, 2 * d + 1, c) - own,
                                         own - nb_average<PHYS, DIM>(P, B.aux, cell, 2 * d, c));
        }
        cell_sync<C>();
        if (troubled) {
#pragma unroll
            for (int c = 0; c < M; ++c) {
                double v = fma(sP1[lc][0][c], T.xg[a], B.aux[(size_t)cell * M + c]);
                if constexpr (DIM == 2) v = fma(sP1[lc][1][c], T.xg[b], v);
                u[c] = v;
            }
        }
    }
    if (node == 0 && active) {
        if (B.tflags && (P.ind_stage == 0 || P.ind_stage == 3)) B.tflags[cell] = troubled ? 1 : 0;
        if (troubled) atomicAdd(B.ntrb, 1ull);
    }
    double pts[C::PPT][M];
    float rhi;
    const bool cleared = limit_block(P, B, S, lc, node, active, u, pts, false, true, true, rhi);
    post_rate<C>(P, B, S, lc, node, active, cleared, rhi, pts);
    store_node<DIM, N, PHYS>(P, B.unew, cell, node, active, u);
}

template <int DIM, int N, int PHYS>
__global__ void __launch_bounds__(kWarpThreads) k_trouble(Params P, Bufs B) {
    trouble_body<DIM, N, PHYS>(P, B, blockIdx.x);
}

// MLP features of every cell (2D Euler) and the plain indicator's decision (tflags).
// Features, per component: the 3x3 neighbourhood of cell averages (neighbours across a
// boundary follow its condition) minus their mean over den = max(range, M hx hy) +
// 1e-6 max|v|, and the cell's first Legendre moments over the same den.  Layout
// [cell][44]: 36 normalised averages ([comp][9], row-major, centre 4), then 8
// normalised moments ([comp][x, y]).  Reads unew and the averages in aux.
// The 36 stencil features of a 2D Euler cell (per component the 3x3 averages minus their
// mean, times scale = 1 / (max(range, M hx hy) + 1e-6 max|v|)) from the cell averages
// aux[cell][m]; v receives the stencil averages and scale the per-component factor.
template <int PHYS>
__device__ __forceinline__ void stencil_features(const Params &P, const double *aux, int cell, float *f,
                                                 double (&v)[9][ncomp(PHYS, 2)], double (&scale)[ncomp(PHYS, 2)]) {
    constexpr int DIM = 2, M = ncomp(PHYS, 2);
    // 3x3 stencil; a position outside the domain takes the nearest in-domain cell's
    // average with the boundary state of each crossed side applied (x side first)
#pragma unroll
    for (int dy = -1; dy <= 1; ++dy)
#pragma unroll
        for (int dx = -1; dx <= 1; ++dx) {
            int cx = cell;
            bool xout = false, yout = false;
            if (dx != 0) {
                int nb = neighbour(P, cell, dx < 0 ? 0 : 1);
                if (nb >= 0) cx = nb; else xout = true;
            }
            int cy = cx;
            if (dy != 0) {
                int nb = neighbour(P, cx, dy < 0 ? 2 : 3);
                if (nb >= 0) cy = nb; else yout = true;
            }
            double val[M], tmp[M];
#pragma unroll
            for (int c = 0; c < M; ++c) val[c] = aux[(size_t)cy * M + c];
            if (xout) {
                boundary_state<PHYS, DIM>(P, dx < 0 ? 0 : 1, val, tmp);
#pragma unroll
                for (int c = 0; c < M; ++c) val[c] = tmp[c];
            }
            if (yout) {
                boundary_state<PHYS, DIM>(P, dy < 0 ? 2 : 3, val, tmp);
#pragma unroll
                for (int c = 0; c < M; ++c) val[c] = tmp[c];
            }
#pragma unroll
            for (int c = 0; c < M; ++c) v[(dy + 1) * 3 + (dx + 1)][c] = val[c];
        }
    // per component: (v - mean) / den and slopes / den, den = max(range, M hx hy) + 1e-6 max|v|
    const double thr = P.thr_feat;
#pragma unroll
    for (int c = 0; c < M; ++c) {
        unsigned long long kmx = kKeyNegInf, kmn = kKeyPosInf, kab = 0ull;
        int E = 0;
#pragma unroll
        for (int q = 0; q < 9; ++q) {
            E = max(E, fx_exp(v[q][c]));
            if (!isnan_bits(v[q][c])) {  // fmax / fmin ignore NaN
                const unsigned long long k = ordbits(v[q][c]);
                kmx = umax64(kmx, k);
                kmn = umin64(kmn, k);
                kab = umax64(kab, dbits(v[q][c]) & 0x7fffffffffffffffull);
            }
        }
        const double mx = ordbits_inv(kmx), mn = ordbits_inv(kmn), amax = bitsd(kab);
        const double den = fmax(mx - mn, thr) + (1e-6 * amax + 1e-30);
        scale[c] = recip_nr(den);
        if (E < 1900) {
            // 9 (v - mean) exactly in fixed point, times scale / 9 as a product of sums of two floats, rounded
            // once: the FP64 sums, division, products and conversions took 38 FP64 instructions a component
            long long m[9], sum = 0;
#pragma unroll
            for (int q = 0; q < 9; ++q) {
                m[q] = fx_whole(v[q][c], E) >> 2;
                sum += m[q];
            }
            float sh, sl;  // 2^(E - 1079) scale / 9 for mantissas in units of 2^-60
            two_floats(scale[c] * (1.0 / 9.0) * bitsd((unsigned long long)(E + 4) << 52), sh, sl);
#pragma unroll
            for (int q = 0; q < 9; ++q) {
                float dh, dl;
                two_floats_fx(9 * m[q] - sum, dh, dl);
                const float p = __fmul_rn(dh, sh);
                f[c * 9 + q] = p + (fmaf(dh, sh, -p) + fmaf(dh, sl, dl * sh));
            }
            continue;
        }
        double mean = 0.0;
#pragma unroll
        for (int q = 0; q < 9; ++q) mean += v[q][c];
        mean /= 9.0;
#pragma unroll
        for (int q = 0; q < 9; ++q) f[c * 9 + q] = (float)((v[q][c] - mean) * scale[c]);
    }
}

template <int DIM, int N, int PHYS>
__device__ __forceinline__ void features_body(const Params &P, const Bufs &B, int blk) {
    constexpr int M = ncomp(PHYS, DIM);
    constexpr int NN = DIM == 2 ? N * N : N;
    const int cell = blk * blockDim.x + threadIdx.x;
    if constexpr (DIM != 2 || PHYS != PH_EULER) {
        return;
    } else {
        if (cell >= P.ncell) return;
        const NodalTables &T = c_tab[N - 2];
        double v[9][M], scale[M];
        stencil_features<PHYS>(P, B.aux, cell, B.feat + (size_t)cell * 44, v, scale);
        float *f = B.feat + (size_t)cell * 44;
        // the first moments, and the plain indicator's decision for this cell (the troubled-cell kernel's
        // arithmetic): the label of harvested features and the fallback of the learned flags
        int trouble = 0;
#pragma unroll
        for (int c = 0; c < M; ++c) {
            const double *u = B.unew + ((size_t)c * P.ncell + cell) * NN;
            double w[NN];
            int En = 0;
#pragma unroll
            for (int q = 0; q < NN; ++q) {
                w[q] = u[q];
                En = max(En, fx_exp(w[q]));
            }
            FxSum s[2] = {{0, 0}, {0, 0}}, r[2] = {{0, 0}, {0, 0}}, l[2] = {{0, 0}, {0, 0}};
#pragma unroll
            for (int q = 0; q < NN; ++q) {
                const Fx x = fx_of(w[q], En);
#pragma unroll
                for (int d = 0; d < 2; ++d) {
                    fx_mac(s[d], x, T.pm2x[d][q]);
                    fx_mac(r[d], x, T.trw2x[d][0][q]);
                    fx_mac(l[d], x, T.trw2x[d][1][q]);
                }
            }
#pragma unroll
            for (int d = 0; d < 2; ++d) {
                const double m = En == 0x7ff ? NAN : fx_double(fx_sum(s[d]), fx_shift(En, kFxAvg));
                f[36 + 2 * c + d] = (float)(m * scale[c]);
                const double lo = v[d == 0 ? 3 : 1][c], hi = v[d == 0 ? 5 : 7][c];
                int t = tvb_pair(fx_sum(r[d]), fx_sum(l[d]), En, v[4][c], lo, hi, P.thr[d]);
                if (t == 2) t = tvb_pair_64<2, N>(u, d, v[4][c], lo, hi, P.thr[d]);
                if (t) trouble = 1;
            }
        }
        if (B.tflags) B.tflags[cell] = trouble;
    }
}

template <int DIM, int N, int PHYS>
__global__ void k_features(Params P, Bufs B) {
    features_body<DIM, N, PHYS>(P, B, blockIdx.x);
}

template <int DIM, int N, int PHYS>
cudaError_t launch_one(int kernel, cudaStream_t st, const Params &P, const Bufs &B) {
    using C = CfgW<DIM, N, PHYS>;
    const int nblocks = (P.ncell + C::NCB - 1) / C::NCB;
    switch (kernel) {
    case K_INNER:
        if (PHYS != PH_EULER || P.fx.on)  // scalar laws out of the range: eval_G_fx's own fallback
            k_inner<DIM, N, PHYS, true><<<nblocks, C::NT, 0, st>>>(P, B);
        else
            k_inner<DIM, N, PHYS, PHYS != PH_EULER><<<nblocks, C::NT, 0, st>>>(P, B);
        break;
    case K_FINAL:
        if (!B.tsum) {
            k_final<DIM, N, PHYS, RECOMPUTED><<<nblocks, C::NT, 0, st>>>(P, B);
        } else if (DIM == 2 && B.fc) {
            const size_t points = 2 * (size_t)P.ncell * N;
            k_faces<N, PHYS><<<(unsigned)((points + 127) / 128), 128, 0, st>>>(P, B);
            k_final<DIM, N, PHYS, FACES><<<nblocks, C::NT, 0, st>>>(P, B);
        } else {
            k_final<DIM, N, PHYS, STORED><<<nblocks, C::NT, 0, st>>>(P, B);
        }
        break;
    case K_LIMIT: k_limit<DIM, N, PHYS><<<nblocks, C::NT, 0, st>>>(P, B); break;
    case K_TROUBLE: k_trouble<DIM, N, PHYS><<<nblocks, C::NT, 0, st>>>(P, B); break;
    case K_FEATURES: k_features<DIM, N, PHYS><<<(P.ncell + 127) / 128, 128, 0, st>>>(P, B); break;
    case K_A0:
    case K_MARGINS: k_scan<DIM, N, PHYS><<<nblocks, C::NT, 0, st>>>(P, B); break;
    case K_AVG: {
        int tot = P.ncell * C::M;
        k_avg<DIM, N, PHYS><<<(tot + 255) / 256, 256, 0, st>>>(P, B);
        break;
    }
    default: return cudaErrorInvalidValue;
    }
    return cudaGetLastError();
}

template <int DIM>
cudaError_t launch_dim(int kernel, int n, int phys, cudaStream_t st, const Params &P, const Bufs &B) {
#define CRKDG_CASE(NV, PV) \
    if (n == NV && phys == PV) return launch_one<DIM, NV, PV>(kernel, st, P, B);
    CRKDG_CASE(2, PH_ADV) CRKDG_CASE(2, PH_BURG) CRKDG_CASE(2, PH_EULER)
    CRKDG_CASE(3, PH_ADV) CRKDG_CASE(3, PH_BURG) CRKDG_CASE(3, PH_EULER)
    CRKDG_CASE(4, PH_ADV) CRKDG_CASE(4, PH_BURG) CRKDG_CASE(4, PH_EULER)
#undef CRKDG_CASE
    return cudaErrorInvalidValue;
}

}  // namespace crkdg
