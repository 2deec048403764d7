// lbm_fp64.cuh -- the node update of the FP64 step (Eqs. e4-e7, e16-e18,
// SEC-VON-11), written for the fewest FP64 instructions.
//
// GB300 issues one FP64 warp instruction per SM in 16 cycles (1/64 of the
// FP32 rate), so the FP64 step takes as long as its FP64 instruction count.
// This form needs 99 of them a node: 54 for moments and equilibrium, 45 for
// the five-point update.  The shared templates of lbm_device.cuh, whose
// operation order the FP32 modes are tied to, take 124.  What is saved:
//  * sums and differences of opposite pairs serve density and momentum;
//  * the equilibrium is formed from density-weighted moments -- rho,
//    p = rho T, g = rho u / c1 and g.u / c1 -- so that most products with
//    rho fall away, and B v.u needs no product with u either;
//  * omega and the speeds are folded into the constants (Fp64Step);
//  * the factor (b + 2) T + u^2 of both velocity sets' B is formed once;
//  * (v.u)^2 of the diagonals comes from u^2 and 2 ux uy;
//  * the reciprocal of the density is one cubic Newton step from the
//    hardware's approximation.
#pragma once

#include <cmath>

#include "lbm_device.cuh"

namespace lbm {

// Constants of the FP64 step; w[i][s] as in Model.  With U = u / c1,
// g = rho U, p = rho T, and q = g.U = rho u^2 / c1^2:
struct Fp64Step {
    double w[9][5];
    double kap;              // d / c1
    double te, t1, t2;       // eta0^2 / b, c1^2 / b, c2^2 / b:  p = te f_0 + t1 s14 + t2 s58 - t1 q
    double k0;               // omega A_0 / T
    double vp;               // (b + 2) / c1^2:  V = (vp p + q) / rho
    double a1r, a1p, a1q;    // omega rho A_1..4 = a1r rho + a1p p + a1q q
    double a5r, a5p, a5q;    // omega rho A_5..8 + the u^2 part of its D (v.u)^2
    double h1;               // omega D_1..4 c1^4 = omega / 2
    double b1c, b1v;         // omega c1^2 B_1..4 = b1c + b1v V
    double b5c, b5v;         // omega c1 d B_5..8
    double k5;               // 2 omega D_5 c1^2 d^2
};

// Unevaluated sum of two doubles, about 106 bits (Dekker / Knuth error-free
// sums and products), for the constants above on the host.
struct Wide {
    double hi, lo;
    Wide(double h = 0.0, double l = 0.0) : hi(h), lo(l) {}
    static Wide sum(double a, double b) {
        const double s = a + b, t = s - a;
        return Wide(s, (a - (s - t)) + (b - t));
    }
    friend Wide operator+(Wide a, Wide b) {
        Wide s = sum(a.hi, b.hi);
        return sum(s.hi, s.lo + (a.lo + b.lo));
    }
    friend Wide operator*(Wide a, Wide b) {
        const double p = a.hi * b.hi;
        return sum(p, std::fma(a.hi, b.hi, -p) + (a.hi * b.lo + a.lo * b.hi));
    }
    friend Wide operator-(Wide a) { return Wide(-a.hi, -a.lo); }
    friend Wide operator-(Wide a, Wide b) { return a + (-b); }
    friend Wide operator/(Wide a, Wide b) {
        const double q = a.hi / b.hi;
        const Wide r = a - b * Wide(q);
        return sum(q, (r.hi + r.lo) / b.hi);
    }
};

// Each constant is formed in Wide arithmetic from the parameters and rounded
// once: rounded step by step, their mutual errors act as a small source of
// mass and energy at every node and step (on the 256 x 64 double Mach
// reflection to t = 0.2, 2560 steps, the error in rho against extended
// precision is 1.2e-13 rms this way and 4.2e-13 with constants formed in
// plain double; the templates' update has 2.2e-13).
inline Fp64Step fp64_step(const Model<double>& M, double b_, double tau, double dt, double c1_, double c2_,
                          double eta0) {
    Fp64Step C;
    for (int i = 0; i < 9; ++i)
        for (int s = 0; s < 5; ++s) C.w[i][s] = M.w[i][s];
    const Wide b(b_), c1(c1_), c2(c2_), om = Wide(dt) / Wide(tau);
    const Wide d = c2 / Wide(1.4142135623730951, -9.667293313452913e-17);  // c2 / sqrt(2)
    const Wide c1s = c1 * c1, c2s = c2 * c2, es = Wide(eta0) * Wide(eta0), cd = c1 * d, two(2.0);
    const Wide gap = c1s - c2s;
    const Wide q1 = Wide(4.0) * gap, q5 = -q1;                     // denominators of A (Eq. e17)
    const Wide d1 = two * c1s * gap, d5 = -(two * c2s * gap);      // and of B (Eq. e18)
    const Wide D5 = Wide(1.0) / (two * c2s * c2s), bm = (b - two) / es;
    C.kap = (d / c1).hi;
    C.te = (es / b).hi;
    C.t1 = (c1s / b).hi;
    C.t2 = (c2s / b).hi;
    C.k0 = (om * bm).hi;
    C.vp = ((b + two) / c1s).hi;
    C.a1r = (-(om * c2s / q1)).hi;
    C.a1p = (om * (bm * c2s + two) / q1).hi;
    C.a1q = (om * c2s / q1).hi;                                    // A's u^2 term (c2^2 / c1^2) / q1, times c1^2
    C.a5r = (-(om * c1s / q5)).hi;
    C.a5p = (om * (bm * c1s + two) / q5).hi;
    C.a5q = (om * ((c1s / c2s) / q5 + D5 * d * d) * c1s).hi;
    C.h1 = (om / two).hi;
    C.b1c = (-(om * c1s * c2s / d1)).hi;
    C.b1v = (om * c1s * c1s / d1).hi;                              // B = (-c^2 + c1^2 V) / d
    C.b5c = (-(om * cd * c1s / d5)).hi;
    C.b5v = (om * cd * c1s / d5).hi;
    C.k5 = (two * om * D5 * cd * cd).hi;
    return C;
}

// The constants of the FP64 adjoint step (adjoint_collision).
struct Fp64Adjoint : Fp64Step {
    double k5h;        // k5 / 2
    double inv_omega;  // tau / dt
};

// 1 / a by one step of Chebyshev's third-order method (J. F. Traub, Iterative
// Methods for the Solution of Equations, 1964) for 1/x - a = 0, x (1 + e + e^2)
// with e = 1 - a x, from the hardware approximation x.  With |e| <= 2^-20 the
// step leaves a relative error of e^3 <= 2^-60, and the roundings before the
// last one at most 2^-53 |e| each: within 0.51 ulp of 1 / a for 2^-1022 <= |a| <
// 2^1022.  Zeros, subnormals, infinities and NaN give NaN, and from 2^1022 on
// x may be flushed to zero; fp64_health reports all of these.  (Falling back on the
// library's reciprocal there costs registers: 10 % of the adjoint step.)
__device__ __forceinline__ double fp64_rcp(double a) {
    double x;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(x) : "d"(a));
    const double e = __fma_rn(-a, x, 1.0);
    return __fma_rn(x, __fma_rn(e, e, e), x);
}

// The bits of health() without FP64 comparisons (they would take the FP64
// pipe): rho > 0 and p > 0 from the sign, and V = ((b + 2) T + u^2) / c1^2 is
// finite only if T, u and 1 / rho are.  A density whose reciprocal fp64_rcp does
// not form counts as non-physical.
__device__ __forceinline__ unsigned fp64_health(double rho, double p, double V) {
    const bool finite = (__double2hiint(V) & 0x7ff00000) != 0x7ff00000;
    const bool dense = (unsigned)__double2hiint(rho) - 0x00100000u < 0x7fd00000u - 0x00100000u;
    if (!dense || !finite) return ST_NONPHYSICAL;
    return __double_as_longlong(p) > 0 ? 0u : ST_T_NONPOS;
}

// E / b of a node: the rest population and the sums of the two velocity sets.
__device__ __forceinline__ double fp64_energy(const Fp64Step& C, double f0, double s14, double s58) {
    return __fma_rn(C.te, f0, __fma_rn(C.t1, s14, C.t2 * s58));
}

// Relaxation terms omega f^eq_i of a node; returns its health bits.
__device__ __forceinline__ unsigned fp64_relaxation(const Fp64Step& C, const double (&f)[9], double (&r)[9]) {
    // differences along +x, +y and the two diagonals, sums of the pairs
    const double ax = f[3] - f[1], ay = f[4] - f[2], ar = f[7] - f[5], am = f[6] - f[8];
    const double s14 = (f[1] + f[3]) + (f[2] + f[4]);
    const double s58 = (f[5] + f[7]) + (f[6] + f[8]);
    const double rho = (f[0] + s14) + s58;
    const double inv = fp64_rcp(rho);
    const double gx = __fma_rn(C.kap, ar + am, ax), gy = __fma_rn(C.kap, ar - am, ay);
    const double Ux = gx * inv, Uy = gy * inv;
    const double xx = gx * Ux, yy = gy * Uy, xy = gx * Uy;
    const double q = xx + yy;
    const double p = __fma_rn(-C.t1, q, fp64_energy(C, f[0], s14, s58));
    const double V = __fma_rn(C.vp, p, q) * inv;
    r[0] = C.k0 * p;
    {
        const double A = __fma_rn(C.a1p, p, __fma_rn(C.a1q, q, C.a1r * rho));
        const double B = __fma_rn(C.b1v, V, C.b1c);
        const double sx = __fma_rn(C.h1, xx, A), sy = __fma_rn(C.h1, yy, A);
        r[1] = __fma_rn(-B, gx, sx);
        r[3] = __fma_rn(B, gx, sx);
        r[2] = __fma_rn(-B, gy, sy);
        r[4] = __fma_rn(B, gy, sy);
    }
    {
        const double A = __fma_rn(C.a5p, p, __fma_rn(C.a5q, q, C.a5r * rho));
        const double B = __fma_rn(C.b5v, V, C.b5c);
        const double sr = __fma_rn(C.k5, xy, A), sm = __fma_rn(-C.k5, xy, A);
        const double gr = gx + gy, gm = gx - gy;
        r[5] = __fma_rn(-B, gr, sr);
        r[7] = __fma_rn(B, gr, sr);
        r[6] = __fma_rn(B, gm, sm);
        r[8] = __fma_rn(-B, gm, sm);
    }
    return fp64_health(rho, p, V);
}

// f' = w0 c + w1 e + w2 w + w3 n + w4 s + r (Eq. SEC-VON-11, folded weights).
__device__ __forceinline__ double fp64_update(const Fp64Step& C, int i, double r, double c, double e, double w,
                                              double n, double s) {
    double acc = __fma_rn(C.w[i][0], c, r);
    acc = __fma_rn(C.w[i][1], e, acc);
    acc = __fma_rn(C.w[i][2], w, acc);
    acc = __fma_rn(C.w[i][3], n, acc);
    return __fma_rn(C.w[i][4], s, acc);
}

}  // namespace lbm
