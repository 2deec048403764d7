// lbm_eig.cuh -- eigenvalues of a small dense complex matrix in FP64, one
// matrix per thread: reduction to upper Hessenberg form by Givens rotations,
// then the shifted QR iteration on the Hessenberg matrix (Wilkinson shift
// from the trailing 2 x 2 block, deflation at negligible subdiagonal entries,
// ad hoc shifts after 10 and 20 stalled sweeps).  This is the textbook
// algorithm for the complex Schur form (Golub & Van Loan, Matrix
// Computations, Sec. 7.5), restricted to what the spectral radius needs: the
// rotations act only on the active diagonal block, since the eigenvalues do
// not depend on the blocks outside it.  Compiles for host and device.
//
// On the GPU the FP64 pipe bounds it (1/64 of the FP32 rate), comparisons and
// conversions included, so everything but the rotations themselves is kept
// off it or short: a rotation is formed with two reciprocal square roots (24
// instructions; hypot and divisions took about 135, more than applying it to
// a 9 x 9 matrix's columns), deflation is decided in FP32, and zero tests
// look at the exponent.  The iteration runs in FP32 first, at a thirtieth of
// the cost: its eigenvalues as first shifts make most deflate after two sweeps
// (a warp's rotated pairs of entries 1250 -> 875).  63488 matrices of the
// stability scan, with the host's part: 6.55 ms with divisions and hypot, 4.56
// without, 3.95 with FP32 shifts.
#pragma once

#include <math.h>
#include <string.h>

#ifdef __CUDACC__
#define LBM_HD __host__ __device__ __forceinline__
#else
#define LBM_HD inline
#endif

namespace lbm {

template <typename R>
struct cx {
    R re, im;
};
using cplx = cx<double>;

// clang-format off
template <typename R> LBM_HD cx<R> cadd(cx<R> a, cx<R> b) { return cx<R>{a.re + b.re, a.im + b.im}; }
template <typename R> LBM_HD cx<R> csub(cx<R> a, cx<R> b) { return cx<R>{a.re - b.re, a.im - b.im}; }
template <typename R> LBM_HD cx<R> cmul(cx<R> a, cx<R> b) {
    return cx<R>{a.re * b.re - a.im * b.im, a.re * b.im + a.im * b.re};
}
template <typename R> LBM_HD cx<R> cconj(cx<R> a) { return cx<R>{a.re, -a.im}; }
template <typename R> LBM_HD cx<R> cscale(cx<R> a, R s) { return cx<R>{a.re * s, a.im * s}; }
template <typename R> LBM_HD R cabs2(cx<R> a) { return a.re * a.re + a.im * a.im; }
// clang-format on

// The upper half of a double's bits: its sign, exponent and leading digits.
LBM_HD int high_bits(double a) {
#ifdef __CUDA_ARCH__
    return __double2hiint(a);
#else
    long long v;
    memcpy(&v, &a, sizeof v);
    return (int)(v >> 32);
#endif
}

// |a| rounded towards zero to FP32 by integer operations: 0 below 2^-126,
// infinite or NaN from 2^128.
LBM_HD float narrow_abs(double a) {
    unsigned long long v;
#ifdef __CUDA_ARCH__
    v = (unsigned long long)__double_as_longlong(a);
#else
    memcpy(&v, &a, sizeof v);
#endif
    v &= 0x7fffffffffffffffull;
    const unsigned long long low = 897ull << 52, high = (896ull + 255ull) << 52;
    const unsigned bits = v < low ? 0u : v >= high ? 0x7fc00000u : (unsigned)((v - (896ull << 52)) >> 29);
    float f;
#ifdef __CUDA_ARCH__
    f = __uint_as_float(bits);
#else
    memcpy(&f, &bits, sizeof f);
#endif
    return f;
}
LBM_HD float narrow_abs1(cplx a) { return narrow_abs(a.re) + narrow_abs(a.im); }
LBM_HD float narrow_abs1(cx<float> a) { return fabsf(a.re) + fabsf(a.im); }

LBM_HD bool negative(double a) { return high_bits(a) < 0; }
LBM_HD bool negative(float a) { return a < 0.0f; }

// A square so small (below about 2^-960) that the number counts as zero; a
// NaN of either sign does not.
LBM_HD bool tiny_square(double a2) { return (unsigned)high_bits(a2) < (63u << 20); }
LBM_HD bool tiny_square(float a2) { return a2 < 1e-30f; }

// 1 / sqrt(a), a > 0 and not tiny, by one step of Chebyshev's third-order
// method (J. F. Traub, Iterative Methods for the Solution of Equations, 1964)
// for 1/y^2 - a = 0, y (1 + e / 2 + 3 e^2 / 8) with e = 1 - a y^2, from the
// hardware approximation y.  With y good to 2^-20 the step leaves a relative
// error of 5 e^3 / 16 <= 2^-58; with the rounding of a y and the last one the
// result lies within 1.03 ulp.
LBM_HD double rsqrt_pos(double a) {
#ifdef __CUDA_ARCH__
    double y;
    asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(a));
    const double e = __fma_rn(-(a * y), y, 1.0);
    return __fma_rn(y * e, __fma_rn(0.375, e, 0.5), y);
#else
    return 1.0 / sqrt(a);
#endif
}

LBM_HD float rsqrt_pos(float a) {
#ifdef __CUDA_ARCH__
    return rsqrtf(a);
#else
    return 1.0f / sqrtf(a);
#endif
}

// a / b as a conj(b) / |b|^2 (b not tiny; the quotients here are of order
// one, so the squares neither overflow nor lose b).
template <typename R>
LBM_HD cx<R> cdiv(cx<R> a, cx<R> b) {
    const R ri = rsqrt_pos(cabs2(b));
    return cscale(cmul(a, cconj(b)), ri * ri);
}

// Principal square root: sqrt(z) = sqrt((|z| + x) / 2) + i sgn(y) sqrt((|z| - x) / 2),
// with the smaller part formed as y / (2 * larger) to avoid cancellation.
template <typename R>
LBM_HD cx<R> csqrt_p(cx<R> z) {
    const R m2 = cabs2(z);
    if (tiny_square(m2)) return cx<R>{0, 0};
    const R m = m2 * rsqrt_pos(m2);
    const R h = R(0.5) * (m + (negative(z.re) ? -z.re : z.re)), ri = rsqrt_pos(h);
    const R big = h * ri, small = R(0.5) * z.im * ri;
    if (!negative(z.re)) return cx<R>{big, small};
    return negative(z.im) ? cx<R>{-small, -big} : cx<R>{small, big};
}

// Rotation G = [[c, s], [-conj(s), c]] (c real, c^2 + |s|^2 = 1) with
// G (x, y)^T = (r, 0)^T.
template <typename R>
struct Givens {
    R c;
    cx<R> s;
};

template <typename R>
LBM_HD Givens<R> givens(cx<R> x, cx<R> y) {
    const R y2 = cabs2(y);
    if (tiny_square(y2)) return Givens<R>{1, cx<R>{0, 0}};
    const R x2 = cabs2(x);
    if (tiny_square(x2)) return Givens<R>{0, cconj(cscale(y, rsqrt_pos(y2)))};  // s = conj(y) / |y|
    const R ri = rsqrt_pos(x2 + y2), xi = rsqrt_pos(x2);
    // c = |x| / r, s = (x / |x|) conj(y) / r
    return Givens<R>{x2 * xi * ri, cmul(cscale(x, xi * ri), cconj(y))};
}

// Rows p, p + 1 of H (n x n, row-major, leading dimension ld), columns
// c0 .. c1: (a, b) -> (c a + s b, -conj(s) a + c b).
template <typename R>
LBM_HD void rot_rows(cx<R>* H, int ld, int p, int c0, int c1, Givens<R> g) {
    for (int j = c0; j <= c1; ++j) {
        const cx<R> a = H[p * ld + j], b = H[(p + 1) * ld + j];
        H[p * ld + j] = cadd(cscale(a, g.c), cmul(g.s, b));
        H[(p + 1) * ld + j] = csub(cscale(b, g.c), cmul(cconj(g.s), a));
    }
}

// Columns p, p + 1 of H, rows r0 .. r1, multiplied from the right by G^H:
// (a, b) -> (c a + conj(s) b, -s a + c b).
template <typename R>
LBM_HD void rot_cols(cx<R>* H, int ld, int p, int r0, int r1, Givens<R> g) {
    for (int i = r0; i <= r1; ++i) {
        const cx<R> a = H[i * ld + p], b = H[i * ld + p + 1];
        H[i * ld + p] = cadd(cscale(a, g.c), cmul(cconj(g.s), b));
        H[i * ld + p + 1] = csub(cscale(b, g.c), cmul(g.s, a));
    }
}

// Reduce H (n x n) to upper Hessenberg form by unitary similarity.
LBM_HD void hessenberg(cplx* H, int n) {
    for (int k = 0; k + 2 < n; ++k)
        for (int j = n - 1; j >= k + 2; --j) {
            const Givens<double> g = givens(H[(j - 1) * n + k], H[j * n + k]);
            rot_rows(H, n, j - 1, k, n - 1, g);
            H[j * n + k] = cplx{0.0, 0.0};
            rot_cols(H, n, j - 1, 0, n - 1, g);
        }
}

// Eigenvalues of the upper Hessenberg matrix H (destroyed) into ev[0..n).
// guess (may be null): an approximation of each eigenvalue, the first shift
// for the one at its place.  Returns the number of QR sweeps, or -1 if a block
// did not converge within kMaxSweeps sweeps (the unconverged eigenvalues are
// then NaN).
template <typename R>
LBM_HD int hessenberg_eigenvalues(cx<R>* H, int n, cx<R>* ev, const cx<float>* guess) {
    constexpr int kMaxSweeps = 60;  // per eigenvalue
    constexpr float kEps = sizeof(R) == 8 ? 2.220446049250313e-16f : 1.1920929e-7f;
    float anorm = 0.0f;
    for (int k = 0; k < n * n; ++k) anorm = fmaxf(anorm, narrow_abs1(H[k]));
    int hi = n - 1, its = 0, total = 0;
    while (hi >= 0) {
        if (hi == 0) {
            ev[0] = H[0];
            break;
        }
        // smallest l such that the block l..hi has no negligible subdiagonal
        int l = hi;
        while (l > 0) {
            float s = narrow_abs1(H[(l - 1) * n + l - 1]) + narrow_abs1(H[l * n + l]);
            if (s == 0.0f) s = anorm;
            if (narrow_abs1(H[l * n + l - 1]) <= kEps * s) {
                H[l * n + l - 1] = cx<R>{0, 0};
                break;
            }
            --l;
        }
        if (l == hi) {  // 1 x 1 block splits off
            ev[hi] = H[hi * n + hi];
            --hi;
            its = 0;
            continue;
        }
        if (its == kMaxSweeps) {
            for (int k = 0; k <= hi; ++k) ev[k] = cx<R>{R(NAN), R(NAN)};
            return -1;
        }
        // shift
        cx<R> mu;
        const cx<R> a = H[(hi - 1) * n + hi - 1], b = H[(hi - 1) * n + hi];
        const cx<R> c = H[hi * n + hi - 1], d = H[hi * n + hi];
        if (guess && its == 0 && isfinite(guess[hi].re + guess[hi].im)) {
            mu = cx<R>{guess[hi].re, guess[hi].im};
        } else if (its == 10 || its == 20) {
            mu = cadd(d, cx<R>{R(fabs(c.re) + (hi >= 2 ? fabs(H[(hi - 1) * n + hi - 2].re) : 0)), 0});
        } else {
            // eigenvalue of [[a, b], [c, d]] nearer to d: d - bc / (p + disc),
            // p = (a - d) / 2, disc = sqrt(p^2 + bc) signed to enlarge |p + disc|
            const cx<R> p = cscale(csub(a, d), R(0.5));
            const cx<R> bc = cmul(b, c);
            cx<R> disc = csqrt_p(cadd(cmul(p, p), bc));
            if (negative(p.re * disc.re + p.im * disc.im)) disc = cx<R>{-disc.re, -disc.im};
            const cx<R> den = cadd(p, disc);
            mu = tiny_square(cabs2(den)) ? d : csub(d, cdiv(bc, den));
        }
        // one explicit-shift QR sweep on the block l..hi: H - mu I = Q R, H <- R Q + mu I
        for (int k = l; k <= hi; ++k) H[k * n + k] = csub(H[k * n + k], mu);
        Givens<R> gs[16];
        for (int k = l; k < hi; ++k) {
            gs[k - l] = givens(H[k * n + k], H[(k + 1) * n + k]);
            rot_rows(H, n, k, k, hi, gs[k - l]);
            H[(k + 1) * n + k] = cx<R>{0, 0};
        }
        for (int k = l; k < hi; ++k) rot_cols(H, n, k, l, (k + 2 <= hi ? k + 2 : hi), gs[k - l]);
        for (int k = l; k <= hi; ++k) H[k * n + k] = cadd(H[k * n + k], mu);
        ++its;
        ++total;
    }
    return total;
}

// FP64 to FP32 by integer operations, rounded towards zero.
LBM_HD float narrow(double a) {
    const float m = narrow_abs(a);
    return negative(a) ? -m : m;
}

// Spectral radius of H (n x n, n <= 9, destroyed); NaN if the iteration does
// not converge.  Entries far from one are scaled by a power of two, so that
// squares stay in range.
LBM_HD double spectral_radius(cplx* H, int n) {
    int m = 0;
    for (int k = 0; k < n * n; ++k) {
        const int re = high_bits(H[k].re) & 0x7fffffff, im = high_bits(H[k].im) & 0x7fffffff;
        m = m > re ? m : re;
        m = m > im ? m : im;
    }
    if (m >= 0x7ff00000) return NAN;
    const int e = (m >> 20) - 1023;
    const int shift = e > 60 || e < -60 ? e : 0;
    if (shift)
        for (int k = 0; k < n * n; ++k) H[k] = cplx{scalbn(H[k].re, -shift), scalbn(H[k].im, -shift)};
    hessenberg(H, n);
    cplx ev[9];
    {
        // the whole iteration in FP32 for the first shifts (above)
        cx<float> A[81], guess[9];
        for (int k = 0; k < n * n; ++k) A[k] = cx<float>{narrow(H[k].re), narrow(H[k].im)};
        hessenberg_eigenvalues<float>(A, n, guess, nullptr);
        if (hessenberg_eigenvalues<double>(H, n, ev, guess) < 0) return NAN;
    }
    double r2 = 0.0;
    for (int k = 0; k < n; ++k) r2 = fmax(r2, cabs2(ev[k]));
    const double r = sqrt(r2);
    return shift ? scalbn(r, shift) : r;
}

}  // namespace lbm
