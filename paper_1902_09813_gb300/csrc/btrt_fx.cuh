// btrt_fx.cuh -- the FP64 collision in 64-bit block fixed point.
//
// GB300 issues fewer than two FP64 operations per SM and clock (0.527 T op/s
// measured), so a collision of 50 FP64 operations takes 29 clocks per node while
// nine tenths of the issue slots stay empty; HBM would allow one node per 7 clocks.
// The collision of Eq. 6 is a linear map of the nine populations (plus a few
// per-node terms), so it can run on the integer pipes instead: the populations of
// one node are brought to one common exponent E (the largest among them), as 64-bit
// integers in units of 2^(E - 58), their moments are exact integer sums, products
// with the collision's constants are 64 x 64-bit products rounded to a unit, and
// each result is rounded once to FP64 on its way out.
//
// Precision: the largest population has its 53 bits in the integer with five to
// spare, so every intermediate carries an error of about one unit, 2^-58 of the
// largest population, where FP64 arithmetic rounds each intermediate of that size
// to 2^-53.  The four-times-smaller axis populations and the sixteen-times-smaller
// diagonal ones keep errors at or below those of the FP64 form; their sum is exact
// (r_0 is formed as the total minus the other eight).
// Range: largest populations of exponent 64 .. 2040 (about 1e-289 .. 1e306), or nodes that
// are zero throughout; the others (and infinities and NaN) take the FP64 form
// (collide_f64_slow).
#pragma once

#include <math.h>
#include <stdint.h>
#include <string.h>

#ifdef __CUDACC__
#define BTRT_HD __host__ __device__ __forceinline__
#else
#define BTRT_HD inline
#endif

namespace btrt {

using fx = long long;

constexpr unsigned int kFxExpMin = 64u << 20, kFxExpMax = 2040u << 20, kFxExpMask = 0x7ff00000u;

// A constant C as (hi 2^32 + lo) = C 2^64, lo signed; |C| < 1/2.
struct FxConst {
    int hi, lo;
};
// v / div to the nearest unit: the integer division adds no rounding of its own to v's.
inline FxConst fx_const(double v, int div) {
    int e;
    const __int128 m = (__int128)(long long)ldexp(frexp(v, &e), 53);   // v = m 2^(e - 53)
    const int sh = 49 - e;                                             // (m 2^60 / div) 2^(e - 49) = v 2^64 / div
    const __int128 q = m * ((__int128)1 << 60) / div;
    const long long c = sh < 120 ? (long long)((q + ((__int128)1 << (sh - 1))) >> sh) : 0;
    FxConst k;
    k.lo = (int)(unsigned int)(unsigned long long)c;
    k.hi = (int)((c - (long long)k.lo) >> 32);
    return k;
}

BTRT_HD unsigned long long fx_bits(double v) {
#ifdef __CUDA_ARCH__
    return (unsigned long long)__double_as_longlong(v);
#else
    unsigned long long b;
    memcpy(&b, &v, 8);
    return b;
#endif
}
BTRT_HD double fx_double(unsigned long long b) {
#ifdef __CUDA_ARCH__
    return __longlong_as_double((long long)b);
#else
    double v;
    memcpy(&v, &b, 8);
    return v;
#endif
}
// Exponent field of v, in place in the high word.
BTRT_HD unsigned int fx_exp(double v) { return (unsigned int)(fx_bits(v) >> 32) & kFxExpMask; }

// v in units of 2^(E - TOP) (E = em >> 20, biased as in FP64), truncated toward
// zero: the mantissa with its hidden bit at the top of the word, shifted down by
// E + 63 - TOP - e.  D2Q9: TOP = 58, nine populations then sum below 2^63; D3Q19: 57.
// Shifts of 64 and more give 0 (also for zeros and subnormals, whose
// hidden bit is not there: E >= 64 shifts them out).  e <= E + 62 - TOP.
template <int TOP = 58> BTRT_HD fx fx_from(double v, unsigned int em) {
    const unsigned long long b = fx_bits(v);
    const unsigned int sh = (em + ((63u - TOP) << 20) - ((unsigned int)(b >> 32) & kFxExpMask)) >> 20;
    unsigned long long m = (b << 11) | 0x8000000000000000ull;
#ifdef __CUDA_ARCH__
    asm("shr.u64 %0, %0, %1;" : "+l"(m) : "r"(sh));   // PTX clamps the amount at 64
#else
    m = sh < 64 ? m >> sh : 0;
#endif
    const fx s = (fx)b >> 63;
    return ((fx)m ^ s) - s;
}

// The FP64 value nearest to v 2^(E - TOP) (ties away from zero).
template <int TOP = 58> BTRT_HD double fx_to(fx v, unsigned int em) {
    const fx s = v >> 63;
    const unsigned long long a = (unsigned long long)((v ^ s) - s);
    unsigned int hi = (unsigned int)(a >> 32), lo = (unsigned int)a, up = em + ((62u - TOP) << 20);
    if (hi == 0) {
        hi = lo;
        lo = 0;
        up -= 32u << 20;
    }
#ifdef __CUDA_ARCH__
    const unsigned int lz = (unsigned int)__clz((int)hi);
    const unsigned int mh = __funnelshift_l(lo, hi, lz), ml = lo << (lz & 31);
#else
    const unsigned int lz = hi ? (unsigned int)__builtin_clz(hi) : 32u;
    const unsigned long long n = hi ? (((unsigned long long)hi << 32) | lo) << lz : 0ull;
    const unsigned int mh = (unsigned int)(n >> 32), ml = (unsigned int)n;
#endif
    // mantissa with its hidden bit at bit 52, rounded; the hidden bit adds one to the exponent field
    unsigned long long r = ((((unsigned long long)mh << 32) | ml) >> 11) + ((ml >> 10) & 1u);
    r += (unsigned long long)(up - (lz << 20)) << 32;
    r |= (unsigned long long)s & 0x8000000000000000ull;
    return fx_double((int)mh < 0 ? r : 0ull);
}

// The same with two FP64 additions (ties to even): the words of v enter the
// mantissas of 2^84 and 2^52, the constants leave again, and only the second
// addition rounds.  The FP64 adder is otherwise idle here, but ten conversions
// would make it the bound.
template <int TOP = 58> BTRT_HD double fx_to_add(fx v, unsigned int em) {
    const unsigned long long u = (unsigned long long)v;
    const double b = fx_double(0x4530000000000000ull | ((u >> 32) ^ 0x80000000ull));
    const double a = fx_double(0x4330000000000000ull | (u & 0xffffffffull));
    const double r = (b - 19342822341709703277445120.0) + a;   // 2^84 + 2^63 + 2^52
    const unsigned long long rb = fx_bits(r);
    const unsigned int rh = (unsigned int)(rb >> 32);
    return fx_double((unsigned long long)(rh ? rh + em - ((1023u + TOP) << 20) : 0u) << 32 | (rb & 0xffffffffull));
}

// x as h 2^32 + l with l signed, for the products below.
struct FxArg {
    int h, l;
};
BTRT_HD FxArg fx_arg(fx x) {
    FxArg a;
    a.l = (int)(unsigned int)(unsigned long long)x;
    a.h = (int)(x >> 32) + (int)((unsigned int)a.l >> 31);
    return a;
}

// Sum of products C_k x_k, |C_k| < 1/2: p counts units, t 2^-32 units (the products
// of the two low words, at most a quarter of a unit per term, are left out).  t
// starts at half a unit of the result, which rounds it.  The host checks that t
// stays in range for the constants it hands out (fx_flux_fits).
struct FxSum {
    fx p, t;
};
BTRT_HD FxSum fx_sum() {
    FxSum s;
    s.p = 0;
    s.t = 1ll << 31;
    return s;
}
BTRT_HD void fx_add(FxSum &s, const FxArg &x, const FxConst &c) {
    s.t += (fx)x.h * c.lo;
    s.t += (fx)x.l * c.hi;
    s.p += (fx)x.h * c.hi;
}
BTRT_HD fx fx_value(const FxSum &s) { return s.p + (fx)(int)(s.t >> 32); }
BTRT_HD fx fx_mul(const FxArg &x, const FxConst &c) {
    const fx t = (1ll << 31) + (fx)x.h * c.lo + (fx)x.l * c.hi;
    return (fx)x.h * c.hi + (fx)(int)(t >> 32);
}
// Whether the sum qx jx + qy jy + cp phi + cg phi^{n-1} keeps t below 2^63 for every
// node the integer path takes: populations below 2^59 units (high words below 2^27;
// each enters the first three products with the coefficient ex qx + ey qy + cp),
// phi^{n-1} below 2^62.
inline bool fx_flux_fits(const FxConst &qx, const FxConst &qy, const FxConst &cp, const FxConst &cg) {
    const int ex[9] = {0, 1, 0, -1, 0, 1, -1, -1, 1}, ey[9] = {0, 0, 1, 0, -1, 1, 1, -1, -1};
    auto mag = [](double v) { return v < 0 ? -v : v; };
    double t = 17179869184.0 + 1073741824.0 * mag(cg.lo);
    for (int i = 0; i < 9; ++i) t += 134217728.0 * mag((double)ex[i] * qx.lo + (double)ey[i] * qy.lo + cp.lo);
    t += 2147483648.0 * (mag(qx.hi) + mag(qy.hi) + mag(cp.hi) + mag(cg.hi) + 4.0);
    return t < 9223372036854775808.0;
}

// x / 9, rounded to a unit.
BTRT_HD fx fx_ninth(fx x) {
    const FxConst c = {0x1c71c71c, 0x71c71c72};   // 2^64 / 9
    return fx_mul(fx_arg(x), c);
}

// The constant-coefficient collision's constants (see collide_fold for the scheme
// and the names): V/6 takes -(K1 - k0 I)/6 on the first moments, (K1 u^ + g)/6 on
// phi and -g/6 on phi^{n-1}, g = (I - K1/2) u^; the second-order block takes
// (k2 - k0)/18 on (3/2) sigma and (k2 - k0)/4 on delta and Pi_xy; om2 = (1 - k0)/2.
struct FxFold {
    FxConst Qxx, Qxy, Qyy, Px, Py, gx, gy, d18, d4, om2;
    FxConst ux, uy, k06;   // per-node coefficients: u^ and k0/6
    int ok;          // kFxOk* bits; a form whose bit is not set takes the FP64 collision
    int ush;         // u^ is its constant times 2^ush
    double trh, detA;      // half the trace and the determinant of A0^
};
// om2, u^ and k0/6 fit; the constant-coefficient form's fit; bgx = bgy; c3 != 0
enum { kFxOkGeneral = 1, kFxOkLinear = 2, kFxSameB = 4, kFxC3 = 8 };

// A constant as the products see it.
inline double fx_real(const FxConst &c) { return ldexp((double)c.hi, -32) + ldexp((double)c.lo, -64); }

// Whether every sum of fx_collide_linear stays in its word, beyond what fx_density and
// fx_flux_fits cover: the fluxes V/6 and the results, as linear maps of the populations
// (at most 1, in units of 2^59), phi^{n-1} (4) and the source (2), the word ending at 16.
inline bool fx_linear_fits(const FxFold &q) {
    const int ex[9] = {0, 1, 0, -1, 0, 1, -1, -1, 1}, ey[9] = {0, 0, 1, 0, -1, 1, 1, -1, -1};
    const double Qxx = fx_real(q.Qxx), Qxy = fx_real(q.Qxy), Qyy = fx_real(q.Qyy);
    const double Px = fx_real(q.Px), Py = fx_real(q.Py), gx = fx_real(q.gx), gy = fx_real(q.gy);
    const double d18 = fx_real(q.d18), d4 = fx_real(q.d4), om = 2.0 * fx_real(q.om2);
    double top = 6.0 * (fabs(Qxx) + fabs(Qxy)) + 9.0 * fabs(Px) + 4.0 * fabs(gx);
    top = fmax(top, 6.0 * (fabs(Qyy) + fabs(Qxy)) + 9.0 * fabs(Py) + 4.0 * fabs(gy)) + 0.5;   // X, Y: 2 max(|X|, |Y|) < 16
    bool fits = top < 8.0;
    for (int i = 0; i < 9; ++i) {
        const double w = i == 0 ? 4.0 / 9 : (i <= 4 ? 1.0 / 9 : 1.0 / 36);
        const int axis = i >= 1 && i <= 4, diag = i > 4;
        double sum = 2.0 * w + 4.0 * 18.0 * w * fabs(ex[i] * gx + ey[i] * gy) + 0.01;
        for (int k = 0; k < 9; ++k) {
            const double jx = ex[k], jy = ey[k], pxy = ex[k] * ey[k], del = ex[k] * ex[k] - ey[k] * ey[k];
            const double s32 = k == 0 ? -1.0 : (k <= 4 ? 0.5 : 2.0), ks = d18 * s32;
            const double X = Qxx * jx + Qxy * jy + Px, Y = Qxy * jx + Qyy * jy + Py;
            double r = (k == i ? om : 0.0) + w * (1.0 - om) + 18.0 * w * (ex[i] * X + ey[i] * Y);
            r += i == 0 ? 8.0 * ks : -ks;
            if (axis) r -= (ex[i] * ex[i] - ey[i] * ey[i]) * d4 * del;
            if (diag) r -= ex[i] * ey[i] * d4 * pxy;
            sum += fabs(r);
        }
        fits = fits && sum < 16.0;
    }
    return fits;
}

// The fold of a lattice: Q = K1 - k0 I (xx, xy, yy), P = K1 u^ + g, g, k2 - k0, 1 - k0, u^
// and k0.  A constant that does not fit (or is not finite), or a sum that could leave its
// word, clears the form's bit: the kernels then keep the FP64 collision.
// Per-node coefficients need no such test (units of 2^59, |u^| < 1): over k0 and k2 in
// (0, 2) the populations' part of a result, with k0 j/6 of the flux, and the source take
// at most 9.9 (rest direction), 4 (axes) and 1.8; C - phi, tested against 2, takes 1.8, 0.5
// and 0.5; the rest of the flux, (K1 E + B's change)/6, enters the axes with 2 (9.7 + 13 |u^| + 2)/6
// = 8.3, since K1's eigenvalues lie in (0, 2) and E is tested against 4.
inline FxFold fx_fold(const double (&Q)[3], const double (&P)[2], const double (&g)[2], double dk, double om,
                      const double (&u)[2], double k0) {
    // a constant holds less than a half: from there on it is half of u^, and the product doubled
    const int ush = fabs(u[0]) >= 0.4999 || fabs(u[1]) >= 0.4999 ? 1 : 0;
    const double us = ush ? 0.5 : 1.0;
    const double v[13] = {-Q[0], -Q[1], -Q[2], P[0], P[1], -g[0], -g[1], dk, dk, om, us * u[0], us * u[1], k0};
    const int div[13] = {6, 6, 6, 6, 6, 6, 6, 18, 4, 2, 1, 1, 6};
    FxConst k[13];
    bool fit[13], lin = true;
    for (int i = 0; i < 13; ++i) {
        fit[i] = fabs(v[i]) < 0.4999 * div[i];
        k[i] = fx_const(fit[i] ? v[i] : 0.0, div[i]);
        if (i < 10) lin = lin && fit[i];
    }
    FxFold q = {k[0], k[1], k[2], k[3], k[4], k[5], k[6], k[7], k[8], k[9], k[10], k[11], k[12], 0, ush, 0.0, 0.0};
    lin = lin && fx_flux_fits(q.Qxx, q.Qxy, q.Px, q.gx) && fx_flux_fits(q.Qxy, q.Qyy, q.Py, q.gy) && fx_linear_fits(q);
    // the low products of k0 j/6 + B's change/6 (up to 15 units) sum below 2^63 up to k0 = 1.9
    const bool gen = fit[9] && fit[10] && fit[11] && fit[12] && (!ush || k0 < 1.9);
    q.ok = (gen ? kFxOkGeneral : 0) | (lin ? kFxOkLinear : 0);
    return q;
}

// Sums whose terms may pass 2^63 (the caller tests the result before it is used).
BTRT_HD fx fx_plus(fx a, fx b) { return (fx)((unsigned long long)a + (unsigned long long)b); }
BTRT_HD fx fx_minus(fx a, fx b) { return (fx)((unsigned long long)a - (unsigned long long)b); }
BTRT_HD fx fx_times2(fx a, int sh) { return (fx)((unsigned long long)a << sh); }   // a 2^sh
// |phi| below LIMIT (in units of 2^32).
template <int LIMIT> BTRT_HD bool fx_below(fx phi) {
    return (unsigned int)((int)(phi >> 32) + LIMIT) < 2u * (unsigned int)LIMIT;
}

// a = k0 phi + source of a node; false when it could leave its word.  With k0 = 1 it
// cannot (nine populations below 2^59 units and a source below 2^60; in three dimensions
// nineteen below 2^58, and 2^59).  Otherwise half of it is formed again from the high
// words of its terms, which fits: three cut words, three units of 2^32 off.
template <bool K0ONE, bool SOURCE, int TOP>
BTRT_HD bool fx_density(fx phi, const FxArg &ph, const FxConst &om2, double src, unsigned int em, fx &a) {
    const fx s = SOURCE ? fx_from<TOP>(src, em) : 0;
    if (K0ONE) {
        a = phi + s;
        return true;
    }
    const fx om = fx_mul(ph, om2);
    a = fx_plus(fx_minus(phi, 2 * om), s);
    const int half = ((int)(phi >> 32) >> 1) - (int)(om >> 32) + ((int)(s >> 32) >> 1);
    constexpr unsigned int most = (1u << 30) - 4u;
    return (unsigned int)half + most < 2u * most;
}

// Populations after the collision from the node's integer moments: a = k0 phi +
// source, z the term of C(phi) != phi, X, Y = V/6, ks = (k2 - k0) sigma / 12, and the
// two anisotropic second-order terms t1 = (k2 - k0) delta / 4, t5 = (k2 - k0) Pi_xy / 4.
BTRT_HD void fx_expand(fx a, fx z, fx X, fx Y, fx ks, fx t1, fx t5, fx (&r)[9]) {
    const fx b = fx_ninth(a);
    const fx zk = z - ks;
    const fx T1 = b + zk, T5 = (b >> 2) + zk;
    r[0] = fx_minus(a, 4 * (T1 + T5));  // the other eight sum to 4 (T1 + T5)
    const fx A1 = T1 - t1, A2 = T1 + t1;
    r[1] = A1 + 2 * X;
    r[3] = A1 - 2 * X;
    r[2] = A2 + 2 * Y;
    r[4] = A2 - 2 * Y;
    const fx P = T5 - t5, M = T5 + t5;
    const fx Vp = (X + Y) >> 1, Vm = (X - Y) >> 1;
    r[5] = P + Vp;
    r[7] = P - Vp;
    r[6] = M - Vm;
    r[8] = M + Vm;
}

// Integer moments of a node.
struct FxMoments {
    fx phi, jx, jy, pxy, del, s32;   // s32 = (3/2) sigma = (a13 + a24)/2 + 2 (diagonals) - d0
};
BTRT_HD FxMoments fx_moments(const fx (&D)[9]) {
    FxMoments m;
    const fx a13 = D[1] + D[3], a24 = D[2] + D[4];
    const fx s57 = D[5] + D[7], s68 = D[6] + D[8];
    const fx d57 = D[5] - D[7], d68 = D[6] - D[8];
    const fx sd = s57 + s68, a1324 = a13 + a24;
    m.phi = D[0] + sd + a1324;
    m.jx = (D[1] - D[3]) + (d57 - d68);
    m.jy = (D[2] - D[4]) + (d57 + d68);
    m.pxy = s57 - s68;
    m.del = a13 - a24;
    m.s32 = (a1324 >> 1) + 2 * sd - D[0];
    return m;
}

// The common exponent of a node's populations; false outside the range.
template <int N> BTRT_HD bool fx_common_exp(const double (&d)[N], unsigned int &em) {
    em = fx_exp(d[0]);
#pragma unroll
    for (int i = 1; i < N; ++i) {
        const unsigned int e = fx_exp(d[i]);
        em = em > e ? em : e;
    }
    return em - kFxExpMin <= kFxExpMax - kFxExpMin;
}

// Whether a node is zero throughout (its results then are as well).
template <int N> BTRT_HD bool fx_all_zero(const double (&d)[N], double phi_prev, double src) {
    unsigned long long any = fx_bits(phi_prev) | fx_bits(src);
#pragma unroll
    for (int i = 0; i < N; ++i) any |= fx_bits(d[i]);
    return (any << 1) == 0;
}
// A node whose largest population is out of the range: large values take the FP64 form, and
// so do tiny ones, for its gradual underflow; zeros are done.  On the device the
// out-of-line FP64 forms of the one-step sweeps look for those: with the test in line the
// 8192^2 sweep took 38.56 ms instead of 37.48.  ZEROS: in line all the same (many steps per
// launch: the 64^2 hill 0.959 ms against 0.977).
template <bool ZEROS, int N>
BTRT_HD bool fx_out_of_range(const double (&d)[N], double phi_prev, double src, double &phi_out) {
#ifdef __CUDA_ARCH__
    if (!ZEROS) return false;
#endif
    phi_out = 0.0;
    return fx_all_zero(d, phi_prev, src);
}

// The outputs of a node, (1 - k0) D_i + r_i, as FP64; the first NADD by the FP64
// adder (fx_to_add), the others by integer instructions.
template <bool K0ONE, int NADD, int TOP = 58, int N>
BTRT_HD void fx_store(const fx (&D)[N], const fx (&r)[N], const FxConst &om2, unsigned int em, double (&d)[N]) {
#pragma unroll
    for (int i = 0; i < N; ++i) {
        const fx v = K0ONE ? r[i] : r[i] + 2 * fx_mul(fx_arg(D[i]), om2);
        d[i] = i < NADD ? fx_to_add<TOP>(v, em) : fx_to<TOP>(v, em);
    }
}

// Populations that the FP64 adder converts in the constant-coefficient collision:
// the 8192^2 manufactured solution (20 steps) measured 52.7 / 49.0 / 49.4 ms with 0 / 3 / 5
// (four rows per thread) and 38.8 / 38.2 / 42.0 with 4 / 5 / 6 at six blocks per SM,
// 37.5 / 38.1 with 4 / 5 at five.
#ifndef BTRT_FX_NADD
#define BTRT_FX_NADD 4
#endif

// The constant-coefficient collision of one node: d in, post-collision populations
// out; src is the node's source term (0 when there is none).  Returns false, with
// d untouched, when the node's values leave the range (the caller takes the FP64
// form): the exponents of the populations, or phi^{n-1} or the source more than four
// times or twice the largest population.
template <bool K0ONE, bool SOURCE, bool ZEROS = false>
BTRT_HD bool fx_collide_linear(const FxFold &q, double (&d)[9], double phi_prev, double src, double &phi_out) {
    unsigned int em;
    const bool in = fx_common_exp(d, em);
    if (!in || fx_exp(phi_prev) > em + (2u << 20))
        return !in && fx_out_of_range<ZEROS>(d, phi_prev, SOURCE ? src : 0.0, phi_out);
    if (SOURCE && fx_exp(src) > em + (1u << 20)) return false;
    fx D[9];
#pragma unroll
    for (int i = 0; i < 9; ++i) D[i] = fx_from(d[i], em);
    const FxMoments m = fx_moments(D);
    const FxArg jx = fx_arg(m.jx), jy = fx_arg(m.jy), ph = fx_arg(m.phi), pp = fx_arg(fx_from(phi_prev, em));
    FxSum sx = fx_sum(), sy = fx_sum();
    fx_add(sx, jx, q.Qxx);
    fx_add(sx, jy, q.Qxy);
    fx_add(sx, ph, q.Px);
    fx_add(sx, pp, q.gx);
    fx_add(sy, jx, q.Qxy);
    fx_add(sy, jy, q.Qyy);
    fx_add(sy, ph, q.Py);
    fx_add(sy, pp, q.gy);
    const fx ks = fx_mul(fx_arg(m.s32), q.d18), t1 = fx_mul(fx_arg(m.del), q.d4), t5 = fx_mul(fx_arg(m.pxy), q.d4);
    fx a, r[9];
    if (!fx_density<K0ONE, SOURCE, 58>(m.phi, ph, q.om2, src, em, a)) return false;
    fx_expand(a, 0, fx_value(sx), fx_value(sy), ks, t1, t5, r);
    fx_store<K0ONE, BTRT_FX_NADD>(D, r, q.om2, em, d);
    phi_out = fx_to(m.phi, em);
    return true;
}

// ---------------------------------------------------------------- D3Q19
// Velocity order as in btrt_sweep3.cuh: rest; +-x, +-y, +-z; xy, xz and yz diagonals
// with signs (+,+) (-,+) (+,-) (-,-).  Units of 2^(E - 57): nineteen populations
// below 2^58 sum below 2^63.
constexpr int kFxTop3 = 57;

// V/6 takes -(K1 - k0 I)/6 on the first moments, (K1 u^ + g)/6 on phi, -g/6 on
// phi^{n-1}; (k2 - k0)/12 acts on 3 h_a, (k2 - k0)/24 on 3 t3, (k2 - k0)/4 on Pi_ab
// (collide3 for the scheme and the names).
struct FxFold3 {
    FxConst Q[6];    // xx, xy, xz, yy, yz, zz
    FxConst P[3], g[3], d12, d24, d4, om2;
    int ok;          // kFxOk* bits
    int pad;
};

// As fx_flux_fits: populations below 2^58 units, phi^{n-1} below 2^61.
inline bool fx_flux_fits3(const FxConst &qx, const FxConst &qy, const FxConst &qz, const FxConst &cp, const FxConst &cg) {
    auto mag = [](double v) { return v < 0 ? -v : v; };
    double t = 17179869184.0 + 536870912.0 * mag(cg.lo);
    for (int x = -1; x <= 1; ++x)
        for (int y = -1; y <= 1; ++y)
            for (int z = -1; z <= 1; ++z)
                if (x * x + y * y + z * z <= 2)
                    t += 67108864.0 * mag((double)x * qx.lo + (double)y * qy.lo + (double)z * qz.lo + cp.lo);
    t += 2147483648.0 * (mag(qx.hi) + mag(qy.hi) + mag(qz.hi) + mag(cp.hi) + mag(cg.hi) + 5.0);
    return t < 9223372036854775808.0;
}

// As fx_linear_fits: populations at most 1 (in units of 2^58), phi^{n-1} 4, the source 2,
// the word ending at 32.
inline bool fx_linear_fits3(const FxFold3 &q) {
    const int c[19][3] = {{0, 0, 0},  {1, 0, 0},  {-1, 0, 0}, {0, 1, 0},   {0, -1, 0}, {0, 0, 1},  {0, 0, -1},
                          {1, 1, 0},  {-1, 1, 0}, {1, -1, 0}, {-1, -1, 0}, {1, 0, 1},  {-1, 0, 1}, {1, 0, -1},
                          {-1, 0, -1}, {0, 1, 1}, {0, -1, 1}, {0, 1, -1},  {0, -1, -1}};
    const int at[3][3] = {{0, 1, 2}, {1, 3, 4}, {2, 4, 5}};
    double Q[3][3], P[3], g[3], top = 0.0;
    for (int a = 0; a < 3; ++a) {
        P[a] = fx_real(q.P[a]);
        g[a] = fx_real(q.g[a]);
        double t = 19.0 * fabs(P[a]) + 4.0 * fabs(g[a]) + 0.5;
        for (int b = 0; b < 3; ++b) {
            Q[a][b] = fx_real(q.Q[at[a][b]]);
            t += 10.0 * fabs(Q[a][b]);
        }
        top = fmax(top, t);
    }
    bool fits = top < 16.0;   // X, Y, Z: twice the largest < 32
    const double d4 = fx_real(q.d4), om = 2.0 * fx_real(q.om2);
    for (int i = 0; i < 19; ++i) {
        const double w = i == 0 ? 1.0 / 3 : (i <= 6 ? 1.0 / 18 : 1.0 / 36);
        double cg = 0.0;
        for (int a = 0; a < 3; ++a) cg += c[i][a] * g[a];
        double sum = 2.0 * w + 4.0 * 18.0 * w * fabs(cg) + 0.01;
        for (int k = 0; k < 19; ++k) {
            // w (a + 3 c.V - (9/2) (k2 - k0) (c c : N - t3)), N = sum c c d - phi I / 3, t3 = tr N / 3
            double V = 0.0, H = 0.0, e2 = 0.0, t3 = 0.0;
            for (int a = 0; a < 3; ++a) {
                double X = P[a];
                for (int b = 0; b < 3; ++b) {
                    X += Q[a][b] * c[k][b];
                    H += c[i][a] * c[i][b] * (c[k][a] * c[k][b] - (a == b ? 1.0 / 3 : 0.0));
                }
                V += c[i][a] * X;
                e2 += c[k][a] * c[k][a];
            }
            t3 = (e2 - 1.0) / 3.0;
            sum += fabs((k == i ? om : 0.0) + w * (1.0 - om) + 18.0 * w * V - 18.0 * w * d4 * (H - t3));
        }
        fits = fits && sum < 32.0;
    }
    return fits;
}

// As fx_fold: Q = K1 - k0 I (xx, xy, xz, yy, yz, zz), P = K1 u^ + g, g, k2 - k0, 1 - k0.
inline FxFold3 fx_fold3(const double (&Q)[6], const double (&P)[3], const double (&g)[3], double dk, double om) {
    const double v[16] = {-Q[0], -Q[1], -Q[2], -Q[3], -Q[4], -Q[5], P[0], P[1], P[2], -g[0], -g[1], -g[2], dk, dk, dk, om};
    const int div[16] = {6, 6, 6, 6, 6, 6, 6, 6, 6, 6, 6, 6, 12, 24, 4, 2};
    FxConst k[16];
    bool ok = true;
    for (int i = 0; i < 16; ++i) {
        const bool fits = fabs(v[i]) < 0.4999 * div[i];
        k[i] = fx_const(fits ? v[i] : 0.0, div[i]);
        ok = ok && fits;
    }
    FxFold3 q = {};
    for (int i = 0; i < 6; ++i) q.Q[i] = k[i];
    for (int i = 0; i < 3; ++i) {
        q.P[i] = k[6 + i];
        q.g[i] = k[9 + i];
    }
    q.d12 = k[12];
    q.d24 = k[13];
    q.d4 = k[14];
    q.om2 = k[15];
    ok = ok && fx_flux_fits3(k[0], k[1], k[2], k[6], k[9]) && fx_flux_fits3(k[1], k[3], k[4], k[7], k[10]) &&
         fx_flux_fits3(k[2], k[4], k[5], k[8], k[11]) && fx_linear_fits3(q);
    q.ok = (fabs(om) < 0.9998 ? kFxOkGeneral : 0) | (ok ? kFxOkLinear : 0);
    return q;
}

struct FxMoments3 {
    fx phi, jx, jy, jz, pxy, pxz, pyz;
    fx hx, hy, t3;   // 3 h_x, 3 h_y (h_z = -h_x - h_y) and 3 t3
};
BTRT_HD FxMoments3 fx_moments3(const fx (&D)[19]) {
    FxMoments3 m;
    const fx ax = D[1] + D[2], ay = D[3] + D[4], az = D[5] + D[6];
    const fx xyp = D[7] + D[8], xym = D[9] + D[10], xyd = D[7] - D[8], xye = D[9] - D[10];
    const fx xzp = D[11] + D[12], xzm = D[13] + D[14], xzd = D[11] - D[12], xze = D[13] - D[14];
    const fx yzp = D[15] + D[16], yzm = D[17] + D[18], yzd = D[15] - D[16], yze = D[17] - D[18];
    const fx sxy = xyp + xym, sxz = xzp + xzm, syz = yzp + yzm;
    m.jx = (D[1] - D[2]) + (xyd + xye) + (xzd + xze);
    m.jy = (D[3] - D[4]) + (xyp - xym) + (yzd + yze);
    m.jz = (D[5] - D[6]) + (xzp - xzm) + (yzp - yzm);
    m.pxy = xyd - xye;
    m.pxz = xzd - xze;
    m.pyz = yzd - yze;
    const fx Pxx = ax + sxy + sxz, Pyy = ay + sxy + syz, Pzz = az + sxz + syz;
    const fx S = Pxx + Pyy + Pzz, sd = sxy + sxz + syz;
    m.phi = D[0] + (S - sd);            // the diagonals count twice in S
    m.hx = 2 * Pxx - Pyy - Pzz;
    m.hy = 2 * Pyy - Pxx - Pzz;
    m.t3 = sd - D[0];                   // S - phi
    return m;
}

// Populations from a = k0 phi + source, z (the term of C(phi) != phi on the diagonals),
// X = V/6, Hx, Hy = (k2 - k0) h / 4, K = (k2 - k0) t3 / 8, t_ab = (k2 - k0) Pi_ab / 4.
BTRT_HD void fx_expand3(fx a, fx z, fx X, fx Y, fx Z, fx Hx, fx Hy, fx K, fx txy, fx txz, fx tyz, fx (&r)[19]) {
    const fx b = fx_ninth(a) >> 1;                // a / 18
    const fx Hz = -(Hx + Hy), G = (b >> 1) + z - K;
    r[0] = fx_minus(a - 6 * b, 12 * G);           // the axis directions sum to 6 b, the diagonals to 12 G
    const fx bx = b - Hx, by = b - Hy, bz = b - Hz;
    r[1] = bx + X;
    r[2] = bx - X;
    r[3] = by + Y;
    r[4] = by - Y;
    r[5] = bz + Z;
    r[6] = bz - Z;
    const fx gx = Hx >> 1, gy = Hy >> 1, gz = -(gx + gy);
    const fx xy = G + gz, xz = G + gy, yz = G + gx;
    const fx xyp = (X + Y) >> 1, xym = (X - Y) >> 1, xzp = (X + Z) >> 1, xzm = (X - Z) >> 1;
    const fx yzp = (Y + Z) >> 1, yzm = (Y - Z) >> 1;
    r[7] = xy - txy + xyp;
    r[10] = xy - txy - xyp;
    r[8] = xy + txy - xym;
    r[9] = xy + txy + xym;
    r[11] = xz - txz + xzp;
    r[14] = xz - txz - xzp;
    r[12] = xz + txz - xzm;
    r[13] = xz + txz + xzm;
    r[15] = yz - tyz + yzp;
    r[18] = yz - tyz - yzp;
    r[16] = yz + tyz - yzm;
    r[17] = yz + tyz + yzm;
}

// Populations of D3Q19 that the FP64 adder converts: 3.45 / 3.29 / 3.27 / 3.51 ms with
// 0 / 5 / 8 / 12 on the 128^3 hill (20 steps).
#ifndef BTRT_FX_NADD3
#define BTRT_FX_NADD3 8
#endif

// As fx_collide_linear.
template <bool K0ONE, bool SOURCE>
BTRT_HD bool fx_collide_linear3(const FxFold3 &q, double (&d)[19], double phi_prev, double src, double &phi_out) {
    unsigned int em;
    const bool in = fx_common_exp(d, em);
    if (!in || fx_exp(phi_prev) > em + (2u << 20))
        return !in && fx_out_of_range<false>(d, phi_prev, SOURCE ? src : 0.0, phi_out);
    if (SOURCE && fx_exp(src) > em + (1u << 20)) return false;
    fx D[19];
#pragma unroll
    for (int i = 0; i < 19; ++i) D[i] = fx_from<kFxTop3>(d[i], em);
    const FxMoments3 m = fx_moments3(D);
    const FxArg jx = fx_arg(m.jx), jy = fx_arg(m.jy), jz = fx_arg(m.jz), ph = fx_arg(m.phi);
    const FxArg pp = fx_arg(fx_from<kFxTop3>(phi_prev, em));
    FxSum sx = fx_sum(), sy = fx_sum(), sz = fx_sum();
    fx_add(sx, jx, q.Q[0]);
    fx_add(sx, jy, q.Q[1]);
    fx_add(sx, jz, q.Q[2]);
    fx_add(sx, ph, q.P[0]);
    fx_add(sx, pp, q.g[0]);
    fx_add(sy, jx, q.Q[1]);
    fx_add(sy, jy, q.Q[3]);
    fx_add(sy, jz, q.Q[4]);
    fx_add(sy, ph, q.P[1]);
    fx_add(sy, pp, q.g[1]);
    fx_add(sz, jx, q.Q[2]);
    fx_add(sz, jy, q.Q[4]);
    fx_add(sz, jz, q.Q[5]);
    fx_add(sz, ph, q.P[2]);
    fx_add(sz, pp, q.g[2]);
    fx a, r[19];
    if (!fx_density<K0ONE, SOURCE, kFxTop3>(m.phi, ph, q.om2, src, em, a)) return false;
    fx_expand3(a, 0, fx_value(sx), fx_value(sy), fx_value(sz), fx_mul(fx_arg(m.hx), q.d12), fx_mul(fx_arg(m.hy), q.d12),
               fx_mul(fx_arg(m.t3), q.d24), fx_mul(fx_arg(m.pxy), q.d4), fx_mul(fx_arg(m.pxz), q.d4),
               fx_mul(fx_arg(m.pyz), q.d4), r);
    fx_store<K0ONE, BTRT_FX_NADD3, kFxTop3>(D, r, q.om2, em, d);
    phi_out = fx_to<kFxTop3>(m.phi, em);
    return true;
}

}  // namespace btrt
