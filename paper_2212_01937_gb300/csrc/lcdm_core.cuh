// Distance integrals of one (cosmology, redshift) pair and their reverse-mode
// derivatives, in either precision.
//
// The reduction is that of eqs. (3.7)-(3.9) / (B.1)-(B.3); it is written in
// coordinates in which everything that does not depend on z is a constant of
// the row.  Divided by N^2 (N = sqrt(E^2(0)) times the normalisation of the
// roots), Carlson's arguments are
//   s1 = n_A n_B + n_P n_P*,  u = n_P n_A + n_P* n_B (and u*),  n_j = sqrt(1 + z q_j),
//   x1 = s1^2, y = u^2, and p = u_A5^2 for the third-kind integral of eq. (3.8),
// and all their differences are constants of the row times z^2:
//   the deviations X_i of (x1, y, y*) from their mean satisfy
//     X^3 + e2 z^4 X - e3 z^6 = 0,  e2 = -I / (3 S0^2),  e3 = -J / (27 S0^3)
//   with I, J the invariants of the quartic E^2(x) and S0 = E^2(x = 1);
//   p = s5 - d,  s5 = (n_B |n_P|^2 + (1+z) n_A)^2 / (1+z),  d = OL/S0 z^2 (1+eps)^2 n_A^2 / (1+z);
//   mean - p = m z^2,  (p - x1)(p - y)(p - y*) = -k^2 (OL/S0) z^6,
//   k = 3 k2,  eps = -1/rho_A.
// (p is a ratio of sums of positive numbers but for the subtraction of d, and
// it is positive wherever E^2 > 0 between the limits: R_C(s5, p) diverges like
// p^-1/2 while t is finite.  So no principal values occur.)
// With eps = q_A = 0 and the cubic's real root in the place of B the same
// formulas are those of App. B.1 (the radiationless case), so there is one
// path for all root kinds.
//
// Consequences for the duplication (Carlson's algorithm, the paper's ref. [10]):
//  * the sequence is carried without the division by four (x <- x + lambda):
//    differences are then constant and the truncated series are polynomials
//    in w = z^2 dev / A with constants of the row as coefficients, so a degree more
//    costs one multiply-add (and a larger deviation may be left: fewer steps).
//    dev is the row's largest deviation over z^2: with it in w the coefficients
//    are at most of order one (a power of dev up to the eleventh leaves single
//    precision where E^2(0) is small, a sum of densities of 1e-5 or a lower limit
//    at which the universe loiters);
//  * the stopping rule is one multiplication: z^2 max|deviation| <= tol A;
//  * y y* = x1 S^2 after the first step, so a step takes two square roots
//    (one more per third-kind track) and no division by a difference;
//  * the R_C(1, 1+e) argument of a third-kind track is const z^6 / d^2.
// Gradients are taken in reverse through the stored sequence (s1, S, P and
// sqrt(p) of each step): its cost does not depend on the number of
// parameters, and nothing is divided by a difference of arguments.
#pragma once
#include "lcdm_math.cuh"

namespace lcdm {

// Row record of the core (T = float or double).  Tangent slots k = 0..5:
// Om, OL, Or, Ok, Os, Ox (the first ncol - 1 used).
enum CoreField {
    C_QA = 0, C_QB, C_QR, C_QRL,          // q_j = -1/r_j; the pair: real and imaginary part, or the two reals
    C_QI, C_QIL, C_C2, C_KIND,            // (QRL, QIL: low words in single precision); c2 = 2 / sqrt(S0);
                                          // KIND: 1 for a complex pair, 0 for two reals
    C_DH, C_TH, C_IH0, C_OK,              // c/H0 [Mpc], 1/H0 [Gyr], 1/H0, Omega_k0
    C_DF, C_B = 13,                       // DF: max deviation / z^2 from the mean of three; B: series of R_F (10)
    C_RS = 23,                            // -1 / (2 S0) with free S0, 0 under the closure
    C_DJ = 24, C_EPS, C_K2, C_K3,         // DJ: max deviation from the mean of five (t track)
    C_A = 28,                             // series of the t track's R_J (10)
    C_FREE0 = 38, C_FREE1,
    // absorption distance (values)
    X_HX = 40, X_LX, X_PX, X_DX,          // p0 - x1 = -hx z^2; p0 = (..)^2 - lx z^2 w_B; pi/z^4; max deviation
    X_C0, X_T1, X_G1, X_G2,
    X_G3, X_G4, X_G5, X_SY,
    X_N0, X_N1, X_N2, X_FREE,
    X_AB, X_LAM, X_SQ, X_PQ,              // q_P + q_P*, q_P q_P*
    X_S = 60,                             // series at p0, at x1, and their divided differences, by degree (3 x 10)
    C_TAN = 92, C_TSTRIDE = 28,           // tangents of slot k at C_TAN + 28 k:
    CT_QA = 0, CT_QB, CT_QR, CT_QI, CT_B, CT_EPS = 14, CT_K2, CT_K3, CT_A = 17, CT_END = 27,
    NCORE = C_TAN + 6 * C_TSTRIDE
};
enum { CORE_NS = 10 };       // room for the series' coefficients in the record: degrees 2 to 11
enum { CORE_NS_ONCE = 6 };   // used where a record serves one evaluation (the limit at infinity): there the
                             // coefficients cost more than the steps they save, and instead of their
                             // tangents the record holds (e2, e3, m) and theirs
enum { C_E2 = C_B + 6, C_E3 = C_B + 7, C_M = C_A + 6, CT_E2 = CT_B, CT_E3 = CT_B + 1, CT_M = CT_A };

// ----------------------------------------------------- two pairs in a thread ---
// Two single-precision numbers in one 64-bit register pair: this part's packed
// add, multiply and fused multiply-add do both in one issue slot (of the two
// cycles that their 64 lane operations take), and the pair kernels are bound by
// issue.  Written without a rounding modifier, so that a product and a sum
// contract as for plain floats.
struct F2 { float x, y; };
LCDM_HD F2 mkf2(float x, float y) { F2 r; r.x = x; r.y = y; return r; }
#ifdef __CUDA_ARCH__
LCDM_HD uint64_t f2_bits(F2 a) { uint64_t r; asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a.x), "f"(a.y)); return r; }
LCDM_HD F2 f2_of(uint64_t u) { F2 r; asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(u)); return r; }
LCDM_HD F2 operator*(F2 a, F2 b) {
    uint64_t r;
    asm("mul.ftz.f32x2 %0, %1, %2;" : "=l"(r) : "l"(f2_bits(a)), "l"(f2_bits(b)));
    return f2_of(r);
}
LCDM_HD F2 operator+(F2 a, F2 b) {
    uint64_t r;
    asm("add.ftz.f32x2 %0, %1, %2;" : "=l"(r) : "l"(f2_bits(a)), "l"(f2_bits(b)));
    return f2_of(r);
}
LCDM_HD F2 operator-(F2 a, F2 b) {
    uint64_t r;
    asm("sub.ftz.f32x2 %0, %1, %2;" : "=l"(r) : "l"(f2_bits(a)), "l"(f2_bits(b)));
    return f2_of(r);
}
#else
LCDM_HD F2 operator*(F2 a, F2 b) { return mkf2(a.x * b.x, a.y * b.y); }
LCDM_HD F2 operator+(F2 a, F2 b) { return mkf2(a.x + b.x, a.y + b.y); }
LCDM_HD F2 operator-(F2 a, F2 b) { return mkf2(a.x - b.x, a.y - b.y); }
#endif
LCDM_HD F2 operator-(F2 a) { return mkf2(-a.x, -a.y); }
template <> struct CstImpl<F2> { static LCDM_HD F2 make(double v) { return mkf2((float)v, (float)v); } };

// What the core asks of its scalar beside arithmetic: the record's type, a
// record entry as a scalar, |a|, a selection by sign, and comparisons (of both
// numbers: all of them, or any).
template <class T> struct Scalar {
    typedef T rec;
    static LCDM_HD T of(T v) { return v; }
};
template <> struct Scalar<F2> {
    typedef float rec;
    static LCDM_HD F2 of(float v) { return mkf2(v, v); }
};
LCDM_HD float abs_(float a) { return fabsf(a); }
LCDM_HD double abs_(double a) { return fabs(a); }
LCDM_HD F2 abs_(F2 a) { return mkf2(fabsf(a.x), fabsf(a.y)); }
template <class T> LCDM_HD T sel_ge0(T c, T a, T b) { return c >= cst<T>(0.0) ? a : b; }
LCDM_HD F2 sel_ge0(F2 c, F2 a, F2 b) { return mkf2(c.x >= 0.f ? a.x : b.x, c.y >= 0.f ? a.y : b.y); }
template <class T> LCDM_HD bool all_le(T a, T b) { return a <= b; }
LCDM_HD bool all_le(F2 a, F2 b) { return a.x <= b.x && a.y <= b.y; }
template <class T> LCDM_HD bool any_gt(T a, T b) { return a > b; }
LCDM_HD bool any_gt(F2 a, F2 b) { return a.x > b.x || a.y > b.y; }
// bits of the numbers that are not <= (NaN included)
template <class T> LCDM_HD int not_le(T a, T b) { return a <= b ? 0 : 1; }
LCDM_HD int not_le(F2 a, F2 b) { return (a.x <= b.x ? 0 : 1) | (a.y <= b.y ? 0 : 2); }
// (in double a comparison would hold the FP64 pipe: both sides in single)
LCDM_HD float cmp_(float a) { return a; }
LCDM_HD float cmp_(double a) { return (float)a; }
LCDM_HD F2 cmp_(F2 a) { return a; }
LCDM_HD float times_(float k, float a) { return k * a; }
LCDM_HD F2 times_(float k, F2 a) { return mkf2(k, k) * a; }

// ------------------------------------------------------------- arithmetic ---
// 1/sqrt, sqrt and 1/x of positive normal numbers.  Single precision: the
// hardware approximations (within two ulp).  Double precision: one step of
// Householder's third-order method from the hardware's 20-bit approximation
// (error 2^-60 before rounding), written out for each: with y ~ x^-1/2, t = x y
// and e = 1 - t y,  x^-1/2 = y + y e (1/2 + 3 e / 8),  x^1/2 = t + t e (1/2 + 3 e / 8);
// with y ~ 1/x, e = 1 - x y,  1/x = y + y (e + e^2).  Five, five and three FP64
// instructions; CUDA's square root issues about 9, its division 9, rsqrt 5.5.
LCDM_HD float rsq(float x) { return srsqrt(x); }
LCDM_HD float sqt(float x) { return x * srsqrt(x); }
LCDM_HD F2 rsq(F2 x) { return mkf2(srsqrt(x.x), srsqrt(x.y)); }
LCDM_HD F2 sqt(F2 x) { return x * rsq(x); }
#ifdef __CUDA_ARCH__
LCDM_HD double rsq_seed(double x) {
    double y;
    asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
    return y;
}
#endif
LCDM_HD double rsq(double x) {
#ifdef __CUDA_ARCH__
    const double y = rsq_seed(x), e = fma(-(x * y), y, 1.0);
    return fma(y * e, fma(0.375, e, 0.5), y);
#else
    return 1.0 / sqrt(x);
#endif
}
LCDM_HD double sqt(double x) {
#ifdef __CUDA_ARCH__
    const double y = rsq_seed(x), t = x * y, e = fma(-t, y, 1.0);
    return fma(t * e, fma(0.375, e, 0.5), t);
#else
    return sqrt(x);
#endif
}
LCDM_HD float rcp_(float x) {
#ifdef __CUDA_ARCH__
    float y;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
#else
    return 1.0f / x;
#endif
}
LCDM_HD F2 rcp_(F2 x) { return mkf2(rcp_(x.x), rcp_(x.y)); }
LCDM_HD double rcp_(double x) {
#ifdef __CUDA_ARCH__
    double y;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
    const double e = fma(-x, y, 1.0);
    return fma(y, fma(e, e, e), y);
#else
    return 1.0 / x;
#endif
}

template <class T> struct CoreTol;
template <> struct CoreTol<float> {
    // largest deviation left to the series of degree ns + 1 (its truncation:
    // about dup^(ns + 2) / 100); relative deviation s of R_C's; largest s1 taken
    // without scaling
    static constexpr float dup = 0.25f, once = 0.15f, rc = 0.1f, big = 65536.0f, e_series = 0.1f;
    enum { maxit = 24, ns = 8 };
};
template <> struct CoreTol<F2> : CoreTol<float> {};
template <> struct CoreTol<double> {
    // (big: the stopping tests compare z^2 times the deviation in single precision)
    static constexpr double dup = 0.05, once = 0.009, rc = 0.008, big = 1e9, e_series = 0.03;
    enum { maxit = 40, ns = 10 };
};

// R_C(1, 1 + e) and its derivative by closed relations, for e beyond the
// series; b = sqrt(1 + e)
template <class T> struct RcE { T v, d; };
template <class T> LCDM_NI RcE<T> rc1_far(T e, T b) {
    T a = cst<T>(1.0), tm = cst<T>(1.0);
    const T b0 = b;
    T U = a * a + cst<T>(2.0) * b * b;
#pragma unroll 1
    for (int m = 0; m < CoreTol<T>::maxit && !(fabs(e) <= CoreTol<T>::rc * U); m++) {
        const T n = a + b, q = cst<T>(2.0) * b * n;
        a = n;
        b = sqt(q);
        U = a * a + cst<T>(2.0) * b * b;
        tm = tm + tm;
    }
    const T s = e * rcp_(U);
    const T ser = cst<T>(1.0) + s * s * (cst<T>(0.3) + s * (cst<T>(1.0 / 7) + s * (cst<T>(0.375)
                  + s * (cst<T>(9.0 / 22) + s * (cst<T>(159.0 / 208) + s * cst<T>(1.125))))));
    RcE<T> r;
    r.v = tm * ser * rsq(U * cst<T>(1.0 / 3));
    // 2 e dR_C/de = 1/(1+e) - R_C (from Euler's relation and the derivative along x and y together)
    r.d = (rcp_(b0 * b0) - r.v) * cst<T>(0.5) / e;
    return r;
}
// R_C(1, 1+e) = sum (-e)^n / (2n+1), with its derivative (GRAD)
LCDM_HD RcE<float> rc1_core(float e, bool grad) {
    if (fabsf(e) <= CoreTol<float>::e_series) {
        RcE<float> r;
        const float w = -e;
        float s = 1.0f / 13, ds = 0.f;
#pragma unroll
        for (int n = 5; n >= 0; n--) { ds = ds * w + s; s = 1.0f / (2 * n + 1) + w * s; }
        r.v = s;
        r.d = -ds;
        return r;
    }
    return rc1_far<float>(e, sqt(1.0f + e));
}
LCDM_HD RcE<F2> rc1_core(F2 e, bool grad) {
    RcE<F2> r;
    if (all_le(abs_(e), cst<F2>(CoreTol<float>::e_series))) {
        const F2 w = -e;
        F2 s = cst<F2>(1.0 / 13), ds = cst<F2>(0.0);
#pragma unroll
        for (int n = 5; n >= 0; n--) {
            if (grad) ds = ds * w + s;
            s = cst<F2>(1.0 / (2 * n + 1)) + w * s;
        }
        r.v = s;
        r.d = -ds;
        return r;
    }
    const RcE<float> a = rc1_core(e.x, grad), b = rc1_core(e.y, grad);
    r.v = mkf2(a.v, b.v);
    r.d = mkf2(a.d, b.d);
    return r;
}
LCDM_HD RcE<double> rc1_core(double e, bool grad) {
    // e falls by 64 or more per step: most steps need a few terms only
    const double w = -e;
    const double ae = fabs(e);
    RcE<double> r;
    if (ae <= 3e-5) {
        r.v = 1.0 + w * (1.0 / 3 + w * (0.2 + w * (1.0 / 7)));
        r.d = grad ? -(1.0 / 3 + w * (0.4 + w * (3.0 / 7 + w * (4.0 / 9)))) : 0.0;
        return r;
    }
    if (ae <= CoreTol<double>::e_series) {
        double s = 1.0 / 25, ds = 0.0;
#pragma unroll
        for (int n = 11; n >= 0; n--) {
            if (grad) ds = ds * w + s;
            s = 1.0 / (2 * n + 1) + w * s;
        }
        r.v = s;
        r.d = -ds;
        return r;
    }
    return rc1_far<double>(e, sqt(1.0 + e));
}
// (R_C(1, 1+e) - 1) / e
template <class T> LCDM_HD T rc1m1_core(T e) {
    constexpr int NT = sizeof(T) == 4 ? 6 : 12;
    const T w = -e;
    if (sizeof(T) == 8 && fabs(e) <= cst<T>(3e-5))
        return cst<T>(-1.0 / 3) + w * (cst<T>(-0.2) + w * (cst<T>(-1.0 / 7) + w * cst<T>(-1.0 / 9)));
    if (fabs(e) <= CoreTol<T>::e_series) {
        T s = cst<T>(-1.0 / (2 * NT + 3));
#pragma unroll
        for (int n = NT; n >= 1; n--) s = cst<T>(-1.0 / (2 * n + 1)) + w * s;
        return s;
    }
    return (rc1_far<T>(e, sqt(cst<T>(1.0) + e)).v - cst<T>(1.0)) / e;
}
LCDM_HD F2 rc1m1_core(F2 e) {
    if (all_le(abs_(e), cst<F2>(CoreTol<float>::e_series))) {
        const F2 w = -e;
        F2 s = cst<F2>(-1.0 / 15);
#pragma unroll
        for (int n = 6; n >= 1; n--) s = cst<F2>(-1.0 / (2 * n + 1)) + w * s;
        return s;
    }
    return mkf2(rc1m1_core<float>(e.x), rc1m1_core<float>(e.y));
}
// [R_C(1, 1-w) - (1-w)^-1/2] / w  (see phi_rc) for 0 <= w < 1, so = sqrt(1-w)
// (which cancels if formed from w near 1).  Beyond the series' range R_C's
// duplication is carried on the difference itself: with a = sqrt(x), b =
// sqrt(y), x - y = w, and b' = sqrt(2 b (a + b)) of the next step,
//   F = R_C - 1/b = 2 F' - 2 w / ((a + b) b' (2 b + b')),
// a sum of numbers of one sign.
template <class T> LCDM_HD T phi_core(T w, T so) {
    constexpr int NT = sizeof(typename Scalar<T>::rec) == 4 ? 9 : 17;
    T a = cst<T>(1.0), b = so, sum = cst<T>(0.0), t = cst<T>(1.0), ia = cst<T>(1.0), v = w;
#pragma unroll 1
    for (int m = 0; m < CoreTol<T>::maxit && any_gt(v, cst<T>(0.1)); m++) {
        const T n = a + b, q = cst<T>(2.0) * b * n, c = sqt(q);
        sum = sum - cst<T>(2.0) * t * rcp_(n * c * (cst<T>(2.0) * b + c));
        a = n;
        b = c;
        t = t + t;
        ia = rcp_(a);
        v = w * (ia * ia);
    }
    constexpr double cs[17] = LCDM_PHI_CS;
    T acc = cst<T>(cs[NT - 1]);
#pragma unroll
    for (int n = NT - 1; n >= 1; n--) acc = acc * v + cst<T>(cs[n - 1]);
    return sum + t * acc * (ia * ia * ia);
}

// 1 + z q: rounded once in double precision; in single precision in
// double-float arithmetic from q's two words (it cancels for the pair near
// z = Re r_P close to the no-Big-Bang boundary)
LCDM_HD double one_plus(double q, double, double z) { return fma(q, z, 1.0); }
LCDM_HD float one_plus(float q, float ql, float z) {
    const float p = q * z, e1 = fmaf(q, z, -p);
    const df64 s = two_sum(1.0f, p);
    return s.hi + (s.lo + fmaf(ql, z, e1));
}
LCDM_HD F2 one_plus(F2 q, F2 ql, F2 z) { return mkf2(one_plus(q.x, ql.x, z.x), one_plus(q.y, ql.y, z.y)); }
// w - n^2, rounded once
LCDM_HD float fms_(float n, float w) { return fmaf(-n, n, w); }
LCDM_HD double fms_(double n, double w) { return fma(-n, n, w); }
LCDM_HD F2 fms_(F2 n, F2 w) { return mkf2(fms_(n.x, w.x), fms_(n.y, w.y)); }
// power of two near 1/z for very large z (or s1, which is of z's size where E^2(0) is 1)
LCDM_HD float scale_of(float z) { return z < 1e38f ? pow2i<float>(-even_exponent(z)) : 0.0f; }
LCDM_HD double scale_of(double z) {
    int e;
    frexp(z, &e);
    return z < 1e300 ? pow2i<double>(-e) : 0.0;
}

// the scaling of a pair, 1 unless its s1 is very large
LCDM_HD float scaling(float z) { return z > CoreTol<float>::big ? scale_of(z) : 1.0f; }
LCDM_HD double scaling(double z) { return z > CoreTol<double>::big ? scale_of(z) : 1.0; }
LCDM_HD F2 scaling(F2 z) { return mkf2(scaling(z.x), scaling(z.y)); }
template <class T> LCDM_HD T unscale(T h) { return cst<T>(1.0) / h; }
LCDM_HD F2 unscale(F2 h) { return mkf2(1.0f / h.x, 1.0f / h.y); }

// Four consecutive record entries from a multiple of four (records are 16-byte
// aligned): one 128-bit load in single precision, two in double.
template <class T> struct Quad { T v[4]; };
LCDM_HD Quad<float> quad(const float* p) {
    Quad<float> q;
#ifdef __CUDA_ARCH__
    const float4 f = __ldg(reinterpret_cast<const float4*>(p));
    q.v[0] = f.x; q.v[1] = f.y; q.v[2] = f.z; q.v[3] = f.w;
#else
    for (int i = 0; i < 4; i++) q.v[i] = p[i];
#endif
    return q;
}
LCDM_HD Quad<double> quad(const double* p) {
    Quad<double> q;
#ifdef __CUDA_ARCH__
    const double2 a = __ldg(reinterpret_cast<const double2*>(p)), b = __ldg(reinterpret_cast<const double2*>(p) + 1);
    q.v[0] = a.x; q.v[1] = a.y; q.v[2] = b.x; q.v[3] = b.y;
#else
    for (int i = 0; i < 4; i++) q.v[i] = p[i];
#endif
    return q;
}

template <class T> LCDM_HD Quad<T> quad_as(const typename Scalar<T>::rec* p) {
    const Quad<typename Scalar<T>::rec> f = quad(p);
    Quad<T> q;
#pragma unroll
    for (int i = 0; i < 4; i++) q.v[i] = Scalar<T>::of(f.v[i]);
    return q;
}

// a w + c with c a record entry.  Two pairs: two plain multiply-adds, which take
// c as it is (a packed one wants it in both halves of a register pair; X's 24
// coefficients made so spilled: 2.74 against 2.72 ms for 1e8 pairs)
template <class T> LCDM_HD T horner(T a, T w, T c) { return a * w + c; }
LCDM_HD F2 horner(F2 a, F2 w, float c) { return mkf2(a.x * w.x + c, a.y * w.y + c); }

// ------------------------------------------------------------------- core ---
// A closing series 1 + w^2 (c_2 + c_3 w + ...) from ns coefficients at rec[i],
// i = 0 or 1 modulo 4, and with it (D) the derivative of the bracket.
template <class T> struct SerVal { T v, d; };
template <bool D, int N, class T> LCDM_HD SerVal<T> series(const typename Scalar<T>::rec* rec, int i, T w) {
    T c[12];
    const int skip = i & 3;
#pragma unroll
    for (int q = 0; q < (N + skip + 3) / 4; q++) {
        const Quad<T> k = quad_as<T>(rec + (i - skip) + 4 * q);
#pragma unroll
        for (int l = 0; l < 4; l++)
            if (4 * q + l >= skip && 4 * q + l - skip < 12) c[4 * q + l - skip] = k.v[l];
    }
    SerVal<T> r;
    r.v = c[N - 1];
    r.d = cst<T>(0.0);
#pragma unroll
    for (int j = N - 2; j >= 0; j--) {
        if (D) r.d = r.d * w + r.v;
        r.v = r.v * w + c[j];
    }
    return r;
}

// The steps taken, for the reverse pass: s1, S and P of the duplication (sqrt(p)
// of the t track), and R_C's a and b.  Apart from the pair's other state: it is
// indexed by the step and lives in local memory (of which only the steps taken
// are touched), where it would take everything in the same object with it (51
// local loads and stores per pair instead of 8).
template <class T, bool REV, bool WT> struct CoreTape {
    enum { N = REV ? (int)CoreTol<T>::maxit : 1, NR = REV && WT ? (int)CoreTol<T>::maxit : 1, NQ = NR };
    T s1[N], S[N], P[N], q[NQ], ra[NR], rb[NR];
};

// One pair.  WT: the time coordinate; WX: the absorption distance (values
// only); REV: keep what the reverse pass needs; INF: the upper limit at
// infinity.  There n_j / sqrt(z) -> sqrt(q_j), every u grows like z, and with
// the homogeneity of R_F, R_C and R_J the powers of z cancel: z stands for 1
// and 1 + z q_j for q_j, and eq. (3.8)'s R_C has the factor (1 + eps) n_A (in
// the radiationless case n_A = 0: that term falls off like z^-1/2).
template <class T, bool WT, bool WX, bool REV, bool INF = false> struct CorePair {
    typedef CoreTape<T, REV, WT> Tape;
    enum { NS = INF ? (int)CORE_NS_ONCE : (int)CoreTol<T>::ns };
    typedef typename Scalar<T>::rec R;
    const R* rc;
    T z, zh, z2, h, cz;
    bool cplx, big;
    // square roots of the linear factors and their reciprocals
    T rA, nA, rB, nB, Pn, iP, wr, wi, nr, ni;   // real pair: nr, ni = n_1, n_2; wr, wi = their reciprocals
    T s1, uR, uI;                               // real pair: u_1, u_2
    int m;                                      // duplication steps taken
    T tm;                                       // 2^m
    T T3, RF, RJ, rF, wF, sF, rJ, wJ, sJs;      // 3 A, results, 1/sqrt(A), w, series
    T p, izh, d5, a5, RCp, g, kB, ig;           // t
    int mr;
    T U, sc, rcr, tr;
    T X;
    T Ichi, It;
    // adjoints of the row's constants
    T qA_, qB_, qR_, qI_, bF_, eps_, k2_, k3_, bJ_;
    T e2_, e3_, m_;   // INF: in the place of the series' coefficients

    LCDM_HD void forward(T zin, const R* rec, Tape& tape, int* fail) {
        rc = rec;
        z = zin;
        const T one = cst<T>(1.0);
        const Quad<T> k0 = quad_as<T>(rc + C_QA), k1 = quad_as<T>(rc + C_QI);
        cplx = rc[C_KIND] != R(0);
        const T wA = INF ? k0.v[0] : one + k0.v[0] * z, wB = INF ? k0.v[1] : one + k0.v[1] * z;
        rA = rsq(wA);
        if (INF && !any_gt(wA, cst<T>(0.0))) rA = cst<T>(0.0);
        nA = wA * rA;
        rB = rsq(wB);
        nB = wB * rB;
        const T qR = k0.v[2], qI = k1.v[0], c2 = k1.v[2];
        Quad<T> kT;
        if (WT) kT = quad_as<T>(rc + C_DJ);
        T S, P, T30;
        if (cplx) {
            wr = INF ? qR : one_plus(qR, k0.v[3], z);
            wi = qI * z;
            const T r2 = wr * wr + wi * wi;
            iP = rsq(r2);
            Pn = r2 * iP;
            // n_P: the larger part by a square root, the other by division
            const T hh = (Pn + abs_(wr)) * cst<T>(0.5), rh = rsq(hh);
            const T t = hh * rh, o = wi * cst<T>(0.5) * rh;
            nr = sel_ge0(wr, t, o);
            ni = sel_ge0(wr, o, t);
            uR = nr * (nA + nB);
            uI = ni * (nA - nB);
        } else {
            const T w1 = INF ? qR : one_plus(qR, k0.v[3], z), w2 = INF ? qI : one_plus(qI, k1.v[1], z);
            wr = rsq(w1);
            wi = rsq(w2);
            nr = w1 * wr;
            ni = w2 * wi;
            Pn = nr * ni;
            iP = wr * wi;
            uR = nr * nA + ni * nB;
            uI = ni * nA + nr * nB;
        }
        if (WX && sizeof(R) == 4) {
            // the absorption distance is a difference of terms twice its size:
            // one Newton step takes the approximate square roots to half an ulp
            const T hf = cst<T>(0.5);
            nA = nA + hf * rA * fms_(nA, wA);
            nB = nB + hf * rB * fms_(nB, wB);
        }
        s1 = nA * nB + Pn;
        zh = z;
        z2 = z * z;
        const T z1 = INF ? one : one + z;
        if (WT) {
            izh = INF ? one : rsq(z1);
            a5 = (nB * Pn + z1 * nA) * izh;
        }
        T aX = cst<T>(0.0), lX = cst<T>(0.0);
        Quad<T> kX;
        if (WX) {
            kX = quad_as<T>(rc + X_HX);
            aX = nA * Pn + nB;
            lX = kX.v[1] * wB;
        }
        // powers of large arguments (very large z, or a small E^2(0)) would leave
        // the range: everything is homogeneous and is scaled by a power of two
        big = any_gt(s1, cst<T>(CoreTol<T>::big));
        h = one;
        if (big) {
            h = scaling(s1);
            s1 = s1 * h; uR = uR * h; uI = uI * h;
            if (WT) a5 = a5 * h;
            if (WX) aX = aX * h;
            zh = z * h;
            z2 = zh * zh;
            zh = z * h;
        }
        if (cplx) {
            S = uR + uR;
            P = uR * uR + uI * uI;
            T30 = cst<T>(2.0) * (uR * uR - uI * uI);
        } else {
            S = uR + uI;
            P = uR * uI;
            T30 = uR * uR + uI * uI;
        }
        T x = s1 * s1;
        T3 = x + T30;
        T sJ = cst<T>(0.0), kz = cst<T>(0.0), k9 = kz, opE = cst<T>(0.0);
        p = cst<T>(0.0);
        if (WT) {
            opE = one + kT.v[1];
            d5 = kT.v[3] * z2 * (opE * opE) * (wA * (izh * izh));
            p = a5 * a5 - d5;
            kz = kT.v[2] * (z2 * zh);
            k9 = cst<T>(-9.0) * kT.v[3];
        }
        T p0 = cst<T>(0.0), hX = cst<T>(0.0), piX = cst<T>(0.0), sD = cst<T>(0.0), sDD = cst<T>(0.0), x0 = x, rp0 = cst<T>(0.0);
        if (WX) {
            p0 = aX * aX - lX * z2;
            if (big) {
                // the z^3 of both terms cancel (lambda y_B^2 q_B = S0 q_A q_P q_P*): the
                // polynomial w_A |w_P|^2 - lx w_B z^2 without it
                const Quad<T> kB = quad_as<T>(rc + X_AB);
                const T qA = k0.v[0], p1 = qA + kB.v[2], p2 = qA * kB.v[2] + kB.v[3] - kX.v[1];
                const T pb = p2 * z2 + (p1 * zh + h) * h + cst<T>(2.0) * (nA * (nB * h)) * (Pn * h) + wB * h * h;
                p0 = sel_ge0(z - cst<T>(CoreTol<T>::big), pb, p0);
            }
            piX = kX.v[2] * (z2 * z2);
            hX = -(kX.v[0] * z2);
        }
        T pX = p0;
        const float it = (float)(1.0 / (INF ? CoreTol<T>::once : CoreTol<T>::dup));
        const auto z2c = cmp_(z2);
        const auto dF = times_((float)rc[C_DF] * it * 3.0f, z2c);
        const auto dJ = times_(WT ? (float)rc[C_DJ] * it * 5.0f : 0.0f, z2c);
        const auto dD = times_(WX ? (float)rc[X_DX] * it * 5.0f : 0.0f, z2c);
        T S1 = s1;
        tm = one;
        T q0 = cst<T>(0.0);
        m = 0;
#pragma unroll 1
        for (; m < CoreTol<T>::maxit; m++) {
            // (compared in single precision: in double each comparison would hold
            // the FP64 pipe)
            bool conv = all_le(dF, cmp_(T3));
            if (WT) conv = conv && all_le(dJ, cmp_(T3 + p + p));
            if (WX) conv = conv && all_le(dD, cmp_(T3 + pX + pX)) && all_le(dD, cmp_(T3 + x + x));
            if (conv) break;
            const T lam = S1 * S + P;
            const T xl = x + lam;
            if (WT) {
                const T sq = sqt(p);
                if (m == 0) q0 = sq;
                const T gg = p + (sq * S + P);
                const T id = rcp_((sq + S1) * gg);
                const T v = kz * id, e = k9 * (v * v);
                sJ = sJ + tm * rc1_core(e, false).v * id;
                if (REV) tape.q[m] = sq;
                p = p + lam;
            }
            if constexpr (WX) {
                // R_D: 1 / (s1 (x + lambda)); divided difference of the p0 track against it
                const T ix = rcp_(S1 * xl);
                sD = sD + tm * ix;
                const T sq = sqt(pX);
                if (m == 0) rp0 = sq;
                const T gg = pX + (sq * S + P), qs = sq + S1;
                const T id = rcp_(qs * gg);
                const T eh = (piX * id) * id, e = hX * eh;
                sDD = sDD + tm * (eh * rc1m1_core(e) * id
                                  - ((gg + cst<T>(2.0) * S1 * (qs + S)) * id) * (id * gg) * ix * cst<T>(0.5));   // (id^2 may flush to zero)
                pX = pX + lam;
            }
            if (REV) {
                tape.s1[m] = S1;
                tape.S[m] = S;
                if (WT) tape.P[m] = P;
            }
            x = xl;
            T3 = T3 + cst<T>(3.0) * lam;
            const T n1 = sqt(x);
            const T Q = S * (S + cst<T>(2.0) * (S1 + n1));
            P = n1 * S;
            S = sqt(Q);
            S1 = n1;
            tm = tm + tm;
        }
        if (m == CoreTol<T>::maxit) {
            // not converged (of two pairs: those that are not)
            *fail |= not_le(dF, cmp_(T3));
            if (WT) *fail |= not_le(dJ, cmp_(T3 + p + p));
            if (WX) *fail |= not_le(dD, cmp_(T3 + pX + pX)) | not_le(dD, cmp_(T3 + x + x));
        }
        // closing series in w = z^2 / A
        {
            const T A = T3 * cst<T>(1.0 / 3);
            rF = rsq(A);
            wF = (INF ? z2 : z2 * Scalar<T>::of(rc[C_DF])) * (rF * rF);
            const T s = series<false, NS>(rc, C_B, wF).v;
            sF = one + s * (wF * wF);
            RF = tm * sF * rF;
        }
        cz = c2 * zh;
        Ichi = cz * RF;
        if (WT) {
            const T A = (T3 + p + p) * cst<T>(0.2);
            rJ = rsq(A);
            wJ = (INF ? z2 : z2 * kT.v[0]) * (rJ * rJ);
            const T s = series<false, NS>(rc, C_A, wJ).v;
            sJs = one + s * (wJ * wJ);
            RJ = tm * sJs * (rJ * rJ * rJ) + cst<T>(6.0) * sJ;
            // R_C(s5, p), Carlson's duplication on the square roots a = sqrt(s5), b = sqrt(p)
            T a = a5, b = m > 0 ? q0 : sqt(p);
            U = a * a + cst<T>(2.0) * (b * b);
            tr = one;
            mr = 0;
            const T ad = abs_(d5);
#pragma unroll 1
            for (; mr < CoreTol<T>::maxit; mr++) {
                if (REV) { tape.ra[mr] = a; tape.rb[mr] = b; }
                if (all_le(ad, cst<T>(CoreTol<T>::rc) * U)) break;
                const T n = a + b, q = cst<T>(2.0) * b * n;
                a = n;
                b = sqt(q);
                U = a * a + cst<T>(2.0) * (b * b);
                tr = tr + tr;
            }
            if (mr == CoreTol<T>::maxit) *fail |= not_le(ad, cst<T>(CoreTol<T>::rc) * U);
            const T iA = cst<T>(3.0) * rcp_(U);
            sc = -d5 * iA * cst<T>(1.0 / 3);
            T ser = cst<T>(159.0 / 208) + sc * cst<T>(1.125);
            ser = cst<T>(9.0 / 22) + sc * ser;
            ser = cst<T>(0.375) + sc * ser;
            ser = cst<T>(1.0 / 7) + sc * ser;
            ser = cst<T>(0.3) + sc * ser;
            ser = one + sc * sc * ser;
            rcr = rsq(U * cst<T>(1.0 / 3));
            RCp = tr * ser * rcr * izh;
            const T eps = kT.v[1];
            g = abs_(opE) * nA;
            if (INF) {
                It = cz * (RCp * g - eps * RF - kT.v[2] * z2 * RJ);
            } else {
                ig = rcp_(g + one);
                kB = (one + (one + eps) * z1) * ig;
                It = cz * (RCp + eps * (RCp * kB - RF) - kT.v[2] * z2 * RJ);
            }
        }
        if constexpr (WX) {
            const T iA2 = cst<T>(5.0) * rcp_(T3 + x + x);
            const T A2 = (T3 + x + x) * cst<T>(0.2), A1 = (T3 + pX + pX) * cst<T>(0.2);
            const T r1 = rsq(A1), r2 = rsq(A2);
            const T sx = Scalar<T>::of(rc[X_DX]);
            const T i1 = r1 * r1, w1 = (z2 * sx) * i1, u2 = z2 * iA2, w2 = u2 * sx, ww = cst<T>(-0.4) * w1 * u2;
            // series at p0 and at x1, and the divided difference of the brackets
            // (coefficients by degree: at p0, at x1, their divided difference)
            constexpr int N = CoreTol<T>::ns;
            T v1 = cst<T>(0.0), v2 = cst<T>(0.0), e = cst<T>(0.0);
            R q[3 * CORE_NS + 2];
#pragma unroll
            for (int j = 0; j < (3 * N + 3) / 4; j++) {
                const Quad<R> f = quad(rc + X_S + 4 * j);
#pragma unroll
                for (int i = 0; i < 4; i++) q[4 * j + i] = f.v[i];
            }
#pragma unroll
            for (int j = N - 1; j >= 0; j--) {
                e = e * w1 + horner(v2, ww, -q[3 * j + 2]);
                v1 = horner(v1, w1, q[3 * j]);
                v2 = horner(v2, w2, q[3 * j + 1]);
            }
            const T ser1 = one + v1 * (w1 * w1);
            const T dser = iA2 * (cst<T>(-0.4) * (w1 + w2) * w1 * v1 + w2 * (sx * e));
            const T q1 = A1 * r1, q2 = A2 * r2;
            const T r13 = r1 * i1, r23 = r2 * iA2;
            const T dA = cst<T>(-0.4) * (A1 + q1 * q2 + A2) * rcp_(q1 + q2) * r13 * r23;
            const T DJ = tm * (dA * ser1 + r23 * dser) + cst<T>(6.0) * sDD;
            const T RD = tm * (one + v2 * (w2 * w2)) * r23 + cst<T>(3.0) * sD;
            if (m == 0) rp0 = sqt(p0);
            // the arguments, and with them s1, x0, p0 and the integrals, are scaled by
            // powers of h (1 but for very large z): what falls off like 1/z is formed
            // from them as they are, with one h in front (unscaled, z^4 and x1 leave
            // single precision from z = 1e10 on)
            const T ih = big ? unscale(h) : one;
            const Quad<T> c0 = quad_as<T>(rc + X_C0), c3 = quad_as<T>(rc + X_G3), cN = quad_as<T>(rc + X_N0), cB = quad_as<T>(rc + X_AB);
            const T irA = rA, syd = c3.v[3] * (nA * Pn * rB + one), isy = rcp_(syd);
            const T T0 = c0.v[0] * irA * (k0.v[1] * Pn * rcp_(nB + one) + (cB.v[2] + z * cB.v[3]) * rcp_(Pn + one)
                                           - k0.v[0] * rcp_(nA + one));
            const T t1 = c0.v[1] * RF + z2 * (c0.v[2] * RD + c0.v[3] * z2 * DJ);
            const T wy = z * isy, wy2 = wy * wy;
            // y / yd = S0 p0 / (yB^2 n_B^2 yd), the part of yd beside lam z^2
            const T t2 = c3.v[0] * wy2 * phi_core(cB.v[1] * wy2, (rp0 * rB) * (c3.v[3] * (isy * ih))) * isy;
            const T as = nA * s1;
            const T num = x0 * (cN.v[1] * z + cN.v[0]) + cN.v[2] * z2;
            const T t3 = c3.v[1] * num * (nB * rcp_(rp0 * as * (as + cB.v[0] * rp0)));
            const T t4 = c3.v[2] * nB * irA * rcp_(s1);
            X = z * (T0 + t2 + h * (t1 + t3 + t4));
        }
    }

    // 1 / E(z) = E(0)^-1 / (n_A n_B |n_P|^2)
    LCDM_HD T inv_E() const { return Scalar<T>::of(rc[C_C2] * R(0.5)) * (rA * rB * iP); }

    // Adjoints of the row's constants for the cotangents ci, ti of Ichi, It.
    LCDM_HD void reverse(T ci, T ti, const Tape& tape) {
        const T one = cst<T>(1.0), two = cst<T>(2.0), half = cst<T>(0.5);
        T RF_ = ci * cz, T_ = cst<T>(0.0), p_ = cst<T>(0.0), cJ = cst<T>(0.0), del_ = cst<T>(0.0), a_ = cst<T>(0.0),
          b_ = cst<T>(0.0), d_ = cst<T>(0.0), nA_ = cst<T>(0.0), wA_ = cst<T>(0.0);
        Quad<T> kT;
        if (WT) kT = quad_as<T>(rc + C_DJ);
        const T eps = WT ? kT.v[1] : cst<T>(0.0), z1 = INF ? one : one + z;
        eps_ = k2_ = k3_ = bJ_ = cst<T>(0.0);
        if (WT) {
            const T b = ti * cz;
            const T RCp_ = INF ? b * g : b * (one + eps * kB);
            RF_ = RF_ - b * eps;
            const T bk = b * z2;
            const T RJ_ = -bk * kT.v[2];
            k2_ = -bk * RJ;
            const T opE = one + eps, ao = abs_(opE), sA = sel_ge0(opE, nA, -nA);
            if (INF) {
                eps_ = b * (RCp * sA - RF);
                nA_ = b * RCp * ao;
            } else {
                // kB = (2 + z + eps (1+z)) / (|1+eps| n_A + 1)
                const T er = b * eps * RCp * ig;
                eps_ = b * (RCp * kB - RF) + er * (z1 - kB * sA);
                nA_ = -er * kB * ao;
            }
            // R_C: series, then the steps in reverse
            const T rcb = RCp_ * izh * tr * rcr;          // cotangent of the series
            const T iU = cst<T>(1.0 / 3) * (rcr * rcr);   // 1 / U
            T ser = cst<T>(1.125), ds = cst<T>(0.0);
            ds = ser; ser = cst<T>(159.0 / 208) + sc * ser;
            ds = ds * sc + ser; ser = cst<T>(9.0 / 22) + sc * ser;
            ds = ds * sc + ser; ser = cst<T>(0.375) + sc * ser;
            ds = ds * sc + ser; ser = cst<T>(1.0 / 7) + sc * ser;
            ds = ds * sc + ser; ser = cst<T>(0.3) + sc * ser;
            // f = 1 + s^2 q(s): f' = s (2 q + s q')
            const T sd = sc * (two * ser + sc * ds), sv = one + sc * sc * ser;
            d_ = -rcb * sd * iU;
            const T U_ = -rcb * iU * (sc * sd + half * sv);
            T ax = tape.ra[mr < Tape::NR ? mr : 0], bx = tape.rb[mr < Tape::NR ? mr : 0];
            a_ = two * ax * U_;
            b_ = cst<T>(4.0) * bx * U_;
#pragma unroll 1
            for (int i = mr - 1; i >= 0; i--) {
                const T a0 = tape.ra[i], b0 = tape.rb[i];
                const T Q_ = b_ * half * rcp_(bx);
                const T n_ = a_ + two * b0 * Q_;
                b_ = two * (a0 + b0) * Q_ + n_;
                a_ = n_;
                bx = b0;
            }
            p_ = b_ * half * rcp_(bx);                    // b = sqrt(p)
            // R_J: closing series
            const SerVal<T> sv2 = series<true, NS>(rc, C_A, wJ);
            const T s = sv2.v, s2 = sv2.d;
            const T r2 = rJ * rJ, c = RJ_ * tm * r2 * rJ;
            bJ_ = c;
            const T A_ = -c * r2 * (wJ * wJ * (two * s + wJ * s2) + cst<T>(1.5) * sJs);
            T_ = A_ * cst<T>(0.2);
            // the sequence's final p: its cotangent joins the chain (p differs
            // from the initial p by the sum of the lambdas)
            cJ = cst<T>(6.0) * RJ_;
            pf_ = A_ * cst<T>(0.4);
        }
        {
            const SerVal<T> sv2 = series<true, NS>(rc, C_B, wF);
            const T s = sv2.v, s2 = sv2.d;
            const T c = RF_ * tm * rF;
            bF_ = c;
            T_ = T_ - c * (rF * rF) * cst<T>(1.0 / 3) * (wF * wF * (two * s + wF * s2) + half * sF);
        }
        // the duplication in reverse: cotangents of (s1, S, P), x and p
        T s_ = cst<T>(0.0), S_ = cst<T>(0.0), P_ = cst<T>(0.0), x_ = cst<T>(0.0);
        T ps_ = WT ? pf_ : cst<T>(0.0);
        T kz = cst<T>(0.0), k9 = kz, tk = tm;
        if (WT) {
            kz = kT.v[2] * (z2 * zh);
            k9 = cst<T>(-9.0) * kT.v[3];
        }
        T n1 = one, n1s = one;   // the next step's sqrt(x) and S
#pragma unroll 1
        for (int i = m - 1; i >= 0; i--) {
            const T a = tape.s1[i], Sm = tape.S[i], Pm = WT ? tape.P[i] : cst<T>(0.0);
            tk = tk * half;
            T Sn_ = cst<T>(0.0), an_ = cst<T>(0.0);
            if (i < m - 1) {
                // next: n1 = sqrt(x'), P' = n1 S, S' = sqrt(S (S + 2 (a + n1)))
                const T Q_ = S_ * half * rcp_(n1s);
                const T t = two * Sm * Q_;
                const T n_ = s_ + P_ * Sm + t;
                Sn_ = P_ * n1 + Q_ * two * (Sm + a + n1);
                an_ = t;
                x_ = x_ + n_ * half * rcp_(n1);
            }
            n1 = a;
            n1s = Sm;
            const T lam_ = x_ + ps_ + cst<T>(3.0) * T_;
            s_ = an_ + lam_ * Sm;
            S_ = Sn_ + lam_ * a;
            P_ = lam_;
            if (WT) {
                const T sq = tape.q[i], gg = sq * (sq + Sm) + Pm, qs = sq + a;
                const T id = rcp_(qs * gg), v = kz * id, vv = v * v, e = k9 * vv;
                const RcE<T> r = rc1_core(e, true);
                const T c = cJ * tk * id;                 // cotangent of rc
                del_ = del_ + c * r.d * vv;
                // 1/d: rc d(1/d) + rc' 2 delta id d(1/d), d(1/d) = -id^2 dd
                const T dd = -c * id * (r.v + two * e * r.d);
                const T g_ = dd * qs, q_ = dd * gg + g_ * Sm;
                s_ = s_ + dd * gg;
                S_ = S_ + g_ * sq;
                P_ = P_ + g_;
                ps_ = ps_ + g_ + q_ * half * rcp_(sq);
            }
        }
        // initial values: x = s1^2, 3 A = x + y + y*, p = a5^2 - d5; e = -9 k3 v^2, v = k2 z^3 / d
        s_ = s_ + two * s1 * (x_ + T_);
        T nB_, Pn_ = cst<T>(0.0), h5_ = cst<T>(0.0);
        if (WT) {
            p_ = p_ + ps_;
            a_ = a_ + two * a5 * p_;
            d_ = d_ - p_;
            const R k2 = rc[C_K2];
            const T ik2 = Scalar<T>::of(fabs(k2) > R(1e-30) ? rcp_(k2) : R(0)), k3 = kT.v[3];
            k2_ = k2_ - cst<T>(18.0) * k3 * del_ * ik2;
            const T opE = one + eps, wA = nA * nA;
            const T f = z2 * (izh * izh) * opE;
            k3_ = d_ * f * opE * wA - cst<T>(9.0) * del_;
            eps_ = eps_ + d_ * k3 * two * f * wA;
            wA_ = d_ * k3 * f * opE;
            h5_ = a_ * izh;
            if (big) h5_ = h5_ * h;
        }
        T uR_, uI_;
        if (cplx) {
            uR_ = two * S_ + two * uR * P_ + cst<T>(4.0) * uR * T_;
            uI_ = two * uI * P_ - cst<T>(4.0) * uI * T_;
        } else {
            uR_ = S_ + uI * P_ + two * uR * T_;
            uI_ = S_ + uR * P_ + two * uI * T_;
        }
        if (big) { s_ = s_ * h; uR_ = uR_ * h; uI_ = uI_ * h; }
        Pn_ = s_;
        nA_ = nA_ + s_ * nB;
        nB_ = s_ * nA;
        if (WT) {
            Pn_ = Pn_ + h5_ * nB;
            nB_ = nB_ + h5_ * Pn;
            nA_ = nA_ + h5_ * z1;
        }
        if (cplx) {
            const T tr_ = uR_ * nr, ti_ = uI_ * ni;
            nA_ = nA_ + tr_ + ti_;
            nB_ = nB_ + tr_ - ti_;
            const T r_ = uR_ * (nA + nB), i_ = uI_ * (nA - nB);
            // n_P = sqrt(w_P), Pn = |w_P|
            const T hp = half * iP;
            qR_ = (Pn_ * wr * iP + hp * (nr * r_ - ni * i_)) * z;
            qI_ = (Pn_ * wi * iP + hp * (ni * r_ + nr * i_)) * z;
        } else {
            nA_ = nA_ + uR_ * nr + uI_ * ni;
            nB_ = nB_ + uR_ * ni + uI_ * nr;
            qR_ = (uR_ * nA + uI_ * nB + Pn_ * ni) * half * wr * z;
            qI_ = (uR_ * nB + uI_ * nA + Pn_ * nr) * half * wi * z;
        }
        qA_ = (nA_ * half * rA + wA_) * z;
        qB_ = nB_ * half * rB * z;
        if (INF) series_adjoint();
    }
    T pf_;

    // INF: the closing series' adjoints taken through to (e2, e3, m), where a
    // record of coefficient tangents would be used once.  R_F to degree 7:
    //   1 - E2/10 + E3/14 + E2^2/24 - 3 E2 E3/44 - 5 E2^3/208 + 3 E3^2/104 + E2^2 E3/16, E_i = e_i w^i;
    // R_J alike in E2 .. E5 (DLMF 19.36.2), which are polynomials of (m, e2, e3) (rj_coefs).
    LCDM_HD void series_adjoint() {
        {
            const T w = wF, ww = w * w, E2 = Scalar<T>::of(rc[C_E2]) * ww, E3 = Scalar<T>::of(rc[C_E3]) * (ww * w);
            e2_ = bF_ * ww * (cst<T>(-0.1) + E2 * cst<T>(1.0 / 12) - E3 * cst<T>(3.0 / 44) - E2 * E2 * cst<T>(15.0 / 208)
                              + E2 * E3 * cst<T>(0.125));
            e3_ = bF_ * ww * w * (cst<T>(1.0 / 14) - E2 * cst<T>(3.0 / 44) + E3 * cst<T>(3.0 / 52) + E2 * E2 * cst<T>(1.0 / 16));
        }
        if (WT) {
            const T w = wJ, ww = w * w, m = Scalar<T>::of(rc[C_M]) * w, e2 = Scalar<T>::of(rc[C_E2]) * ww, e3 = Scalar<T>::of(rc[C_E3]) * (ww * w);
            const T mm = m * m, P = m * cst<T>(0.6), P2 = P * P, P3 = P2 * P;
            const T E2 = e2 - mm * cst<T>(0.6);
            const T Q = e3 - m * e2 * cst<T>(0.4) - mm * m * cst<T>(0.064);
            const T E3 = Q + cst<T>(2.0) * E2 * P + cst<T>(4.0) * P3;
            const T W = cst<T>(2.0) * Q + E2 * P + cst<T>(3.0) * P3, E4 = W * P, E5 = Q * P2;
            const T g5 = cst<T>(3.0 / 26) - E2 * cst<T>(9.0 / 68);
            const T g4 = cst<T>(-3.0 / 22) + E2 * cst<T>(3.0 / 20) - E3 * cst<T>(9.0 / 68);
            const T g3 = cst<T>(1.0 / 6) - E2 * cst<T>(9.0 / 52) + E3 * cst<T>(3.0 / 20) + E2 * E2 * cst<T>(45.0 / 272)
                         - E4 * cst<T>(9.0 / 68);
            const T gW = g4 * P;
            const T g2 = cst<T>(-3.0 / 14) + E2 * cst<T>(9.0 / 44) - E3 * cst<T>(9.0 / 52) - E2 * E2 * cst<T>(3.0 / 16)
                         + E4 * cst<T>(3.0 / 20) + E2 * E3 * cst<T>(45.0 / 136) - E5 * cst<T>(9.0 / 68)
                         + cst<T>(2.0) * g3 * P + gW * P;
            const T gQ = g5 * P2 + cst<T>(2.0) * gW + g3;
            const T gP = cst<T>(2.0) * g5 * Q * P + g4 * W + gW * (E2 + cst<T>(9.0) * P2) + g3 * (cst<T>(2.0) * E2 + cst<T>(12.0) * P2);
            const T c = bJ_;
            m_ = c * w * (cst<T>(0.6) * gP - cst<T>(1.2) * m * g2 - gQ * (cst<T>(0.4) * e2 + cst<T>(0.192) * mm));
            e2_ = e2_ + c * ww * (g2 - cst<T>(0.4) * m * gQ);
            e3_ = e3_ + c * ww * w * gQ;
        }
    }

    LCDM_HD T thirds(const R* t) const {
        return eps_ * Scalar<T>::of(t[CT_EPS]) + k2_ * Scalar<T>::of(t[CT_K2]) + k3_ * Scalar<T>::of(t[CT_K3]);
    }
    // sum over the row's constants of adjoint times tangent, direction k
    LCDM_HD T along(int k) const {
        const R* t = rc + C_TAN + C_TSTRIDE * k;
        if (INF) {
            const Quad<T> f = quad_as<T>(t);
            T r = qA_ * f.v[0] + qB_ * f.v[1] + (qR_ * f.v[2] + qI_ * f.v[3]) + e2_ * Scalar<T>::of(t[CT_E2]) + e3_ * Scalar<T>::of(t[CT_E3]);
            if (WT) r = r + thirds(t) + m_ * Scalar<T>::of(t[CT_M]);
            return r;
        }
        const Quad<T> t0 = quad_as<T>(t);
        const T b = series<false, NS>(t, CT_B, wF).v;
        T r = qA_ * t0.v[0] + qB_ * t0.v[1] + (qR_ * t0.v[2] + qI_ * t0.v[3]) + bF_ * (wF * wF) * b;
        if (WT) {
            const T a = series<false, NS>(t, CT_A, wJ).v;
            r = r + thirds(t) + bJ_ * (wJ * wJ) * a;
        }
        return r;
    }
};

}  // namespace lcdm
