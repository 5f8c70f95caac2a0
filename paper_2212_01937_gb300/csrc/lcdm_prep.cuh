// Root preparation, one or four lanes per cosmology, FP64: factorise E^2 (eq. 3.2),
// classify the roots, choose the root labels, precompute the per-cosmology
// constants and the root tangents (App. A, eqs. A.1-A.4).
#pragma once
#include "lcdm_between.cuh"
#include "lcdm_corerec.cuh"
#include "lcdm_kernels.cuh"

namespace lcdm {

// ---------------------------------------------------------------- roots -----
struct cd { double re, im; };
LCDM_HD cd cmk(double r, double i) { cd c; c.re = r; c.im = i; return c; }
LCDM_HD cd cadd(cd a, cd b) { return cmk(a.re + b.re, a.im + b.im); }
LCDM_HD cd csub(cd a, cd b) { return cmk(a.re - b.re, a.im - b.im); }
LCDM_HD cd cmul(cd a, cd b) { return cmk(a.re * b.re - a.im * b.im, a.re * b.im + a.im * b.re); }
// One copy of the double-precision division for all of the preparation: each
// '/' would otherwise carry its own copy of the division's slow path.
LCDM_NI double ddiv(double a, double b) { return a / b; }

LCDM_HD cd cdiv(cd a, cd b) {
    double s = fabs(b.re) > fabs(b.im) ? fabs(b.re) : fabs(b.im);
    double is = ddiv(1.0, s);
    double br = b.re * is, bi = b.im * is, inv = ddiv(is, br * br + bi * bi);
    return cmk((a.re * br + a.im * bi) * inv, (a.im * br - a.re * bi) * inv);
}
LCDM_HD double cabs_(cd a) { return hypot(a.re, a.im); }
LCDM_HD cd csqrt_(cd a) {
    double r = cabs_(a);
    if (a.re >= 0) { double t = sqrt(0.5 * (r + a.re)); return cmk(t, t > 0 ? a.im * ddiv(0.5, t) : 0.0); }
    double t = sqrt(0.5 * (r - a.re));
    return cmk(fabs(a.im) * ddiv(0.5, t), a.im < 0 ? -t : t);
}

LCDM_HD double cnorm(cd a) { return a.re * a.re + a.im * a.im; }
// 1/b with one real division (the polynomial's values stay far inside the
// double range for the normalised coefficients used here)
LCDM_HD cd crcp(cd b) {
    double s = ddiv(1.0, cnorm(b));
    return cmk(b.re * s, -b.im * s);
}

// p(x) = sum_k c[k] x^k (degree n, c[n] = 1) and p'(x) by Horner's rule
LCDM_HD void horner(const double* c, int n, cd x, cd& p, cd& dp) {
    p = cmk(c[n], 0); dp = cmk(0, 0);
#pragma unroll 1
    for (int k = n - 1; k >= 0; k--) { dp = cadd(cmul(dp, x), p); p = cadd(cmul(p, x), cmk(c[k], 0)); }
}

// Error-free transformations: Knuth's sum, and the product by the fused
// multiply-add (a b = p + e exactly).
LCDM_HD void two_sum_d(double a, double b, double& s, double& e) {
    s = a + b;
    const double bb = s - a;
    e = (a - (s - bb)) + (b - bb);
}
LCDM_HD void two_prod_d(double a, double b, double& p, double& e) {
    p = a * b;
    e = fma(a, b, -p);
}

// p(x) = sum_k a[k] x^k (degree n) and p'(x) at complex x by the compensated
// Horner scheme (Graillat, Langlois and Louvet): the rounding error of every
// Horner step is carried, exactly, into a second Horner recurrence, so the
// value is as accurate as if it had been evaluated in twice the working
// precision.  Newton's method on it then finds a root to the last bit even
// where p' is small, as at the near-double roots of the no-Big-Bang boundary.
LCDM_HD void horner_comp(const double* a, int n, cd x, cd& p, cd& dp) {
    cd h = cmk(a[n], 0), q = cmk(0, 0);
    dp = cmk(0, 0);
#pragma unroll 1
    for (int k = n - 1; k >= 0; k--) {
        dp = cadd(cmul(dp, x), h);
        double p1, e1, p2, e2, p3, e3, p4, e4, s1, e5, s2, e6, t1, e7;
        two_prod_d(h.re, x.re, p1, e1);
        two_prod_d(h.im, x.im, p2, e2);
        two_prod_d(h.re, x.im, p3, e3);
        two_prod_d(h.im, x.re, p4, e4);
        two_sum_d(p1, -p2, s1, e5);
        two_sum_d(p3, p4, s2, e6);
        two_sum_d(s1, a[k], t1, e7);
        q = cadd(cmul(q, x), cmk(((e1 - e2) + e5) + e7, (e3 + e4) + e6));
        h = cmk(t1, s2);
    }
    p = cadd(h, q);
}

// Newton steps on the polynomial with the given (not normalised) coefficients,
// evaluated by horner_comp; a step is kept only while |p| decreases.
LCDM_HD void polish_root(const double* a, int n, cd& x) {
    cd p, dp;
    horner_comp(a, n, x, p, dp);
#pragma unroll 1
    for (int it = 0; it < 2; it++) {
        if ((dp.re == 0 && dp.im == 0) || (p.re == 0 && p.im == 0)) return;
        const cd xn = csub(x, cdiv(p, dp));
        cd pn, dpn;
        horner_comp(a, n, xn, pn, dpn);
        if (!(cnorm(pn) < cnorm(p))) return;
        x = xn; p = pn; dp = dpn;
    }
}

// (pr + i pi) / (er + i ei).  Divided by the larger part first: with a root of
// 1e6 (Om / Or) the polynomial's value is 1e24, and its products with the
// derivative leave single precision from a root of 3e5 on.  Approximate
// reciprocals: the quotient is needed to 1e-7 (one row's preparation and 1e4 FP64
// pairs 33.2 -> 31.6 us).
LCDM_HD void fquot(float pr, float pi, float er, float ei, float& wr, float& wi) {
    const float i = rcp_(fmaxf(fabsf(er), fabsf(ei)));
    er *= i;
    ei *= i;
    pr *= i;
    pi *= i;
    const float ie = rcp_(er * er + ei * ei);
    wr = (pr * er + pi * ei) * ie;
    wi = (pi * er - pr * ei) * ie;
}

// One Newton step from one compensated evaluation, the quotient in single
// precision: enough for a root known to about 1e-15 / separation (the step
// leaves 1e-7 of that error), without polish_root's confirming evaluations.
LCDM_HD void polish_once(const double* a, int n, cd& x) {
    cd p, dp;
    horner_comp(a, n, x, p, dp);
    const float pr = (float)p.re, pi = (float)p.im, dr = (float)dp.re, di = (float)dp.im;
    float wr, wi;
    fquot(pr, pi, dr, di, wr, wi);
    if (!(fabsf(wr) + fabsf(wi) < 1e30f)) return;
    x = cmk(x.re - (double)wr, x.im - (double)wi);
}

// A double as a float after division by 2^e (by its bits: no FP64 instruction),
// 0 or a huge number beyond the float's range; and a double's binary exponent.
// With e = the larger exponent of a number's parts, ratios of its size can be
// compared in single precision wherever it lies.
LCDM_HD int exponent_of(double v) { return (int)((__double_as_longlong(v) >> 52) & 0x7ff) - 1023; }
LCDM_HD float scaled(double v, int e) {
    const long long b = __double_as_longlong(v);
    const int x = (int)((b >> 52) & 0x7ff), k = x - e;   // biased exponents of v and of the quotient
    if (x == 0 || k < 1023 - 100) return 0.0f;   // (zero has no leading one: a root at exactly zero is real)
    if (k > 1023 + 100) return 1e30f;
    return (float)__longlong_as_double((b & ~(0x7ffLL << 52)) | ((long long)k << 52));
}
LCDM_HD int exponent_of(cd z) {
    const int a = exponent_of(z.re), b = exponent_of(z.im);
    return a > b ? a : b;
}
// |Im z| <= 1e-12 |z|
LCDM_HD bool negligible_im(cd z) {
    const int e = exponent_of(z);
    const float x = scaled(z.re, e), y = scaled(z.im, e);
    return fabsf(y) <= 1e-12f * sqrtf(x * x + y * y);
}

// Single-precision elementary functions for the starting circles only (no
// accuracy needed there): the fast hardware approximations on the device.
LCDM_HD float flog(float x) {
#ifdef __CUDA_ARCH__
    return __logf(x);
#else
    return logf(x);
#endif
}
LCDM_HD float fexp(float x) {
#ifdef __CUDA_ARCH__
    return __expf(x);
#else
    return expf(x);
#endif
}
LCDM_HD float fcos(float x) {
#ifdef __CUDA_ARCH__
    return __cosf(x);
#else
    return cosf(x);
#endif
}
LCDM_HD float fsin(float x) {
#ifdef __CUDA_ARCH__
    return __sinf(x);
#else
    return sinf(x);
#endif
}

// Starting points of the root iteration for the monic polynomial c (degree
// n <= 4): circles whose radii come from the Newton polygon of log|c_k|, so
// that a root near -Om/Or and the O(1) roots both start close.
LCDM_HD void start_points(const float* c, int n, float* zr, float* zi) {
    // upper convex hull of (k, log|c_k|); single precision is enough for the start
    float lg[5];
    int idx[5], m = 0;
    for (int k = 0; k <= n; k++) lg[k] = c[k] != 0.f ? flog(fabsf(c[k])) : -1e30f;
    for (int k = 0; k <= n; k++) {
        if (c[k] == 0.f) continue;
        while (m >= 2) {
            int a = idx[m - 2], b = idx[m - 1];
            // remove b if it lies below the segment a-k
            if ((lg[b] - lg[a]) * (k - a) <= (lg[k] - lg[a]) * (b - a)) m--; else break;
        }
        idx[m++] = k;
    }
    int r = 0;
    for (int e = 0; e + 1 < m; e++) {
        int a = idx[e], b = idx[e + 1], w = b - a;
        float rad = fexp((lg[a] - lg[b]) / w);
        for (int j = 0; j < w && r < 4; j++) {
            float ang = 6.2831853f * j / w + 6.2831853f * a / n + 0.4f;
            zr[r] = rad * fcos(ang);
            zi[r++] = rad * fsin(ang);
        }
    }
    for (; r < 4; r++) { zr[r] = 0.5f * r + 0.1f; zi[r] = 0.3f; }  // (zero constant term etc.)
}

// Starting points in closed form, to about 1e-6: the big root of the quartic by
// the fixed point A = -(a_3 + a_2/A + a_1/A^2 + a_0/A^3) / a_4 (it contracts by
// a_4 a_2 / a_3^2, ~1e-4 for any realistic radiation density), the others (all
// of a cubic's) by Cardano's formulas on the deflated cubic.  Returns false
// where that is not good: the fixed point has not settled, the other roots are
// not small beside A, or one of them is so small that the shift a/3 costs its
// digits, or the discriminant, of the roots' sixth power, may leave the range.
LCDM_HD bool closed_start(const float* al, int n, float* zr, float* zi) {
    float g3 = al[3], g2 = al[2], g1 = al[1], g0 = al[0];
    int k = 0;
    bool good = true;
    float A = 0.f;
    if (n == 4) {
        const float i4 = -1.0f / al[4];
        A = al[3] * i4;
        float prev = A;
#pragma unroll
        for (int it = 0; it < 3; it++) {
            const float iA = 1.0f / A;
            prev = A;
            A = (al[3] + iA * (al[2] + iA * (al[1] + iA * al[0]))) * i4;
        }
        good = fabsf(A - prev) < 1e-4f * fabsf(A);
        zr[0] = A;
        zi[0] = 0.f;
        k = 1;
        const float eps = -1.0f / A;
        g1 = al[1] - eps * g0;
        g2 = al[2] - eps * g1;
        g3 = al[3] - eps * g2;
    }
    const float i3 = 1.0f / g3, a = g2 * i3, b = g1 * i3, c = g0 * i3;
    const float sh = a * (1.0f / 3), p3 = (b - a * sh) * (1.0f / 3), h = 0.5f * (c - sh * b) + sh * sh * sh;
    const float disc = h * h + p3 * p3 * p3;
    float r0, r1, r2, im = 0.f;
    if (disc >= 0.f) {
        const float w = -(h + copysignf(sqrtf(disc), h));
        const float u = w == 0.f ? 0.f : copysignf(fexp(flog(fabsf(w)) * (1.0f / 3)), w);
        const float v = u == 0.f ? 0.f : -p3 / u;
        r0 = (u + v) - sh;
        r1 = r2 = -0.5f * (u + v) - sh;
        im = 0.8660254f * fabsf(u - v);
    } else {
        const float m = sqrtf(-p3), q = fminf(1.0f, fmaxf(-1.0f, -h / (m * m * m))), th = acosf(q) * (1.0f / 3);
        r0 = 2.0f * m * fcos(th) - sh;
        r1 = 2.0f * m * fcos(th + 2.0943951f) - sh;
        r2 = 2.0f * m * fcos(th - 2.0943951f) - sh;
    }
    zr[k] = r0; zi[k] = 0.f;
    zr[k + 1] = r1; zi[k + 1] = im;
    zr[k + 2] = r2; zi[k + 2] = -im;
    if (n == 3) { zr[3] = 0.f; zi[3] = 0.f; }
    const float q0 = fabsf(r0), q1 = fabsf(r1) + im, q2 = fabsf(r2) + im;
    const float lo = fminf(q0, fminf(q1, q2)), hi = fmaxf(q0, fmaxf(q1, q2));
    // (false for anything not finite, too)
    return good && lo > 1e-2f * (fabsf(sh) + hi) && lo > 1e-5f && hi < 1e5f && (n == 3 || hi < 0.05f * fabsf(A));
}

// Roots of the monic polynomial c (degree n <= 4) by the simultaneous
// Aberth-Ehrlich iteration, G lanes per polynomial (G = 1 or 4): lane s of a
// group of G consecutive lanes owns roots s, s + G, ... and reads the others'
// current values by shuffles.  Four lanes cut the dependent chain of one
// cosmology (few cosmologies: latency-bound); one lane does no repeated work
// (many cosmologies: bound by the FP64 pipe).  Every lane of the warp must
// call this (groups with active == false take part in the shuffles without
// updating).
//
// On this part every FP64 instruction of a warp holds its sub-partition for
// 64 cycles (19 per SM when all four issue), whatever the number of active
// lanes or independent operations, so what counts is the number of FP64
// instructions.  Hence: single precision first, to about 1e-6, in closed form
// where that is good and by the iteration from Newton-polygon circles where it
// is not (its six to nine sweeps of 250 instructions were most of the kernel's
// time); then sweeps in
// which only what decides the accuracy is double, the polynomial's and its
// derivative's values (26 instructions) and the differences of the roots; the
// correction itself, a number known to 1e-7 of its size, is single.  A sweep
// leaves 1e-7 of the error (or its cube), so two usually end it; comparisons
// are made in single precision or on the bits.  (4096 rows, kernel time: 0.070
// ms with double corrections, confirmations and hypot; 0.031 ms so, with the
// closed-form starts.)
// Coefficients of the monic polynomial beyond 1e6 (Or0 below 3e-7 for Om0 = 0.3:
// |A|^4 would near the end of single precision) or OL0 = 0 take the sweeps in
// double throughout, from the circles.
//
// A root closer than a tenth of its modulus to another (near-multiple roots,
// as near the no-Big-Bang boundary) is polished on the original coefficients
// (the monic ones carry the rounding of the division by alpha_n) by the
// compensated scheme; an isolated one is within an ulp or two after the
// sweeps.  For single-precision distances the polish starts at a hundredth
// (`near`): the roots' error there is 1e-13 without it.
// On return every lane of the group holds all n roots in z.
template <int G>
__device__ void group_roots(const double* c, const double* alpha, int n, bool active, float near, cd* z) {
    constexpr int R = 4 / G;   // roots per lane
    const unsigned full = 0xffffffffu;
    const int s = threadIdx.x & (G - 1);
    float cf[5], zr[R], zi[R];
    bool usual = true;
#pragma unroll
    for (int k = 0; k <= 4; k++) {
        cf[k] = k <= n ? (float)c[k] : 0.f;
        usual = usual && fabsf(cf[k]) < 1e6f;
    }
    usual = usual && fabsf(cf[0]) > 1e-20f;
    float st_r[4], st_i[4], af[5];
#pragma unroll
    for (int k = 0; k <= 4; k++) af[k] = (float)alpha[k];
    const bool good = usual && closed_start(af, n, st_r, st_i);
    // (a lane beyond the last row, or of an invalid one, takes no part)
    if (!__all_sync(full, good || !active)) {
        float pr[4], pi[4];
        start_points(cf, n, pr, pi);
#pragma unroll
        for (int k = 0; k < 4; k++)
            if (!good) { st_r[k] = pr[k]; st_i[k] = pi[k]; }
    }
#pragma unroll
    for (int r = 0; r < R; r++) {
        zr[r] = G == 1 ? st_r[r] : (s == 0 ? st_r[0] : s == 1 ? st_r[1] : s == 2 ? st_r[2] : st_r[3]);
        zi[r] = G == 1 ? st_i[r] : (s == 0 ? st_i[0] : s == 1 ? st_i[1] : s == 2 ? st_i[2] : st_i[3]);
    }
    double zre[R], zim[R];
#pragma unroll
    for (int r = 0; r < R; r++) { zre[r] = zr[r]; zim[r] = zi[r]; }
    {
        bool done = !active || good;
#pragma unroll 1
        for (int itf = 0; itf < 100; itf++) {
            if (__all_sync(full, done)) break;
            float ar[4], ai[4];
#pragma unroll
            for (int k = 0; k < 4; k++) {
                ar[k] = G == 1 ? zr[k / G] : __shfl_sync(full, zr[k / G], k % G, G);
                ai[k] = G == 1 ? zi[k / G] : __shfl_sync(full, zi[k / G], k % G, G);
            }
            int small = 1;
#pragma unroll
            for (int r = 0; r < R; r++) {
                const int j = r * G + s;
                if (done || j >= n) continue;
                const float xr0 = ar[j], xi0 = ai[j];
                float pr = cf[4], pi = 0.f, dr = 0.f, di = 0.f;   // (cf[4] = 0 for a cubic)
#pragma unroll
                for (int k = 3; k >= 0; k--) {
                    float ndr = dr * xr0 - di * xi0 + pr, ndi = dr * xi0 + di * xr0 + pi;
                    float npr = pr * xr0 - pi * xi0 + cf[k], npi = pr * xi0 + pi * xr0;
                    dr = ndr; di = ndi; pr = npr; pi = npi;
                }
                if ((pr == 0.f && pi == 0.f) || !(fabsf(dr) + fabsf(di) > 1e-30f)) continue;
                float rr, ri;
                fquot(pr, pi, dr, di, rr, ri);   // p / p'
                float sr = 0.f, si = 0.f;
#pragma unroll
                for (int k = 0; k < 4; k++) {
                    if (k == j || k >= n) continue;
                    float xr = xr0 - ar[k], xi = xi0 - ai[k], x2 = xr * xr + xi * xi;
                    if (!(x2 > 0.f)) continue;
                    float ix = 1.0f / x2;
                    sr += xr * ix; si -= xi * ix;
                }
                float qr = 1.f - (rr * sr - ri * si), qi = -(rr * si + ri * sr);
                float qn = qr * qr + qi * qi;
                if (!(qn > 0.f)) continue;
                float iq = 1.0f / qn;
                float wr = (rr * qr + ri * qi) * iq, wi = (ri * qr - rr * qi) * iq;
                zr[r] = xr0 - wr; zi[r] = xi0 - wi;
                if (!(wr * wr + wi * wi < 1e-12f * (zr[r] * zr[r] + zi[r] * zi[r]) + 1e-30f)) small = 0;
            }
            if (G > 1) {
                small &= __shfl_xor_sync(full, small, 1, G);
                small &= __shfl_xor_sync(full, small, 2, G);
            }
            if (small) done = true;
        }
#pragma unroll
        for (int r = 0; r < R; r++)
            if (isfinite(zr[r]) && isfinite(zi[r])) { zre[r] = zr[r]; zim[r] = zi[r]; }
    }
    // the roots' separation relative to their moduli (float): isolated or not
    float sep = 1.0f;
    {
        float ar[4], ai[4];
#pragma unroll
        for (int k = 0; k < 4; k++) {
            ar[k] = G == 1 ? (float)zre[k / G] : __shfl_sync(full, (float)zre[k / G], k % G, G);
            ai[k] = G == 1 ? (float)zim[k / G] : __shfl_sync(full, (float)zim[k / G], k % G, G);
        }
#pragma unroll
        for (int j = 0; j < 4; j++) {
#pragma unroll
            for (int k = 0; k < 4; k++) {
                if (k == j || j >= n || k >= n) continue;
                const float dr = ar[j] - ar[k], di = ai[j] - ai[k], q = dr * dr + di * di, mj = ar[j] * ar[j] + ai[j] * ai[j];
                if (!(q > sep * sep * mj)) sep = sqrtf(q / mj);
            }
        }
        if (!(sep > 0.f)) sep = 0.f;
    }
    const bool iso = sep > 0.1f;
    // (a group's lanes agree; the others take the next block for nothing)
    if (!__all_sync(full, iso || !active)) {
        // Single precision (the closed form's discriminant, or the sweeps) knows
        // two nearly equal roots only to about 1e-3 of their size: it cannot tell
        // two reals from a conjugate pair, and may return them equal, both real,
        // or exactly conjugate.  The sweeps keep real approximations real and
        // mirror images mirror images (the polynomial is real), so from such
        // starts roots of the other kind are out of reach.  Two approximations
        // that are each other's nearest, with a mean near the real axis, restart
        // at 45 degrees to it through that mean: there the iteration is Halley's
        // for the square root of the pair's discriminant, which reaches either
        // kind (a distance ten times too large costs two sweeps).
        float cr[4], ci[4], dist[4];
        int near_to[4];
#pragma unroll
        for (int k = 0; k < 4; k++) {
            cr[k] = G == 1 ? (float)zre[k / G] : __shfl_sync(full, (float)zre[k / G], k % G, G);
            ci[k] = G == 1 ? (float)zim[k / G] : __shfl_sync(full, (float)zim[k / G], k % G, G);
        }
#pragma unroll
        for (int j = 0; j < 4; j++) {
            dist[j] = 3e38f;
            near_to[j] = -1;
#pragma unroll
            for (int k = 0; k < 4; k++) {
                if (k == j || k >= n) continue;
                const float xr = cr[j] - cr[k], xi = ci[j] - ci[k], q = sqrtf(xr * xr + xi * xi);
                if (q < dist[j]) { dist[j] = q; near_to[j] = k; }
            }
        }
#pragma unroll
        for (int r = 0; r < R; r++) {
#pragma unroll
            for (int j = 0; j < 4; j++) {
                if (j != r * G + s || j >= n) continue;
                const float m = fabsf(cr[j]) + fabsf(ci[j]);
                if (!(dist[j] < 0.1f * m && fabsf(ci[j]) < 0.1f * m)) continue;
#pragma unroll
                for (int k = 0; k < 4; k++) {
                    if (k != near_to[j] || near_to[k] != j) continue;
                    const float h = 0.70710678f * fmaxf(0.5f * dist[j], 1e-3f * m), sg = j < k ? h : -h;
                    zre[r] = (double)(0.5f * (cr[j] + cr[k]) + sg);
                    zim[r] = (double)sg;
                }
            }
        }
    }
    {
        bool done = !active;
        float prev = 3e38f;
#pragma unroll 1
        for (int it = 0; it < 200; it++) {
            double br[4], bi[4];
#pragma unroll
            for (int k = 0; k < 4; k++) {
                br[k] = G == 1 ? zre[k / G] : __shfl_sync(full, zre[k / G], k % G, G);
                bi[k] = G == 1 ? zim[k / G] : __shfl_sync(full, zim[k / G], k % G, G);
            }
            float worst = 0.f;
#pragma unroll
            for (int r = 0; r < R; r++) {
                const int j = r * G + s;
                if (done || j >= n) continue;
                const double x = br[j], y = bi[j];
                if (usual) {
                    // value and derivative by Horner's rule (the monic quartic's first two steps by hand)
                    cd p, dp;
                    if (n == 4) {
                        p = cmk(x + c[3], y);
                        dp = cmk(x + p.re, y + y);
                    } else {
                        p = cmk(1.0, 0.0);
                        dp = cmk(0.0, 0.0);
                    }
#pragma unroll
                    for (int k = 2; k >= 0; k--) {
                        if (n == 4 ? k < 2 : true)
                            dp = cmk(fma(dp.re, x, fma(-dp.im, y, p.re)), fma(dp.re, y, fma(dp.im, x, p.im)));
                        p = cmk(fma(p.re, x, fma(-p.im, y, c[k])), fma(p.re, y, p.im * x));
                    }
                    const float pr = (float)p.re, pi = (float)p.im, dr = (float)dp.re, di = (float)dp.im;
                    float sr = 0.f, si = 0.f;
#pragma unroll
                    for (int k = 0; k < 4; k++) {
                        if (k == j || k >= n) continue;
                        const float xr = (float)(x - br[k]), xi = (float)(y - bi[k]), x2 = xr * xr + xi * xi;
                        if (!(x2 > 0.f)) continue;
                        const float ix = 1.0f / x2;
                        sr += xr * ix;
                        si -= xi * ix;
                    }
                    // w = p / (p' - p S)
                    float wr, wi;
                    fquot(pr, pi, dr - (pr * sr - pi * si), di - (pr * si + pi * sr), wr, wi);
                    if (pr == 0.f && pi == 0.f) continue;
                    zre[r] = x - (double)wr;
                    zim[r] = y - (double)wi;
                    const float xf = (float)x, yf = (float)y, rel = (wr * wr + wi * wi) / (xf * xf + yf * yf);
                    if (!(rel <= worst)) worst = rel;   // a NaN counts as the worst
                } else {
                    cd zj = cmk(x, y), p, dp;
                    horner(c, n, zj, p, dp);
                    if (p.re == 0 && p.im == 0) continue;
                    cd ratio = cmul(p, crcp(dp));
                    cd sm = cmk(0, 0);
#pragma unroll 1
                    for (int k = 0; k < n; k++)
                        if (k != j) sm = cadd(sm, crcp(csub(zj, cmk(br[k], bi[k]))));
                    cd w = cmul(ratio, crcp(csub(cmk(1, 0), cmul(ratio, sm))));
                    zj = csub(zj, w);
                    zre[r] = zj.re; zim[r] = zj.im;
                    const float rel = (float)(cnorm(w) * ddiv(1.0, cnorm(zj) + 1e-300));
                    if (!(rel <= worst)) worst = rel;
                }
            }
            if (G > 1) {
#pragma unroll
                for (int o = 1; o < G; o <<= 1) {
                    const float v = __shfl_xor_sync(full, worst, o, G);
                    if (!(v <= worst)) worst = v;
                }
            }
            if (!done) {
                // |w| below 1e-9 |z| (usual: 1e-7 of it is left), or no longer shrinking
                if (worst < (usual ? 1e-18f : 1e-30f)) done = true;
                else if (it >= 4 && worst >= 0.25f * prev && worst < 1e-16f) done = true;
                prev = worst;
            }
            if (__all_sync(full, done)) break;
        }
    }
    // A root whose imaginary part is negligible (|Im| <= 1e-12 |z|: the
    // classification's test) is put on the real axis; then the polish.
    {
        double cr[4], ci[4];
#pragma unroll
        for (int k = 0; k < 4; k++) {
            cr[k] = G == 1 ? zre[k / G] : __shfl_sync(full, zre[k / G], k % G, G);
            ci[k] = G == 1 ? zim[k / G] : __shfl_sync(full, zim[k / G], k % G, G);
        }
#pragma unroll
        for (int r = 0; r < R; r++) {
            const int j = r * G + s;
            if (!active || j >= n) continue;
            cd zj = cmk(zre[r], zim[r]);
            const int ez = exponent_of(zj);
            const float mx = scaled(zj.re, ez), my = scaled(zj.im, ez), mz = sqrtf(mx * mx + my * my);
            if (fabsf(my) <= 1e-12f * mz) zj.im = 0.0;
            // a single root at zero (OL0 = 0 beside Ox0) is one exactly: the sweeps
            // end somewhere below 1e-100, off the axis
            if (c[0] == 0.0 && c[1] != 0.0 && fabs(zj.re) + fabs(zj.im) < 1e-100) zj = cmk(0.0, 0.0);
            float d = 1.0f;   // distance to the nearest other root over the modulus
#pragma unroll
            for (int k = 0; k < 4; k++) {
                if (k == j || k >= n) continue;
                const float xr = scaled(cr[k] - cr[j], ez), xi = scaled(ci[k] - ci[j], ez);
                const float q = sqrtf(xr * xr + xi * xi) / mz;
                if (!(q >= d)) d = q;
            }
            // (of a conjugate pair only the upper member is used)
            if (!(d > near) && (zj.im >= 0.0)) {
                if (d > 1e-4f) polish_once(alpha, n, zj); else polish_root(alpha, n, zj);
            }
            zre[r] = zj.re; zim[r] = zj.im;
        }
    }
#pragma unroll
    for (int k = 0; k < 4; k++)
        z[k] = G == 1 ? cmk(zre[k / G], zim[k / G])
                      : cmk(__shfl_sync(full, zre[k / G], k % G, G), __shfl_sync(full, zim[k / G], k % G, G));
}

// Root solve and classification of one cosmology, parameter row p[ncol] =
// (H0, Om, OL, Or[, Ok[, Os, Ox]]): the labelled roots in r and, with
// `tangents`, their derivatives dr[slot][k] (slots: A and B of a quartic, B of
// a cubic, then the pair; 1: each lane of a group gets the directions k equal
// to its own number modulo G, 2: every lane gets all).  Returns the status code.  Called by the G lanes of
// a group together (see group_roots); `active` is false for lanes past the
// last cosmology.
template <int G>
__device__ int prep_roots(const double* p, int ncol, bool active, int tangents, float near, RowRoots& r,
                          cd (*dr)[RF_KT], bool& labelled) {
    r.H0 = p[0]; r.Om = p[1]; r.OL = p[2]; r.Or = p[3];
    r.Ok = ncol >= 5 ? p[4] : 1.0 - r.Om - r.OL - r.Or;
    // the further components of fn4 (7-column rows): Os (w = -1/3) scales as
    // (1+z)^2 like curvature but stays out of the curvature map, Ox (w = -2/3)
    // as (1+z); with them every density is an independent direction
    r.Os = ncol >= 7 ? p[5] : 0.0;
    r.Ox = ncol >= 7 ? p[6] : 0.0;
    r.ncol = ncol;
    const double Om = r.Om, OL = r.OL, Or = r.Or, Ok = r.Ok, Os = r.Os, Ox = r.Ox;
    labelled = false;
    int st = ST_OK;
    const int K = ncol - 1;
    const bool finite = isfinite(r.H0) && isfinite(Om) && isfinite(OL) && isfinite(Or) && isfinite(Ok) &&
                        isfinite(Os) && isfinite(Ox);
    const int n = Or > 0 ? 4 : 3;
    r.quartic = n == 4;
    r.cpair = 0;
    if (!finite || !(r.H0 > 0) || Or < 0 || (n == 3 && !(Om > 0))) st = ST_INVALID;
    cd z[4];
    double alpha[5] = {OL, Ox, Ok + Os, Om, Or};
    double an = alpha[n];
    double c[5] = {0.0, 0.0, 0.0, 0.0, 0.0};
    c[n] = 1.0;
    if (st == ST_OK) {
        const double ian = an < 1e-280 ? ddiv(1.0, an) : rcp_(an);
        for (int k = 0; k <= n; k++) c[k] = alpha[k] * ian;
        c[n] = 1.0;
    }
    // A triple root at rho = 0 (x = 1 + z = 0): OL = Ox = Ok + Os = 0 to within
    // the rounding of the closure, so that E^2 = x^3 (Or x + Om) (flat matter +
    // radiation; Einstein-de Sitter when Or = 0).  The root iteration cannot
    // separate a triple root (its error would be of order eps^(1/3)), so the
    // roots are set exactly: rho = 0 three times and rho_A = -Om/Or.  The
    // reductions (3.7)-(3.9) / (B.1)-(B.3) then hold with the repeated roots
    // (the factors d_ij that vanish only multiply terms that drop out).  The
    // root derivatives of App. A are singular at a multiple root, so the
    // tangent slots of such a row are NaN (no gradient).
    const double dtol = 8.0 * 2.220446049250313e-16 * (fabs(Om) + fabs(Or) + fabs(OL) + fabs(Ok) + 1.0);
    const bool triple0 = st == ST_OK && fabs(OL) <= dtol && fabs(Ox) <= dtol && fabs(Ok + Os) <= dtol;
    group_roots<G>(c, alpha, n, active && st == ST_OK && !triple0, near, z);   // every lane, outside any divergent branch
    if (triple0) {
        z[0] = cmk(n == 4 ? -Om / Or : 0.0, 0.0);
        for (int i = 1; i < 4; i++) z[i] = cmk(0.0, 0.0);
    }
    if (st == ST_OK) {
        // Classification: real when the imaginary part is negligible (compared
        // in single precision; other comparisons on the bits: a double's
        // comparison holds the FP64 pipe like any other FP64 instruction).
        // Reals come first, by decreasing |rho| (fn15: largest roots of
        // E^2(z+1)), then complex ones, then the cubic's absent fourth.
        long long key[4];
        int nreal = 0;
        #pragma unroll
        for (int i = 0; i < 4; i++) {
            const bool real = i < n && (triple0 || negligible_im(z[i]));
            if (real) {
                z[i].im = 0;
                nreal++;
                if (__double_as_longlong(z[i].re) >= __double_as_longlong(1.0)) st = ST_NO_BIG_BANG;   // real root at z >= 0 (Sec. 3, Fig. 1)
            }
            key[i] = real ? __double_as_longlong(z[i].re) & INT64_MAX : i < n ? -1 : -2;
        }
        auto order = [&](int i, int j) {
            if (key[j] > key[i]) {
                const long long t = key[i]; key[i] = key[j]; key[j] = t;
                const cd u = z[i]; z[i] = z[j]; z[j] = u;
            }
        };
        order(0, 1); order(2, 3); order(0, 2); order(1, 3); order(1, 2);
        const int ncx = n - nreal;
        cd A = cmk(0, 0), Bv = cmk(0, 0), P1 = cmk(0, 0), P2 = cmk(0, 0);
        const bool cpair = ncx == 2 && nreal == n - 2;
        if (n == 4) { A = z[0]; Bv = z[1]; P1 = z[2]; P2 = z[3]; }
        else { Bv = z[0]; P1 = z[1]; P2 = z[2]; }
        if (cpair) {
            if (__double_as_longlong(P1.im) < 0) P1 = P2;   // the member with the positive imaginary part
        } else if (ncx != 0 && st == ST_OK) {
            st = ST_UNSUPPORTED;   // e.g. two complex pairs (no real root)
        }
        if (st != ST_OK && st != ST_NO_BIG_BANG) return st;
        labelled = true;
        r.cpair = cpair;
        r.A = A.re;
        r.B = Bv.re;
        r.pr = P1.re;
        r.pi = cpair ? P1.im : P2.re;
        // division by rho_A in eq. (3.8)
        if (n == 4 && A.re == 0.0 && !triple0) st = st == ST_OK ? ST_DEGENERATE : st;
        if (n == 3 && Bv.re == 0.0 && !triple0) st = st == ST_OK ? ST_DEGENERATE : st;
        cd rho[4];
        int nr = 0;
        if (n == 4) rho[nr++] = A;
        rho[nr++] = Bv;
        rho[nr++] = P1;
        rho[nr++] = cpair ? cmk(P1.re, -P1.im) : P2;
        int degen = 0;
        if (!tangents) {
            // (two equal labelled roots: the reduction's differences vanish)
            #pragma unroll 1
            for (int j = 0; j < nr; j++)
                for (int m2 = 0; m2 < j; m2++)
                    if (rho[j].re == rho[m2].re && rho[j].im == rho[m2].im) degen = 1;
            if (degen && !triple0) st = (st == ST_OK) ? ST_DEGENERATE : st;
            return st;
        }
        // App. A (eqs. A.2-A.4): d rho_j / d c_i = -rho_j^i / prod_{m != j} (rho_j - rho_m).
        // Summed over the coefficients c_i = alpha_i / alpha_n of the monic
        // polynomial this is
        //   d rho_j / d theta_k = -(dE^2/dtheta_k)(rho_j) / (alpha_n prod_{m != j} (rho_j - rho_m)),
        // with dE^2/dOm = x^3, dE^2/dOL = 1, dE^2/dOr = x^4, dE^2/dOk = dE^2/dOs = x^2,
        // dE^2/dOx = x, and -x^2 added to the first three under the closure.
        // With G lanes per cosmology, lane j of the group takes root j and
        // the group exchanges the results (the G lanes of a group take the
        // same branches: one cosmology).
        const int sg = G > 1 ? (int)(threadIdx.x & (G - 1)) : 0;
        cd mine[RF_KT];
        #pragma unroll
        for (int k = 0; k < RF_KT; k++) mine[k] = cmk(0, 0);
        #pragma unroll 1
        for (int j = 0; j < nr; j++) {
            if (G > 1 && j != sg) continue;
            const cd x = rho[j];
            cd e2p = cmk(-an, 0);
            #pragma unroll 1
            for (int m2 = 0; m2 < nr; m2++)
                if (m2 != j) e2p = cmul(e2p, csub(x, rho[m2]));
            const bool degenerate = e2p.re == 0 && e2p.im == 0;
            if (degenerate) degen = 1;
            // inv = -1 / (alpha_n prod), y = x^2 inv
            const double ie = rcp_(cnorm(e2p));
            const cd inv = degenerate ? cmk(nan(""), nan("")) : cmk(e2p.re * ie, -(e2p.im * ie));
            const cd y = cmul(x, cmul(x, inv));
            if (ncol == 4) {
                // x^3 - x^2 = x^2 (x-1), 1 - x^2 = -(x-1)(x+1), x^4 - x^2 = x^2 (x-1)(x+1)
                const cd u = cmk(x.re - 1.0, x.im), t = cmul(u, cmk(x.re + 1.0, x.im)), w = cmul(t, inv);
                mine[0] = cmul(y, u);
                mine[1] = cmk(-w.re, -w.im);
                mine[2] = cmul(y, t);
            } else {
                const cd y3 = cmul(y, x);
                mine[0] = y3;
                mine[1] = inv;
                mine[2] = cmul(y3, x);
                mine[3] = y;
                mine[4] = y;
                mine[5] = cmul(x, inv);
            }
            if (n == 3) mine[2] = cmk(nan(""), nan(""));  // no Or direction in a cubic
            if (G == 1)
                for (int k = 0; k < K; k++) dr[j][k] = mine[k];
        }
        if (G > 1) {
            const unsigned gmask = ((1u << G) - 1) << ((threadIdx.x & 31) & ~(G - 1));
            #pragma unroll
            for (int o = 1; o < G; o <<= 1) degen |= __shfl_xor_sync(gmask, degen, o, G);
            if (tangents == 1) {
                // transposed: at step d lane l reads lane l + d's direction l
                #pragma unroll 1
                for (int h = 0; h < K; h += G)
                    #pragma unroll 1
                    for (int d = 0; d < G; d++) {
                        const int from = (sg + d) & (G - 1), give = h + ((sg - d) & (G - 1));
                        const cd v = give < K ? mine[give] : cmk(0, 0);
                        const cd g = cmk(__shfl_sync(gmask, v.re, from, G), __shfl_sync(gmask, v.im, from, G));
                        if (h + sg < K) dr[from][h + sg] = g;
                    }
            } else {
                #pragma unroll 1
                for (int j = 0; j < nr; j++)
                    #pragma unroll 1
                    for (int k = 0; k < K; k++)
                        dr[j][k] = cmk(__shfl_sync(gmask, mine[k].re, j, G), __shfl_sync(gmask, mine[k].im, j, G));
            }
        }
        if (degen && !triple0) st = (st == ST_OK) ? ST_DEGENERATE : st;
    }
    return st;
}

// The record of the X-tangent kernel (RecField) from the labelled roots.
__device__ __noinline__ void legacy_record(const RowRoots& r, const cd (*dr)[RF_KT], bool labelled, double* rec) {
    const double H0 = r.H0, Om = r.Om, OL = r.OL, Or = r.Or, Ok = r.Ok, Os = r.Os, Ox = r.Ox;
    const int ncol = r.ncol, K = ncol - 1, n = r.quartic ? 4 : 3;
    const bool cpair = r.cpair;
    // slot A of this record is the cubic's only special root
    const cd A = cmk(r.quartic ? r.A : r.B, 0.0), Bv = cmk(r.quartic ? r.B : 0.0, 0.0);
    const cd P1 = cmk(r.pr, cpair ? r.pi : 0.0), P2 = cmk(cpair ? 0.0 : r.pi, 0.0);
    for (int i = 0; i < NREC; i++) rec[i] = 0;
    if (labelled) {
        rec[RF_A] = A.re - 1.0;
        rec[RF_B] = (n == 4 ? Bv.re : 1.0) - 1.0;
        if (cpair) { rec[RF_PRE] = P1.re - 1.0; rec[RF_PIM] = P1.im; }
        else { rec[RF_PRE] = P1.re - 1.0; rec[RF_PIM] = P2.re - 1.0; }
        rec[RF_YA] = sqrt(-rec[RF_A]);
        rec[RF_YB] = sqrt(-rec[RF_B]);
        if (cpair) { cd y = csqrt_(cmk(-rec[RF_PRE], -rec[RF_PIM])); rec[RF_YPRE] = y.re; rec[RF_YPIM] = y.im; }
        else { rec[RF_YPRE] = sqrt(-rec[RF_PRE]); rec[RF_YPIM] = sqrt(-rec[RF_PIM]); }
        // big-root quantities of the quartic, scaled by lam = Or (see quartic_integrals)
        if (n == 4) {
            double rA = A.re;                  // rho_A
            rec[RF_LAM] = Or;
            rec[RF_AA] = -Or * (rA - 1.0);
            rec[RF_MA] = Or * rA;
            const double irA = ddiv(1.0, rA);
            rec[RF_EPSA] = -irA;
            rec[RF_RHOA] = rA;
            // Tangents of m_A = lam rho_A = y from the scaled quartic
            //   F(y) = y^4 + Om y^3 + (Ok + Os) Or y^2 + Ox Or^2 y + OL Or^3 = Or^3 E^2(rho_A) = 0,
            // dy = -(dF/dtheta) / (dF/dy), a ratio of O(1) terms: in the Or
            // direction rho_A d lam and lam d rho_A are each O(Om/Or) and cancel.
            // a_A = -lam (rho_A - 1) = -y + lam.
            const double y = Or * rA, Oks = Ok + Os;
            const double iFy = ddiv(1.0, y * y * (4.0 * y + 3.0 * Om) + 2.0 * Oks * Or * y + Ox * Or * Or);
            const double cl = ncol == 4 ? 1.0 : 0.0, FOk = Or * y * y;
            const double Fth[RF_KT] = {y * y * y - cl * FOk, Or * Or * Or - cl * FOk,
                                       Oks * y * y + 2.0 * Ox * Or * y + 3.0 * OL * Or * Or - cl * FOk, FOk, FOk,
                                       Or * Or * y};
            #pragma unroll 1
            for (int k = 0; k < K; k++) {
                double dl = (k == 2) ? 1.0 : 0.0, dA = dr[0][k].re;
                const double dy = -Fth[k] * iFy;
                rec[RF_DLAM + k] = dl;
                rec[RF_DAA + k] = dl - dy;
                rec[RF_DMA + k] = dy;
                rec[RF_DEPSA + k] = dA * (irA * irA);
                rec[RF_DRHOA + k] = dA;
            }
        }
        // q_j = -1/r_j (dq_j = dr_j / r_j^2) for the normalised Carlson arguments
        {
            double rA = A.re - 1.0;
            const double iA = rA != 0.0 ? ddiv(1.0, rA) : 0.0;
            rec[RF_QA] = -iA;
            for (int k = 0; k < K; k++) rec[RF_DQA + k] = dr[0][k].re * (iA * iA);
            if (n == 4) {
                double rB = Bv.re - 1.0;
                const double iB = rB != 0.0 ? ddiv(1.0, rB) : 0.0;
                rec[RF_QB] = -iB;
                for (int k = 0; k < K; k++) rec[RF_DQB + k] = dr[1][k].re * (iB * iB);
            }
            const int jq = n == 4 ? 2 : 1;
            if (cpair) {
                cd r = cmk(P1.re - 1.0, P1.im);
                cd q = cdiv(cmk(-1.0, 0.0), r);
                rec[RF_QPRE] = q.re;
                rec[RF_QPIM] = q.im;
                const cd q2 = cmul(q, q);   // dq = dr / r^2 = q^2 dr
                for (int k = 0; k < K; k++) {
                    cd dq = cmul(dr[jq][k], q2);
                    rec[RF_DQPRE + k] = dq.re;
                    rec[RF_DQPIM + k] = dq.im;
                }
            } else {
                double r1 = P1.re - 1.0, r2 = P2.re - 1.0;
                const double i1 = r1 != 0.0 ? ddiv(1.0, r1) : 0.0, i2 = r2 != 0.0 ? ddiv(1.0, r2) : 0.0;
                rec[RF_QPRE] = -i1;
                rec[RF_QPIM] = -i2;
                for (int k = 0; k < K; k++) {
                    rec[RF_DQPRE + k] = dr[jq][k].re * (i1 * i1);
                    rec[RF_DQPIM + k] = dr[jq + 1][k].re * (i2 * i2);
                }
            }
        }
        #pragma unroll 1
        for (int k = 0; k < K; k++) {
            rec[RF_DA + k] = dr[0][k].re;
            rec[RF_DB + k] = n == 4 ? dr[1][k].re : 0.0;
            int jp = n == 4 ? 2 : 1;
            if (cpair) { rec[RF_DPRE + k] = dr[jp][k].re; rec[RF_DPIM + k] = dr[jp][k].im; }
            else { rec[RF_DPRE + k] = dr[jp][k].re; rec[RF_DPIM + k] = dr[jp + 1][k].re; }
        }
    }
    // prefactors: alpha_m^-1/2 (Or for the quartic, Om for the cubic, eq. 3.2 / fn13)
    double amh = ddiv(1.0, sqrt(n == 4 ? Or : Om));
    rec[RF_AMH] = amh;
    rec[RF_OK] = Ok;
    rec[RF_H0] = H0;
    const double iH0 = ddiv(1.0, H0);
    rec[RF_DH] = LCDM_C_KMS * iH0;
    rec[RF_TH] = LCDM_HUBBLE_GYR * iH0;
    rec[RF_KIND] = !labelled ? 0 : n == 4 ? (cpair ? 0 : 1) : (cpair ? 2 : 3);
    // N = sqrt(E^2(0) / alpha_n): E^2(0) = Om + OL + Or + Ok (+ Os + Ox), exactly 1 under the closure
    const double S0 = ncol == 4 ? 1.0 : Om + OL + Or + Ok + Os + Ox;
    const double iOm = ddiv(1.0, Om);
    const double nrm = n == 4 ? sqrt(S0) : sqrt(S0 * iOm);
    const double inrm = ddiv(1.0, nrm);
    rec[RF_NRM] = nrm;
    #pragma unroll 1
    for (int k = 0; k < K; k++) {
        const double dS = ncol == 4 ? 0.0 : 1.0, dOm = k == 0 ? 1.0 : 0.0;
        rec[RF_DNRM + k] = n == 4 ? 0.5 * dS * inrm : 0.5 * (dS * Om - S0 * dOm) * inrm * (iOm * iOm);
        if (n == 3 && k == 2) rec[RF_DNRM + k] = nan("");
    }
    #pragma unroll 1
    for (int k = 0; k < K; k++) {
        rec[RF_DAMH + k] = 0;
        if (n == 4 && k == 2) rec[RF_DAMH + k] = -0.5 * amh * amh * amh;
        if (n == 3 && k == 0) rec[RF_DAMH + k] = -0.5 * amh * amh * amh;
        if (n == 3 && k == 2) rec[RF_DAMH + k] = nan("");
        rec[RF_DOK + k] = ncol == 4 ? -1.0 : (k == 3 ? 1.0 : 0.0);
    }
}

// The core's record of one cosmology: lane 0 of the group writes the values,
// lane k mod G the tangents of direction k.
template <int G, class T>
__device__ void write_core(const RowRoots& r, const cd (*dr)[RF_KT], int lane, bool time, bool absorb, bool tangents, int ns,
                           T* rec) {
    if (lane == 0) {
        core_values<T>(r, time, absorb, ns, rec);
        const double iH0 = r.H0 < 1e-280 ? ddiv(1.0, r.H0) : rcp_(r.H0);
        put(rec, C_DH, LCDM_C_KMS * iH0);
        put(rec, C_TH, LCDM_HUBBLE_GYR * iH0);
        put(rec, C_IH0, iH0);
    }
    if (!tangents) return;
    const int b = r.quartic ? 1 : 0;
    #pragma unroll 1
    for (int k = lane; k < r.ncol - 1; k += G)
        core_tangent<T>(r, time, ns, k, dr[0][k].re, dr[b][k].re, dr[b + 1][k].re, r.cpair ? dr[b + 1][k].im : dr[b + 2][k].re,
                        rec);
}

struct PrepArgs {
    ShiftArgs shift;        // general limits: the rows are shifted first (shift.z1 null: they are not)
    const double* params;   // [B][ncol]
    int64_t B;
    int ncol;
    int tangents;           // the root derivatives are needed
    int ns;                 // series coefficients the core will use
    int time;               // the time coordinate's constants are needed
    int absorb;             // the absorption distance's constants are needed
    double* recD;           // [B][NREC] record of the X-tangent kernel, and its (hi, lo) copy (optional)
    float2* recF;
    float* coreF;           // [B][NCORE] record of the core, single or double precision (optional; beside
                            // recD without tangents)
    double* coreD;
    int32_t* status;
    double* grad;           // [B][ncol], [B]: initialised to 0 (NaN for a bad status), optional
    double* loglike;
};

// G lanes per cosmology (see group_roots).  Launched with 32-thread blocks
// over G B threads.
template <int G> __global__ void prep_kernel(PrepArgs a) {
    const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int64_t b = t / G;
    const int j = (int)(t % G);
    const bool inb = b < a.B;
    const int ncol = a.ncol;
    // lanes past the end work on a copy of the last row and write nothing
    const int64_t bb = inb ? b : a.B - 1;
    double shifted[4];
    if (a.shift.z1) shift_row(a.shift, bb, inb && j == 0, shifted);
    const double* prow = a.shift.z1 ? shifted : a.params + bb * ncol;
    RowRoots r;
    cd dr[4][RF_KT];
    bool labelled;
    const int st = prep_roots<G>(prow, ncol, inb, a.tangents ? (a.recD ? 2 : 1) : 0, a.coreF && !a.recD ? 0.01f : 0.1f, r, dr,
                                 labelled);
    if (!inb) return;
    if (a.recD) {
        double rec[NREC];
        legacy_record(r, dr, labelled, rec);
        double* rd = a.recD + b * NREC;
        float2* rf = a.recF + b * NREC;
        #pragma unroll 1
        for (int i = j; i < NREC; i += G) {
            rd[i] = rec[i];
            if (!a.recF) continue;
            float h = (float)rec[i];
            rf[i] = make_float2(h, (float)(rec[i] - (double)h));
        }
    }
    if (st == ST_OK && (a.coreF || a.coreD)) {
        r.finish(a.time);
        const bool tangents = a.tangents && !a.recD;
        if (a.coreF) write_core<G, float>(r, dr, j, a.time, a.absorb, tangents, a.ns, a.coreF + b * NCORE);
        else write_core<G, double>(r, dr, j, a.time, a.absorb, tangents, a.ns, a.coreD + b * NCORE);
    }
    if (j != 0) return;
    a.status[b] = st;
    double init = st == ST_OK ? 0.0 : nan("");
    if (a.grad)
        for (int k = 0; k < ncol; k++) a.grad[b * ncol + k] = init;
    if (a.loglike) a.loglike[b] = init;
}

}  // namespace lcdm
