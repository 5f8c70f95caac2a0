// The row record of the core (lcdm_core.cuh) from a cosmology's roots.
#pragma once
#include "lcdm_core.cuh"

namespace lcdm {

// largest deviation of the three, and of the five, arguments from their mean, over z^2
LCDM_HD float dev3(double e2, double e3) {
    const float a = sqrtf((float)fabs(e2)), b = cbrtf(4.0f * (float)fabs(e3));
    return a > b ? a : b;
}
LCDM_HD float dev5(float d3, double m) {
    const float am = (float)fabs(m);
    const float a = 0.6f * am, b = d3 + 0.4f * am;
    return a > b ? a : b;
}

// Roots of E^2(x), x = 1 + z, as classified by the preparation: the big root A
// (quartic only), B, and the pair (conjugate: P = (pr, +-pi); two reals: pr, pi),
// with derivatives along the K density directions.
struct RowRoots {
    double H0, Om, OL, Or, Ok, Os, Ox;
    int ncol, quartic, cpair;
    double A, B, pr, pi;
    // set by finish(): q_j = -1/(rho_j - 1) (0 for the cubic's absent root; the
    // pair: real and imaginary part, or the two), eps = -1/rho_A, 1/S0
    double qA, qB, q1, q2, eps, S0, iS0;
    // the invariants e2 = -I / (3 S0^2), e3 = -J / (27 S0^3), the largest deviation
    // of the three arguments over z^2; with `time` also k (k2 = k / 3), m and the
    // five's.  (Every lane of a group needs them.)
    double e2, e3, k, m;
    float d3, d5;

    // (for a valid row: every real root below 1, S0 > 0)
    LCDM_HD void finish(bool time = true) {
        qA = quartic ? rcp_(1.0 - A) : 0.0;
        eps = quartic ? -1.0 / A : 0.0;
        qB = rcp_(1.0 - B);
        // one reciprocal for the pair
        const double a = pr - 1.0, b = cpair ? pi : pi - 1.0;
        const double i = -rcp_(cpair ? a * a + b * b : a * b);
        q1 = (cpair ? a : b) * i;
        q2 = (cpair ? -b : a) * i;
        S0 = ncol == 4 ? 1.0 : Om + OL + Or + Ok + Os + Ox;
        iS0 = ncol == 4 ? 1.0 : rcp_(S0);
        const double C = Ok + Os, iS2 = iS0 * iS0;
        const double I = 12.0 * Or * OL - 3.0 * Om * Ox + C * C;
        const double J = 2.0 * C * C * C - 9.0 * Om * C * Ox + 27.0 * Or * Ox * Ox + 27.0 * Om * Om * OL - 72.0 * Or * C * OL;
        e2 = I * (-1.0 / 3) * iS2;
        e3 = J * (-1.0 / 27) * (iS2 * iS0);
        d3 = dev3(e2, e3);
        if (!time) return;
        // E^2(x) / (1 - x / rho_A) = g0 + g1 x + g2 x^2 + g3 x^3
        const double g0 = OL, g1 = Ox - eps * g0, g2 = C - eps * g1, g3 = Om - eps * g2;
        k = (-g3 + eps * (g2 - eps * (g1 - eps * g0))) * iS0;
        m = (g2 + eps * (3.0 * eps * g0 - 2.0 * g1)) * (iS0 * (1.0 / 3));
        d5 = dev5(d3, m);
    }
};

// derivative of the density parameters (Om, OL, Or, Ok + Os, Ox) along direction k
struct RowDir { double dOm, dOL, dOr, dOk, dOx, dS; };
LCDM_HD RowDir row_dir(int ncol, int k) {
    RowDir d;
    d.dOm = k == 0; d.dOL = k == 1; d.dOr = k == 2; d.dOx = k == 5;
    d.dOk = k == 3 || k == 4 ? 1.0 : (ncol == 4 ? -1.0 : 0.0);
    d.dS = ncol == 4 ? 0.0 : 1.0;
    return d;
}

// The closing series' ns <= 10 coefficients from degree 2 (single-precision records:
// in single precision; they enter the results times the squared deviation and
// higher powers, at most a twentieth).  With the arguments' deviations X_i from
// their mean (sum 0) the series are sum_N c_N T_N, c_N = 1/(2N+1) for R_F and
// 3/(2N+3) for R_J (DLMF 19.19), where sum_N T_N t^N = prod_i (1 - t X_i)^-1/2
// = Q(t)^-1/2, Q = 1 + E2 t^2 - E3 t^3 + E4 t^4 - E5 t^5; from 2 Q S' = -Q' S,
//   N T_N = - sum_j (N - j/2) q_j T_{N-j}.
template <class S> struct SeriesBase { typedef typename Base<S>::type type; };
template <class T> struct SeriesBase<DD<T> > { typedef T type; };
template <class S> LCDM_HD S zero_like(const S& a) { return a * typename SeriesBase<S>::type(0); }
// R_F: b_2 .. b_11 from (e2, e3)
template <class S> LCDM_HD void rf_coefs(const S& e2, const S& e3, int ns, S* b) {
    typedef typename SeriesBase<S>::type B;
    S t[CORE_NS + 2];
    t[0] = zero_like(e2) + B(1);
    t[1] = zero_like(e2);
#pragma unroll
    for (int n = 2; n < CORE_NS + 2; n++) {
        if (n >= ns + 2) break;
        S v = t[n - 2] * e2 * B(-(n - 1.0) / n);
        if (n >= 3) v = v + t[n - 3] * e3 * B((n - 1.5) / n);
        t[n] = v;
        b[n - 2] = v * B(1.0 / (2 * n + 1));
    }
}
// R_J: a_2 .. a_11; m = (mean of three - p) / z^2
template <class S> LCDM_HD void rj_coefs(const S& m, const S& e2, const S& e3, int ns, S* a) {
    typedef typename SeriesBase<S>::type B;
    const S m2 = m * m;
    const S E2 = e2 - m2 * B(0.6);
    const S Q = e3 - m * e2 * B(0.4) - m2 * m * B(0.064);
    const S P = m * B(0.6), P2 = P * P, P3 = P2 * P;
    const S E3 = Q + E2 * P * B(2.0) + P3 * B(4.0);
    const S E4 = (Q * B(2.0) + E2 * P + P3 * B(3.0)) * P;
    const S E5 = Q * P2;
    S t[CORE_NS + 2];
    t[0] = zero_like(E2) + B(1);
    t[1] = zero_like(E2);
#pragma unroll
    for (int n = 2; n < CORE_NS + 2; n++) {
        if (n >= ns + 2) break;
        S v = t[n - 2] * E2 * B(-(n - 1.0) / n);
        if (n >= 3) v = v + t[n - 3] * E3 * B((n - 1.5) / n);
        if (n >= 4) v = v - t[n - 4] * E4 * B((n - 2.0) / n);
        if (n >= 5) v = v + t[n - 5] * E5 * B((n - 2.5) / n);
        t[n] = v;
        a[n - 2] = v * B(3.0 / (2 * n + 3));
    }
}
// 1 / dev, the scale of the series' variable (1 where a record serves one
// evaluation; 0 without deviations)
template <class T> LCDM_HD T dev_scale(float dev, int ns) {
    return ns <= CORE_NS_ONCE ? (T)1 : dev > 0.0f ? (T)1 / (T)dev : (T)0;
}

template <class T> LCDM_HD void put(T* rec, int i, double v) { rec[i] = (T)v; }
LCDM_HD void put_lo(float* rec, int i, double v) { rec[i] = (float)(v - (double)(float)v); }
LCDM_HD void put_lo(double* rec, int i, double) { rec[i] = 0.0; }

// values (directions are added by core_tangent)
template <class T> LCDM_HD void core_values(const RowRoots& r, bool time, bool absorb, int ns, T* rec) {
    const double Oks = r.Ok + r.Os, S0 = r.S0, iS0 = r.iS0, sS = r.ncol == 4 ? 1.0 : sqrt(S0), isS = sS * iS0;
    const double qA = r.qA, qB = r.qB, q1 = r.q1, q2 = r.q2, eps = r.eps;
    put(rec, C_QA, qA); put(rec, C_QB, qB);
    put(rec, C_QR, q1); put_lo(rec, C_QRL, q1);
    put(rec, C_QI, q2); put_lo(rec, C_QIL, q2);
    put(rec, C_C2, 2.0 * isS);
    put(rec, C_OK, r.Ok);
    put(rec, C_KIND, r.cpair ? 1.0 : 0.0);
    put(rec, C_RS, r.ncol == 4 ? 0.0 : -0.5 * iS0);
    put(rec, C_FREE0, 0.0); put(rec, C_FREE1, 0.0);
    const T f2 = (T)r.e2, f3 = (T)r.e3;
    T b[CORE_NS];
    // (normalised by the largest deviation: see lcdm_core.cuh)
    const T u3 = dev_scale<T>(r.d3, ns);
    rf_coefs<T>((f2 * u3) * u3, ((f3 * u3) * u3) * u3, ns, b);
#pragma unroll
    for (int j = 0; j < CORE_NS; j++)
        if (j < ns) rec[C_B + j] = b[j];
    rec[C_DF] = (T)r.d3;
    if (ns <= CORE_NS_ONCE) { put(rec, C_E2, r.e2); put(rec, C_E3, r.e3); }
    if (time) {
        put(rec, C_EPS, eps);
        put(rec, C_K2, r.k * (1.0 / 3));
        put(rec, C_K3, r.OL * iS0);
        if (ns <= CORE_NS_ONCE) put(rec, C_M, r.m);
        const T u5 = dev_scale<T>(r.d5, ns);
        rj_coefs<T>((T)r.m * u5, (f2 * u5) * u5, ((f3 * u5) * u5) * u5, ns, b);
#pragma unroll
        for (int j = 0; j < CORE_NS; j++)
            if (j < ns) rec[C_A + j] = b[j];
        rec[C_DJ] = (T)r.d5;
    }
    if (!absorb) return;
    const double S = r.cpair ? 2.0 * r.pr : r.pr + r.pi, Q = r.cpair ? r.pr * r.pr + r.pi * r.pi : r.pr * r.pi;
    const double pB = r.cpair ? (r.pr - r.B) * (r.pr - r.B) + r.pi * r.pi : (r.pr - r.B) * (r.pi - r.B);
    const double yB = 1.0 - r.B, mA = r.quartic ? r.Or * r.A : -r.Om, rs = r.B + S, iS3 = iS0 * isS;
    const double X1 = mA * iS0 * (1.0 / 3) * ((S - 2.0 * r.B) + eps * (2.0 * Q - r.B * S));
    double hx = 0.0;
    if (r.quartic) {
        const double aA = -r.Or * (r.A - 1.0), iaA = rcp_(aA), aB = aA - r.Or * yB, c = 1.0 - eps * rs;
        const double rE1 = -(mA * (2.0 * S + eps * (Q + r.B * r.B + r.B * S)));
        hx = r.Or * pB * iS0;
        put(rec, X_LX, r.Or * yB * yB * iS0);
        put(rec, X_PX, pB * aB * aB * (iS0 * iS0));
        put(rec, X_C0, sS * iaA);
        put(rec, X_T1, (2.0 * r.B * r.B - pB) * isS);
        put(rec, X_G1, pB * rE1 * (1.0 / 3) * iS3);
        put(rec, X_G2, -c * aB * mA * pB * pB * (1.0 / 3) * (iS3 * iS0));
        put(rec, X_G3, c * mA);
        put(rec, X_G4, c * yB * mA * iS3 * (iaA * iaA));
        put(rec, X_G5, rE1 * yB * isS * iaA);
        put(rec, X_SY, sS * rcp_(yB));
        put(rec, X_N0, S0 * (2.0 * aA * yB - r.Or * yB * yB));
        put(rec, X_N1, S0 * aA);
        put(rec, X_N2, aB * aB * pB);
        put(rec, X_AB, aB * iaA);
        put(rec, X_LAM, r.Or);
    } else {
        put(rec, X_LX, 0.0); put(rec, X_PX, 0.0);
        put(rec, X_C0, (2.0 / 3) * sS / r.Om);
        put(rec, X_T1, (2.0 / 3) * (3.0 * r.B * r.B - pB) * isS);
        put(rec, X_G1, (4.0 / 9) * rs * pB * r.Om * iS3);
        put(rec, X_G2, 0.0); put(rec, X_G3, 0.0); put(rec, X_G4, 0.0);
        put(rec, X_G5, (4.0 / 3) * rs * yB * isS);
        put(rec, X_SY, 1.0);
        put(rec, X_N0, 0.0); put(rec, X_N1, 0.0); put(rec, X_N2, 0.0);
        put(rec, X_AB, 0.0); put(rec, X_LAM, 0.0);
    }
    put(rec, X_FREE, 0.0);
    put(rec, X_HX, hx);
    const float dA = dev5(r.d3, X1 + hx), dD = dev5(r.d3, X1), dX = dA > dD ? dA : dD;
    rec[X_DX] = (T)dX;
    if (r.cpair) { put(rec, X_SQ, 2.0 * q1); put(rec, X_PQ, q1 * q1 + q2 * q2); }
    else { put(rec, X_SQ, q1 + q2); put(rec, X_PQ, q1 * q2); }
    // the series at p0 (offset X1 + hx) and at x1 (offset X1), and their divided differences
    DD<T> ad[CORE_NS];
    const T uX = dev_scale<T>(dX, ns), g2 = (f2 * uX) * uX, g3 = ((f3 * uX) * uX) * uX;
    rj_coefs<DD<T> >(mkdd<T>((T)(X1 + hx) * uX, (T)X1 * uX, uX), mkdd<T>(g2, g2, (T)0), mkdd<T>(g3, g3, (T)0), ns, ad);
#pragma unroll
    for (int j = 0; j < CORE_NS; j++) {
        if (j >= ns) break;
        rec[X_S + 3 * j] = ad[j].v1;
        rec[X_S + 3 * j + 1] = ad[j].v2;
        rec[X_S + 3 * j + 2] = ad[j].d;
    }
    rec[X_S + 3 * CORE_NS] = rec[X_S + 3 * CORE_NS + 1] = (T)0;
}

// tangents of direction k; dA, dB, (dpr, dpi): the roots' derivatives along it
template <class T>
LCDM_HD void core_tangent(const RowRoots& r, bool time, int ns, int k, double dA, double dB, double dpr, double dpi, T* rec) {
    T* t = rec + C_TAN + C_TSTRIDE * k;
    const RowDir d = row_dir(r.ncol, k);
    const double Oks = r.Ok + r.Os, iS0 = r.iS0, eps = r.eps;
    put(t, CT_QA, r.quartic ? dA * (r.qA * r.qA) : 0.0);
    put(t, CT_QB, dB * (r.qB * r.qB));
    if (r.cpair) {
        // dq = q^2 dr
        const double s1 = r.q1 * r.q1 - r.q2 * r.q2, s2 = 2.0 * r.q1 * r.q2;
        put(t, CT_QR, s1 * dpr - s2 * dpi);
        put(t, CT_QI, s1 * dpi + s2 * dpr);
    } else {
        put(t, CT_QR, dpr * (r.q1 * r.q1));
        put(t, CT_QI, dpi * (r.q2 * r.q2));
    }
    // e2 = -I / (3 S0^2), e3 = -J / (27 S0^3) by the invariants' partial derivatives
    const double Om = r.Om, OL = r.OL, Or = r.Or, c = Oks, Ox = r.Ox, c2 = c * c, iS2 = iS0 * iS0;
    double dI = 2.0 * c * d.dOk, dJ = (6.0 * c2 - 9.0 * Om * Ox - 72.0 * Or * OL) * d.dOk;
    if (k == 0) { dI -= 3.0 * Ox; dJ += 54.0 * Om * OL - 9.0 * c * Ox; }
    if (k == 1) { dI += 12.0 * Or; dJ += 27.0 * Om * Om - 72.0 * Or * c; }
    if (k == 2) { dI += 12.0 * OL; dJ += 27.0 * Ox * Ox - 72.0 * c * OL; }
    if (k == 5) { dI -= 3.0 * Om; dJ += 54.0 * Or * Ox - 9.0 * Om * c; }
    double de2 = dI * (-1.0 / 3), de3 = dJ * (-1.0 / 27);
    if (r.ncol != 4) {
        de2 = (de2 * iS0 - 2.0 * r.e2) * iS0;
        de3 = (de3 * iS2 - 3.0 * r.e3) * iS0;
    }
    const T e2 = (T)r.e2, e3 = (T)r.e3;
    typedef Dual<T, 1> F;
    F b[CORE_NS];
    // the invariants and their derivatives, normalised by dev u = 1 (a constant of the row here)
    auto f2 = [&](T u) { F f; f.v = (e2 * u) * u; f.d[0] = ((T)de2 * u) * u; return f; };
    auto f3 = [&](T u) { F f; f.v = ((e3 * u) * u) * u; f.d[0] = ((T)(de3 * u) * u) * u; return f; };
    const bool once = ns <= CORE_NS_ONCE;
    if (once) {
        put(t, CT_E2, de2);
        put(t, CT_E3, de3);
    } else {
        const T u = dev_scale<T>(r.d3, ns);
        rf_coefs<F>(f2(u), f3(u), ns, b);
#pragma unroll
        for (int j = 0; j < CORE_NS; j++)
            if (j < ns) t[CT_B + j] = b[j].d[0];
    }
    if (time) {
        // k S0 = -Om + 2 eps C - 3 eps^2 Ox + 4 eps^3 OL, 3 m S0 = C - 3 eps Ox + 6 eps^2 OL (C = Ok + Os):
        // the recursion of finish() multiplied out
        const double ee = eps * eps, de = r.quartic ? dA * ee : 0.0;
        const double kv = r.k, mv = r.m;
        const double dk = (-d.dOm + 2.0 * eps * d.dOk - ee * (3.0 * d.dOx - 4.0 * eps * d.dOL)
                           + (2.0 * c - eps * (6.0 * Ox - 12.0 * eps * OL)) * de - kv * d.dS) * iS0;
        const double dm = (d.dOk - eps * (3.0 * d.dOx - 6.0 * eps * d.dOL) - (3.0 * Ox - 12.0 * eps * OL) * de
                           - 3.0 * mv * d.dS) * (iS0 * (1.0 / 3));
        put(t, CT_EPS, de);
        put(t, CT_K2, dk * (1.0 / 3));
        put(t, CT_K3, (d.dOL - OL * iS0 * d.dS) * iS0);
        if (once) {
            put(t, CT_M, dm);
        } else {
            F fm;
            const T u = dev_scale<T>(r.d5, ns);
            fm.v = (T)mv * u; fm.d[0] = (T)dm * u;
            rj_coefs<F>(fm, f2(u), f3(u), ns, b);
#pragma unroll
            for (int j = 0; j < CORE_NS; j++)
                if (j < ns) t[CT_A + j] = b[j].d[0];
        }
    }
    put(t, CT_END, 0.0);
}

}  // namespace lcdm
