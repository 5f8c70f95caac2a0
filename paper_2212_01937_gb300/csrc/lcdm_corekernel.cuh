// The pair kernel on the core (lcdm_core.cuh): values, vector-Jacobian
// products, the Gaussian log-likelihood, and Jacobians.
//
// Bound by instruction issue (FP32) or by the FP64 pipe: per pair some 250
// (values of d_C, t, mu) to 600 (with their gradient) instructions against
// 8 to 32 bytes of memory traffic.  One thread per pair, warps over
// contiguous ranges; a lane keeps its row's end and record pointer in
// registers and looks the row up only when it leaves it.
#pragma once
#include "lcdm_core.cuh"
#include "lcdm_kernels.cuh"

namespace lcdm {

// S_k(D) = D s(u), u = Ok D^2, s(u) = sum u^n / (2n+1)!; dS/dD = s + 2 u s',
// dS/dOk = D^3 s'.  One Horner pass gives s and s'; beyond the series' range
// (it cancels for u < -4, and needs more terms for large u) curv_map's closed
// forms.
template <class T> LCDM_HD void curv_core(T D, T Ok, bool want_d, T& S, T& SD, T& Sk) {
    const T u = Ok * D * D;
    constexpr bool F = sizeof(T) == 4;
    constexpr int NT = F ? 9 : 11;
    if (u <= (F ? (T)8 : (T)2) && u >= (F ? (T)-4 : (T)-2)) {
        constexpr double cs[11] = {1.0, 1.0 / 6, 1.0 / 120, 1.0 / 5040, 1.0 / 362880, 1.0 / 39916800,
                                   1.0 / 6227020800.0, 1.0 / 1307674368000.0, 1.0 / 355687428096000.0,
                                   1.0 / 121645100408832000.0, 1.0 / 51090942171709440000.0};
        T s = (T)cs[NT - 1], ds = 0;
#pragma unroll
        for (int i = NT - 2; i >= 0; i--) {
            if (want_d) ds = ds * u + s;
            s = (T)cs[i] + u * s;
        }
        S = D * s;
        SD = s + (T)2 * u * ds;
        Sk = D * D * D * ds;
        return;
    }
    curv_map<T>(D, Ok, S, SD, Sk);
}

// mu = 5 log10(d_L) + 25.  Single precision: the exponent's part and the special
// function unit's log2 of the mantissa in [sqrt(1/2), sqrt(2)), whose absolute
// error of 2^-22 there is a tenth of the last place of mu ~ 40 (applied to d_L
// itself it would be 2^-22 of a log2 of 14).  8 instructions; 15 with a series
// in (m - 1) / (m + 1), 3.63 against 3.58 ms for 1.4e8 pairs of mu and its
// gradient; rms error over z = 0.01 to 10 1.26e-6 mag against 1.28e-6, and
// 1.41e-6 with log10f.  Zero, negative and non-finite distances go to log10f.
LCDM_HD double mu_of(double dL) { return 5.0 * log10(dL) + 25.0; }
__device__ __forceinline__ float mu_of(float dL) {
    uint32_t b;
    memcpy(&b, &dL, sizeof b);
    if (b - 0x00800000u >= 0x7f000000u) return 5.0f * log10f(dL) + 25.0f;
    const int e = (int)(b - 0x3f3504f3u) >> 23;   // the mantissa in [sqrt(1/2), sqrt(2))
    const uint32_t mb = b - ((uint32_t)e << 23);
    float m;
    memcpy(&m, &mb, sizeof m);
    float l;
    asm("lg2.approx.ftz.f32 %0, %1;" : "=f"(l) : "f"(m));
    return fmaf((float)e, 1.50514997831990598f, fmaf(l, 1.50514997831990598f, 25.0f));
}

// acc += c.  Double-float: one error-free sum; its error joins the low word,
// which is not renormalised (it stays far below the high word's last place
// times the number of terms, and the flush adds both in double).
__device__ __forceinline__ void acc_add(double& a, double c) { a += c; }
__device__ __forceinline__ void acc_add(df64& a, float c) {
    const df64 s = two_sum(a.hi, c);
    a = mkdf(s.hi, LCDM_FADD(a.lo, s.lo));
}

// The map of a general-limits row: z' = (z2 - z1) / s.  Single precision: hi is
// exact near z1 (Sterbenz), and its sign decides the domain test; lo is z1 - hi
// rounded, which keeps the sign of the tie z2 == hi.
template <class T> struct LimitMap;
template <> struct LimitMap<float> {
    float hi, lo, is, s;
    __device__ __forceinline__ void load(const float4* rowf, const double*, const double*, int row) {
        const float4 r = __ldg(rowf + row);
        hi = r.x; lo = r.y; is = r.z; s = r.w;
    }
    __device__ __forceinline__ float dz(float z2) const { return (z2 - hi) - lo; }
    __device__ __forceinline__ float zp(float d) const { return d * is; }
};
template <> struct LimitMap<double> {
    double z1, s;
    __device__ __forceinline__ void load(const float4*, const double* z1s, const double* scale, int row) {
        z1 = __ldg(z1s + row); s = __ldg(scale + row);
    }
    __device__ __forceinline__ double dz(double z2) const { return z2 - z1; }
    __device__ __forceinline__ double zp(double d) const { return d / s; }
};

struct CoreArgs {
    PairArgs p;
    const void* rec;    // [B][NCORE]
    void* grad_z;       // [nnz] derivative with respect to each pair's redshift, optional
    const float4* rowf; // [B] (z1 hi, z1 lo, 1/s, s) of general limits (single precision)
    const double* z1;   // [B] lower limits, s = 1 + z1 (double precision)
    const double* scale;
};

// What a kernel produces beside the outputs: the per-row sums (of cotangents
// times derivatives, or of the log-likelihood), per-pair Jacobians, or the
// sums and the derivatives with respect to each redshift.  (Kernels of their
// own: the redshift derivatives cost the others 4 % in registers.)
// CORE_BETWEEN: the sums, for pairs given by an upper limit z2 above the row's
// own lower limit (general limits, lcdm_between.cuh): z' = (z2 - z1) / s, the
// outputs' factors and the domain test z2 >= z1 are applied here.  (Two maps
// over the pairs did that before: 0.04 ms of the 0.15 ms of 4 M values.)
enum CoreMode { CORE_SUM = 0, CORE_JAC = 1, CORE_DZ = 2, CORE_BETWEEN = 3 };

// Registers per thread: blocks of 256 threads per SM the compiler aims at.
// Single precision: one block more or less cost 2 to 10 % (0.78 -> 0.88 ms for
// the value and gradient kernels of 25 M pairs at 3 and 2 blocks, 0.83 at 6 and
// 5).  Double precision is bound by the FP64 pipe, which two warps per
// sub-partition fill: no cap (two blocks: 4 % slower by the spills).
template <int PREC, int K, bool WT, bool WX, int MODE>
struct CoreBlocks { enum { value = PREC == 1 ? (K == 0 ? (WX ? 3 : 4) : (MODE == CORE_JAC ? 2 : 3)) : 1 }; };

template <int PREC, int K, bool WT, bool WX, int MODE>
__global__ void __launch_bounds__(256, CoreBlocks<PREC, K, WT, WX, MODE>::value) core_kernel(CoreArgs ca) {
    constexpr bool JAC = MODE == CORE_JAC, DZ = MODE == CORE_DZ, BT = MODE == CORE_BETWEEN;
    typedef typename std::conditional<PREC == 0, double, float>::type T;
    typedef typename std::conditional<PREC == 0, double, df64>::type AccT;
    constexpr int NV = K + 2;   // H0, K density directions, log-likelihood
    const PairArgs& a = ca.p;
    const int lane = threadIdx.x & 31;
    const int64_t warp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int64_t start = warp * a.chunk;
    const int64_t end = max(start, min(start + a.chunk, a.nnz));
    const bool loglike = a.mobs != nullptr;
    const bool reduce = !JAC && ((a.grad != nullptr) || (a.loglike != nullptr));
    const T inv_sig = (T)(1.0 / a.sigma);
    const T lnorm = (T)(-log(a.sigma * 2.5066282746310002));
    const T Mobs = (T)a.M;
    const T c5 = (T)(5.0 / 2.302585092994045684);
    __shared__ AccT acc_s[JAC ? 1 : NV * ACC_STRIDE];
    AccT* acc = acc_s + (JAC ? 0 : threadIdx.x);
    if (reduce) {
#pragma unroll
        for (int i = 0; i < NV; i++) acc[i * ACC_STRIDE] = cst<AccT>(0.0);
    }
    int acc_row = -1;   // (a row's index fits 32 bits: its record alone takes 1040 bytes)
    int64_t wf = -1, wl = -1;
    if (a.part && reduce && warp < a.det_cap) {
        // deterministic reduction: the warp's first and last rows, its slots zeroed
        if (start < end) {
            wf = row_of(a, a.base + start);
            wl = row_of(a, a.base + end - 1);
        }
        if (lane < 2 * DET_SLOT) a.part[warp * 2 * DET_SLOT + lane] = 0.0;
        if (lane < 2) a.wrow[warp * 2 + lane] = lane == 0 ? wf : wl;
        __syncwarp();
        __threadfence_block();
    }
    // Within the warp's range everything is counted in 32 bits from its first
    // pair (a range of 2^31 pairs would not fit the memory).
    const int len = (int)(end - start), nb = (len + 31) / 32;
    const int s_it = a.interleave ? 1 : 32;
    const int64_t p0 = a.base + start;
    int row = -1, rend = INT32_MIN, zoff = 0;   // the lane's row, its end, and what takes a pair to its redshift (shared)
    const T* rec = nullptr;
    int st = 0;
    LimitMap<T> lm;
    // outputs that need the curvature map
    const bool map = loglike || (a.outmask & ((1 << O_DM) | (1 << O_DL) | (1 << O_MU))) ||
                     ((K > 0 || DZ) && (a.cot[O_DM] || a.cot[O_DL] || a.cot[O_MU] || a.jac[O_DM] || a.jac[O_DL] || a.jac[O_MU]));
    // Derivatives with respect to the redshift (the upper limit): by the
    // fundamental theorem the integrands there, from E(z) = sqrt(S0) n_A n_B |n_P|^2,
    //   d chi/dz = (c/H0)/E, d t/dz = 1/(H0 (1+z) E), d d_abs/dz = (c/H0)(1+z)^2/E,
    //   d d_M/dz = (c/H0) S_k'/E, d d_L/dz = d_M + (1+z) d d_M/dz,
    //   d mu/dz = 5/ln 10 (1/(1+z) + S_k'/(E S_k))  (0 at z = 0, where mu = -inf);
    // a kernel of its own read d_C, mu and the row again: 0.20 ms per 4 M pairs.
    T* const gz = DZ ? reinterpret_cast<T*>(ca.grad_z) + p0 : nullptr;
    const bool want_mu = loglike || (a.outmask & (1 << O_MU));
    const T* const zs = reinterpret_cast<const T*>(a.z) + p0;
    int off = a.interleave ? lane * nb : lane;
    for (int it = 0; it < nb; it++, off += s_it) {
        const bool active = off < len;
        const int o = active ? off : len - 1;
        if (o >= rend) {
            const int64_t pp = p0 + o;
            int64_t e;
            if (a.layout == LAYOUT_CSR) {
                int64_t r = row;
                if (r < 0) {
                    r = row_search(a.offsets, a.B, pp);
                } else {
                    int steps = 0;
                    while (r < a.B - 1 && __ldg(a.offsets + r + 1) <= pp && steps < 8) { r++; steps++; }
                    if (r < a.B - 1 && __ldg(a.offsets + r + 1) <= pp) r = row_search(a.offsets, a.B, pp);
                }
                row = (int)r;
                e = r < a.B - 1 ? __ldg(a.offsets + r + 1) - p0 : INT32_MAX;
            } else {
                const int64_t r = pp / a.nrow;
                row = (int)r;
                e = (r + 1) * a.nrow - p0;
                if (a.layout == LAYOUT_SHARED) zoff = row;
            }
            rend = e < INT32_MAX ? (int)e : INT32_MAX;
            rec = reinterpret_cast<const T*>(ca.rec) + (int64_t)row * NCORE;
            st = row_status(a.status, row);
            if (BT) lm.load(ca.rowf, ca.z1, ca.scale, row);
        }
        const int64_t zi = a.layout == LAYOUT_SHARED ? o - (int64_t)zoff * a.nrow : o;
        T z = __ldg(zs + zi);
        bool inside = true;   // (an interval with z2 < z1 gives NaN and adds nothing)
        if (BT) {
            const T d = lm.dz(z);
            inside = d >= (T)0;
            z = inside ? lm.zp(d) : (T)0;
        }
        T gcot[N_OUT];
        T mob = (T)0;
        if constexpr (K > 0 && !JAC) {
            // loaded ahead of the evaluation, which hides their latency
#pragma unroll
            for (int i = 0; i < N_OUT; i++)
                gcot[i] = (reduce && !loglike && a.cot[i] && i != O_X && (i != O_T || WT)) ? load_io<T>(a.cot[i], p0 + o) : (T)0;
        }
        if (!JAC && loglike) mob = __ldg(reinterpret_cast<const T*>(a.mobs) + p0 + zi);
        int fail = 0;
        const bool zero = z == (T)0;
        T c[NV];
#pragma unroll
        for (int i = 0; i < NV; i++) c[i] = 0;
        if (st == ST_OK) {
            typedef CorePair<T, WT, WX, (K > 0)> E;
            E e;
            typename E::Tape tape;
            e.forward(zero ? (T)1 : z, rec, tape, &fail);
            const T D = zero ? (T)0 : e.Ichi;
            const Quad<T> ku = quad(rec + C_DH);   // c/H0, 1/H0 [Gyr], 1/H0, Ok
            const T DH = ku.v[0], tH = ku.v[1], iH0 = ku.v[2];
            const T z1 = (T)1 + z;
            T S = 0, SD = 0, Sk = 0;
            if (map) curv_core<T>(D, ku.v[3], K > 0 || DZ, S, SD, Sk);
            T v[N_OUT];
            v[O_DC] = DH * D;
            v[O_T] = WT ? (zero ? (T)0 : tH * e.It) : (T)0;
            v[O_X] = WX ? (zero ? (T)0 : DH * e.X) : (T)0;
            v[O_DM] = DH * S;
            v[O_DL] = z1 * v[O_DM];
            v[O_MU] = want_mu ? mu_of(v[O_DL]) : (T)0;
            if (BT) {
                v[O_DC] = v[O_DC] * lm.s;
                v[O_DM] = v[O_DM] * lm.s;
                v[O_X] = v[O_X] * (lm.s * lm.s * lm.s);
            }
            if (fail || (BT && !inside)) {
                const T nan = (T)CUDART_NAN;
#pragma unroll
                for (int i = 0; i < N_OUT; i++) v[i] = nan;
                if (fail && active) atomicMax(a.status + row, (int)ST_NOCONV);
            }
            if (active) {
#pragma unroll
                for (int i = 0; i < N_OUT; i++)
                    if ((i != O_X || WX) && (i != O_T || WT) && (a.outmask & (1 << i)))
                        (reinterpret_cast<T*>(a.out[i]) + p0)[o] = v[i];
            }
            if (DZ && active) {
                const T iE = zero ? rec[C_C2] * (T)0.5 : e.inv_E();
                const T ix = rcp_(z1), dM = SD * iE;
                T g;
                if (loglike) {
                    const T r = (mob - v[O_MU] - Mobs) * inv_sig;
                    g = zero ? (T)0 : r * inv_sig * c5 * (ix + dM / S);
                } else {
                    auto ct = [&](int i) { return a.cot[i] ? load_io<T>(a.cot[i], p0 + o) : (T)0; };
                    g = DH * (ct(O_DC) * iE + ct(O_X) * (z1 * z1 * iE) + ct(O_DM) * dM + ct(O_DL) * (S + z1 * dM))
                        + tH * ct(O_T) * (iE * ix);
                    if (a.cot[O_MU]) g = g + (zero ? (T)0 : ct(O_MU) * c5 * (ix + dM / S));
                }
                gz[o] = fail ? (T)CUDART_NAN : g;
            }
            if constexpr (JAC) {
                // one reverse pass per integral, contracted with the tangents
                const T bad = fail ? (T)CUDART_NAN : (T)0;
                const int64_t pj = (p0 + o) * a.ncol;
                T dc[K];
                const bool jchi = a.jac[O_DC] || a.jac[O_DM] || a.jac[O_DL] || a.jac[O_MU];
                if (jchi) {
                    e.reverse((T)1, (T)0, tape);
                    const T fr = e.Ichi * rec[C_RS];
#pragma unroll
                    for (int k = 0; k < K; k++) dc[k] = zero ? (T)0 : e.along(k) + fr;
                    const T ism = c5 / S;
#pragma unroll
                    for (int i = 0; i < N_OUT; i++) {
                        if (i == O_T || i == O_X || !a.jac[i] || !active) continue;
                        T* jp = reinterpret_cast<T*>(a.jac[i]) + pj;
                        jp[0] = (i == O_MU ? -c5 * iH0 : -v[i] * iH0) + bad;
#pragma unroll
                        for (int k = 0; k < K; k++) {
                            const T dOk = a.ncol == 4 ? (T)-1 : (k == 3 ? (T)1 : (T)0);
                            T d = i == O_DC ? dc[k] : SD * dc[k] + Sk * dOk;
                            d = i == O_MU ? (zero ? (T)0 : d * ism) : d * (i == O_DL ? z1 * DH : DH);
                            jp[1 + k] = d + bad;
                        }
                    }
                }
                if (WT && a.jac[O_T]) {
                    e.reverse((T)0, (T)1, tape);
                    const T fr = e.It * rec[C_RS];
                    T* jp = reinterpret_cast<T*>(a.jac[O_T]) + pj;
                    T dt[K];
#pragma unroll
                    for (int k = 0; k < K; k++) dt[k] = zero ? (T)0 : tH * (e.along(k) + fr);
                    if (active) {
                        jp[0] = -v[O_T] * iH0 + bad;
#pragma unroll
                        for (int k = 0; k < K; k++) jp[1 + k] = dt[k] + bad;
                    }
                }
                continue;
            }
            if (reduce && active && !fail && inside) {
                T lin = 0, gm = 0;   // cotangent sums: of H0's linear outputs, of mu
                T ci = 0, cs = 0, ti = 0;
                if (loglike) {
                    const T r = (mob - v[O_MU] - Mobs) * inv_sig;
                    gm = r * inv_sig;
                    c[K + 1] = (T)-0.5 * r * r + lnorm;
                }
                if constexpr (K > 0) {
                    if (!loglike) {
                        if (BT) {
                            // (v holds the scaled outputs: their sum below keeps the plain cotangents)
                            lin = gcot[O_DC] * v[O_DC] + gcot[O_DM] * v[O_DM];
                            gcot[O_DC] = gcot[O_DC] * lm.s;
                            gcot[O_DM] = gcot[O_DM] * lm.s;
                        }
                        gm = gcot[O_MU];
                        cs = DH * (gcot[O_DM] + z1 * gcot[O_DL]);
                        ci = DH * gcot[O_DC];
                        if (WT) ti = tH * gcot[O_T];
                        if (!BT) lin = gcot[O_DC] * v[O_DC] + gcot[O_DM] * v[O_DM];
                        lin = lin + gcot[O_DL] * v[O_DL];
                        if (WT) lin = lin + gcot[O_T] * v[O_T];
                    }
                    c[0] = -(lin + c5 * gm) * iH0;
                    if (!zero && a.grad) {
                        if (gm != (T)0) cs = cs + gm * (c5 / S);
                        ci = ci + cs * SD;
                        e.reverse(ci, ti, tape);
                        const T fr = (e.Ichi * ci + (WT ? e.It * ti : (T)0)) * rec[C_RS];
                        const T co = cs * Sk;
#pragma unroll
                        for (int k = 0; k < K; k++) {
                            const T dOk = a.ncol == 4 ? (T)-1 : (k == 3 ? (T)1 : (T)0);
                            c[1 + k] = e.along(k) + fr + co * dOk;
                        }
                    }
                }
            }
        } else if (active) {
            const T nan = (T)CUDART_NAN;
#pragma unroll
            for (int i = 0; i < N_OUT; i++) {
                if (a.outmask & (1 << i)) (reinterpret_cast<T*>(a.out[i]) + p0)[o] = nan;
                if (DZ && i == 0) gz[o] = nan;
                if (JAC && a.jac[i]) {
                    T* jp = reinterpret_cast<T*>(a.jac[i]) + (p0 + o) * a.ncol;
                    for (int k = 0; k <= K; k++) jp[k] = nan;
                }
            }
        }
        if (!reduce) continue;
        // per-lane accumulation while the whole warp stays on one row
        const int r0 = __shfl_sync(0xffffffffu, row, 0);
        const bool uniform = __all_sync(0xffffffffu, row == r0);
        if (uniform && r0 == acc_row) {
            if (K > 0 && a.grad) {
#pragma unroll
                for (int i = 0; i <= K; i++) acc_add(acc[i * ACC_STRIDE], c[i]);
            }
            if (loglike) acc_add(acc[(K + 1) * ACC_STRIDE], c[K + 1]);
            continue;
        }
        if (acc_row >= 0) flush_row<NV, K>(acc, acc_row, a, lane, warp, wf, wl);
        if (uniform) {
#pragma unroll
            for (int i = 0; i < NV; i++) acc[i * ACC_STRIDE] = cst<AccT>(0.0) + c[i];
            acc_row = r0;
        } else {
            double cd_[NV];
#pragma unroll
            for (int i = 0; i < NV; i++) cd_[i] = (double)c[i];
            if (seg_reduce<NV>(cd_, row) && active) add_row(a, row, cd_, K + 1, warp, wf, wl);
#pragma unroll
            for (int i = 0; i < NV; i++) acc[i * ACC_STRIDE] = cst<AccT>(0.0);
            acc_row = -1;
        }
    }
    if (reduce && acc_row >= 0) flush_row<NV, K>(acc, acc_row, a, lane, warp, wf, wl);
}

// ------------------------------------------------- two pairs in a thread -----
// Per-lane sums of the two packed pairs, each double-float.
struct Acc2 { F2 hi, lo; };
template <> struct CstImpl<Acc2> {
    static LCDM_HD Acc2 make(double) { Acc2 a; a.hi = a.lo = mkf2(0.f, 0.f); return a; }
};
__device__ __forceinline__ double acc_to_double(Acc2 a) {
    return ((double)a.hi.x + (double)a.lo.x) + ((double)a.hi.y + (double)a.lo.y);
}
// a += c: Knuth's error-free sum of the high words, both at once
__device__ __forceinline__ void acc_add(Acc2& a, F2 c) {
    const F2 s = a.hi + c, bb = s - a.hi;
    const F2 e = (a.hi - (s - bb)) + (c - bb);
    a.hi = s;
    a.lo = a.lo + e;
}

__device__ __forceinline__ void curv_core(F2 D, float Ok, bool want_d, F2& S, F2& SD, F2& Sk) {
    const F2 u = mkf2(Ok, Ok) * (D * D);
    if (fmaxf(u.x, u.y) <= 8.f && fminf(u.x, u.y) >= -4.f) {
        constexpr double cs[9] = {1.0, 1.0 / 6, 1.0 / 120, 1.0 / 5040, 1.0 / 362880, 1.0 / 39916800,
                                  1.0 / 6227020800.0, 1.0 / 1307674368000.0, 1.0 / 355687428096000.0};
        F2 s = cst<F2>(cs[8]), ds = cst<F2>(0.0);
#pragma unroll
        for (int i = 7; i >= 0; i--) {
            if (want_d) ds = ds * u + s;
            s = cst<F2>(cs[i]) + u * s;
        }
        S = D * s;
        SD = s + cst<F2>(2.0) * u * ds;
        Sk = D * D * D * ds;
        return;
    }
    curv_core<float>(D.x, Ok, want_d, S.x, SD.x, Sk.x);
    curv_core<float>(D.y, Ok, want_d, S.y, SD.y, Sk.y);
}

// (one block more or less per SM: 2 and 33 % slower on 25 M pairs' values and
// gradients; with X two blocks, at 128 registers)
template <int K, bool WX> struct Core2Blocks { enum { value = K == 0 && !WX ? 3 : 2 }; };

// The single-precision sums and values with two pairs of a row in a thread:
// the arithmetic is that of core_kernel on packed numbers (F2), and what it
// does per pair beside arithmetic (the row, the record, the loop) is done once
// for two.  Bound by issue like core_kernel (75 % of cycles there, at 241
// instructions per pair of values and 527 with the gradient): 1.42e8 ragged
// pairs of mu and its gradient 4.43 -> 3.49 ms, 25 M pairs over a shared set
// 0.78 -> 0.62 ms, 1e8 pairs of d_C, t and X 3.18 -> 2.75 ms.  A warp takes two 32-pair batches at a time while every lane's two
// pairs lie in one row, else one (the second number is then a copy).
template <int K, bool WT, bool WX, int MODE>
__global__ void __launch_bounds__(256, Core2Blocks<K, WX>::value) core2_kernel(CoreArgs ca) {
    constexpr bool DZ = MODE == CORE_DZ, BT = MODE == CORE_BETWEEN;
    constexpr int NV = K + 2;
    constexpr unsigned full = 0xffffffffu;
    const PairArgs& a = ca.p;
    const int lane = threadIdx.x & 31;
    const int64_t warp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int64_t start = warp * a.chunk;
    const int64_t end = max(start, min(start + a.chunk, a.nnz));
    const bool loglike = a.mobs != nullptr;
    const bool reduce = (a.grad != nullptr) || (a.loglike != nullptr);
    const float inv_sig = (float)(1.0 / a.sigma);
    const float lnorm = (float)(-log(a.sigma * 2.5066282746310002));
    const float Mobs = (float)a.M;
    const float c5 = (float)(5.0 / 2.302585092994045684);
    __shared__ Acc2 acc_s[NV * ACC_STRIDE];
    Acc2* acc = acc_s + threadIdx.x;
    if (reduce) {
#pragma unroll
        for (int i = 0; i < NV; i++) acc[i * ACC_STRIDE] = cst<Acc2>(0.0);
    }
    int acc_row = -1;
    int64_t wf = -1, wl = -1;
    if (a.part && reduce && warp < a.det_cap) {
        if (start < end) {
            wf = row_of(a, a.base + start);
            wl = row_of(a, a.base + end - 1);
        }
        if (lane < 2 * DET_SLOT) a.part[warp * 2 * DET_SLOT + lane] = 0.0;
        if (lane < 2) a.wrow[warp * 2 + lane] = lane == 0 ? wf : wl;
        __syncwarp();
        __threadfence_block();
    }
    const int len = (int)(end - start), nb = (len + 31) / 32;
    const int s_it = a.interleave ? 1 : 32;
    const int64_t p0 = a.base + start;
    int row = -1, rend = INT32_MIN, zoff = 0;
    const float* rec = nullptr;
    int st = 0;
    LimitMap<float> lm;
    const bool map = loglike || (a.outmask & ((1 << O_DM) | (1 << O_DL) | (1 << O_MU))) ||
                     ((K > 0 || DZ) && (a.cot[O_DM] || a.cot[O_DL] || a.cot[O_MU]));
    float* const gz = DZ ? reinterpret_cast<float*>(ca.grad_z) + p0 : nullptr;
    const bool want_mu = loglike || (a.outmask & (1 << O_MU));
    const float* const zs = reinterpret_cast<const float*>(a.z) + p0;
    int off = a.interleave ? lane * nb : lane;
    for (int it = 0; it < nb;) {
        const bool act0 = off < len;
        const int o0 = act0 ? off : len - 1;
        if (o0 >= rend) {
            const int64_t pp = p0 + o0;
            int64_t e;
            if (a.layout == LAYOUT_CSR) {
                int64_t r = row;
                if (r < 0) {
                    r = row_search(a.offsets, a.B, pp);
                } else {
                    int steps = 0;
                    while (r < a.B - 1 && __ldg(a.offsets + r + 1) <= pp && steps < 8) { r++; steps++; }
                    if (r < a.B - 1 && __ldg(a.offsets + r + 1) <= pp) r = row_search(a.offsets, a.B, pp);
                }
                row = (int)r;
                e = r < a.B - 1 ? __ldg(a.offsets + r + 1) - p0 : INT32_MAX;
            } else {
                const int64_t r = pp / a.nrow;
                row = (int)r;
                e = (r + 1) * a.nrow - p0;
                if (a.layout == LAYOUT_SHARED) zoff = row;
            }
            rend = e < INT32_MAX ? (int)e : INT32_MAX;
            rec = reinterpret_cast<const float*>(ca.rec) + (int64_t)row * NCORE;
            st = row_status(a.status, row);
            if (BT) lm.load(ca.rowf, ca.z1, ca.scale, row);
        }
        const int off1 = off + s_it;
        const bool has1 = it + 1 < nb && off1 < len;
        const bool two = __all_sync(full, !has1 || off1 < rend);
        const bool act1 = two && has1;
        const int o1 = act1 ? off1 : o0;
        it += two ? 2 : 1;
        off += two ? 2 * s_it : s_it;
        const int64_t zb = a.layout == LAYOUT_SHARED ? (int64_t)zoff * a.nrow : 0;
        F2 z = mkf2(__ldg(zs + (o0 - zb)), __ldg(zs + (o1 - zb)));
        bool in0 = true, in1 = true;
        if (BT) {
            const float d0 = lm.dz(z.x), d1 = lm.dz(z.y);
            in0 = d0 >= 0.f;
            in1 = d1 >= 0.f;
            z = mkf2(in0 ? lm.zp(d0) : 0.f, in1 ? lm.zp(d1) : 0.f);
        }
        F2 gcot[N_OUT];
        F2 mob = mkf2(0.f, 0.f);
        auto cotangent = [&](int i) {
            return mkf2(load_io<float>(a.cot[i], p0 + o0), load_io<float>(a.cot[i], p0 + o1));
        };
        if constexpr (K > 0) {
#pragma unroll
            for (int i = 0; i < N_OUT; i++)
                gcot[i] = (reduce && !loglike && a.cot[i] && i != O_X && (i != O_T || WT)) ? cotangent(i) : mkf2(0.f, 0.f);
        }
        if (loglike) {
            const float* mo = reinterpret_cast<const float*>(a.mobs) + p0;
            mob = mkf2(__ldg(mo + (o0 - zb)), __ldg(mo + (o1 - zb)));
        }
        F2 c[NV];
#pragma unroll
        for (int i = 0; i < NV; i++) c[i] = mkf2(0.f, 0.f);
        if (st == ST_OK) {
            int fail = 0;
            const bool z0 = z.x == 0.f, z1_ = z.y == 0.f;
            typedef CorePair<F2, WT, WX, (K > 0)> E;
            E e;
            typename E::Tape tape;
            e.forward(mkf2(z0 ? 1.f : z.x, z1_ ? 1.f : z.y), rec, tape, &fail);
            auto zeroed = [&](F2 v) { return mkf2(z0 ? 0.f : v.x, z1_ ? 0.f : v.y); };
            const F2 D = zeroed(e.Ichi);
            const Quad<float> ku = quad(rec + C_DH);   // c/H0, 1/H0 [Gyr], 1/H0, Ok
            const F2 DH = mkf2(ku.v[0], ku.v[0]), tH = mkf2(ku.v[1], ku.v[1]), iH0 = mkf2(ku.v[2], ku.v[2]);
            const F2 z1 = cst<F2>(1.0) + z;
            F2 S = mkf2(0.f, 0.f), SD = S, Sk = S;
            if (map) curv_core(D, ku.v[3], K > 0 || DZ, S, SD, Sk);
            F2 v[N_OUT];
            v[O_DC] = DH * D;
            v[O_T] = WT ? zeroed(tH * e.It) : mkf2(0.f, 0.f);
            v[O_X] = WX ? zeroed(DH * e.X) : mkf2(0.f, 0.f);
            v[O_DM] = DH * S;
            v[O_DL] = z1 * v[O_DM];
            v[O_MU] = want_mu ? mkf2(mu_of(v[O_DL].x), mu_of(v[O_DL].y)) : mkf2(0.f, 0.f);
            if (BT) {
                const F2 s = mkf2(lm.s, lm.s);
                v[O_DC] = v[O_DC] * s;
                v[O_DM] = v[O_DM] * s;
                v[O_X] = v[O_X] * (s * s * s);
            }
            if (fail || (BT && !(in0 && in1))) {
                const float nan = CUDART_NAN_F;
                const bool b0 = (fail & 1) || !in0, b1 = (fail & 2) || !in1;
#pragma unroll
                for (int i = 0; i < N_OUT; i++) v[i] = mkf2(b0 ? nan : v[i].x, b1 ? nan : v[i].y);
                if (((fail & 1) && act0) || ((fail & 2) && act1)) atomicMax(a.status + row, (int)ST_NOCONV);
            }
#pragma unroll
            for (int i = 0; i < N_OUT; i++)
                if ((i != O_X || WX) && (i != O_T || WT) && (a.outmask & (1 << i))) {
                    float* p = reinterpret_cast<float*>(a.out[i]) + p0;
                    if (act0) p[o0] = v[i].x;
                    if (act1) p[o1] = v[i].y;
                }
            if (DZ) {
                const float i0 = rec[C_C2] * 0.5f;
                F2 iE = e.inv_E();
                iE = mkf2(z0 ? i0 : iE.x, z1_ ? i0 : iE.y);
                const F2 ix = rcp_(z1), dM = SD * iE;
                F2 g;
                if (loglike) {
                    const F2 r = (mob - v[O_MU] - mkf2(Mobs, Mobs)) * mkf2(inv_sig, inv_sig);
                    g = zeroed(r * mkf2(inv_sig * c5, inv_sig * c5) * (ix + dM * rcp_(S)));
                } else {
                    auto ct = [&](int i) { return a.cot[i] ? cotangent(i) : mkf2(0.f, 0.f); };
                    g = DH * (ct(O_DC) * iE + ct(O_X) * (z1 * z1 * iE) + ct(O_DM) * dM + ct(O_DL) * (S + z1 * dM))
                        + tH * ct(O_T) * (iE * ix);
                    if (a.cot[O_MU]) g = g + zeroed(ct(O_MU) * mkf2(c5, c5) * (ix + dM * rcp_(S)));
                }
                if (act0) gz[o0] = (fail & 1) ? CUDART_NAN_F : g.x;
                if (act1) gz[o1] = (fail & 2) ? CUDART_NAN_F : g.y;
            }
            const bool m0 = act0 && !(fail & 1) && in0, m1 = act1 && !(fail & 2) && in1;
            if (reduce && (m0 || m1)) {
                F2 lin = mkf2(0.f, 0.f), gm = lin, ci = lin, cs = lin, ti = lin;
                auto masked = [&](F2 w) { return mkf2(m0 ? w.x : 0.f, m1 ? w.y : 0.f); };
                if (loglike) {
                    const F2 r = (mob - v[O_MU] - mkf2(Mobs, Mobs)) * mkf2(inv_sig, inv_sig);
                    gm = r * mkf2(inv_sig, inv_sig);
                    c[K + 1] = masked(cst<F2>(-0.5) * r * r + mkf2(lnorm, lnorm));
                }
                if constexpr (K > 0) {
                    if (!loglike) {
                        lin = gcot[O_DC] * v[O_DC] + gcot[O_DM] * v[O_DM] + gcot[O_DL] * v[O_DL];
                        if (BT) {
                            // (v holds the scaled outputs)
                            const F2 s = mkf2(lm.s, lm.s);
                            gcot[O_DC] = gcot[O_DC] * s;
                            gcot[O_DM] = gcot[O_DM] * s;
                        }
                        gm = gcot[O_MU];
                        cs = DH * (gcot[O_DM] + z1 * gcot[O_DL]);
                        ci = DH * gcot[O_DC];
                        if (WT) {
                            ti = tH * gcot[O_T];
                            lin = lin + gcot[O_T] * v[O_T];
                        }
                    }
                    c[0] = masked(-((lin + mkf2(c5, c5) * gm) * iH0));
                    const bool n0 = m0 && !z0, n1 = m1 && !z1_;
                    if (a.grad && (n0 || n1)) {
                        if (gm.x != 0.f || gm.y != 0.f) {
                            const F2 q = gm * (mkf2(c5, c5) * rcp_(S));
                            cs = cs + mkf2(gm.x != 0.f ? q.x : 0.f, gm.y != 0.f ? q.y : 0.f);
                        }
                        ci = ci + cs * SD;
                        e.reverse(ci, ti, tape);
                        F2 fr = e.Ichi * ci;
                        if (WT) fr = fr + e.It * ti;
                        fr = fr * mkf2(rec[C_RS], rec[C_RS]);
                        const F2 co = cs * Sk;
#pragma unroll
                        for (int k = 0; k < K; k++) {
                            const float dOk = a.ncol == 4 ? -1.f : (k == 3 ? 1.f : 0.f);
                            const F2 w = e.along(k) + fr + co * mkf2(dOk, dOk);
                            c[1 + k] = mkf2(n0 ? w.x : 0.f, n1 ? w.y : 0.f);
                        }
                    }
                }
            }
        } else {
            const float nan = CUDART_NAN_F;
#pragma unroll
            for (int i = 0; i < N_OUT; i++) {
                if (a.outmask & (1 << i)) {
                    float* p = reinterpret_cast<float*>(a.out[i]) + p0;
                    if (act0) p[o0] = nan;
                    if (act1) p[o1] = nan;
                }
            }
            if (DZ) {
                if (act0) gz[o0] = nan;
                if (act1) gz[o1] = nan;
            }
        }
        if (!reduce) continue;
        const int r0 = __shfl_sync(full, row, 0);
        const bool uniform = __all_sync(full, row == r0);
        if (uniform && r0 == acc_row) {
            if (K > 0 && a.grad) {
#pragma unroll
                for (int i = 0; i <= K; i++) acc_add(acc[i * ACC_STRIDE], c[i]);
            }
            if (loglike) acc_add(acc[(K + 1) * ACC_STRIDE], c[K + 1]);
            continue;
        }
        if (acc_row >= 0) flush_row<NV, K>(acc, acc_row, a, lane, warp, wf, wl);
        if (uniform) {
#pragma unroll
            for (int i = 0; i < NV; i++) {
                Acc2 f = cst<Acc2>(0.0);
                f.hi = c[i];
                acc[i * ACC_STRIDE] = f;
            }
            acc_row = r0;
        } else {
            double cd_[NV];
#pragma unroll
            for (int i = 0; i < NV; i++) cd_[i] = (double)c[i].x + (double)c[i].y;
            if (seg_reduce<NV>(cd_, row) && act0) add_row(a, row, cd_, K + 1, warp, wf, wl);
#pragma unroll
            for (int i = 0; i < NV; i++) acc[i * ACC_STRIDE] = cst<Acc2>(0.0);
            acc_row = -1;
        }
    }
    if (reduce && acc_row >= 0) flush_row<NV, K>(acc, acc_row, a, lane, warp, wf, wl);
}

// Rows in which a pair's duplication did not converge (a non-finite redshift)
// have a bad status: all their redshift derivatives are NaN.  One warp per row.
template <class T> __global__ void nan_rows_kernel(PairArgs a, T* gz) {
    const int64_t row = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    if (row >= a.B || a.status[row] != ST_NOCONV) return;
    const int64_t p0 = a.layout == LAYOUT_CSR ? a.offsets[row] : row * a.nrow;
    const int64_t p1 = a.layout == LAYOUT_CSR ? a.offsets[row + 1] : p0 + a.nrow;
    for (int64_t p = p0 + (threadIdx.x & 31); p < p1; p += 32) gz[p] = (T)CUDART_NAN;
}

}  // namespace lcdm
