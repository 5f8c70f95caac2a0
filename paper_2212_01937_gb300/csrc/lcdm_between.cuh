// General integration limits (eqs. 2.3-2.5 from z1 to z2) and the upper
// limit at infinity, on top of the z1 = 0 path.
//
// For a lower limit z1 the substitution 1+z = (1+z1)(1+z') maps the integrals
// over [z1, z2] onto integrals over [0, z'] of a closed cosmology: with
// s = 1+z1 and E1 = E^2(z1),
//   Omega'_m = Omega_m s^3 / E1, Omega'_L = Omega_L / E1, Omega'_r = Omega_r s^4 / E1,
//   Omega'_k = Omega_k s^2 / E1, H0' = H0 sqrt(E1), z' = (z2 - z1) / s,
// the roots move to r' = (r - z1) / s, and
//   chi(z1, z2) = s chi'(0, z'),  t(z1, z2) = t'(0, z'),  d_abs(z1, z2) = s^3 d_abs'(0, z'),
//   d_M(z1, z2) = s d_M'(z'),  and d_L'(z') = (1+z2) d_M(z1, z2) / (1+z1)^2 is the
//   luminosity distance of a source at z2 seen by a comoving observer at z1.
// Substituted into the definitions of Sec. 3.1 this is eqs. (3.7)-(3.9) with
// X_m = sqrt(z2 - r_m), Y_m = sqrt(z1 - r_m), every factor of s cancelling:
// the same formulas, evaluated in the observer's own coordinate.  So the
// per-pair kernels run unchanged on the shifted cosmology (one row each) and
// small kernels here do the per-row shift, the per-pair map of z and of the
// cotangents, the output scaling, and the chain rule of the gradient.
//
// The shifted Omega' sum to one identically (E^2(z1) / E1), so the shifted
// row takes the closure form (H0', Om', OL', Or') with Ok' = 1 - Om' - OL' -
// Or', and the same three-direction tangents as a closure row: because
// sum_i dOmega'_i / dtheta = 0, the chain rule needs only the closure
// derivatives d/dOmega'_a - d/dOk' (a = m, L, r).
#pragma once
#include <cuda_runtime.h>
#include <math_constants.h>
#include <stdint.h>

#include "lcdm_core.cuh"

namespace lcdm {

struct ShiftArgs {
    const double* params;   // [B][ncol]
    const double* z1;       // [B]
    int64_t B;
    int ncol;
    double* jac;            // [B][4][ncol] d (H0', Om', OL', Or') / d params, optional
    double* scale;          // [B] s = 1 + z1 (NaN for an invalid row)
    float4* rowf;           // [B] (z1 hi, z1 lo, 1/s, s) in float32 for the FP32 pair maps
};

// The shifted row q = (H0', Om', OL', Or') of row b (closure form); `write`: also
// its Jacobian and constants.  Part of the root preparation (a kernel of its
// own took 7 us of the 97 of 4096 rows x 1024 pairs).
__device__ __forceinline__ void shift_row(const ShiftArgs& a, int64_t b, bool write, double* q) {
    const int nc = a.ncol;
    const double* p = a.params + b * nc;
    const double H0 = p[0], Om = p[1], OL = p[2], Or = p[3];
    const double Ok = nc == 5 ? p[4] : 1.0 - Om - OL - Or;
    const double z1 = a.z1[b];
    const double s = 1.0 + z1, s2 = s * s, s3 = s2 * s, s4 = s2 * s2;
    // E^2(z1), eq. (2.2); exactly 1 at z1 = 0 under the closure
    const double E1 = (z1 == 0.0 && nc == 4) ? 1.0 : Or * s4 + Om * s3 + Ok * s2 + OL;
    if (!(z1 >= 0.0) || !isfinite(z1) || !(E1 > 0.0) || !isfinite(E1)) {
        const double nan = CUDART_NAN;
        for (int i = 0; i < 4; i++) q[i] = nan;
        if (!write) return;
        if (a.jac)
            for (int i = 0; i < 4 * nc; i++) a.jac[b * 4 * nc + i] = nan;
        a.scale[b] = nan;
        a.rowf[b] = make_float4(nan, nan, nan, nan);
        return;
    }
    const double irE = E1 > 1e-280 && E1 < 1e280 ? rsq(E1) : 1.0 / sqrt(E1), rE = E1 * irE, iE = irE * irE;
    const double pw[4] = {s3, 1.0, s4, s2};       // powers of s for (Om, OL, Or, Ok)
    q[0] = H0 * rE;
    q[1] = Om * s3 * iE;
    q[2] = OL * iE;
    q[3] = Or * s4 * iE;
    if (!write) return;
    if (a.jac) {
        // derivatives: column 0 is H0; the Omega columns act on (Om, OL, Or[, Ok]),
        // with dOk = -1 for each of the first three under the closure
        double* J = a.jac + b * 4 * nc;
        J[0] = rE;
        for (int i = 0; i < 3; i++) J[(1 + i) * nc] = 0.0;
        for (int c = 1; c < nc; c++) {
            const double dE = pw[c - 1] - (nc == 4 ? s2 : 0.0);
            J[c] = 0.5 * H0 * dE * irE;
            for (int i = 0; i < 3; i++) J[(1 + i) * nc + c] = ((i == c - 1 ? pw[i] : 0.0) - q[1 + i] * dE) * iE;
        }
    }
    a.scale[b] = s;
    // z1 as an unevaluated float sum hi + lo, so that z2 - z1 and the sign test
    // z2 >= z1 come out right in float32 arithmetic when z2 is close to z1
    const float hi = (float)z1;
    a.rowf[b] = make_float4(hi, (float)(z1 - (double)hi), (float)rcp_(s), (float)s);
}

struct PairMapArgs {
    const int64_t* offsets; // CSR offsets, or null for the dense layout
    int64_t nrow;           // pairs per row (dense)
    int64_t nnz;
    int64_t B;
    int fp64;               // z, outputs and cotangents are float64 (else float32)
    const double* z1;       // [B]
    const double* scale;    // [B]
    const float4* rowf;     // [B] float32 row constants (FP32 maps)
    const void* z2;         // [nnz]
    void* zp;               // [nnz] z' = (z2 - z1) / s
    const void* cot[6];     // user cotangents
    void* cotp[6];          // mapped cotangents (d_C, X, d_M, mu; null = not needed)
    void* out[6];           // outputs scaled in place
};

struct LimitArgs {
    const double* rec;      // [B][NCORE] core records of the shifted cosmologies
    int32_t* status;
    int64_t B;
    const double* scale;
    double* chi;            // [B] chi(z1, inf), Mpc (may be null)
    double* age;            // [B] t(z1, inf), Gyr (may be null)
    const double* cot_chi;  // [B] (VJP; may be null)
    const double* cot_age;
    const double* jac;      // [B][4][ncol] d (shifted parameters) / d params (VJP)
    int ncol;
    double* grad;           // [B][ncol] (VJP)
};

cudaError_t launch_shift(const ShiftArgs& a, cudaStream_t s);
cudaError_t launch_pair_pre(const PairMapArgs& a, cudaStream_t s);
cudaError_t launch_pair_post(const PairMapArgs& a, cudaStream_t s);
cudaError_t launch_chain(const double* jac, const double* gradp, int64_t B, int ncol, double* grad,
                         cudaStream_t s);
cudaError_t launch_limits(const LimitArgs& a, bool tangents, cudaStream_t s);

}  // namespace lcdm
