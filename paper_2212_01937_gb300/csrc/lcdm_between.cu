// Kernels of the general-limits path (see lcdm_between.cuh): the per-row
// shift of the parameters, the per-pair maps, the gradient chain rule, and
// the upper limit at infinity (age and horizon, FP64, one thread per row).
#include <math_constants.h>

#include "lcdm_between.cuh"
#include "lcdm_core.cuh"
#include "lcdm_kernels.cuh"

namespace lcdm {

// The row shift alone, for the per-pair maps.
__global__ void shift_kernel(ShiftArgs a) {
    const int64_t b = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (b >= a.B) return;
    double q[4];
    shift_row(a, b, true, q);
}

cudaError_t launch_shift(const ShiftArgs& a, cudaStream_t s) {
    if (a.B <= 0) return cudaSuccess;
    shift_kernel<<<(unsigned)((a.B + 127) / 128), 128, 0, s>>>(a);
    return cudaGetLastError();
}

// ------------------------------------------------------- per-pair maps -----
// (where X has tangents; other plans map in the pair kernel, see LimitMap)
// Each warp takes a contiguous run of pairs, lane l every 32nd pair from l
// (coalesced); the row of a lane's first pair comes from a binary search of
// the CSR offsets, later rows from stepping forward.
struct RowWalk {
    const int64_t* off;
    int64_t B, nrow, row;
    __device__ int64_t at(int64_t p) {
        if (!off) {
            if (row < 0) row = p / nrow;
            while ((row + 1) * nrow <= p) row++;
            return row;
        }
        if (row < 0) {
            int64_t lo = 0, hi = B;   // off[lo] <= p < off[hi]
            while (hi - lo > 1) {
                int64_t mid = (lo + hi) >> 1;
                if (__ldg(off + mid) <= p) lo = mid; else hi = mid;
            }
            row = lo;
        }
        while (row < B - 1 && __ldg(off + row + 1) <= p) row++;
        return row;
    }
};

#define LCDM_MAP_BLOCK 256
#define LCDM_MAP_BLOCKS_PER_SM 8

__device__ __forceinline__ void warp_run(int64_t nnz, int64_t& p0, int64_t& p1) {
    const int64_t nw = (int64_t)gridDim.x * (blockDim.x / 32);
    const int64_t w = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) / 32;
    int64_t chunk = (nnz + nw - 1) / nw;
    chunk = (chunk + 31) / 32 * 32;
    p0 = min(nnz, w * chunk);
    p1 = min(nnz, p0 + chunk);
}

// z' = (z2 - z1) / s, the domain test z2 >= z1, and the output / cotangent
// factors (s for d_C and d_M, s^3 for d_abs, 1 otherwise), in the pass type
template <class T> struct RowMap;
template <> struct RowMap<float> {
    float hi, lo, is, s;
    __device__ RowMap(const PairMapArgs& a, int64_t b) {
        const float4 r = a.rowf[b];
        hi = r.x; lo = r.y; is = r.z; s = r.w;
    }
    // (z2 - hi) is exact near z1 (Sterbenz) and its sign is exact; lo is
    // |z1 - hi| rounded, which keeps the sign of the tie z2 == hi
    __device__ float dz(float z2) const { return (z2 - hi) - lo; }
    __device__ float zp(float d) const { return d * is; }
    __device__ float f(int o) const { return o == 2 ? s * s * s : ((o == 0 || o == 3) ? s : 1.0f); }
};
template <> struct RowMap<double> {
    double z1, s;
    __device__ RowMap(const PairMapArgs& a, int64_t b) : z1(a.z1[b]), s(a.scale[b]) {}
    __device__ double dz(double z2) const { return z2 - z1; }
    __device__ double zp(double d) const { return d / s; }
    __device__ double f(int o) const { return o == 2 ? s * s * s : ((o == 0 || o == 3) ? s : 1.0); }
};

template <class T> __global__ void __launch_bounds__(LCDM_MAP_BLOCK) pair_pre_kernel(PairMapArgs a) {
    int64_t p0, p1;
    warp_run(a.nnz, p0, p1);
    RowWalk rw{a.offsets, a.B, a.nrow, -1};
    for (int64_t p = p0 + (threadIdx.x & 31); p < p1; p += 32) {
        const RowMap<T> m(a, rw.at(p));
        const T d = m.dz(reinterpret_cast<const T*>(a.z2)[p]);
        // an interval with z2 < z1 is outside the domain: evaluated at z' = 0,
        // its outputs are set to NaN afterwards and it adds nothing to the gradient
        const bool ok = d >= (T)0;
        reinterpret_cast<T*>(a.zp)[p] = ok ? m.zp(d) : (T)0;
#pragma unroll
        for (int o = 0; o < 6; o++)
            if (a.cotp[o]) {
                const T g = reinterpret_cast<const T*>(a.cot[o])[p];
                reinterpret_cast<T*>(a.cotp[o])[p] = ok ? m.f(o) * g : (T)0;
            }
    }
}

template <class T> __global__ void __launch_bounds__(LCDM_MAP_BLOCK) pair_post_kernel(PairMapArgs a) {
    int64_t p0, p1;
    warp_run(a.nnz, p0, p1);
    RowWalk rw{a.offsets, a.B, a.nrow, -1};
    for (int64_t p = p0 + (threadIdx.x & 31); p < p1; p += 32) {
        const RowMap<T> m(a, rw.at(p));
        const bool ok = m.dz(reinterpret_cast<const T*>(a.z2)[p]) >= (T)0;
        // t, d_L and mu need no factor: they are touched only to mark a pair
        // outside the domain
#pragma unroll
        for (int o = 0; o < 6; o++)
            if (a.out[o]) {
                T* v = reinterpret_cast<T*>(a.out[o]) + p;
                if (!ok) *v = (T)CUDART_NAN;
                else if (o == 0 || o == 2 || o == 3) *v = m.f(o) * *v;
            }
    }
}

static unsigned map_grid(int64_t nnz) {
    int dev = 0, sms = 1;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    const int64_t need = (nnz + LCDM_MAP_BLOCK - 1) / LCDM_MAP_BLOCK, cap = (int64_t)sms * LCDM_MAP_BLOCKS_PER_SM;
    return (unsigned)(need < cap ? (need > 0 ? need : 1) : cap);
}

cudaError_t launch_pair_pre(const PairMapArgs& a, cudaStream_t s) {
    if (a.nnz <= 0) return cudaSuccess;
    if (a.fp64) pair_pre_kernel<double><<<map_grid(a.nnz), LCDM_MAP_BLOCK, 0, s>>>(a);
    else pair_pre_kernel<float><<<map_grid(a.nnz), LCDM_MAP_BLOCK, 0, s>>>(a);
    return cudaGetLastError();
}

cudaError_t launch_pair_post(const PairMapArgs& a, cudaStream_t s) {
    if (a.nnz <= 0) return cudaSuccess;
    if (a.fp64) pair_post_kernel<double><<<map_grid(a.nnz), LCDM_MAP_BLOCK, 0, s>>>(a);
    else pair_post_kernel<float><<<map_grid(a.nnz), LCDM_MAP_BLOCK, 0, s>>>(a);
    return cudaGetLastError();
}

// ------------------------------------------------------ gradient chain -----
// grad[c] = sum_a gradp[a] d params4[a] / d params[c] of one row.  Entries
// with a zero Jacobian are skipped, so that the NaN Omega_r' component of a
// radiationless row (no such direction in the cubic) reaches only the
// Omega_r column, as on the z1 = 0 path.
__device__ __forceinline__ void chain_row(const double* J, const double* g, int ncol, double* grad) {
    for (int c = 0; c < ncol; c++) {
        double acc = 0.0;
        for (int i = 0; i < 4; i++) {
            const double j = J[i * ncol + c];
            if (j != 0.0) acc += g[i] * j;
        }
        grad[c] = acc;
    }
}

__global__ void chain_kernel(const double* __restrict__ jac, const double* __restrict__ gradp, int64_t B,
                             int ncol, double* __restrict__ grad) {
    const int64_t b = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (b >= B) return;
    chain_row(jac + b * 4 * ncol, gradp + b * 4, ncol, grad + b * ncol);
}

cudaError_t launch_chain(const double* jac, const double* gradp, int64_t B, int ncol, double* grad,
                         cudaStream_t s) {
    if (B <= 0) return cudaSuccess;
    chain_kernel<<<(unsigned)((B + 127) / 128), 128, 0, s>>>(jac, gradp, B, ncol, grad);
    return cudaGetLastError();
}

// ------------------------------------------------- upper limit at infinity -
// One thread per row of the shifted cosmology: chi'(0, inf) and t'(0, inf)
// in FP64, with the closure gradient w.r.t. (Om', OL', Or') by one reverse
// pass when GRAD.  Bound by the FP64 pipe.
template <bool GRAD> __global__ void __launch_bounds__(128) limits_kernel(LimitArgs a) {
    const int64_t b = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (b >= a.B) return;
    const double* rec = a.rec + b * NCORE;
    const double nan = CUDART_NAN;
    double chi = nan, age = nan;
    int st = a.status[b];
    if (st == ST_OK) {
        typedef CorePair<double, true, false, GRAD, true> E;
        E e;
        typename E::Tape tape;
        int fail = 0;
        e.forward(1.0, rec, tape, &fail);
        const double s = a.scale[b], DH = rec[C_DH], tH = rec[C_TH];
        if (fail) {
            a.status[b] = st = ST_NOCONV;
        } else {
            chi = s * DH * e.Ichi;
            age = tH * e.It;
            if (GRAD) {
                const double gc = a.cot_chi ? a.cot_chi[b] : 0.0, ga = a.cot_age ? a.cot_age[b] : 0.0;
                double g[4];
                g[0] = -(gc * chi + ga * age) * rec[C_IH0];
                e.reverse(gc * s * DH, ga * tH, tape);
                for (int k = 0; k < 3; k++) g[1 + k] = e.along(k);
                chain_row(a.jac + b * 4 * a.ncol, g, a.ncol, a.grad + b * a.ncol);
            }
        }
    }
    if (st != ST_OK && GRAD)
        for (int k = 0; k < a.ncol; k++) a.grad[b * a.ncol + k] = nan;
    if (a.chi) a.chi[b] = chi;
    if (a.age) a.age[b] = age;
}

cudaError_t launch_limits(const LimitArgs& a, bool tangents, cudaStream_t s) {
    if (a.B <= 0) return cudaSuccess;
    const unsigned grid = (unsigned)((a.B + 127) / 128);
    if (tangents) limits_kernel<true><<<grid, 128, 0, s>>>(a);
    else limits_kernel<false><<<grid, 128, 0, s>>>(a);
    return cudaGetLastError();
}

}  // namespace lcdm
