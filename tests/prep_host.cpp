// The root preparation (csrc/lcdm_prep.cuh), one lane per cosmology, and the
// core on its records, compiled for the host.  The device's built-ins are
// stood in for by their meaning in a warp of one lane.
#define LCDM_HD inline
#define LCDM_NI inline
#include <cmath>
#include <cstdint>
#include <cstring>
using std::fabs;
using std::fma;
using std::frexp;
using std::hypot;
using std::isfinite;
using std::nan;
using std::sqrt;
#include <cuda_runtime.h>
#undef __noinline__
#define __noinline__
#define __launch_bounds__(...)

static struct { unsigned x; } threadIdx, blockIdx, blockDim;
template <class T> static T __ldg(const T* p) { return *p; }
template <class T> static T __shfl_sync(unsigned, T v, int, int = 32) { return v; }
template <class T> static T __shfl_xor_sync(unsigned, T v, int, int = 32) { return v; }
template <class T> static T __shfl_down_sync(unsigned, T v, int, int = 32) { return v; }
template <class T> static T __shfl_up_sync(unsigned, T v, int, int = 32) { return v; }
static int __all_sync(unsigned, int v) { return v; }
static unsigned __ballot_sync(unsigned, int v) { return v; }
static int __clz(int v) { return v ? __builtin_clz(v) : 32; }
static int __ffs(unsigned v) { return __builtin_ffs(v); }
static void __syncwarp(unsigned = 0) {}
static void __syncthreads() {}
static void __threadfence_block() {}
template <class T> static T atomicMax(T* p, T v) { const T o = *p; *p = v > o ? v : o; return o; }
template <class T> static T atomicAdd(T* p, T v) { const T o = *p; *p += v; return o; }
static long long __double_as_longlong(double d) { long long r; memcpy(&r, &d, 8); return r; }
static double __longlong_as_double(long long d) { double r; memcpy(&r, &d, 8); return r; }
static int __float_as_int(float f) { int r; memcpy(&r, &f, 4); return r; }
static float __int_as_float(int i) { float r; memcpy(&r, &i, 4); return r; }
template <class T> static T min(T a, T b) { return a < b ? a : b; }
template <class T> static T max(T a, T b) { return a > b ? a : b; }
#include "lcdm_prep.cuh"

using namespace lcdm;

// status[B], kind[B] (0 quartic with a pair, 1 four reals, 2 cubic with a pair,
// 3 three reals), roots[B][4] in x = 1 + z (A, B, the pair: re, im or the two)
extern "C" void prep_rows(const double* p, int64_t B, int ncol, float near, int32_t* status, int32_t* kind, double* roots) {
    for (int64_t b = 0; b < B; b++) {
        RowRoots r;
        cd dr[4][RF_KT];
        bool labelled;
        memset(&r, 0, sizeof r);
        status[b] = prep_roots<1>(p + b * ncol, ncol, true, 1, near, r, dr, labelled);
        kind[b] = (r.quartic ? 0 : 2) + (r.cpair ? 0 : 1);
        roots[4 * b] = r.A; roots[4 * b + 1] = r.B; roots[4 * b + 2] = r.pr; roots[4 * b + 3] = r.pi;
    }
}

template <class T> static void values(const RowRoots& r, int n, const double* z, double* out) {
    T rec[NCORE];
    core_values<T>(r, true, true, CoreTol<T>::ns, rec);
    for (int i = 0; i < n; i++) {
        CorePair<T, true, true, false> e;
        typename CorePair<T, true, true, false>::Tape tape;
        int fail = 0;
        e.forward((T)z[i], rec, tape, &fail);
        out[4 * i] = e.Ichi; out[4 * i + 1] = e.It; out[4 * i + 2] = e.X; out[4 * i + 3] = fail;
    }
}

// one row from its parameters: out[n][4] = chi, t, X (in c/H0, 1/H0, c/H0), failed; returns the status
extern "C" int prep_pairs(const double* p, int ncol, int fp64, int n, const double* z, double* out) {
    RowRoots r;
    cd dr[4][RF_KT];
    bool labelled;
    const int st = prep_roots<1>(p, ncol, true, 0, fp64 ? 0.1f : 0.01f, r, dr, labelled);
    if (st != ST_OK) return st;
    r.finish();
    if (fp64) values<double>(r, n, z, out);
    else values<float>(r, n, z, out);
    return st;
}
