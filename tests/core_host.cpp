// The core's arithmetic (csrc/lcdm_core.cuh, lcdm_corerec.cuh) compiled for the
// host: records from given roots, and the integrals with their gradients.
#define LCDM_HD inline
#define LCDM_NI inline
#include <cmath>
using std::fabs;
using std::fma;
using std::frexp;
using std::sqrt;
#include "lcdm_corerec.cuh"

using namespace lcdm;

static RowRoots row(const double* p, int ncol, int quartic, int cpair, const double* r) {
    RowRoots R;
    R.H0 = p[0]; R.Om = p[1]; R.OL = p[2]; R.Or = p[3];
    R.Ok = ncol >= 5 ? p[4] : 1.0 - p[1] - p[2] - p[3];
    R.Os = ncol >= 7 ? p[5] : 0.0;
    R.Ox = ncol >= 7 ? p[6] : 0.0;
    R.ncol = ncol; R.quartic = quartic; R.cpair = cpair;
    R.A = r[0]; R.B = r[1]; R.pr = r[2]; R.pi = r[3];
    R.finish();
    return R;
}

// out[n][4]: chi, t, X (in units of c/H0, 1/H0, c/H0), failed; grad[n][2][K] of chi and t
template <class T> static void pairs(const RowRoots& R, const double* dr, int n, const T* z, double* out, double* grad) {
    const int K = R.ncol - 1, ns = CoreTol<T>::ns;
    T rec[NCORE];
    core_values<T>(R, true, true, ns, rec);
    for (int k = 0; k < K; k++) core_tangent<T>(R, true, ns, k, dr[4 * k], dr[4 * k + 1], dr[4 * k + 2], dr[4 * k + 3], rec);
    for (int i = 0; i < n; i++) {
        int fail = 0;
        typedef CorePair<T, true, true, false> V;
        V v;
        typename V::Tape none;
        v.forward(z[i], rec, none, &fail);
        out[4 * i] = v.Ichi; out[4 * i + 1] = v.It; out[4 * i + 2] = v.X; out[4 * i + 3] = fail;
        typedef CorePair<T, true, false, true> G;
        for (int q = 0; q < 2; q++) {
            G g;
            typename G::Tape tape;
            g.forward(z[i], rec, tape, &fail);
            g.reverse((T)(q == 0), (T)(q == 1), tape);
            for (int k = 0; k < K; k++) grad[(2 * i + q) * K + k] = g.along(k) + (q ? g.It : g.Ichi) * rec[C_RS];
        }
    }
}

extern "C" void core_pairs(const double* p, int ncol, int quartic, int cpair, const double* roots, const double* dr, int fp64,
                           int n, const double* z, double* out, double* grad) {
    const RowRoots R = row(p, ncol, quartic, cpair, roots);
    if (fp64) {
        pairs<double>(R, dr, n, z, out, grad);
    } else {
        float* f = new float[n];
        for (int i = 0; i < n; i++) f[i] = (float)z[i];
        pairs<float>(R, dr, n, f, out, grad);
        delete[] f;
    }
}

// z -> infinity (double, closure rows): out[2] = chi, t; grad[2][3]
extern "C" void core_limit(const double* p, int quartic, int cpair, const double* roots, const double* dr, double* out,
                           double* grad) {
    const RowRoots R = row(p, 4, quartic, cpair, roots);
    double rec[NCORE];
    core_values<double>(R, true, false, CORE_NS_ONCE, rec);
    for (int k = 0; k < 3; k++)
        core_tangent<double>(R, true, CORE_NS_ONCE, k, dr[4 * k], dr[4 * k + 1], dr[4 * k + 2], dr[4 * k + 3], rec);
    typedef CorePair<double, true, false, true, true> E;
    for (int q = 0; q < 2; q++) {
        E e;
        E::Tape tape;
        int fail = 0;
        e.forward(1.0, rec, tape, &fail);
        e.reverse(q == 0, q == 1, tape);
        out[q] = fail ? 0.0 : (q ? e.It : e.Ichi);
        for (int k = 0; k < 3; k++) grad[3 * q + k] = e.along(k);
    }
}
