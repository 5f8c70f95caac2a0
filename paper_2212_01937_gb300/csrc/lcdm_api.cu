// Host side of liblcdm: argument checks, workspace carving, launch shapes,
// the launch-shape autotuner, and the extern "C" entry points of include/lcdm.h.
#include <atomic>
#include <cmath>
#include <map>
#include <mutex>
#include <tuple>

#include "../../include/lcdm.h"
#include "lcdm_between.cuh"
#include "lcdm_launch.cuh"
#include "lcdm_prep.cuh"

using namespace lcdm;

namespace {

std::atomic<int64_t> g_launches{0};

size_t align256(size_t x) { return (x + 255) & ~size_t(255); }

// largest batch whose root preparation uses four lanes per cosmology
#define LCDM_PREP_GROUP_MAX_B 16384

// Row records: those of the core (NCORE floats or doubles per row), and beside
// them those of the X-tangent kernel (FP64, in single precision also their (hi,
// lo) copy): a call that differentiates X and has other work on the core uses
// both from one preparation.
size_t core_bytes(int64_t B, int prec) { return align256((size_t)B * NCORE * (prec == 0 ? sizeof(double) : sizeof(float))); }
size_t record_bytes(int64_t B, int prec) {
    return core_bytes(B, prec) + align256((size_t)B * NREC * sizeof(double)) +
           (prec == 1 ? align256((size_t)B * NREC * sizeof(float2)) : 0);
}
// (one size for either precision)
size_t ws_bytes_for(int64_t B) {
    const size_t d = record_bytes(B, 0), f = record_bytes(B, 1);
    return d > f ? d : f;
}
int prec_of(const lcdm_opts* o) { return o->precision == LCDM_FP64 ? 0 : 1; }

bool opts_ok(const lcdm_opts* o) {
    return o && (o->ncol == 4 || o->ncol == 5 || o->ncol == 7) &&
           (o->precision == LCDM_FP64 || o->precision == LCDM_FP32_MIXED) &&
           o->layout >= LCDM_LAYOUT_CSR && o->layout <= LCDM_LAYOUT_SHARED && o->block >= 0 && o->block <= 256 &&
           (o->block % 32) == 0 && o->blocks_per_sm >= 0 && o->blocks_per_sm <= 64 && o->lane_map >= LCDM_MAP_TUNED &&
           o->lane_map <= LCDM_MAP_INTERLEAVED && (o->deterministic == 0 || o->deterministic == 1);
}

int num_sms();

// Partial sums of the deterministic reduction: per launched warp, the sums
// of its first and last rows (DET_NV values each) and those rows' indices.
// At most 64 resident warps per SM are ever launched.
#define DET_NV (RF_KT + 2)
size_t det_warps() { return (size_t)64 * num_sms(); }
size_t det_bytes() {
    return align256(det_warps() * 2 * DET_NV * sizeof(double)) + align256(det_warps() * 2 * sizeof(int64_t));
}

struct Carved {
    char* core;                  // the core's records
    double* recD;                // those of the X-tangent kernel
    float2* recF;                // (null in double precision)
    double* part = nullptr;      // deterministic mode: [warps][2][DET_NV]
    int64_t* wrow = nullptr;     // [warps][2]
};

Carved carve_records(char* p, int64_t B, int prec) {
    Carved c;
    c.core = p;
    c.recD = p ? (double*)(p + core_bytes(B, prec)) : nullptr;
    c.recF = p && prec == 1 ? (float2*)((char*)c.recD + align256((size_t)B * NREC * sizeof(double))) : nullptr;
    return c;
}

// need: the bytes the call asks of its workspace, 0: those of every record
lcdm_status carve(void* ws, size_t ws_bytes, int64_t B, int prec, Carved& c, int det = 0, size_t need = 0) {
    const size_t rec = ws_bytes_for(B);
    if (need == 0) need = rec + (det ? det_bytes() : 0);
    if (!ws || ((uintptr_t)ws & 255) != 0 || ws_bytes < need) return LCDM_ERR_WORKSPACE;
    c = carve_records((char*)ws, B, prec);
    if (det) {
        c.part = (double*)((char*)ws + rec);
        c.wrow = (int64_t*)((char*)c.part + align256(det_warps() * 2 * DET_NV * sizeof(double)));
    }
    return LCDM_OK;
}

// SM count of the current device, looked up once per device
#define LCDM_MAX_DEVICES 64
std::atomic<int> g_num_sms[LCDM_MAX_DEVICES];

int current_device() {
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= LCDM_MAX_DEVICES) dev = 0;
    return dev;
}

int num_sms() {
    const int dev = current_device();
    int n = g_num_sms[dev].load();
    if (n <= 0) {
        if (cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || n <= 0) n = 1;
        g_num_sms[dev].store(n);
    }
    return n;
}

const PairsTable& table(int prec, int K) {
    static PairsTable t[2][4];
    static std::once_flag once;
    std::call_once(once, [] {
        t[0][0] = table_f64_k0(); t[0][1] = table_f64_k3(); t[0][2] = table_f64_k4(); t[0][3] = table_f64_k6();
        t[1][0] = table_mix_k0(); t[1][1] = table_mix_k3(); t[1][2] = table_mix_k4(); t[1][3] = table_mix_k6();
    });
    return t[prec][K == 0 ? 0 : (K == 3 ? 1 : (K == 4 ? 2 : 3))];
}

// tuned launch shapes: key (device, precision, K, kernel (entry_index), layout, log2 npairs)
typedef std::tuple<int, int, int, int, int, int> TuneKey;
struct Tuned { int block, bps, lane_map; };
std::map<TuneKey, Tuned> g_tuned;
std::mutex g_tune_mu;

int log2_bucket(int64_t n) {
    int b = 0;
    while (n > 1) { n >>= 1; b++; }
    return b;
}

struct Plan {
    PairArgs args;
    const void* core;       // the core's records
    void* grad_z;           // [npairs] derivatives with respect to the redshifts, optional
    const float4* rowf;     // general limits: the rows' maps (null: limits from 0)
    const double* z1;
    const double* scale;
    int legacy;             // the tangent launch is the X-tangent kernel's
    int time, absorb;       // the core's records need the constants of t, of the absorption distance
    int prec, K, wt, wx;
    int64_t npairs;
    // outputs wanted as values only while other outputs need tangents: the
    // time coordinate and the absorption distance each run their own R_J
    // track, whose tangents would be computed for nothing; such outputs are
    // written by a second, tangent-free launch (split_mask: LCDM_T, LCDM_X bits)
    int split_mask;
};

lcdm_status check_pairs_args(const double* params, int64_t B, const int64_t* offsets, const void* z, int64_t n,
                             int32_t* status, const lcdm_opts* opts) {
    if (!opts_ok(opts) || !params || !status || B <= 0 || n < 0) return LCDM_ERR_INVALID;
    if (opts->layout == LCDM_LAYOUT_CSR && !offsets) return LCDM_ERR_INVALID;
    if (n > 0 && !z) return LCDM_ERR_INVALID;
    return LCDM_OK;
}

// Builds the kernel arguments; any of out / jac / cot / mobs may be null.
lcdm_status make_plan(const double* params, int64_t B, const int64_t* offsets, const void* z, int64_t n,
                      void* const* out, void* const* jac, const void* const* cot, const void* mobs, double M,
                      double sigma, double* grad, double* loglike, int32_t* status, const lcdm_opts* opts,
                      const Carved& cv, Plan& P) {
    PairArgs& a = P.args;
    memset(&a, 0, sizeof(a));
    a.recD = cv.recD;
    a.recF = cv.recF;
    P.core = cv.core;
    P.grad_z = nullptr;
    P.rowf = nullptr;
    P.z1 = P.scale = nullptr;
    a.part = cv.part;
    a.wrow = cv.wrow;
    a.det_cap = cv.part ? (int64_t)det_warps() : 0;
    a.status = status;
    a.offsets = offsets;
    a.z = z;
    a.layout = opts->layout;
    a.B = B;
    a.ncol = opts->ncol;
    a.nrow = n;
    P.npairs = opts->layout == LCDM_LAYOUT_CSR ? n : B * n;
    a.nnz = P.npairs;
    bool tangents = grad != nullptr;
    int wt = 0, wx = 0;
    for (int i = 0; i < LCDM_NOUT; i++) {
        a.out[i] = out ? out[i] : nullptr;
        a.jac[i] = jac ? jac[i] : nullptr;
        a.cot[i] = cot ? cot[i] : nullptr;
        if (a.out[i]) a.outmask |= 1 << i;
        if (a.jac[i]) tangents = true;
        bool used = a.out[i] || a.jac[i] || a.cot[i];
        if (used && i == LCDM_T) wt = 1;
        if (used && i == LCDM_X) wx = 1;
    }
    P.split_mask = 0;
    if (mobs) { tangents = tangents || grad != nullptr; }
    a.mobs = mobs;
    a.M = M;
    a.sigma = sigma;
    a.grad = grad;
    a.loglike = loglike;
    P.prec = opts->precision == LCDM_FP64 ? 0 : 1;
    P.K = tangents ? opts->ncol - 1 : 0;
    if (P.K > 0) {
        for (int i : {LCDM_T, LCDM_X}) {
            if (a.out[i] && !a.jac[i] && !a.cot[i]) {
                P.split_mask |= 1 << i;
                if (i == LCDM_T) wt = 0;
                if (i == LCDM_X) wx = 0;
            }
        }
    }
    P.wt = wt;
    P.wx = wx;
    P.legacy = P.K > 0 && wx;
    P.time = (P.split_mask >> LCDM_T) & 1 || (!P.legacy && wt);
    P.absorb = (P.split_mask >> LCDM_X) & 1 || (P.K == 0 && wx);
    return LCDM_OK;
}

lcdm_status launch_one(Plan& P, int block, int bps, int lane_map, cudaStream_t s);

// Two pairs in a thread where rows are long (a mean of LCDM_PACKED_ROW pairs):
// a batch that crosses a row runs one pair at a time, at the packed kernel's
// registers.  The line is the gradient's (us for 4 M pairs of mu and its gradient
// in rows of 128 / 256 / 512 / 1024, packed and not: 255 222, 220 216, 144 152, 122
// 135); d_C and mu as values cross at 64 (181 190, at 48 221 200; at 1024 66 76).
// Not with t's gradient: two pairs of that do not fit the registers
// (0.41 against 0.39 ms for 4 M pairs of d_C, t and mu).
#define LCDM_PACKED_ROW 256
bool packed_plan(const Plan& P) {
    return P.prec == 1 && !P.legacy && !(P.K > 0 && P.wt) && P.npairs >= P.args.B * LCDM_PACKED_ROW;
}

// index of the plan's kernel in its table (4 and up: per-pair Jacobians, 8 and
// up: with the redshift derivatives, 10 and up: general limits, 14 and up: two
// pairs in a thread)
int entry_index(const Plan& P) {
    bool jac = false;
    for (int i = 0; i < LCDM_NOUT; i++) jac = jac || P.args.jac[i];
    if (packed_plan(P) && !jac) return 14 + (P.rowf ? 8 : P.grad_z ? 4 : 0) + (P.wt ? 2 : 0) + (P.wx ? 1 : 0);
    if (P.rowf) return 10 + (P.wt ? 2 : 0) + (P.wx ? 1 : 0);
    if (P.grad_z && !P.wx && !P.legacy) return 8 + (P.wt ? 1 : 0);
    return (P.wt ? 2 : 0) + (P.wx ? 1 : 0) + (jac ? 4 : 0);
}
TuneKey tune_key(const Plan& P) {
    return TuneKey(current_device(), P.prec, P.K, entry_index(P), P.args.layout, log2_bucket(P.npairs));
}
CoreArgs core_args(const Plan& P) {
    CoreArgs c;
    c.p = P.args;
    c.rec = P.core;
    c.grad_z = P.grad_z;
    c.rowf = P.rowf;
    c.z1 = P.z1;
    c.scale = P.scale;
    return c;
}
const PairsEntry& plan_entry(const Plan& P) {
    const int i = entry_index(P);
    const PairsTable& t = table(P.prec, P.K);
    return i < 4 ? t.e[i] : i < 8 ? t.jac[i - 4] : i < 10 ? t.dz[i - 8] : i < 14 ? t.bt[i - 10] : t.packed[(i - 14) / 4][(i - 14) % 4];
}

}  // namespace

namespace lcdm {
// The deterministic reduction's second pass: the shared rows' partial sums
// added in warp order by one thread (a few thousand additions).
__global__ void det_fixup_kernel(PairArgs a, int64_t nwarps) {
    if (threadIdx.x != 0 || blockIdx.x != 0) return;
    for (int64_t w = 0; w < nwarps && w < a.det_cap; w++) {
        for (int k = 0; k < 2; k++) {
            const int64_t r = a.wrow[w * 2 + k];
            if (r < 0 || (k == 1 && r == a.wrow[w * 2])) continue;
            const double* v = a.part + (w * 2 + k) * DET_SLOT;
            if (a.grad) for (int i = 0; i < a.ncol; i++) a.grad[r * a.ncol + i] += v[i];
            if (a.loglike) a.loglike[r] += v[DET_SLOT - 1];
        }
    }
}

cudaError_t launch_det_fixup(const PairArgs& a, int64_t nwarps, cudaStream_t s) {
    det_fixup_kernel<<<1, 32, 0, s>>>(a, nwarps);
    return cudaGetLastError();
}
}  // namespace lcdm

namespace {

// The value-only outputs of split_mask: a launch of their own (K = 0, their
// tracks only, no reductions).
lcdm_status launch_values(const Plan& P, int lane_map, cudaStream_t s) {
    Plan V = P;
    PairArgs& v = V.args;
    v.outmask = 0;
    V.grad_z = nullptr;
    for (int i = 0; i < LCDM_NOUT; i++) {
        v.jac[i] = nullptr;
        v.cot[i] = nullptr;
        if (!(P.split_mask & (1 << i))) v.out[i] = nullptr;
        if (v.out[i]) v.outmask |= 1 << i;
    }
    v.mobs = nullptr;
    v.grad = nullptr;
    v.loglike = nullptr;
    V.K = 0;
    V.legacy = 0;
    V.wt = (P.split_mask >> LCDM_T) & 1;
    V.wx = (P.split_mask >> LCDM_X) & 1;
    V.split_mask = 0;
    return launch_one(V, 0, 0, lane_map, s);
}
// The redshift derivatives alone: a value launch of chi without outputs.
lcdm_status launch_dz(const Plan& P, int lane_map, cudaStream_t s) {
    Plan D = P;
    for (int i = 0; i < LCDM_NOUT; i++) D.args.out[i] = D.args.jac[i] = nullptr;
    D.args.outmask = 0;
    D.args.grad = nullptr;
    D.K = D.legacy = D.wt = D.wx = D.split_mask = 0;
    return launch_one(D, 0, 0, lane_map, s);
}
// The redshift derivatives come with the plan's main launch, unless that is
// the X-tangent kernel or a value launch with t or X.
bool separate_dz(const Plan& P) { return P.grad_z && (P.legacy || (P.K == 0 && (P.wt || P.wx))); }
// The plan's main launch, without the outputs of split_mask.
lcdm_status launch_main(const Plan& P, int block, int bps, int lane_map, cudaStream_t s) {
    Plan T = P;
    if (separate_dz(P)) T.grad_z = nullptr;
    for (int i = 0; i < LCDM_NOUT; i++)
        if (P.split_mask & (1 << i)) { T.args.out[i] = nullptr; T.args.outmask &= ~(1 << i); }
    T.split_mask = 0;
    return launch_one(T, block, bps, lane_map, s);
}

lcdm_status launch_nan_rows(const Plan& P, cudaStream_t s) {
    if (P.npairs == 0) return LCDM_OK;
    const unsigned grid = (unsigned)((P.args.B * 32 + 127) / 128);
    if (P.prec == 0) nan_rows_kernel<double><<<grid, 128, 0, s>>>(P.args, (double*)P.grad_z);
    else nan_rows_kernel<float><<<grid, 128, 0, s>>>(P.args, (float*)P.grad_z);
    g_launches++;
    return cudaGetLastError() == cudaSuccess ? LCDM_OK : LCDM_ERR_CUDA;
}

// Resident blocks per SM of a pair kernel, queried once per (device, kernel,
// block size): the query is host work on every launch otherwise (the chunked
// host entry point launches twice per chunk).
int cached_occ(const PairsEntry& t, int idx, int prec, int K, int block) {
    static std::mutex mu;
    static std::map<std::tuple<int, int, int, int, int>, int> cache;
    const auto key = std::make_tuple(current_device(), prec, K, idx, block);
    {
        std::lock_guard<std::mutex> lk(mu);
        auto it = cache.find(key);
        if (it != cache.end()) return it->second;
    }
    const int occ = t.occ(block);
    if (occ > 0) {
        std::lock_guard<std::mutex> lk(mu);
        cache[key] = occ;
    }
    return occ;
}

lcdm_status launch_one(Plan& P, int block, int bps, int lane_map, cudaStream_t s) {
    const PairsEntry& t = plan_entry(P);
    if (block == 0 || bps == 0 || lane_map == LCDM_MAP_TUNED) {
        std::lock_guard<std::mutex> lk(g_tune_mu);
        auto it = g_tuned.find(tune_key(P));
        if (it != g_tuned.end()) {
            if (block == 0) block = it->second.block;
            if (bps == 0) bps = it->second.bps;
            if (lane_map == LCDM_MAP_TUNED) lane_map = it->second.lane_map;
        }
    }
    P.args.interleave = lane_map == LCDM_MAP_INTERLEAVED ? 1 : 0;
    if (block == 0) {
        // Full-size blocks (the X-tangent kernels step in lockstep, see
        // pairs_kernel), smaller ones where those would leave SMs idle: a warp
        // alone on its sub-partition issues an FP64 instruction every 64 cycles,
        // one of eight on an SM every 152 (10^4 FP64 pairs: 40 blocks of 256,
        // 20 us; 313 of 32, 10 us).
        block = 256;
        while (block > 32 && P.npairs < (int64_t)block * 2 * num_sms()) block /= 2;
    }
    int occ = cached_occ(t, entry_index(P), P.prec, P.K, block);
    if (occ <= 0) return LCDM_ERR_CUDA;
    if (bps == 0 || bps > occ) bps = occ;
    int64_t warps = (int64_t)num_sms() * bps * (block / 32);
    int64_t chunk = (P.npairs + warps - 1) / warps;
    chunk = ((chunk + 31) / 32) * 32;
    if (chunk < 32) chunk = 32;
    P.args.chunk = chunk;
    int64_t need_warps = (P.npairs + chunk - 1) / chunk;
    int64_t grid = (need_warps * 32 + block - 1) / block;
    if (grid < 1) grid = 1;
    if (P.npairs == 0) return LCDM_OK;
    cudaError_t e = t.launch(core_args(P), (int)grid, block, s);
    g_launches++;
    if (e != cudaSuccess) return LCDM_ERR_CUDA;
    if (P.args.part && (P.args.grad || P.args.loglike)) {
        // the shared rows' partial sums, added in warp order
        e = launch_det_fixup(P.args, need_warps, s);
        g_launches++;
    }
    return e == cudaSuccess ? LCDM_OK : LCDM_ERR_CUDA;
}

int core_ns(int prec) { return prec == 0 ? (int)CoreTol<double>::ns : (int)CoreTol<float>::ns; }
// What a call's records hold.
struct PrepNeed {
    bool legacy;     // the X-tangent kernel's records
    bool core;       // the core's (beside the former: without tangents)
    int prec;        // precision of the core's records
    bool tangents, time, absorb;
    int ns;          // series coefficients of the core's records
};

lcdm_status run_prep(const double* params, int64_t B, const lcdm_opts* opts, const Carved& cv, const PrepNeed& need,
                     int32_t* status, double* grad, double* loglike, cudaStream_t s,
                     const ShiftArgs* shift = nullptr) {
    // One warp per block, so that the FP64 work spreads over as many SMs as
    // possible.  Up to LCDM_PREP_GROUP_MAX_B cosmologies the solve is bound by
    // the latency of one cosmology's dependent FP64 chain and four lanes share
    // each root solve; beyond that the FP64 pipe is the bound and one lane per
    // cosmology does no repeated work.
    PrepArgs a;
    memset(&a.shift, 0, sizeof(a.shift));
    if (shift) a.shift = *shift;
    a.params = params;
    a.B = B;
    a.ncol = opts->ncol;
    a.tangents = need.tangents;
    a.ns = need.ns;
    a.time = need.time;
    a.absorb = need.absorb;
    a.recD = need.legacy ? cv.recD : nullptr;
    a.recF = need.legacy ? cv.recF : nullptr;
    a.coreF = need.core && need.prec == 1 ? (float*)cv.core : nullptr;
    a.coreD = need.core && need.prec == 0 ? (double*)cv.core : nullptr;
    a.status = status;
    a.grad = grad;
    a.loglike = loglike;
    const int block = 32;
    if (B <= LCDM_PREP_GROUP_MAX_B) {
        const int64_t grid = (4 * B + block - 1) / block;
        prep_kernel<4><<<(unsigned)grid, block, 0, s>>>(a);
    } else {
        const int64_t grid = (B + block - 1) / block;
        prep_kernel<1><<<(unsigned)grid, block, 0, s>>>(a);
    }
    g_launches++;
    return cudaGetLastError() == cudaSuccess ? LCDM_OK : LCDM_ERR_CUDA;
}

// The plan's preparation: one launch, also where the tangent launch is the
// X-tangent kernel's and others (value-only outputs, redshift derivatives) run on
// the core.  (One after the other in the same memory: 737 against 636 us for 65536 rows
// of 8 pairs of X with its gradient, and t.)
PrepNeed plan_need(const Plan& P) {
    const bool legacy = P.legacy != 0;
    return PrepNeed{legacy, !legacy || P.split_mask || separate_dz(P), P.prec, P.K > 0, P.time != 0, P.absorb != 0, core_ns(P.prec)};
}

// Preparation and launches of a plan.
lcdm_status run_plan(const Plan& P, const double* params, int64_t B, const lcdm_opts* opts, const Carved& cv,
                     int32_t* status, double* grad, double* loglike, int block, int bps, int lane_map, cudaStream_t s,
                     const ShiftArgs* shift = nullptr) {
    lcdm_status st = run_prep(params, B, opts, cv, plan_need(P), status, grad, loglike, s, shift);
    if (st == LCDM_OK && P.split_mask) st = launch_values(P, lane_map, s);
    if (st == LCDM_OK && separate_dz(P)) st = launch_dz(P, lane_map, s);
    return st == LCDM_OK ? launch_main(P, block, bps, lane_map, s) : st;
}

__global__ void extract_roots(const double* __restrict__ recD, int64_t B, int ncol, double* roots, double* droots,
                              int32_t* kind) {
    int64_t b = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (b >= B) return;
    const double* r = recD + b * NREC;
    int kd = (int)r[RF_KIND];
    bool cpair = kd == 0 || kd == 2, quartic = kd <= 1;
    int K = ncol - 1;
    if (kind) kind[b] = kd;
    // slots: A, B, pair member 1, pair member 2
    double re[4] = {r[RF_A], quartic ? r[RF_B] : -0.0, r[RF_PRE], cpair ? r[RF_PRE] : r[RF_PIM]};
    double im[4] = {0, 0, cpair ? r[RF_PIM] : 0.0, cpair ? -r[RF_PIM] : 0.0};
    if (roots)
        for (int s = 0; s < 4; s++) { roots[(b * 4 + s) * 2] = re[s]; roots[(b * 4 + s) * 2 + 1] = im[s]; }
    if (droots) {
        for (int k = 0; k < K; k++) {
            double dre[4] = {r[RF_DA + k], quartic ? r[RF_DB + k] : 0.0, r[RF_DPRE + k],
                             cpair ? r[RF_DPRE + k] : r[RF_DPIM + k]};
            double dim[4] = {0, 0, cpair ? r[RF_DPIM + k] : 0.0, cpair ? -r[RF_DPIM + k] : 0.0};
            for (int s = 0; s < 4; s++) {
                droots[((b * 4 + s) * 2 + 0) * K + k] = dre[s];
                droots[((b * 4 + s) * 2 + 1) * K + k] = dim[s];
            }
        }
    }
}

lcdm_status pairs_common(const double* params, int64_t B, const int64_t* offsets, const void* z, int64_t n,
                         void* const* out, void* const* jac, const void* const* cot, const void* mobs, double M,
                         double sigma, double* grad, double* loglike, int32_t* status, const lcdm_opts* opts,
                         void* ws, size_t ws_bytes, cudaStream_t stream, size_t need = 0) {
    lcdm_status st = check_pairs_args(params, B, offsets, z, n, status, opts);
    if (st != LCDM_OK) return st;
    Carved cv;
    st = carve(ws, ws_bytes, B, prec_of(opts), cv, opts->deterministic, need);
    if (st != LCDM_OK) return st;
    Plan P;
    st = make_plan(params, B, offsets, z, n, out, jac, cot, mobs, M, sigma, grad, loglike, status, opts, cv, P);
    if (st != LCDM_OK) return st;
    return run_plan(P, params, B, opts, cv, status, grad, loglike, opts->block, opts->blocks_per_sm, opts->lane_map,
                    stream);
}

// ----------------------------------------------------------------------------
// Fixed device scratch for lcdm_distances_static.  The array belongs to this
// translation unit; its device address is looked up once per device with
// cudaGetSymbolAddress (the host-side name is only a stand-in and must never
// be handed to a kernel).
// ----------------------------------------------------------------------------
// (values only: the core's records)
#define LCDM_STATIC_WS_BYTES ((size_t)LCDM_STATIC_MAX_COSMOLOGIES * NCORE * sizeof(double))
static __device__ __align__(256) unsigned char g_static_ws[LCDM_STATIC_WS_BYTES];

static void* g_static_ptr[LCDM_MAX_DEVICES];
static std::mutex g_static_mu;

// Device address of g_static_ws on the current device (set up on first use).
static lcdm_status static_workspace(void** ptr) {
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= LCDM_MAX_DEVICES) return LCDM_ERR_CUDA;
    std::lock_guard<std::mutex> lk(g_static_mu);
    if (!g_static_ptr[dev]) {
        void* p = nullptr;
        if (cudaGetSymbolAddress(&p, g_static_ws) != cudaSuccess || !p) return LCDM_ERR_CUDA;
        g_static_ptr[dev] = p;
    }
    *ptr = g_static_ptr[dev];
    return LCDM_OK;
}

// ----------------------------------------------------------------------------
// Host-buffer entry point: chunked copies on two internal streams per device
// (host-to-device and device-to-host) overlapping the pair kernel of the
// neighbouring chunks on the caller's stream.
// ----------------------------------------------------------------------------
#define LCDM_HOST_MAX_CHUNKS 64
struct HostStreams {
    cudaStream_t up = nullptr, down = nullptr;
    cudaEvent_t ev[2 * LCDM_HOST_MAX_CHUNKS + 3];
    bool ready = false;
};
static HostStreams g_host_streams[LCDM_MAX_DEVICES];
static std::mutex g_host_mu;

lcdm_status host_streams(HostStreams** out) {
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= LCDM_MAX_DEVICES) return LCDM_ERR_CUDA;
    std::lock_guard<std::mutex> lk(g_host_mu);
    HostStreams& h = g_host_streams[dev];
    if (!h.ready) {
        if (cudaStreamCreateWithFlags(&h.up, cudaStreamNonBlocking) != cudaSuccess) return LCDM_ERR_CUDA;
        if (cudaStreamCreateWithFlags(&h.down, cudaStreamNonBlocking) != cudaSuccess) return LCDM_ERR_CUDA;
        for (int i = 0; i < 2 * LCDM_HOST_MAX_CHUNKS + 3; i++)
            if (cudaEventCreateWithFlags(&h.ev[i], cudaEventDisableTiming) != cudaSuccess) return LCDM_ERR_CUDA;
        h.ready = true;
    }
    *out = &h;
    return LCDM_OK;
}

// Device workspace of the host entry point: records, then params, offsets,
// status, grad, z, six cotangent and six output arrays.
struct HostCarve {
    Carved rec;
    double* params;
    int64_t* offsets;
    int32_t* status;
    double* grad;
    char* z;
    char* cot[LCDM_NOUT];
    char* out[LCDM_NOUT];
    size_t bytes;
};

HostCarve host_carve(char* base, int64_t B, int64_t n, int ncol, size_t es) {
    HostCarve c;
    size_t off = 0;
    auto take = [&](size_t bytes) { char* p = base ? base + off : nullptr; off += align256(bytes); return p; };
    c.rec = carve_records(take(ws_bytes_for(B)), B, es == 8 ? 0 : 1);
    c.params = (double*)take((size_t)B * ncol * sizeof(double));
    c.offsets = (int64_t*)take((size_t)(B + 1) * sizeof(int64_t));
    c.status = (int32_t*)take((size_t)B * sizeof(int32_t));
    c.grad = (double*)take((size_t)B * ncol * sizeof(double));
    c.z = take((size_t)n * es);
    for (int i = 0; i < LCDM_NOUT; i++) c.cot[i] = take((size_t)n * es);
    for (int i = 0; i < LCDM_NOUT; i++) c.out[i] = take((size_t)n * es);
    c.bytes = off;
    return c;
}

// Device workspace of the general-limits entry points: records of the
// shifted cosmologies, shifted parameters (closure form, four columns), their
// Jacobian, the scale s = 1+z1,
// the gradient w.r.t. the shifted parameters, z' and the mapped cotangents of
// d_C, X, d_M (scaled) and mu (0 for a pair outside the domain: at z' = 0, where
// such a pair is evaluated, mu alone has a derivative); these five only where X is
// differentiated, see RowMap.
struct BetweenCarve {
    Carved rec;
    double* jac;
    double* scale;
    float4* rowf;
    double* gradp;
    char* zp;
    char* cotp[LCDM_NOUT];
    size_t bytes;
};

BetweenCarve between_carve(char* base, int64_t B, int64_t npairs, int ncol, size_t es) {
    BetweenCarve c;
    size_t off = 0;
    auto take = [&](size_t bytes) { char* p = base ? base + off : nullptr; off += align256(bytes); return p; };
    c.rec = carve_records(take(ws_bytes_for(B)), B, es == 8 ? 0 : 1);
    c.jac = (double*)take((size_t)B * 4 * ncol * sizeof(double));
    c.scale = (double*)take((size_t)B * sizeof(double));
    c.rowf = (float4*)take((size_t)B * sizeof(float4));
    c.gradp = (double*)take((size_t)B * 4 * sizeof(double));
    c.zp = take((size_t)npairs * es);
    for (int i = 0; i < LCDM_NOUT; i++) c.cotp[i] = nullptr;
    c.cotp[LCDM_DC] = take((size_t)npairs * es);
    c.cotp[LCDM_X] = take((size_t)npairs * es);
    c.cotp[LCDM_DM] = take((size_t)npairs * es);
    c.cotp[LCDM_MU] = take((size_t)npairs * es);
    c.bytes = off;
    return c;
}

lcdm_status between_npairs(int64_t B, int64_t n, const lcdm_opts* opts, int64_t* npairs) {
    if (!opts_ok(opts) || B <= 0 || n < 0 || (n > 0 && opts->layout == LCDM_LAYOUT_SHARED))
        return LCDM_ERR_INVALID;
    *npairs = opts->layout == LCDM_LAYOUT_CSR ? n : B * n;
    return LCDM_OK;
}

// The shift of every row to its lower limit, for the preparation.
ShiftArgs between_shift(const double* params, int64_t B, const double* z1, int ncol, const BetweenCarve& w, bool grad) {
    ShiftArgs sa;
    sa.params = params;
    sa.z1 = z1;
    sa.B = B;
    sa.ncol = ncol;
    sa.jac = grad ? w.jac : nullptr;
    sa.scale = w.scale;
    sa.rowf = w.rowf;
    return sa;
}

}  // namespace

extern "C" {

lcdm_status lcdm_between_workspace_size(int64_t B, int64_t n, const lcdm_opts* opts, size_t* bytes) {
    int64_t npairs = 0;
    if (!bytes || between_npairs(B, n, opts, &npairs) != LCDM_OK) return LCDM_ERR_INVALID;
    const size_t es = opts->precision == LCDM_FP64 ? 8 : 4;
    *bytes = between_carve(nullptr, B, npairs, opts->ncol, es).bytes;
    return LCDM_OK;
}

lcdm_status lcdm_distances_between(const double* params, int64_t B, const double* z1, const int64_t* offsets,
                                   const void* z2, int64_t n, const void* const cot[LCDM_NOUT],
                                   void* const out[LCDM_NOUT], double* grad, int32_t* cosmo_status,
                                   const lcdm_opts* opts, void* ws, size_t ws_bytes, cudaStream_t stream) {
    int64_t npairs = 0;
    if (between_npairs(B, n, opts, &npairs) != LCDM_OK || !z1 || (!out && !grad) || (grad && !cot))
        return LCDM_ERR_INVALID;
    if (opts->ncol > 5) return LCDM_ERR_UNSUPPORTED;   // the row shift takes 4 or 5 columns
    if (opts->deterministic && grad) return LCDM_ERR_UNSUPPORTED;
    lcdm_status st = check_pairs_args(params, B, offsets, z2, n, cosmo_status, opts);
    if (st != LCDM_OK) return st;
    const int ncol = opts->ncol;
    const size_t es = opts->precision == LCDM_FP64 ? 8 : 4;
    if (!ws || ((uintptr_t)ws & 255) != 0) return LCDM_ERR_WORKSPACE;
    BetweenCarve w = between_carve((char*)ws, B, npairs, ncol, es);
    if (ws_bytes < w.bytes) return LCDM_ERR_WORKSPACE;
    lcdm_opts o4 = *opts;
    o4.ncol = 4;
    const ShiftArgs shift = between_shift(params, B, z1, ncol, w, grad != nullptr);
    Plan P;
    make_plan(params, B, offsets, z2, n, out, nullptr, grad ? cot : nullptr, nullptr, 0, 1, grad ? w.gradp : nullptr,
              nullptr, cosmo_status, &o4, w.rec, P);
    PairMapArgs m;
    memset(&m, 0, sizeof(m));
    if (!P.legacy) {
        P.rowf = w.rowf;
        P.z1 = z1;
        P.scale = w.scale;
    } else {
        // the kernel of X's tangents takes mapped redshifts and cotangents
        m.offsets = opts->layout == LCDM_LAYOUT_CSR ? offsets : nullptr;
        m.nrow = n;
        m.nnz = npairs;
        m.B = B;
        m.fp64 = opts->precision == LCDM_FP64;
        m.z1 = z1;
        m.scale = w.scale;
        m.rowf = w.rowf;
        m.z2 = z2;
        m.zp = w.zp;
        const void* cotk[LCDM_NOUT];
        for (int i = 0; i < LCDM_NOUT; i++) {
            m.cot[i] = cot[i];
            cotk[i] = cot[i];
            if (cot[i] && w.cotp[i]) { m.cotp[i] = w.cotp[i]; cotk[i] = w.cotp[i]; }
        }
        // (which need the rows' constants before the preparation has run)
        if (launch_shift(shift, stream) != cudaSuccess) return LCDM_ERR_CUDA;
        if (launch_pair_pre(m, stream) != cudaSuccess) return LCDM_ERR_CUDA;
        g_launches += 2;
        make_plan(params, B, offsets, w.zp, n, out, nullptr, cotk, nullptr, 0, 1, w.gradp, nullptr, cosmo_status, &o4,
                  w.rec, P);
    }
    st = run_plan(P, params, B, &o4, w.rec, cosmo_status, grad ? w.gradp : nullptr, nullptr, opts->block,
                  opts->blocks_per_sm, opts->lane_map, stream, &shift);
    if (st != LCDM_OK) return st;
    if (out && P.legacy) {
        for (int i = 0; i < LCDM_NOUT; i++) m.out[i] = out[i];
        if (launch_pair_post(m, stream) != cudaSuccess) return LCDM_ERR_CUDA;
        g_launches++;
    }
    if (grad) {
        if (launch_chain(w.jac, w.gradp, B, ncol, grad, stream) != cudaSuccess) return LCDM_ERR_CUDA;
        g_launches++;
    }
    return LCDM_OK;
}

lcdm_status lcdm_loglike_dz_workspace_size(int64_t B, int64_t n, const lcdm_opts* opts, size_t* bytes) {
    if (!opts_ok(opts) || B <= 0 || n < 0 || !bytes) return LCDM_ERR_INVALID;
    *bytes = ws_bytes_for(B);   // (the redshift derivatives come with the pair kernel)
    return LCDM_OK;
}

lcdm_status lcdm_gauss_loglike_dz(const double* params, int64_t B, const int64_t* offsets, const void* z,
                                  const void* m_obs, int64_t n, double M, double sigma, double* loglike,
                                  double* grad, void* grad_z, void* mu_out, int32_t* cosmo_status,
                                  const lcdm_opts* opts, void* ws, size_t ws_bytes, cudaStream_t stream) {
    if (!m_obs || !loglike || !grad_z || !(sigma > 0) || !std::isfinite(M)) return LCDM_ERR_INVALID;
    lcdm_status st = check_pairs_args(params, B, offsets, z, n, cosmo_status, opts);
    if (st != LCDM_OK) return st;
    if (opts->ncol > 5) return LCDM_ERR_UNSUPPORTED;   // no kernel with redshift derivatives for seven columns
    if (opts->deterministic) return LCDM_ERR_UNSUPPORTED;
    size_t need = 0;
    lcdm_loglike_dz_workspace_size(B, n, opts, &need);
    if (!ws || ((uintptr_t)ws & 255) != 0 || ws_bytes < need) return LCDM_ERR_WORKSPACE;
    Carved cv;
    carve(ws, ws_bytes, B, prec_of(opts), cv);
    void* out[LCDM_NOUT] = {nullptr, nullptr, nullptr, nullptr, nullptr, mu_out};
    Plan P;
    st = make_plan(params, B, offsets, z, n, out, nullptr, nullptr, m_obs, M, sigma, grad, loglike, cosmo_status,
                   opts, cv, P);
    if (st != LCDM_OK) return st;
    P.grad_z = grad_z;
    st = run_plan(P, params, B, opts, cv, cosmo_status, grad, loglike, opts->block, opts->blocks_per_sm, opts->lane_map,
                  stream);
    if (st != LCDM_OK) return st;
    return launch_nan_rows(P, stream);
}

lcdm_status lcdm_distances_vjp_dz(const double* params, int64_t B, const int64_t* offsets, const void* z,
                                  int64_t n, const void* const cot[LCDM_NOUT], void* const out[LCDM_NOUT],
                                  double* grad, void* grad_z, int32_t* cosmo_status, const lcdm_opts* opts,
                                  void* ws, size_t ws_bytes, cudaStream_t stream) {
    if (!cot || !grad_z) return LCDM_ERR_INVALID;
    lcdm_status st = check_pairs_args(params, B, offsets, z, n, cosmo_status, opts);
    if (st != LCDM_OK) return st;
    if (opts->ncol > 5) return LCDM_ERR_UNSUPPORTED;   // no kernel with redshift derivatives for seven columns
    if (opts->deterministic && grad) return LCDM_ERR_UNSUPPORTED;
    size_t need = 0;
    lcdm_loglike_dz_workspace_size(B, n, opts, &need);
    if (!ws || ((uintptr_t)ws & 255) != 0 || ws_bytes < need) return LCDM_ERR_WORKSPACE;
    Carved cv;
    carve(ws, ws_bytes, B, prec_of(opts), cv);
    Plan P;
    st = make_plan(params, B, offsets, z, n, out, nullptr, grad ? cot : nullptr, nullptr, 0, 1, grad, nullptr,
                   cosmo_status, opts, cv, P);
    if (st != LCDM_OK) return st;
    P.grad_z = grad_z;
    if (!grad)   // values and redshift derivatives: the cotangents carry no parameter gradient
        for (int i = 0; i < LCDM_NOUT; i++) P.args.cot[i] = cot[i];
    st = run_plan(P, params, B, opts, cv, cosmo_status, grad, nullptr, opts->block, opts->blocks_per_sm, opts->lane_map,
                  stream);
    if (st != LCDM_OK) return st;
    return launch_nan_rows(P, stream);
}

lcdm_status lcdm_limits(const double* params, int64_t B, const double* z1, double* chi_inf, double* t_inf,
                        const double* cot_chi, const double* cot_t, double* grad, int32_t* cosmo_status,
                        const lcdm_opts* opts, void* ws, size_t ws_bytes, cudaStream_t stream) {
    if (!opts_ok(opts) || B <= 0 || !params || !z1 || !cosmo_status || (!chi_inf && !t_inf && !grad))
        return LCDM_ERR_INVALID;
    if (opts->ncol > 5) return LCDM_ERR_UNSUPPORTED;   // the row shift takes 4 or 5 columns
    const int ncol = opts->ncol;
    if (!ws || ((uintptr_t)ws & 255) != 0) return LCDM_ERR_WORKSPACE;
    BetweenCarve w = between_carve((char*)ws, B, 0, ncol, 8);
    if (ws_bytes < w.bytes) return LCDM_ERR_WORKSPACE;
    lcdm_opts o4 = *opts;
    o4.ncol = 4;
    const ShiftArgs shift = between_shift(params, B, z1, ncol, w, grad != nullptr);
    const PrepNeed need = {false, true, 0, grad != nullptr, true, false, CORE_NS_ONCE};
    lcdm_status st = run_prep(params, B, &o4, w.rec, need, cosmo_status, nullptr, nullptr, stream, &shift);
    if (st != LCDM_OK) return st;
    LimitArgs la;
    la.rec = (const double*)w.rec.core;
    la.status = cosmo_status;
    la.B = B;
    la.scale = w.scale;
    la.chi = chi_inf;
    la.age = t_inf;
    la.cot_chi = cot_chi;
    la.cot_age = cot_t;
    la.jac = w.jac;
    la.ncol = ncol;
    la.grad = grad;
    if (launch_limits(la, grad != nullptr, stream) != cudaSuccess) return LCDM_ERR_CUDA;
    g_launches++;
    return LCDM_OK;
}

lcdm_status lcdm_distances_static(const double* params, int64_t B, const int64_t* offsets, const void* z,
                                  int64_t n, void* const out[LCDM_NOUT], int32_t* cosmo_status,
                                  const lcdm_opts* opts, cudaStream_t stream) {
    if (!out || B > LCDM_STATIC_MAX_COSMOLOGIES) return LCDM_ERR_INVALID;
    lcdm_status st = check_pairs_args(params, B, offsets, z, n, cosmo_status, opts);
    if (st != LCDM_OK) return st;
    void* ws = nullptr;
    st = static_workspace(&ws);
    if (st != LCDM_OK) return st;
    lcdm_opts o = *opts;
    o.deterministic = 0;   // forward values only: there is no reduction
    return pairs_common(params, B, offsets, z, n, out, nullptr, nullptr, nullptr, 0, 1, nullptr, nullptr,
                        cosmo_status, &o, ws, LCDM_STATIC_WS_BYTES, stream, core_bytes(B, prec_of(&o)));
}


lcdm_status lcdm_host_workspace_size(int64_t B, int64_t n, const lcdm_opts* opts, size_t* bytes) {
    if (!opts_ok(opts) || B <= 0 || n < 0 || !bytes) return LCDM_ERR_INVALID;
    const size_t es = opts->precision == LCDM_FP64 ? 8 : 4;
    *bytes = host_carve(nullptr, B, n, opts->ncol, es).bytes;
    return LCDM_OK;
}

lcdm_status lcdm_distances_vjp_host(const double* params, int64_t B, const int64_t* offsets, const void* z,
                                    int64_t n, const void* const cot[LCDM_NOUT], void* const out[LCDM_NOUT],
                                    double* grad, int32_t* cosmo_status, const lcdm_opts* opts, void* dws,
                                    size_t dws_bytes, int32_t nchunks, cudaStream_t stream) {
    if (!opts_ok(opts) || opts->layout != LCDM_LAYOUT_CSR || !params || !offsets || B <= 0 || n < 0 ||
        (n > 0 && !z) || !cot || !grad || !cosmo_status || nchunks < 1 || nchunks > LCDM_HOST_MAX_CHUNKS)
        return LCDM_ERR_INVALID;
    if (offsets[0] != 0 || offsets[B] != n) return LCDM_ERR_INVALID;
    if (opts->deterministic) return LCDM_ERR_UNSUPPORTED;
    for (int64_t r = 0; r < B; r++)
        if (offsets[r + 1] < offsets[r]) return LCDM_ERR_INVALID;
    const int ncol = opts->ncol;
    const size_t es = opts->precision == LCDM_FP64 ? 8 : 4;
    if (!dws || ((uintptr_t)dws & 255) != 0) return LCDM_ERR_WORKSPACE;
    HostCarve d = host_carve((char*)dws, B, n, ncol, es);
    if (dws_bytes < d.bytes) return LCDM_ERR_WORKSPACE;
    HostStreams* hs = nullptr;
    lcdm_status st = host_streams(&hs);
    if (st != LCDM_OK) return st;
    cudaEvent_t* ev = hs->ev;
    bool ok = true;
    auto chk = [&](cudaError_t e) { ok = ok && e == cudaSuccess; };
    // the copies wait for earlier work on the caller's stream (workspace reuse)
    chk(cudaEventRecord(ev[0], stream));
    chk(cudaStreamWaitEvent(hs->up, ev[0], 0));
    chk(cudaMemcpyAsync(d.params, params, (size_t)B * ncol * sizeof(double), cudaMemcpyHostToDevice, hs->up));
    chk(cudaMemcpyAsync(d.offsets, offsets, (size_t)(B + 1) * sizeof(int64_t), cudaMemcpyHostToDevice, hs->up));
    chk(cudaEventRecord(ev[1], hs->up));
    chk(cudaStreamWaitEvent(stream, ev[1], 0));
    if (!ok) return LCDM_ERR_CUDA;
    // one preparation of all rows for every chunk
    {
        Plan P;
        void* const* outs = out;
        make_plan(d.params, B, d.offsets, d.z, n, outs, nullptr, cot, nullptr, 0, 1, d.grad, nullptr, d.status, opts,
                  d.rec, P);
        st = run_prep(d.params, B, opts, d.rec, plan_need(P), d.status, d.grad, nullptr, stream);
        if (st != LCDM_OK) return st;
    }
    // chunk c covers rows [rb[c], rb[c+1]); its share of the pairs ramps up and
    // down, weights min(c + 1, nchunks - c, 3) (1 2 3 ... 3 2 1): the first
    // chunk's input copy and the last chunk's output copy are the parts of the
    // pipeline that nothing overlaps, and each step of the ramp at most doubles
    // (or halves) a chunk, so the next chunk's copy still hides behind the
    // current chunk's kernels
    int64_t rb[LCDM_HOST_MAX_CHUNKS + 1];
    int64_t wcum[LCDM_HOST_MAX_CHUNKS + 1];
    wcum[0] = 0;
    for (int c = 0; c < nchunks; c++) {
        int w = c + 1 < nchunks - c ? c + 1 : nchunks - c;
        wcum[c + 1] = wcum[c] + (w < 3 ? w : 3);
    }
    rb[0] = 0;
    for (int c = 1; c < nchunks; c++) {
        const int64_t target = (int64_t)((double)n * (double)wcum[c] / (double)wcum[nchunks]);
        int64_t lo = rb[c - 1], hi = B;   // first row whose start offset is >= target
        while (lo < hi) {
            int64_t mid = (lo + hi) / 2;
            if (offsets[mid] < target) lo = mid + 1; else hi = mid;
        }
        rb[c] = lo;
    }
    rb[nchunks] = B;
    for (int c = 0; c < nchunks; c++) {
        const int64_t r0 = rb[c], r1 = rb[c + 1];
        const int64_t o0 = offsets[r0], o1 = offsets[r1];
        if (r1 <= r0 || o1 <= o0) continue;
        const size_t nb = (size_t)(o1 - o0) * es, ob = (size_t)o0 * es;
        chk(cudaMemcpyAsync(d.z + ob, (const char*)z + ob, nb, cudaMemcpyHostToDevice, hs->up));
        const void* cotd[LCDM_NOUT] = {nullptr, nullptr, nullptr, nullptr, nullptr, nullptr};
        void* outd[LCDM_NOUT] = {nullptr, nullptr, nullptr, nullptr, nullptr, nullptr};
        for (int i = 0; i < LCDM_NOUT; i++) {
            if (cot[i]) {
                chk(cudaMemcpyAsync(d.cot[i] + ob, (const char*)cot[i] + ob, nb, cudaMemcpyHostToDevice, hs->up));
                cotd[i] = d.cot[i];
            }
            if (out && out[i]) outd[i] = d.out[i];
        }
        chk(cudaEventRecord(ev[2 + 2 * c], hs->up));
        chk(cudaStreamWaitEvent(stream, ev[2 + 2 * c], 0));
        if (!ok) return LCDM_ERR_CUDA;
        Carved rc;
        rc.recD = d.rec.recD + r0 * NREC;
        rc.recF = d.rec.recF ? d.rec.recF + r0 * NREC : nullptr;
        rc.core = d.rec.core + (size_t)r0 * NCORE * es;
        Plan P;
        make_plan(d.params + r0 * ncol, r1 - r0, d.offsets + r0, d.z, o1 - o0, outd, nullptr, cotd, nullptr, 0, 1,
                  d.grad + r0 * ncol, nullptr, d.status + r0, opts, rc, P);
        P.args.base = o0;
        if (P.split_mask) {
            st = launch_values(P, opts->lane_map, stream);
            if (st != LCDM_OK) return st;
        }
        st = launch_main(P, opts->block, opts->blocks_per_sm, opts->lane_map, stream);
        if (st != LCDM_OK) return st;
        chk(cudaEventRecord(ev[3 + 2 * c], stream));
        chk(cudaStreamWaitEvent(hs->down, ev[3 + 2 * c], 0));
        for (int i = 0; i < LCDM_NOUT; i++)
            if (outd[i]) chk(cudaMemcpyAsync((char*)out[i] + ob, d.out[i] + ob, nb, cudaMemcpyDeviceToHost, hs->down));
        if (!ok) return LCDM_ERR_CUDA;
    }
    chk(cudaEventRecord(ev[2 * LCDM_HOST_MAX_CHUNKS + 2], stream));
    chk(cudaStreamWaitEvent(hs->down, ev[2 * LCDM_HOST_MAX_CHUNKS + 2], 0));
    chk(cudaMemcpyAsync(grad, d.grad, (size_t)B * ncol * sizeof(double), cudaMemcpyDeviceToHost, hs->down));
    chk(cudaMemcpyAsync(cosmo_status, d.status, (size_t)B * sizeof(int32_t), cudaMemcpyDeviceToHost, hs->down));
    chk(cudaStreamSynchronize(hs->down));
    return ok ? LCDM_OK : LCDM_ERR_CUDA;
}

lcdm_status lcdm_workspace_size(int64_t B, const lcdm_opts* opts, size_t* bytes) {
    if (!opts_ok(opts) || B <= 0 || !bytes) return LCDM_ERR_INVALID;
    *bytes = ws_bytes_for(B) + (opts->deterministic ? det_bytes() : 0);
    return LCDM_OK;
}

lcdm_status lcdm_roots(const double* params, int64_t B, const lcdm_opts* opts, double* roots, double* droots,
                       int32_t* kind, int32_t* cosmo_status, void* ws, size_t ws_bytes, cudaStream_t stream) {
    if (!opts_ok(opts) || !params || !cosmo_status || B <= 0) return LCDM_ERR_INVALID;
    Carved cv;
    lcdm_status st = carve(ws, ws_bytes, B, prec_of(opts), cv);
    if (st != LCDM_OK) return st;
    const PrepNeed need = {true, false, 0, true, true, false, 0};
    st = run_prep(params, B, opts, cv, need, cosmo_status, nullptr, nullptr, stream);
    if (st != LCDM_OK) return st;
    extract_roots<<<(unsigned)((B + 127) / 128), 128, 0, stream>>>(cv.recD, B, opts->ncol, roots, droots, kind);
    g_launches++;
    return cudaGetLastError() == cudaSuccess ? LCDM_OK : LCDM_ERR_CUDA;
}

lcdm_status lcdm_distances(const double* params, int64_t B, const int64_t* offsets, const void* z, int64_t n,
                           void* const out[LCDM_NOUT], int32_t* cosmo_status, const lcdm_opts* opts, void* ws,
                           size_t ws_bytes, cudaStream_t stream) {
    if (!out) return LCDM_ERR_INVALID;
    return pairs_common(params, B, offsets, z, n, out, nullptr, nullptr, nullptr, 0, 1, nullptr, nullptr,
                        cosmo_status, opts, ws, ws_bytes, stream);
}

lcdm_status lcdm_distances_jac(const double* params, int64_t B, const int64_t* offsets, const void* z, int64_t n,
                               void* const out[LCDM_NOUT], void* const jac[LCDM_NOUT], int32_t* cosmo_status,
                               const lcdm_opts* opts, void* ws, size_t ws_bytes, cudaStream_t stream) {
    if (!jac) return LCDM_ERR_INVALID;
    return pairs_common(params, B, offsets, z, n, out, jac, nullptr, nullptr, 0, 1, nullptr, nullptr,
                        cosmo_status, opts, ws, ws_bytes, stream);
}

lcdm_status lcdm_distances_vjp(const double* params, int64_t B, const int64_t* offsets, const void* z, int64_t n,
                               const void* const cot[LCDM_NOUT], void* const out[LCDM_NOUT], double* grad,
                               int32_t* cosmo_status, const lcdm_opts* opts, void* ws, size_t ws_bytes,
                               cudaStream_t stream) {
    if (!cot || !grad) return LCDM_ERR_INVALID;
    return pairs_common(params, B, offsets, z, n, out, nullptr, cot, nullptr, 0, 1, grad, nullptr, cosmo_status,
                        opts, ws, ws_bytes, stream);
}

lcdm_status lcdm_gauss_loglike(const double* params, int64_t B, const int64_t* offsets, const void* z,
                               const void* m_obs, int64_t n, double M, double sigma, double* loglike, double* grad,
                               void* mu_out, int32_t* cosmo_status, const lcdm_opts* opts, void* ws,
                               size_t ws_bytes, cudaStream_t stream) {
    if (!m_obs || !loglike || !(sigma > 0) || !std::isfinite(M)) return LCDM_ERR_INVALID;
    void* out[LCDM_NOUT] = {nullptr, nullptr, nullptr, nullptr, nullptr, mu_out};
    return pairs_common(params, B, offsets, z, n, out, nullptr, nullptr, m_obs, M, sigma, grad, loglike,
                        cosmo_status, opts, ws, ws_bytes, stream);
}

lcdm_status lcdm_autotune(const double* params, int64_t B, const int64_t* offsets, const void* z, int64_t n,
                          const void* const cot[LCDM_NOUT], void* const out[LCDM_NOUT], double* grad,
                          int32_t* cosmo_status, const lcdm_opts* opts, void* ws, size_t ws_bytes,
                          cudaStream_t stream, int32_t* best_block, int32_t* best_bps, float* best_ms,
                          int32_t* best_map) {
    lcdm_status st = check_pairs_args(params, B, offsets, z, n, cosmo_status, opts);
    if (st != LCDM_OK) return st;
    if (!grad) cot = nullptr;   // forward-only shape
    Carved cv;
    st = carve(ws, ws_bytes, B, prec_of(opts), cv, opts->deterministic);
    if (st != LCDM_OK) return st;
    Plan P;
    st = make_plan(params, B, offsets, z, n, out, nullptr, cot, nullptr, 0, 1, grad, nullptr, cosmo_status, opts, cv,
                   P);
    if (st != LCDM_OK) return st;
    const PairsEntry& t = plan_entry(P);
    cudaEvent_t e0, e1;
    if (cudaEventCreate(&e0) != cudaSuccess || cudaEventCreate(&e1) != cudaSuccess) return LCDM_ERR_CUDA;
    const int blocks[] = {64, 128, 256};
    float best = 1e30f;
    int bb = 128, bbps = 1, bmap = LCDM_MAP_CONTIGUOUS;
    for (int map = LCDM_MAP_CONTIGUOUS; map <= LCDM_MAP_INTERLEAVED; map++) {
        if (opts->lane_map != LCDM_MAP_TUNED && map != opts->lane_map) continue;
        for (int block : blocks) {
            int occ = t.occ(block);
            for (int bps = 1; bps <= occ; bps = (bps * 2 > occ && bps < occ) ? occ : bps * 2) {
                float tot = 0;
                for (int rep = 0; rep < 3; rep++) {
                    // (the preparation is not timed)
                    if (run_prep(params, B, opts, cv, plan_need(P), cosmo_status, grad, nullptr, stream) != LCDM_OK)
                        return LCDM_ERR_CUDA;
                    cudaEventRecord(e0, stream);
                    if (P.split_mask && launch_values(P, map, stream) != LCDM_OK) return LCDM_ERR_CUDA;
                    if (launch_main(P, block, bps, map, stream) != LCDM_OK) return LCDM_ERR_CUDA;
                    cudaEventRecord(e1, stream);
                    cudaEventSynchronize(e1);
                    float ms = 0;
                    cudaEventElapsedTime(&ms, e0, e1);
                    if (rep > 0) tot += ms;
                }
                tot /= 2;
                if (tot < best) { best = tot; bb = block; bbps = bps; bmap = map; }
            }
        }
    }
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    {
        std::lock_guard<std::mutex> lk(g_tune_mu);
        g_tuned[tune_key(P)] = Tuned{bb, bbps, bmap};
    }
    if (best_block) *best_block = bb;
    if (best_bps) *best_bps = bbps;
    if (best_ms) *best_ms = best;
    if (best_map) *best_map = bmap;
    return cudaGetLastError() == cudaSuccess ? LCDM_OK : LCDM_ERR_CUDA;
}

const char* lcdm_status_string(int s) {
    switch (s) {
        case LCDM_OK: return "LCDM_OK";
        case LCDM_ERR_INVALID: return "LCDM_ERR_INVALID: invalid argument";
        case LCDM_ERR_CUDA: return "LCDM_ERR_CUDA: CUDA launch or query failed";
        case LCDM_ERR_WORKSPACE: return "LCDM_ERR_WORKSPACE: workspace missing, too small or not 256-byte aligned";
        case LCDM_ERR_UNSUPPORTED: return "LCDM_ERR_UNSUPPORTED: unsupported combination";
        default: return "unknown lcdm_status";
    }
}

int64_t lcdm_launch_count(void) { return g_launches.load(); }

}  // extern "C"
