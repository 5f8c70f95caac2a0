// Launch helpers for the pair kernel instantiations (one translation unit per
// precision and tangent count, so they compile in parallel).
#pragma once
#include "lcdm_corekernel.cuh"

namespace lcdm {

// One pair kernel: its launch and its resident blocks per SM.  (The kernel of
// X's tangents reads the records in PairArgs.)
struct PairsEntry {
    cudaError_t (*launch)(const CoreArgs& a, int grid, int block, cudaStream_t s);
    int (*occ)(int block);
};

template <int PREC, int K, bool WT> struct TangentX {
    static cudaError_t launch(const CoreArgs& a, int grid, int block, cudaStream_t s) {
        pairs_kernel<PREC, K, WT><<<grid, block, 0, s>>>(a.p);
        return cudaGetLastError();
    }
    static int occ(int block) {
        int n = 0;
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, pairs_kernel<PREC, K, WT>, block, 0) != cudaSuccess)
            return 0;
        return n;
    }
};
template <int PREC, int K, bool WT, bool WX, int MODE = CORE_SUM> struct Core {
    static cudaError_t launch(const CoreArgs& c, int grid, int block, cudaStream_t s) {
        core_kernel<PREC, K, WT, WX, MODE><<<grid, block, 0, s>>>(c);
        return cudaGetLastError();
    }
    static int occ(int block) {
        int n = 0;
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, core_kernel<PREC, K, WT, WX, MODE>, block, 0) != cudaSuccess)
            return 0;
        return n;
    }
};

template <int K, bool WT, bool WX, int MODE = CORE_SUM> struct Core2 {
    static cudaError_t launch(const CoreArgs& c, int grid, int block, cudaStream_t s) {
        core2_kernel<K, WT, WX, MODE><<<grid, block, 0, s>>>(c);
        return cudaGetLastError();
    }
    static int occ(int block) {
        int n = 0;
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, core2_kernel<K, WT, WX, MODE>, block, 0) != cudaSuccess)
            return 0;
        return n;
    }
};

// entries by (WT ? 2 : 0) + (WX ? 1 : 0); jac: the kernels of per-pair
// Jacobians (without X's, whose tangents have a kernel of their own); dz: those
// that also give the redshift derivatives, by WT (four- and five-column rows;
// of the value kernels only the one without t and X); bt: those of general
// limits, like e (the shifted rows have four columns, and X's tangents there go
// through the pair maps)
struct PairsTable {
    PairsEntry e[4], jac[4], dz[2], bt[4];
    PairsEntry packed[3][4];   // two pairs in a thread (single precision, no gradient of t): sums, redshift
                               // derivatives and general limits, each like e
};

template <class E> PairsEntry entry() { PairsEntry e; e.launch = E::launch; e.occ = E::occ; return e; }

template <int PREC> PairsTable value_table() {
    PairsTable t = {};
    t.e[0] = entry<Core<PREC, 0, false, false> >();
    t.e[1] = entry<Core<PREC, 0, false, true> >();
    t.e[2] = entry<Core<PREC, 0, true, false> >();
    t.e[3] = entry<Core<PREC, 0, true, true> >();
    if constexpr (PREC == 1) {
        t.packed[0][0] = entry<Core2<0, false, false> >();
        t.packed[0][1] = entry<Core2<0, false, true> >();
        t.packed[0][2] = entry<Core2<0, true, false> >();
        t.packed[0][3] = entry<Core2<0, true, true> >();
        t.packed[1][0] = entry<Core2<0, false, false, CORE_DZ> >();
        t.packed[2][0] = entry<Core2<0, false, false, CORE_BETWEEN> >();
        t.packed[2][1] = entry<Core2<0, false, true, CORE_BETWEEN> >();
        t.packed[2][2] = entry<Core2<0, true, false, CORE_BETWEEN> >();
        t.packed[2][3] = entry<Core2<0, true, true, CORE_BETWEEN> >();
    }
    t.dz[0] = entry<Core<PREC, 0, false, false, CORE_DZ> >();
    t.bt[0] = entry<Core<PREC, 0, false, false, CORE_BETWEEN> >();
    t.bt[1] = entry<Core<PREC, 0, false, true, CORE_BETWEEN> >();
    t.bt[2] = entry<Core<PREC, 0, true, false, CORE_BETWEEN> >();
    t.bt[3] = entry<Core<PREC, 0, true, true, CORE_BETWEEN> >();
    return t;
}
template <int PREC, int K> PairsTable tangent_table() {
    PairsTable t = {};
    t.e[0] = entry<Core<PREC, K, false, false> >();
    t.e[1] = entry<TangentX<PREC, K, false> >();
    t.e[2] = entry<Core<PREC, K, true, false> >();
    t.e[3] = entry<TangentX<PREC, K, true> >();
    t.jac[0] = entry<Core<PREC, K, false, false, CORE_JAC> >();
    t.jac[1] = t.e[1];
    t.jac[2] = entry<Core<PREC, K, true, false, CORE_JAC> >();
    t.jac[3] = t.e[3];
    if constexpr (PREC == 1) {
        t.packed[0][0] = entry<Core2<K, false, false> >();
        if constexpr (K < 6) t.packed[1][0] = entry<Core2<K, false, false, CORE_DZ> >();
        if constexpr (K == 3) t.packed[2][0] = entry<Core2<K, false, false, CORE_BETWEEN> >();
    }
    if constexpr (K == 3) {
        t.bt[0] = entry<Core<PREC, K, false, false, CORE_BETWEEN> >();
        t.bt[2] = entry<Core<PREC, K, true, false, CORE_BETWEEN> >();
    }
    if constexpr (K < 6) {
        t.dz[0] = entry<Core<PREC, K, false, false, CORE_DZ> >();
        t.dz[1] = entry<Core<PREC, K, true, false, CORE_DZ> >();
    }
    return t;
}

PairsTable table_f64_k0();
PairsTable table_f64_k3();
PairsTable table_f64_k4();
PairsTable table_f64_k6();
PairsTable table_mix_k0();
PairsTable table_mix_k3();
PairsTable table_mix_k4();
PairsTable table_mix_k6();
// second pass of the deterministic reduction (defined with the other kernels)
cudaError_t launch_det_fixup(const PairArgs& a, int64_t nwarps, cudaStream_t s);

}  // namespace lcdm
