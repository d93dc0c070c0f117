// qmc_sums_inst.cuh -- per-translation-unit instantiation of lattice_kernel over the
// transforms (the four public kinds and the two integer-pipe Korobov kinds) for a list of
// families (split across TUs so nvcc compiles them in parallel).
#pragma once
#include "qmc_internal.h"
#include "qmc_sums.cuh"

namespace qmc {

template <int FAM, int TK, int MINB, bool kOne = false>
static cudaError_t launch_one(const LatticeLaunch &lp, int max_d, cudaStream_t s) {
    const uint64_t tiles = lp.end_tile - lp.first_tile;
    const uint64_t grid = tiles < 0x7FFFFFFFull ? tiles : 0x7FFFFFFFull;
    const size_t smem = sizeof(uint64_t) * max_d * lp.m;
    // static and dynamic shared memory together exceed the 48 KB that need no opting in for many
    // shifts and dimensions (the static part is at most 46,160 bytes).  The limit is state of the
    // function that all threads share: always the largest table's size, so that no call lowers it
    // under another one's launch.
    if (smem > 2048) {
        const cudaError_t e = cudaFuncSetAttribute(lattice_kernel<FAM, TK, MINB, kOne>,
                                                   cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                   (int)sizeof(uint64_t) * kMaxDim * kSumsThreads);
        if (e != cudaSuccess) return e;
    }
    if (lp.chain == kChainLater) {
        cudaLaunchAttribute attr{};
        attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr.val.programmaticStreamSerializationAllowed = 1;
        cudaLaunchConfig_t cfg{};
        cfg.gridDim = dim3((unsigned)grid);
        cfg.blockDim = dim3(lp.spb * lp.m);
        cfg.dynamicSmemBytes = smem;
        cfg.stream = s;
        cfg.attrs = &attr;
        cfg.numAttrs = 1;
        return cudaLaunchKernelEx(&cfg, lattice_kernel<FAM, TK, MINB, kOne>, lp);
    }
    lattice_kernel<FAM, TK, MINB, kOne><<<(unsigned)grid, lp.spb * lp.m, smem, s>>>(lp);
    return cudaGetLastError();
}

// Whether a launch under the FP64 Korobov map reads its integral in place (lattice_kernel's kOne):
// single integrals of the separable families; of the polynomial ones, whose loops need the
// registers that uniform operands take, those with an order 0 (sector d = 8, n = 108,863, m = 32: 643
// us, 714 from shared memory) or of at most one wave of blocks (sparse sector d = 6, n = 1021, orders
// 8: 150, 163; at n = 108,863 1647, 1443).
template <int FAM, int MINB>
static bool reads_in_place(const LatticeLaunch &lp) {
    return !lp.items && (!kPolyFamily<FAM> || !lp.one.t.r0 || !lp.one.t.r1 || lp.end_tile - lp.first_tile <= 152 * MINB);
}

template <int FAM, int MINB = kSumsMinBlocks<FAM>>
static cudaError_t launch_family(int tkind, const LatticeLaunch &lp, int max_d, cudaStream_t s) {
    switch (tkind) {
    case QMC_T_NONE: return launch_one<FAM, QMC_T_NONE, MINB>(lp, max_d, s);
    case QMC_T_BAKER: return launch_one<FAM, QMC_T_BAKER, MINB>(lp, max_d, s);
    case QMC_T_KOROBOV:
        if (reads_in_place<FAM, MINB>(lp)) return launch_one<FAM, QMC_T_KOROBOV, MINB, true>(lp, max_d, s);
        return launch_one<FAM, QMC_T_KOROBOV, MINB>(lp, max_d, s);
    case QMC_T_SIDI: return launch_one<FAM, QMC_T_SIDI, MINB>(lp, max_d, s);
    case kTKorobovInt: return launch_one<FAM, kTKorobovInt, MINB>(lp, max_d, s);
    case kTKorobovGen: return launch_one<FAM, kTKorobovGen, MINB>(lp, max_d, s);
    default: return cudaErrorInvalidValue;
    }
}

}  // namespace qmc
