// qmc_sums_inst.cuh -- per-translation-unit instantiation of lattice_kernel over the
// transforms (the four public kinds and the two integer-pipe Korobov kinds) for a list of families
// (split across TUs so nvcc compiles them in parallel).
#pragma once
#include "qmc_internal.h"
#include "qmc_sums.cuh"

namespace qmc {

template <int FAM, int TK>
static cudaError_t launch_one(const LatticeLaunch &lp, int max_d, cudaStream_t s) {
    const uint64_t tiles = lp.end_tile - lp.first_tile;
    const uint64_t grid = tiles < 0x7FFFFFFFull ? tiles : 0x7FFFFFFFull;
    lattice_kernel<FAM, TK><<<(unsigned)grid, lp.spb * lp.m, sizeof(uint64_t) * max_d * lp.m, s>>>(lp);
    return cudaGetLastError();
}

template <int FAM>
static cudaError_t launch_family(int tkind, const LatticeLaunch &lp, int max_d, cudaStream_t s) {
    switch (tkind) {
    case QMC_T_NONE: return launch_one<FAM, QMC_T_NONE>(lp, max_d, s);
    case QMC_T_BAKER: return launch_one<FAM, QMC_T_BAKER>(lp, max_d, s);
    case QMC_T_KOROBOV: return launch_one<FAM, QMC_T_KOROBOV>(lp, max_d, s);
    case QMC_T_SIDI: return launch_one<FAM, QMC_T_SIDI>(lp, max_d, s);
    case kTKorobovInt: return launch_one<FAM, kTKorobovInt>(lp, max_d, s);
    case kTKorobovGen: return launch_one<FAM, kTKorobovGen>(lp, max_d, s);
    default: return cudaErrorInvalidValue;
    }
}

}  // namespace qmc
