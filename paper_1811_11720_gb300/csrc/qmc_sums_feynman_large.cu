// The complex deformed-contour integrand in launches with larger dimensions (or a mix): the
// general form does not fit the two blocks per SM of the others (see kSumsMinBlocks).
#include "qmc_sums_inst.cuh"

namespace qmc {
cudaError_t launch_sums_feynman_large(int tkind, const LatticeLaunch &lp, int max_d, cudaStream_t s) {
    return launch_family<QMC_FEYNMAN, 1>(tkind, lp, max_d, s);
}
}  // namespace qmc
