// The complex deformed-contour integrand, dimensions whose forms are compiled in.
#include "qmc_sums_inst.cuh"

namespace qmc {
cudaError_t launch_sums_feynman(int tkind, const LatticeLaunch &lp, int max_d, cudaStream_t s) {
    if (max_d > kFeynFixedMaxDim) return launch_sums_feynman_large(tkind, lp, max_d, s);
    return launch_family<QMC_FEYNMAN>(tkind, lp, max_d, s);
}
}  // namespace qmc
