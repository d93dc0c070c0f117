// Real sector-like U^a/F^b.
#include "qmc_sums_inst.cuh"

namespace qmc {
cudaError_t launch_sums_sector(int tkind, const LatticeLaunch &lp, int max_d, cudaStream_t s) {
    return launch_family<QMC_SECTOR>(tkind, lp, max_d, s);
}
}  // namespace qmc
