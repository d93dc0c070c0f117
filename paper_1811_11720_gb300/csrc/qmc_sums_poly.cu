// Polynomial families: real sector-like U^a/F^b and the complex deformed-contour integrand.
#include "qmc_sums_inst.cuh"

namespace qmc {
cudaError_t launch_sums_poly(int family, int tkind, const LatticeLaunch &lp, int max_d, cudaStream_t s) {
    switch (family) {
    case QMC_SECTOR: return launch_family<QMC_SECTOR>(tkind, lp, max_d, s);
    case QMC_FEYNMAN: return launch_family<QMC_FEYNMAN>(tkind, lp, max_d, s);
    default: return cudaErrorInvalidValue;
    }
}
}  // namespace qmc
