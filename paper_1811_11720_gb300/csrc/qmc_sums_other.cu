// Genz families 5-6, the minimal-example monomial and the trigonometric test product.
#include "qmc_sums_inst.cuh"

namespace qmc {
cudaError_t launch_sums_other(int family, int tkind, const LatticeLaunch &lp, int max_d, cudaStream_t s) {
    switch (family) {
    case QMC_GENZ_C0: return launch_family<QMC_GENZ_C0>(tkind, lp, max_d, s);
    case QMC_GENZ_DISCONTINUOUS: return launch_family<QMC_GENZ_DISCONTINUOUS>(tkind, lp, max_d, s);
    case QMC_MONOMIAL: return launch_family<QMC_MONOMIAL>(tkind, lp, max_d, s);
    case QMC_TRIG: return launch_family<QMC_TRIG>(tkind, lp, max_d, s);
    default: return cudaErrorInvalidValue;
    }
}
}  // namespace qmc
