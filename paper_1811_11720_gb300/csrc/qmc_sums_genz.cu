// Genz families 1-4 (Sec. 5.2): the benchmark families.
#include "qmc_sums_inst.cuh"

namespace qmc {
cudaError_t launch_sums_genz(int family, int tkind, const LatticeLaunch &lp, int max_d, cudaStream_t s) {
    switch (family) {
    case QMC_GENZ_OSCILLATORY: return launch_family<QMC_GENZ_OSCILLATORY>(tkind, lp, max_d, s);
    case QMC_GENZ_PRODUCT_PEAK: return launch_family<QMC_GENZ_PRODUCT_PEAK>(tkind, lp, max_d, s);
    case QMC_GENZ_CORNER_PEAK: return launch_family<QMC_GENZ_CORNER_PEAK>(tkind, lp, max_d, s);
    case QMC_GENZ_GAUSSIAN: return launch_family<QMC_GENZ_GAUSSIAN>(tkind, lp, max_d, s);
    default: return cudaErrorInvalidValue;
    }
}
}  // namespace qmc
