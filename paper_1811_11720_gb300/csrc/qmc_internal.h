// qmc_internal.h -- host-side declarations shared by the C-ABI and the kernel TUs.
#pragma once
#include <cuda_runtime.h>

#include <cstdint>

#include "qmc_params.cuh"

namespace qmc {

// Launches lattice_kernel<FAM, TK> for the family group compiled in one translation unit;
// max_d: the largest dimension among the integrals (sizes the block's shift table).
// Returns cudaErrorInvalidValue when (family, transform) is not in that group.
cudaError_t launch_sums_genz(int family, int tkind, const LatticeLaunch &lp, int max_d, cudaStream_t s);
cudaError_t launch_sums_other(int family, int tkind, const LatticeLaunch &lp, int max_d, cudaStream_t s);
cudaError_t launch_sums_sector(int tkind, const LatticeLaunch &lp, int max_d, cudaStream_t s);
cudaError_t launch_sums_feynman(int tkind, const LatticeLaunch &lp, int max_d, cudaStream_t s);
cudaError_t launch_sums_feynman_large(int tkind, const LatticeLaunch &lp, int max_d, cudaStream_t s);

struct PointsParams {
    uint64_t n, i_begin, count;
    int d, m;
    // launch shape, set by launch_points: threads per block as rows x cols, steps per thread
    int rows, cols;
    uint32_t steps;
    DimConst dc[kMaxDim];
    const uint64_t *shifts;
    double *out;
};
cudaError_t launch_points(PointsParams p, cudaStream_t s);

// Reduce per-tile partials [tiles][m] (sum, comp) (and the im block) to double-double
// sums [2m] (and [2m..4m) for im), fixed order.
cudaError_t launch_reduce_tiles(const double *partials, uint64_t tiles, int m, int is_complex,
                                double *sums, cudaStream_t s);
cudaError_t launch_finalize(const double *sums, int m, uint64_t n, int is_complex,
                            double *result, double *Q, cudaStream_t s);

cudaError_t launch_evaluate(int family, const Integral &p, double *out, cudaStream_t s);
constexpr int kHistCells = 20480;   // most dim * bins: 160 KB of shared memory
cudaError_t launch_histogram(int family, const Integral &p, int bins, double *hist, double *work,
                             uint32_t nblocks, cudaStream_t s);

int sm_count();

// Batch building blocks shared by qmc_batch_sums and the serving loop.  Item partial
// offsets are relative to `partials`; sums, results and counters are indexed by the items'
// slots.
int fill_batch_item(Integral &it, const qmc_batch_item &b, int m, int spb, uint32_t Lcfg, int fam);
bool batch_family_supported(int fam);
// One launch over items[0..count) of one transform kind, tiles [first_tile, end_tile).
cudaError_t launch_batch(int family, int tkind, int max_d, const Integral *items,
                         const uint64_t *tile_begin, int count, uint64_t first_tile,
                         uint64_t end_tile, int m, int spb, int chain, double *partials,
                         unsigned long long *counters, cudaStream_t s);
cudaError_t launch_batch_reduce(const Integral *d_items, int count, int m, int cplx,
                                const double *partials, double *sums, cudaStream_t s);
cudaError_t launch_batch_finalize(const Integral *d_items, int count, int m, int cplx,
                                  const double *sums, double *results, cudaStream_t s);

}  // namespace qmc
