// qmc_params.cuh -- launch parameters shared by the host dispatch and the kernels.
#pragma once
#include <cstdint>

#include "qmc_gb300.h"
#include "qmc_lattice.cuh"

namespace qmc {

constexpr int kMaxDim = QMC_MAX_DIM;
constexpr int kMaxKorobov = 8;
constexpr int kMaxSidi = 8;
constexpr int kSumsThreads = 256;   // threads per block of the lattice-sum kernel

// Internal transform kind: symmetric Korobov<r,r>, 1 <= r <= kMaxKorobovInt, evaluated in
// integer fixed point (qmc_fixed.cuh).  The public kind stays QMC_T_KOROBOV.
constexpr int kTKorobovInt = 4;
constexpr int kMaxKorobovInt = 6;
// The asymmetric Korobov<r0,r1>, both orders in 1..kMaxKorobovInt, in integer fixed point
// with the orders at run time.
constexpr int kTKorobovGen = 5;

// Korobov<r0,r1> (Eq. (korobov)) as used by the kernels: for u <= 1/2,
//   phi(u) = u^(r0+1) sum_k A[k] u^k,  A[k] = C (-1)^k binom(r1,k) / (r0+k+1), k <= r1,
// and for u > 1/2 the reflection phi(u) = 1 - v^(r1+1) sum_k B[k] v^k with v = 1 - u
// (B: r0 and r1 exchanged).  The weight is C u^r0 (1-u)^r1, C = (r0+r1+1) binom(r0+r1,r0).
struct TransformParams {
    int kind, r0, r1, deg;        // deg = max(r0, r1): Horner length (zero-padded)
    double A[kMaxKorobov + 1];
    double B[kMaxKorobov + 1];
    double C;                     // Korobov constant, or Sidi (pi/2^r) Gamma(r+1)/Gamma((r+1)/2)^2
    union {
        double sidi_c[kMaxSidi + 1];  // Sidi: phi = cr * I_r, I_r via the sin-power reduction
        struct {   // kTKorobovGen: binom(r0 + k, k) 2^kf, and binom(r1 + k, k) by itself, k <= deg
            uint64_t KA[kMaxKorobovInt + 1];
            uint16_t KB[kMaxKorobovInt + 1];
            uint8_t kf;
        };
    };
};

// One integral as the kernels see it: of a launch of its own (passed as a kernel parameter)
// or of a batch (qmc_batch_*: built on the host and kept in the workspace).
struct Integral {
    uint64_t n, i_begin, i_end;
    uint64_t tile_begin, tiles;   // index of the first tile in the launch, number of tiles
    uint64_t partial_off;         // offset of this integral's partials, in doubles
    uint32_t L;                   // points per stream and tile
    int d;
    double cd;                    // Korobov C^d, 1 for the other transforms
    DimConst dc[kMaxDim];
    const uint64_t *shifts;       // [m][d]
    TransformParams t;
    const double *fit;            // [d][6] or nullptr
    // integrand (device pointers; the kernel stages them in shared memory)
    int slot;                     // position of its sums, results and counters in the batch
    const double *c, *w;
    const int64_t *h;
    int nu, nf;
    const double *ucoef, *fcoef;
    const int32_t *uexp, *fexp;
    double pa, pb, lam;
};

// Launches of one batch, one after another in a stream, that share nothing but their inputs: each
// later one may start when all blocks of the one before it have started, and ends after it.
enum { kNoChain = 0, kChainFirst = 1, kChainLater = 2 };

// A launch of the lattice-sum kernel: one integral (items null) or the integrals items[0..count)
// whose tiles, laid end to end, are numbered by tile_begin[0..count]; all of one transform kind.
struct LatticeLaunch {
    Integral one;
    const Integral *items;
    const uint64_t *tile_begin;
    int count;
    int m, spb;                       // shifts, streams per block (blockDim = spb * m)
    int chain;                        // kNoChain, or its place among launches that may overlap
    uint64_t first_tile, end_tile;    // the tiles of this launch
    double *partials;                 // per integral: [tiles][m] (sum, comp) re, then im
    unsigned long long *counters;     // [2] per integral, or nullptr
};

}  // namespace qmc
