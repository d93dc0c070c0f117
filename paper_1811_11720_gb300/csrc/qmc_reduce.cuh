// qmc_reduce.cuh -- fixed-order reductions shared by the single-integral and the batched forms
// (both give the same bits): tile partials to per-shift sums, per-shift sums to mean and error.
#pragma once
#include <cstdint>

namespace qmc {

// A sum as an unnormalized pair: hi is the running double sum, lo collects the rounding errors
// of its additions (TwoSum) and the partials' own compensations.  Eight FP64 operations per
// addition of which only hi's is on the chain from one addition to the next; renormalizing
// after each (double-double addition) costs eleven, nine of them in a chain.
struct SumPair {
    double hi = 0.0, lo = 0.0;
    __device__ __forceinline__ void add(double h, double l) {
        const double s = hi + h;
        const double b = s - hi;
        lo += ((hi - (s - b)) + (h - b)) + l;
        hi = s;
    }
};

constexpr int kRedThreads = 256;

// Folds column `col`'s (sum, compensation) pairs of `tiles` tiles, pair t at base[2 (t m + col)]:
// thread t takes tiles t, t + 256, ... in order, then a fixed halving tree over the threads that
// have any.  Block of kRedThreads; the result is valid in thread 0.
// FP64-bound: a warp addition is eight instructions of ~17 SM cycles.  The tree halves across
// warps in shared memory and only then by shuffles within the first one, at most 12 warp additions
// and none for threads without tiles; a shuffle tree in every warp took 43, and the 8192 blocks of
// a batch of 256 integrals of 16 tiles and 32 shifts 181 us; 30 us now.
__device__ __forceinline__ SumPair fold_tiles(const double *base, uint64_t tiles, int m, int col) {
    __shared__ double part_hi[kRedThreads], part_lo[kRedThreads];
    const double *p = base + 2 * col;   // 8-byte aligned, no more is asked of the caller
    const int tid = threadIdx.x;
    SumPair acc;
#pragma unroll 4
    for (uint64_t t = tid; t < tiles; t += kRedThreads) {
        const double *v = p + 2 * t * (uint64_t)m;
        acc.add(v[0], v[1]);
    }
    const int used = tiles < kRedThreads ? (int)tiles : kRedThreads;
    for (int w = kRedThreads / 2; w >= 32; w >>= 1) {
        if (used <= w) continue;
        if (tid >= w && tid < 2 * w) {
            part_hi[tid] = acc.hi;
            part_lo[tid] = acc.lo;
        }
        __syncthreads();
        if (tid < w) acc.add(part_hi[tid + w], part_lo[tid + w]);
    }
    if (tid < 32) {
        for (int w = 16; w > 0; w >>= 1) {
            if (used <= w) continue;
            const double h = __shfl_down_sync(0xFFFFFFFFu, acc.hi, w);
            const double l = __shfl_down_sync(0xFFFFFFFFu, acc.lo, w);
            acc.add(h, l);
        }
        const double s = acc.hi + acc.lo;   // normalized: |lo| is far below |hi|
        acc.lo = acc.lo - (s - acc.hi);
        acc.hi = s;
    }
    return acc;
}

// Mean and standard error of Q_0..Q_(m-1), value(k) each, by one warp: lane l takes k = l,
// l + 32, ... in order, then a fixed tree.  (Eq. (lattice), Eq. (lattice-error).)
template <class Value>
__device__ __forceinline__ void shift_stats(int m, Value value, double *result) {
    const int lane = threadIdx.x & 31;
    auto all = [](double v) {
        for (int w = 16; w > 0; w >>= 1) v += __shfl_xor_sync(0xFFFFFFFFu, v, w);
        return v;
    };
    double s = 0.0;
    for (int k = lane; k < m; k += 32) s += value(k);
    const double mean = all(s) / (double)m;
    double var = 0.0;
    for (int k = lane; k < m; k += 32) {
        const double dq = value(k) - mean;
        var = fma(dq, dq, var);
    }
    var = all(var) / ((double)m * (double)(m - 1));
    if (lane == 0) {
        result[0] = mean;
        result[1] = sqrt(var);
    }
}

}  // namespace qmc
