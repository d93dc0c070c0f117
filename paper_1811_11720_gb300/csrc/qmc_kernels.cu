// qmc_kernels.cu -- lattice points, fixed-order reductions, evaluate() and the fit
// histogram.
#include <cuda_runtime.h>

#include <cstdint>

#include "qmc_integrands.cuh"
#include "qmc_internal.h"
#include "qmc_lattice.cuh"
#include "qmc_reduce.cuh"
#include "qmc_transforms.cuh"

namespace qmc {

// ---- lattice points (Eq. (lattice), Fig. 1) --------------------------------------------
// The floor is the output's writes (m d doubles per point), so consecutive threads own
// consecutive doubles: thread (row, column) of a block of rows x cols threads keeps the state
// of one coordinate j under one shift k (column = k d + j) and steps it from point to point
// by `rows`, with the constants of `rows` lattice steps taken once as one.  More than 256
// columns are cut into equal chunks (blockIdx.y).  The instructions per double decide how
// near the floor it comes: ~75 with the remainder stepped and all three words rounded, which
// ran at 2.5 TB/s (1,072,187 points, d = 8, m = 4: 111 us; one thread per 64 points, its
// writes scattered: 381 us), ~40 with the short step and the short rounding of
// qmc_lattice.cuh: 61 us, 4.5 TB/s.
constexpr int kPointThreads = 256;

template <bool kShort>
__global__ void __launch_bounds__(kPointThreads) points_kernel(const __grid_constant__ PointsParams p) {
    const int width = p.m * p.d;
    const int row = threadIdx.x / p.cols;
    const int col = blockIdx.y * p.cols + (threadIdx.x - row * p.cols);
    if (col >= width) return;
    const uint64_t off = (uint64_t)blockIdx.x * p.steps * p.rows + row;
    if (off >= p.count) return;
    // this thread's points: off, off + rows, .. (at most `steps`)
    const uint64_t left = (p.count - off + p.rows - 1) / p.rows;
    const uint32_t cnt = left < p.steps ? (uint32_t)left : p.steps;
    const DimConst c = p.dc[col % p.d];
    const uint64_t n = p.n, dsh = p.shifts[col] << 11;   // shifts are [m][d]: row-major columns
    double *o = p.out + off * (uint64_t)width + col;
    const uint64_t stride = (uint64_t)p.rows * width;
    uint64_t fh, fl, rem;
    const uint64_t i0 = p.i_begin + off, rows = (uint64_t)p.rows;
    lattice_state_at(i0, c, n, fh, fl, rem);
    if constexpr (kShort) {
        const uint64_t w = short_step_word(c, n);
        LatticeStep step;   // `rows` steps at once
        lattice_state_at(rows, c, n, step.fz_hi, step.fz_lo, step.remz);
        const uint64_t step_w = rows * w;
        ShortState s{fh, fl, i0 * w};
        for (uint32_t q = 0; q < cnt; ++q) {
            __stcs(o, fixed_to_double(s.f_hi + dsh, s.f_lo, n));
            s.step(step.fz_hi, step.fz_lo, step_w);
            o += stride;
        }
    } else {
        LatticeStep step;
        lattice_state_at(rows, c, n, step.fz_hi, step.fz_lo, step.remz);
        for (uint32_t q = 0; q < cnt; ++q) {
            __stcs(o, fixed_to_double(fh + dsh, fl, n));
            lattice_step(step, n, fh, fl, rem);
            o += stride;
        }
    }
}

cudaError_t launch_points(PointsParams p, cudaStream_t s) {
    if (!p.count) return cudaSuccess;
    const int width = p.m * p.d;
    const int chunks = (width + kPointThreads - 1) / kPointThreads;
    p.cols = (width + chunks - 1) / chunks;
    p.rows = kPointThreads / p.cols;
    // steps per thread: as many as leave two waves of full SMs (a start costs about three
    // steps), at most 64
    const uint64_t passes = (p.count + p.rows - 1) / p.rows;
    const uint64_t want = passes * chunks / (2ull * 152 * 8);
    p.steps = (uint32_t)(want < 1 ? 1 : want > 64 ? 64 : want);
    uint64_t blocks = (passes + p.steps - 1) / p.steps;
    if (blocks > 0x7FFFFFFFull) {   // beyond the grid limit: longer streams
        p.steps = (uint32_t)((passes + 0x7FFFFFFEull) / 0x7FFFFFFFull);
        blocks = (passes + p.steps - 1) / p.steps;
    }
    const dim3 grid((unsigned)blocks, chunks);
    const int threads = p.rows * p.cols;
    if (p.n >> kShortBits) points_kernel<false><<<grid, threads, 0, s>>>(p);
    else points_kernel<true><<<grid, threads, 0, s>>>(p);
    return cudaGetLastError();
}

// ---- fixed-order reductions -------------------------------------------------------------
// One block per (shift, component).
__global__ void __launch_bounds__(kRedThreads) reduce_tiles_kernel(const double *partials,
                                                                   uint64_t tiles, int m,
                                                                   double *sums) {
    const int col = blockIdx.x;           // k + m * component
    const int comp = col / m, k = col % m;
    const SumPair acc = fold_tiles(partials + 2 * (uint64_t)comp * tiles * m, tiles, m, k);
    if (threadIdx.x == 0) {
        double *o = sums + 2 * (uint64_t)comp * m + 2 * k;
        o[0] = acc.hi;
        o[1] = acc.lo;
    }
}

cudaError_t launch_reduce_tiles(const double *partials, uint64_t tiles, int m, int is_complex,
                                double *sums, cudaStream_t s) {
    reduce_tiles_kernel<<<m * (is_complex ? 2 : 1), kRedThreads, 0, s>>>(partials, tiles, m, sums);
    return cudaGetLastError();
}

// Eq. (lattice) and Eq. (lattice-error): Q_k = S_k / n, one thread per shift and component,
// then Qbar and sigma, one warp per component.
constexpr int kFinThreads = 256;

__global__ void __launch_bounds__(kFinThreads)
    finalize_kernel(const double *__restrict__ sums, int m, uint64_t n, int is_complex,
                    double *__restrict__ result, double *__restrict__ Q) {
    __shared__ double q_s[2 * QMC_MAX_SHIFTS];
    const double dn = (double)n;
    const int ncomp = is_complex ? 2 : 1;
    for (int i = threadIdx.x; i < ncomp * m; i += blockDim.x) {
        const int comp = i / m, k = i - comp * m;
        const double *sc = sums + 2 * (size_t)comp * m;
        const double q = (sc[2 * k] + sc[2 * k + 1]) / dn;
        q_s[i] = q;
        if (Q) Q[i] = q;
    }
    if (!is_complex && threadIdx.x < 2) result[2 + threadIdx.x] = 0.0;
    __syncthreads();
    const int comp = threadIdx.x >> 5;
    if (comp >= ncomp) return;
    const double *qc = q_s + (size_t)comp * m;
    shift_stats(m, [&](int k) { return qc[k]; }, result + 2 * comp);
}

cudaError_t launch_finalize(const double *sums, int m, uint64_t n, int is_complex,
                            double *result, double *Q, cudaStream_t s) {
    const int work = m * (is_complex ? 2 : 1);
    const int least = is_complex ? 64 : 32;   // a warp per component
    const int threads = work >= kFinThreads ? kFinThreads : ((work + 31) / 32) * 32;
    finalize_kernel<<<1, threads < least ? least : threads, 0, s>>>(sums, m, n, is_complex, result, Q);
    return cudaGetLastError();
}

// ---- evaluate(): raw f on one shifted lattice, no transform ---------------------------
template <int FAM>
__device__ __forceinline__ void eval_point(const FamilyShared<FAM> &fsh, const double *x, int d,
                                           double &re, double &im, unsigned long long &sf) {
    FamilyAcc<FAM> fa;
    fa.init(fsh);
#pragma unroll
    for (int j = 0; j < kMaxDim; ++j)
        if (j < d) fa.add(j, Mapped{x[j], false}, fsh);
    fa.finish(d, fsh, re, im, sf);
}

constexpr int kEvalThreads = 128;
constexpr uint32_t kEvalChunk = 16;   // points a thread: latency-bound, and a start costs about three steps

template <int FAM>
__global__ void __launch_bounds__(kEvalThreads) evaluate_kernel(const Integral p, double *out) {
    __shared__ FamilyShared<FAM> fsh;
    stage_family<FAM>(p, fsh);
    __syncthreads();
    const int d = p.d;
    const uint64_t count = p.i_end - p.i_begin;
    uint64_t dsh[kMaxDim];
#pragma unroll
    for (int j = 0; j < kMaxDim; ++j) dsh[j] = (j < d) ? (p.shifts[j] << 11) : 0ull;
    for (uint64_t off = ((uint64_t)blockIdx.x * kEvalThreads + threadIdx.x) * kEvalChunk; off < count;
         off += (uint64_t)gridDim.x * kEvalThreads * kEvalChunk) {
        const uint64_t cnt = (count - off < kEvalChunk) ? count - off : kEvalChunk;
        uint64_t fhi[kMaxDim], flo[kMaxDim], rem[kMaxDim];
#pragma unroll
        for (int j = 0; j < kMaxDim; ++j)
            if (j < d) lattice_state_at(p.i_begin + off, p.dc[j], p.n, fhi[j], flo[j], rem[j]);
        for (uint64_t q = 0; q < cnt; ++q) {
            double x[kMaxDim];
#pragma unroll
            for (int j = 0; j < kMaxDim; ++j) {
                x[j] = 0.0;
                if (j < d) {
                    x[j] = fixed_to_double(fhi[j] + dsh[j], flo[j], p.n);
                    lattice_step(lattice_step_of(p.dc[j], p.n), p.n, fhi[j], flo[j], rem[j]);
                }
            }
            double re, im;
            unsigned long long sf = 0;
            eval_point<FAM>(fsh, x, d, re, im, sf);
            if constexpr (FamilyAcc<FAM>::kComplex) {
                out[2 * (off + q)] = re;
                out[2 * (off + q) + 1] = im;
            } else {
                out[off + q] = re;
            }
        }
    }
}

// ---- histogram of |f| per dimension (fit data pass, Sec. 2.4) --------------------------
// Each block walks batches of kHistThreads points: every thread evaluates one, then warp w
// adds the batch to dimensions w, w + 8, ..., 32 points at a time in point order.  Points of
// one group that share a bin (match_any finds them) are first summed in lane order by the
// lowest of them, so the result is deterministic.  Block histograms go to
// work[block][d][bins] and are summed over the blocks in a fixed order by hist_sum_kernel.
// Bound by the evaluations once the adds run 32 wide and the points are spread over enough
// blocks (host: ~512 points each): one thread per dimension adding 128 points one after the
// other, in blocks of 4096, took 519 us for the 1.1e5 evaluations of a d = 5 sector
// integrand, of the 1764 us of the whole fitting call (the sums' fit map since changed too:
// 755 us now).
constexpr int kHistThreads = 256;

template <int FAM>
__global__ void __launch_bounds__(kHistThreads) histogram_kernel(const Integral p, int bins,
                                                                 double *work) {
    extern __shared__ double hsm[];   // [d][bins]
    __shared__ FamilyShared<FAM> fsh;
    __shared__ double val[kHistThreads];
    __shared__ uint16_t bin[kMaxDim][kHistThreads];
    stage_family<FAM>(p, fsh);
    const int d = p.d;
    for (int q = threadIdx.x; q < d * bins; q += kHistThreads) hsm[q] = 0.0;
    __syncthreads();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const uint64_t n = p.n;
    const uint64_t per_block = (n + gridDim.x - 1) / gridDim.x;
    const uint64_t b0 = (uint64_t)blockIdx.x * per_block;
    const uint64_t b1 = (b0 + per_block < n) ? b0 + per_block : n;
    for (uint64_t base = b0; base < b1; base += kHistThreads) {
        const uint64_t i = base + threadIdx.x;
        double v = 0.0;
        if (i < b1) {
            double x[kMaxDim];
#pragma unroll
            for (int j = 0; j < kMaxDim; ++j) {
                x[j] = 0.0;
                if (j < d) {
                    uint64_t fh, fl, rm;
                    lattice_state_at(i, p.dc[j], n, fh, fl, rm);
                    x[j] = fixed_to_double(fh + (p.shifts[j] << 11), fl, n);
                    int b = (int)floor(x[j] * (double)bins);
                    bin[j][threadIdx.x] = (uint16_t)(b >= bins ? bins - 1 : b);
                }
            }
            double re, im;
            unsigned long long sf = 0;
            eval_point<FAM>(fsh, x, d, re, im, sf);
            v = FamilyAcc<FAM>::kComplex ? hypot(re, im) : fabs(re);
        }
        val[threadIdx.x] = v;
        __syncthreads();
        const int lim = b1 - base < kHistThreads ? (int)(b1 - base) : kHistThreads;
        for (int j = warp; j < d; j += kHistThreads / 32) {
            double *h = hsm + j * bins;
            for (int g = 0; g < lim; g += 32) {
                const bool in = g + lane < lim;
                const int b = in ? bin[j][g + lane] : -1;
                double s = in ? val[g + lane] : 0.0;
                const unsigned same = __match_any_sync(0xFFFFFFFFu, b);
                const bool first = lane == __ffs(same) - 1;
                const double mine = s;
                unsigned rest = first ? same & (same - 1) : 0u;   // the others, in lane order
                while (__any_sync(0xFFFFFFFFu, rest != 0)) {
                    const double o = __shfl_sync(0xFFFFFFFFu, mine, rest ? __ffs(rest) - 1 : lane);
                    if (rest) s += o;
                    rest &= rest - 1;
                }
                if (in && first) h[b] += s;
                __syncwarp();
            }
        }
        __syncthreads();
    }
    for (int q = threadIdx.x; q < d * bins; q += kHistThreads)
        work[(size_t)blockIdx.x * d * bins + q] = hsm[q];
}

// Compensated sums over the blocks: kSumParts threads per cell take every kSumParts-th block
// in order, then their (sum, compensation) pairs are added in order.
constexpr int kSumCells = 32, kSumParts = 8;

__device__ __forceinline__ void comp_add(double &s, double &c, double v) {
    const double t = s + v;
    c += (fabs(s) >= fabs(v)) ? (s - t) + v : (v - t) + s;
    s = t;
}

__global__ void __launch_bounds__(kSumCells *kSumParts)
    hist_sum_kernel(const double *work, uint32_t nblocks, int cells, double *hist) {
    __shared__ double part[kSumParts][kSumCells][2];
    const int x = threadIdx.x % kSumCells, y = threadIdx.x / kSumCells;
    const int q = blockIdx.x * kSumCells + x;
    double s = 0.0, c = 0.0;
    if (q < cells) {
#pragma unroll 4
        for (uint32_t b = y; b < nblocks; b += kSumParts) comp_add(s, c, work[(size_t)b * cells + q]);
    }
    part[y][x][0] = s;
    part[y][x][1] = c;
    __syncthreads();
    if (y == 0 && q < cells) {
        for (int k = 1; k < kSumParts; ++k) {
            comp_add(s, c, part[k][x][0]);
            c += part[k][x][1];
        }
        hist[q] = s + c;
    }
}

template <int FAM>
static cudaError_t eval_dispatch_one(const Integral &p, double *out, cudaStream_t s) {
    uint64_t count = p.i_end - p.i_begin;
    uint64_t chunks = (count + kEvalChunk - 1) / kEvalChunk;
    uint32_t blocks = (uint32_t)((chunks + kEvalThreads - 1) / kEvalThreads);
    if (blocks > 65535u * 16u) blocks = 65535u * 16u;
    if (blocks == 0) return cudaSuccess;
    evaluate_kernel<FAM><<<blocks, kEvalThreads, 0, s>>>(p, out);
    return cudaGetLastError();
}

template <int FAM>
static cudaError_t hist_dispatch_one(const Integral &p, int bins, double *hist, double *work,
                                     uint32_t nblocks, cudaStream_t s) {
    // the limit is state of the function that all threads share: always the largest histogram's
    // size, so that no call lowers it under another one's launch
    const size_t smem = (size_t)p.d * bins * sizeof(double);
    cudaError_t e = cudaFuncSetAttribute(histogram_kernel<FAM>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)(kHistCells * sizeof(double)));
    if (e != cudaSuccess) return e;
    histogram_kernel<FAM><<<nblocks, kHistThreads, smem, s>>>(p, bins, work);
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    int cells = p.d * bins;
    hist_sum_kernel<<<(cells + kSumCells - 1) / kSumCells, kSumCells * kSumParts, 0, s>>>(work, nblocks, cells, hist);
    return cudaGetLastError();
}

#define QMC_FAMILY_SWITCH(FN, ...)                                                      \
    switch (family) {                                                                 \
    case QMC_GENZ_OSCILLATORY: return FN<QMC_GENZ_OSCILLATORY>(__VA_ARGS__);            \
    case QMC_GENZ_PRODUCT_PEAK: return FN<QMC_GENZ_PRODUCT_PEAK>(__VA_ARGS__);          \
    case QMC_GENZ_CORNER_PEAK: return FN<QMC_GENZ_CORNER_PEAK>(__VA_ARGS__);            \
    case QMC_GENZ_GAUSSIAN: return FN<QMC_GENZ_GAUSSIAN>(__VA_ARGS__);                  \
    case QMC_GENZ_C0: return FN<QMC_GENZ_C0>(__VA_ARGS__);                              \
    case QMC_GENZ_DISCONTINUOUS: return FN<QMC_GENZ_DISCONTINUOUS>(__VA_ARGS__);        \
    case QMC_MONOMIAL: return FN<QMC_MONOMIAL>(__VA_ARGS__);                            \
    case QMC_TRIG: return FN<QMC_TRIG>(__VA_ARGS__);                                    \
    case QMC_SECTOR: return FN<QMC_SECTOR>(__VA_ARGS__);                                \
    case QMC_FEYNMAN: return FN<QMC_FEYNMAN>(__VA_ARGS__);                              \
    default: return cudaErrorInvalidValue;                                              \
    }

cudaError_t launch_evaluate(int family, const Integral &p, double *out, cudaStream_t s) {
    QMC_FAMILY_SWITCH(eval_dispatch_one, p, out, s)
}

cudaError_t launch_histogram(int family, const Integral &p, int bins, double *hist, double *work,
                             uint32_t nblocks, cudaStream_t s) {
    QMC_FAMILY_SWITCH(hist_dispatch_one, p, bins, hist, work, nblocks, s)
}

int sm_count() {
    int dev = 0, n = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return 0;
    if (cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) return 0;
    return n;
}

}  // namespace qmc
