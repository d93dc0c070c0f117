// qmc_cbc.cu -- fast component-by-component construction of rank-1 lattice generating
// vectors on the GPU (App. A.3 table of generating vectors; the fast CBC of Nuyens and
// Cools, with cuFFT for the cyclic convolutions).
//
// Korobov space of smoothness alpha = 2 with product weights: the squared worst-case error
// of z = (z_1..z_s) on n points is
//     e^2(z) = -1 + (1/n) sum_{k=0}^{n-1} prod_{l<=s} (beta + gamma omega({k z_l / n})),
//     omega(x) = 2 pi^2 (x^2 - x + 1/6),
// and CBC fixes z_1 = 1, then picks each z_j in 1..n-1 minimising e^2 given z_1..z_(j-1).
// Only T(z) = sum_k p(k) omega({k z / n}) depends on the candidate, with p(k) the product of
// the factors of the earlier components.  For prime n and a primitive root g, z = g^a and
// k = g^-b give {k z / n} = {g^(a-b) / n}: T is a cyclic convolution over the group of
// units.  Because g^((n-1)/2) = -1, omega(x) = omega(1 - x) and p(k) = p(n - k), it folds to
// length H = (n-1)/2:
//     T(g^a) = p(0) omega(0) + 2 sum_{b<H} p(g^-b) omega({g^(a-b) / n}),   a < H,
// and the candidates are the representatives min(g^a, n - g^a) <= H.  The cyclic
// convolution of length H is taken from a linear one: with W2 = (W, W) of length 2H and
// P zero-padded, (P * W2)[a + H] = sum_b P[b] W[(a - b) mod H] for a < H, and any transform
// length L >= 2H keeps those indices free of wrap-around; L is chosen 7-smooth so that
// cuFFT runs its mixed-radix kernels whatever the factors of H.  Each component costs one
// real-to-complex FFT of length L, a pointwise product with the (once transformed) W2, one
// complex-to-real FFT, a minimum search and an update of p.
//
// Ties: sums within 1e-14 omega(0) sum_k p(k) of the minimum are ties, and the smallest
// candidate wins (the same reading as the CPU construction that wrote the shipped table).
#include <cuda_runtime.h>
#include <cufft.h>

#include <algorithm>
#include <cmath>
#include <cstdint>
#include <cstring>
#include <memory>
#include <mutex>
#include <new>
#include <vector>

#include "qmc_gb300.h"
#include "qmc_hostutil.h"

namespace qmc {
namespace {

constexpr double kTwoPi2 = 19.739208802178717237668981999752;   // 2 pi^2
constexpr double kTieRtol = 1e-14;
constexpr int kCbcThreads = 256;

__host__ __device__ inline double omega_k(double x) { return kTwoPi2 * (x * x - x + 1.0 / 6.0); }

// Arithmetic modulo n with what it needs precomputed: n < 2^32 takes the quotient from the
// 64-bit reciprocal floor(2^64 / n) (at most 2 low), larger n < 2^53 an FP64 estimate (within 2
// of the exact one); the remainder is then corrected exactly.
struct Modulus {
    uint64_t n, inv;   // inv = floor(2^64 / n) for n < 2^32, else 0
};

__device__ __forceinline__ uint64_t mulmod_dev(uint64_t a, uint64_t b, const Modulus &m) {
    const uint64_t lo = a * b;
    if (m.inv) {
        uint64_t r = lo - __umul64hi(lo, m.inv) * m.n;
        if (r >= 2 * m.n) r -= 2 * m.n;
        return r >= m.n ? r - m.n : r;
    }
    const double qd = floor((double)a * (double)b / (double)m.n);
    const uint64_t q = qd <= 0.0 ? 0ull : (uint64_t)qd;
    long long r = (long long)(lo - q * m.n);   // the exact a b - q n, within (-2n, 3n)
#pragma unroll 1
    for (int it = 0; it < 4 && r < 0; ++it) r += (long long)m.n;
#pragma unroll 1
    for (int it = 0; it < 4 && r >= (long long)m.n; ++it) r -= (long long)m.n;
    return (uint64_t)r;
}

__device__ __forceinline__ uint64_t powmod_dev(uint64_t g, uint64_t e, const Modulus &m) {
    uint64_t r = 1 % m.n, b = g % m.n;
#pragma unroll 1
    while (e) {
        if (e & 1) r = mulmod_dev(r, b, m);
        b = mulmod_dev(b, b, m);
        e >>= 1;
    }
    return r;
}

inline uint64_t mulmod_host(uint64_t a, uint64_t b, uint64_t n) {
    return (uint64_t)((unsigned __int128)a * b % n);
}
inline uint64_t powmod_host(uint64_t g, uint64_t e, uint64_t n) {
    uint64_t r = 1 % n, b = g % n;
    while (e) {
        if (e & 1) r = mulmod_host(r, b, n);
        b = mulmod_host(b, b, n);
        e >>= 1;
    }
    return r;
}

// Deterministic Miller-Rabin for 64-bit integers (the first 12 primes as bases).
bool is_prime_u64(uint64_t n) {
    if (n < 2) return false;
    static const uint64_t small[] = {2, 3, 5, 7, 11, 13, 17, 19, 23, 29, 31, 37};
    for (uint64_t p : small) {
        if (n % p == 0) return n == p;
    }
    uint64_t d = n - 1;
    int r = 0;
    while (!(d & 1)) {
        d >>= 1;
        ++r;
    }
    for (uint64_t a : small) {
        uint64_t x = powmod_host(a, d, n);
        if (x == 1 || x == n - 1) continue;
        bool comp = true;
        for (int i = 1; i < r; ++i) {
            x = mulmod_host(x, x, n);
            if (x == n - 1) {
                comp = false;
                break;
            }
        }
        if (comp) return false;
    }
    return true;
}

// Smallest primitive root of the prime n: g is one when g^((n-1)/q) != 1 for every prime
// factor q of n - 1.
uint64_t primitive_root(uint64_t n) {
    std::vector<uint64_t> qs;
    uint64_t m = n - 1;
    for (uint64_t q = 2; q * q <= m; ++q) {
        if (m % q == 0) {
            qs.push_back(q);
            while (m % q == 0) m /= q;
        }
    }
    if (m > 1) qs.push_back(m);
    for (uint64_t g = 2; g < n; ++g) {
        bool ok = true;
        for (uint64_t q : qs) {
            if (powmod_host(g, (n - 1) / q, n) == 1) {
                ok = false;
                break;
            }
        }
        if (ok) return g;
    }
    return 0;
}

// gp[c] = g^c mod n for c < H; thread t fills [t B, t B + B).
__global__ void cbc_powers_kernel(uint64_t g, Modulus m, uint64_t H, uint64_t B, uint64_t *gp) {
    const uint64_t t = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const uint64_t c0 = t * B;
    if (c0 >= H) return;
    uint64_t x = powmod_dev(g, c0, m);
    const uint64_t c1 = c0 + B < H ? c0 + B : H;
#pragma unroll 1
    for (uint64_t c = c0; c < c1; ++c) {
        gp[c] = x;
        x = mulmod_dev(x, g, m);
    }
}

// w[c] = w[c + H] = omega(g^c / n) for c < H, zero on [2H, L)
__global__ void cbc_omega_kernel(const uint64_t *gp, uint64_t H, uint64_t L, uint64_t n, double *w) {
    for (uint64_t c = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; c < L;
         c += (uint64_t)gridDim.x * blockDim.x) {
        if (c < 2 * H) {
            const uint64_t c0 = c < H ? c : c - H;
            w[c] = omega_k((double)gp[c0] / (double)n);
        } else {
            w[c] = 0.0;
        }
    }
}

// Blocks of the block-wise reductions, and what one component leaves for the next.
constexpr unsigned kCbcBlocks = 152 * 8;

// The choice of the previous component from its blocks' picks: the smallest representative
// (n when there is none) and its T.  Every thread returns the same.
__device__ __forceinline__ uint64_t cbc_choice(const uint64_t *rep, const double *t, unsigned blocks,
                                               uint64_t n, double *t_best) {
    __shared__ uint64_t sr[kCbcThreads];
    __shared__ double st[kCbcThreads];
    uint64_t best = n;
    double bt = 0.0;
    for (unsigned b = threadIdx.x; b < blocks; b += kCbcThreads)
        if (rep[b] < best) {
            best = rep[b];
            bt = t[b];
        }
    sr[threadIdx.x] = best;
    st[threadIdx.x] = bt;
    __syncthreads();
    for (int w = kCbcThreads / 2; w > 0; w >>= 1) {
        if ((int)threadIdx.x < w && sr[threadIdx.x + w] < sr[threadIdx.x]) {
            sr[threadIdx.x] = sr[threadIdx.x + w];
            st[threadIdx.x] = st[threadIdx.x + w];
        }
        __syncthreads();
    }
    *t_best = st[0];
    return sr[0];
}

// Component j: z_1 = 1, later ones the choice of the previous picks.  p[k] *= beta + gamma
// omega({k z / n}) for k <= H (p[k] = the factor for j = 0), and the block sums of p[1..H] (a
// fixed order within a block; the host adds the blocks in order).  z, its T, p[0] and the
// block sums of every component stay on the device until the last one.
__global__ void __launch_bounds__(kCbcThreads)
    cbc_update_kernel(double *p, uint64_t H, Modulus m, double beta, double gamma, int j,
                      unsigned pick_blocks, const uint64_t *rep, const double *rep_t,
                      uint64_t per_block, uint64_t *z_out, double *t_out, double *p0_out, double *sums) {
    __shared__ double s[kCbcThreads];
    uint64_t z = 1;
    double tz = 0.0;
    if (j) z = cbc_choice(rep, rep_t, pick_blocks, m.n, &tz);
    auto update = [&](uint64_t k) {
        const double f = fma(gamma, omega_k((double)mulmod_dev(k, z, m) / (double)m.n), beta);
        const double v = j ? p[k] * f : f;
        p[k] = v;
        return v;
    };
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        p0_out[j] = update(0);
        z_out[j] = z;
        t_out[j] = tz;
    }
    const uint64_t lo = 1 + (uint64_t)blockIdx.x * per_block;
    const uint64_t hi = lo + per_block < H + 1 ? lo + per_block : H + 1;
    double acc = 0.0;
    for (uint64_t k = lo + threadIdx.x; k < hi; k += kCbcThreads) acc += update(k);
    s[threadIdx.x] = acc;
    __syncthreads();
    for (int w = kCbcThreads / 2; w > 0; w >>= 1) {
        if ((int)threadIdx.x < w) s[threadIdx.x] += s[threadIdx.x + w];
        __syncthreads();
    }
    if (threadIdx.x == 0) sums[(uint64_t)j * kCbcBlocks + blockIdx.x] = s[0];
}

// P[b] = p(min(g^-b, n - g^-b)) for b < H (g^-b = n - g^(H - b) for b >= 1, g^0 = 1), zero
// on [H, L).
__global__ void cbc_gather_kernel(const uint64_t *gp, const double *p, uint64_t H, uint64_t L,
                                  uint64_t n, double *P) {
    for (uint64_t b = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; b < L;
         b += (uint64_t)gridDim.x * blockDim.x) {
        if (b >= H) {
            P[b] = 0.0;
            continue;
        }
        uint64_t k = 1;
        if (b) {
            const uint64_t v = gp[H - b];
            k = v < n - v ? v : n - v;
        }
        P[b] = p[k];
    }
}

__global__ void cbc_pointwise_kernel(cufftDoubleComplex *a, const cufftDoubleComplex *b,
                                     uint64_t m) {
    for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < m;
         i += (uint64_t)gridDim.x * blockDim.x) {
        const cufftDoubleComplex x = a[i], y = b[i];
        a[i] = make_cuDoubleComplex(fma(x.x, y.x, -x.y * y.y), fma(x.x, y.y, x.y * y.x));
    }
}

// T[a] = scale raw[a] + off, a < H, with off = p(0) omega(0) of the current p.
__device__ __forceinline__ double cbc_offset(const double *p) { return __dmul_rn(p[0], omega_k(0.0)); }

// Per-block minimum of T.
__global__ void __launch_bounds__(kCbcThreads)
    cbc_min_kernel(const double *raw, const double *p, uint64_t H, double scale, uint64_t per_block,
                   double *out) {
    __shared__ double s[kCbcThreads];
    const double off = cbc_offset(p);
    const uint64_t lo = (uint64_t)blockIdx.x * per_block;
    const uint64_t hi = lo + per_block < H ? lo + per_block : H;
    double m = INFINITY;
    for (uint64_t a = lo + threadIdx.x; a < hi; a += kCbcThreads) m = fmin(m, fma(scale, raw[a], off));
    s[threadIdx.x] = m;
    __syncthreads();
    for (int w = kCbcThreads / 2; w > 0; w >>= 1) {
        if ((int)threadIdx.x < w) s[threadIdx.x] = fmin(s[threadIdx.x], s[threadIdx.x + w]);
        __syncthreads();
    }
    if (threadIdx.x == 0) out[blockIdx.x] = s[0];
}

// Per block: the smallest representative min(g^a, n - g^a) among a with T[a] <= bound, and
// its T (representative n when none).  The bound is the least of the blocks' minima plus the
// tie tolerance of sum_k p(k) (psums: block sums of p[1..H]).
__global__ void __launch_bounds__(kCbcThreads)
    cbc_pick_kernel(const double *raw, const uint64_t *gp, const double *p, uint64_t H, uint64_t n,
                    double scale, uint64_t per_block, const double *mins, unsigned min_blocks,
                    const double *psums, uint64_t *rep_out, double *t_out) {
    __shared__ uint64_t sr[kCbcThreads];
    __shared__ double st[kCbcThreads], sm[kCbcThreads];
    double least = INFINITY, sum = 0.0;
    for (unsigned b = threadIdx.x; b < min_blocks; b += kCbcThreads) least = fmin(least, mins[b]);
    for (unsigned b = threadIdx.x; b < kCbcBlocks; b += kCbcThreads) sum += psums[b];
    sm[threadIdx.x] = least;
    st[threadIdx.x] = sum;
    __syncthreads();
    for (int w = kCbcThreads / 2; w > 0; w >>= 1) {
        if ((int)threadIdx.x < w) {
            sm[threadIdx.x] = fmin(sm[threadIdx.x], sm[threadIdx.x + w]);
            st[threadIdx.x] += st[threadIdx.x + w];
        }
        __syncthreads();
    }
    const double bound = sm[0] + kTieRtol * omega_k(0.0) * (p[0] + 2.0 * st[0]);
    __syncthreads();
    const double off = cbc_offset(p);
    const uint64_t lo = (uint64_t)blockIdx.x * per_block;
    const uint64_t hi = lo + per_block < H ? lo + per_block : H;
    uint64_t best = n;
    double bt = INFINITY;
    for (uint64_t a = lo + threadIdx.x; a < hi; a += kCbcThreads) {
        const double t = fma(scale, raw[a], off);
        if (t <= bound) {
            const uint64_t v = gp[a];
            const uint64_t rep = v < n - v ? v : n - v;
            if (rep < best) {
                best = rep;
                bt = t;
            }
        }
    }
    sr[threadIdx.x] = best;
    st[threadIdx.x] = bt;
    __syncthreads();
    for (int w = kCbcThreads / 2; w > 0; w >>= 1) {
        if ((int)threadIdx.x < w && sr[threadIdx.x + w] < sr[threadIdx.x]) {
            sr[threadIdx.x] = sr[threadIdx.x + w];
            st[threadIdx.x] = st[threadIdx.x + w];
        }
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        rep_out[blockIdx.x] = sr[0];
        t_out[blockIdx.x] = st[0];
    }
}

// Two cuFFT plans of length L, without work areas.  Making them takes two to four milliseconds,
// more than a construction of a middle size runs for (n = 108,863, s = 10: 2.0 ms, of which 0.13
// allocating and freeing), so up to kKept
// pairs wait for the next call of the same device and length; a call takes one out for itself (calls
// from several threads or streams do not share any) and gives it back when its stream has drained.
// The buffers, work area included, are the call's own.
struct Plans {
    int device = -1;
    uint64_t L = 0;
    size_t work_bytes = 0;   // the larger of the two plans' work areas
    cufftHandle fwd = 0, inv = 0;
    bool have_fwd = false, have_inv = false;
    Plans() = default;
    Plans(const Plans &) = delete;
    Plans &operator=(const Plans &) = delete;
    ~Plans() {
        if (have_fwd) cufftDestroy(fwd);
        if (have_inv) cufftDestroy(inv);
    }
    bool make(uint64_t length) {
        long long len = (long long)length;
        size_t wf = 0, wi = 0;
        if (cudaGetDevice(&device) != cudaSuccess) return false;
        L = length;
        if (cufftCreate(&fwd) != CUFFT_SUCCESS) return false;
        have_fwd = true;
        if (cufftCreate(&inv) != CUFFT_SUCCESS) return false;
        have_inv = true;
        if (cufftSetAutoAllocation(fwd, 0) != CUFFT_SUCCESS || cufftSetAutoAllocation(inv, 0) != CUFFT_SUCCESS ||
            cufftMakePlanMany64(fwd, 1, &len, nullptr, 1, 0, nullptr, 1, 0, CUFFT_D2Z, 1, &wf) != CUFFT_SUCCESS ||
            cufftMakePlanMany64(inv, 1, &len, nullptr, 1, 0, nullptr, 1, 0, CUFFT_Z2D, 1, &wi) != CUFFT_SUCCESS)
            return false;
        work_bytes = wf > wi ? wf : wi;
        return true;
    }
    bool use(char *work, cudaStream_t st) {
        return cufftSetWorkArea(fwd, work) == CUFFT_SUCCESS && cufftSetWorkArea(inv, work) == CUFFT_SUCCESS &&
               cufftSetStream(fwd, st) == CUFFT_SUCCESS && cufftSetStream(inv, st) == CUFFT_SUCCESS;
    }
};

constexpr size_t kKept = 2;
std::mutex g_kept_mutex;
// never destroyed: at process exit the driver may be gone before static destructors run
struct Kept {
    std::unique_ptr<Plans> plans[kKept];   // oldest first
};
Kept &kept() {
    static auto *v = new Kept;
    return *v;
}

std::unique_ptr<Plans> take_plans(uint64_t L) {
    int dev = -1;
    if (cudaGetDevice(&dev) != cudaSuccess) return nullptr;
    {
        std::lock_guard<std::mutex> lock(g_kept_mutex);
        for (auto &p : kept().plans)
            if (p && p->device == dev && p->L == L) return std::move(p);
    }
    std::unique_ptr<Plans> p(new (std::nothrow) Plans);
    if (p && !p->make(L)) p.reset();
    return p;
}

void give_back(std::unique_ptr<Plans> p) {
    std::unique_ptr<Plans> old;   // destroyed outside the lock
    std::lock_guard<std::mutex> lock(g_kept_mutex);
    auto &v = kept().plans;
    size_t at = 0;
    while (at < kKept && v[at]) ++at;
    if (at == kKept) {
        old = std::move(v[0]);
        for (at = 0; at + 1 < kKept; ++at) v[at] = std::move(v[at + 1]);
    }
    v[at] = std::move(p);
}

struct DeviceBuffer {
    char *base = nullptr;
    ~DeviceBuffer() {
        if (base) cudaFree(base);
    }
};

// Smallest 2^a 3^b 5^c 7^d >= x.
uint64_t smooth_at_least(uint64_t x) {
    uint64_t best = ~0ull;
    for (uint64_t p7 = 1; p7 < 2 * x; p7 *= 7)
        for (uint64_t p5 = p7; p5 < 2 * x; p5 *= 5)
            for (uint64_t p3 = p5; p3 < 2 * x; p3 *= 3) {
                uint64_t v = p3;
                while (v < x) v *= 2;
                if (v < best) best = v;
            }
    return best;
}

unsigned grid_for(uint64_t work) {
    const uint64_t g = (work + kCbcThreads - 1) / kCbcThreads;
    return (unsigned)(g < 152ull * 64 ? (g ? g : 1) : 152ull * 64);
}

}  // namespace
}  // namespace qmc

using namespace qmc;

extern "C" size_t qmc_cbc_device_bytes(uint64_t n) {
    if (n < 5) return 0;
    const uint64_t H = (n - 1) / 2;
    const uint64_t L = smooth_at_least(2 * H);
    // gp (8 H), p (8 (H + 1)), P/T (8 L), FP and FW (16 (L/2 + 1) each)
    return (size_t)(8 * H + 8 * (H + 1) + 8 * L + 32 * (L / 2 + 1));
}

extern "C" int qmc_cbc_korobov(uint64_t n, int s, double gamma, double beta, uint64_t *z_out,
                               double *e2_out, void *stream) {
    if (!z_out || s < 1 || s > 1024 || n < 5 || n >= (1ull << 53) || !(beta > 0.0) ||
        !(gamma >= 0.0) || !is_prime_u64(n))
        return QMC_ERR_ARG;
    if (const int e = host::device_ok()) return e;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    const uint64_t H = (n - 1) / 2;
    const uint64_t L = smooth_at_least(2 * H);   // transform length
    const uint64_t nc = L / 2 + 1;               // complex outputs of a real FFT of length L
    const uint64_t g = primitive_root(n);
    if (!g) return QMC_ERR_ARG;

    // per-component results and the blocks' partials, then the large arrays
    size_t bytes = 0;
    auto take = [&](size_t count) {
        const size_t at = bytes;
        bytes += (count * 8 + 255) & ~(size_t)255;
        return at;
    };
    const size_t o_z = take(s), o_t = take(s), o_p0 = take(s), o_sums = take((size_t)s * kCbcBlocks),
                 host_bytes = bytes, o_mins = take(kCbcBlocks), o_rep = take(kCbcBlocks),
                 o_rept = take(kCbcBlocks), o_gp = take(H), o_p = take(H + 1), o_P = take(L),
                 o_FP = take(2 * nc), o_FW = take(2 * nc);
    // (declared before the buffer: freeing that waits for whatever is still enqueued)
    std::unique_ptr<Plans> plans = take_plans(L);
    DeviceBuffer buf;
    if (!plans || cudaMalloc(&buf.base, bytes + plans->work_bytes + 256) != cudaSuccess ||
        !plans->use(buf.base + bytes, st))
        return QMC_ERR_CUDA;
    auto at = [&](size_t off) { return buf.base + off; };
    uint64_t *z_d = (uint64_t *)at(o_z), *rep = (uint64_t *)at(o_rep), *gp = (uint64_t *)at(o_gp);
    double *t_d = (double *)at(o_t), *p0_d = (double *)at(o_p0), *sums = (double *)at(o_sums);
    double *mins = (double *)at(o_mins), *rep_t = (double *)at(o_rept), *p = (double *)at(o_p), *P = (double *)at(o_P);
    cufftDoubleComplex *FP = (cufftDoubleComplex *)at(o_FP), *FW = (cufftDoubleComplex *)at(o_FW);

    // powers of g (threads of B powers each: enough threads for the chip first), the
    // transformed omega sequence (P is scratch here)
    const Modulus mod{n, n >> 32 ? 0 : ~0ull / n};   // floor((2^64 - 1) / n) = floor(2^64 / n), n odd
    const uint64_t B = std::max<uint64_t>(1, std::min<uint64_t>(64, H / (152 * 2048)));
    const uint64_t nthr = (H + B - 1) / B;
    cbc_powers_kernel<<<(unsigned)((nthr + kCbcThreads - 1) / kCbcThreads), kCbcThreads, 0, st>>>(g, mod, H, B, gp);
    cbc_omega_kernel<<<grid_for(L), kCbcThreads, 0, st>>>(gp, H, L, n, P);
    if (cudaGetLastError() != cudaSuccess) return QMC_ERR_CUDA;
    if (cufftExecD2Z(plans->fwd, P, FW) != CUFFT_SUCCESS) return QMC_ERR_CUDA;

    const uint64_t per_sum = (H + kCbcBlocks - 1) / kCbcBlocks;
    // the minimum and the pick do not depend on the order: blocks of at least 2048 candidates
    const uint64_t per_min = std::max<uint64_t>(2048, per_sum);
    const unsigned blocks = (unsigned)((H + per_min - 1) / per_min);
    // T[a] = 2 raw[a + H] / L + p(0) omega(0)  (the inverse transform is unnormalised)
    const double scale = 2.0 / (double)L;
    const double *raw = P + H;
    for (int j = 0; j < s; ++j) {
        if (j) {
            cbc_gather_kernel<<<grid_for(L), kCbcThreads, 0, st>>>(gp, p, H, L, n, P);
            if (cufftExecD2Z(plans->fwd, P, FP) != CUFFT_SUCCESS) return QMC_ERR_CUDA;
            cbc_pointwise_kernel<<<grid_for(nc), kCbcThreads, 0, st>>>(FP, FW, nc);
            if (cufftExecZ2D(plans->inv, FP, P) != CUFFT_SUCCESS) return QMC_ERR_CUDA;
            cbc_min_kernel<<<blocks, kCbcThreads, 0, st>>>(raw, p, H, scale, per_min, mins);
            cbc_pick_kernel<<<blocks, kCbcThreads, 0, st>>>(raw, gp, p, H, n, scale, per_min, mins, blocks,
                                                            sums + (size_t)(j - 1) * kCbcBlocks, rep, rep_t);
        }
        cbc_update_kernel<<<kCbcBlocks, kCbcThreads, 0, st>>>(p, H, mod, beta, gamma, j, blocks, rep, rep_t,
                                                              per_sum, z_d, t_d, p0_d, sums);
        if (cudaGetLastError() != cudaSuccess) return QMC_ERR_CUDA;
    }
    std::unique_ptr<char[]> host(new (std::nothrow) char[host_bytes]);
    if (!host || cudaMemcpyAsync(host.get(), buf.base, host_bytes, cudaMemcpyDeviceToHost, st) != cudaSuccess ||
        cudaStreamSynchronize(st) != cudaSuccess)
        return QMC_ERR_CUDA;
    give_back(std::move(plans));
    const uint64_t *hz = (const uint64_t *)(host.get() + o_z);
    const double *ht = (const double *)(host.get() + o_t), *hp0 = (const double *)(host.get() + o_p0);
    const double *hs = (const double *)(host.get() + o_sums);
    double tot = 0.0;   // sum_k p(k) of the components so far
    for (int j = 0; j < s; ++j) {
        if (hz[j] >= n) return QMC_ERR_CUDA;   // non-finite sums
        z_out[j] = hz[j];
        const double before = tot;
        double acc = 0.0;
        for (unsigned b = 0; b < kCbcBlocks; ++b) acc += hs[(size_t)j * kCbcBlocks + b];
        tot = hp0[j] + 2.0 * acc;
        if (e2_out) e2_out[j] = -1.0 + (j ? beta * before + gamma * ht[j] : tot) / (double)n;
    }
    return QMC_OK;
}
