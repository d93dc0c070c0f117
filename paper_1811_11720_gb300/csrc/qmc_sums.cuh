// qmc_sums.cuh -- the lattice-sum kernel (Eq. (lattice)): one integral, or many in one launch.
//
// Work decomposition.  An integral's i-range [i_begin, i_end) is cut into tiles of spb * L
// points; a block of spb * m threads owns one tile.  In a batch the tiles of all integrals
// form one sequence and a block looks up its integral, copies the descriptor to shared
// memory and stages the coefficients; integrals differ in dimension, lattice, fit and
// coefficients, and share the family and the transform kind (template parameters) and m (the
// block shape).  Thread (s, k) evaluates shift k on the L consecutive points of stream s.
// The transform and, where the integrand allows, the integrand's linear and quadratic forms
// run in integer fixed point (qmc_fixed.cuh, qmc_integrands.cuh), and so does its final function
// (qmc_exp.cuh, qmc_cos.cuh); FP64 is left to the sums, the polynomial families' powers and what
// has no fixed-point form.
// Each thread accumulates its L samples in FP64; the tile's per-shift partial is
// the Neumaier-compensated sum over its spb streams in fixed order, written to
// partials[tile][k].  Tiles depend only on the i-range, so the result is bit-identical for
// any grid size and in or out of a batch, and sharding on tile boundaries reproduces the
// same partials.
#pragma once
#include <cstdint>

#include "qmc_fitmap.cuh"
#include "qmc_integrands.cuh"
#include "qmc_transforms.cuh"

namespace qmc {

constexpr uint64_t kInner = 64;   // samples per inner accumulation block (power of two)

__device__ __forceinline__ bool not_finite(double x) {
    return ((unsigned long long)__double_as_longlong(x) & 0x7FF0000000000000ull) ==
           0x7FF0000000000000ull;
}

// Neumaier: add v to (s, c).
__device__ __forceinline__ void neumaier_add(double &s, double &c, double v) {
    double t = s + v;
    if (fabs(s) >= fabs(v)) c += (s - t) + v;
    else c += (v - t) + s;
    s = t;
}

// Fit constants per dimension in shared memory (see apply_fit).
__device__ __forceinline__ void prepare_fit(const double *fit, int d, double *s_fit) {
    const int tid = threadIdx.x;
    for (int j = tid; fit && j < d; j += blockDim.x) {
        const double *a = fit + 6 * j;
        double a2 = fabs(a[2]), a3 = fabs(a[3]);
        double *o = s_fit + kFitStride * j;
        o[0] = a[0];
        o[1] = a[1];
        o[2] = a2 * (a[0] - 1.0);
        o[3] = a3 * (a[1] - 1.0);
        o[4] = a[4];
        o[5] = a[5];
        o[6] = 1.0 - a2 - a3 - a[4] - a[5];
        o[7] = o[2] * a[0];
        o[8] = o[3] * a[1];
        o[9] = 2.0 * o[5];
        o[10] = 3.0 * o[6];
    }
}

// ---- lattice state shared by the warp --------------------------------------------------
// The lanes of a warp are shifts of at most a few streams (one when m is a multiple of 32),
// and the lattice point does not depend on the shift.  So the warp keeps one state per
// (stream, coordinate) pair: lane e and, past 32 pairs, lane e - 32 own pair e in registers,
// step it once per point and publish it to a double-buffered slot of shared memory; every
// lane reads its stream's d coordinates from there, with one __syncwarp per point.  With the
// state per thread instead (streams of m = 20 shifts did that: only m dividing 32 or a
// multiple of 32 shared), each thread steps d coordinates and keeps 3 d words in local
// memory.  More pairs than kPairs (m below ~6 with many dimensions) still do.
constexpr int kPairs = 64;

struct WarpStreams {
    unsigned mask;    // the warp's threads
    int first;        // first stream of the warp, within the block
    int mine;         // this lane's stream, counted from `first`
    int count;        // streams the warp's lanes belong to
};

__device__ __forceinline__ WarpStreams warp_streams(int m) {
    const int tid = threadIdx.x, base = tid & ~31;
    const int last = min(base + 31, (int)blockDim.x - 1);
    WarpStreams w;
    w.mask = last - base == 31 ? 0xFFFFFFFFu : (1u << (last - base + 1)) - 1u;
    w.first = base / m;
    w.mine = tid / m - w.first;
    w.count = last / m - w.first + 1;
    return w;
}

// Words of the state that a transform reads: Korobov<r,r> takes the coordinate as x 2^64 and
// reads the top word, the others (may) round both to u.
template <int TK>
constexpr bool kTopWordOnly = TK == kTKorobovInt;

// The step constants of the d coordinates in shared memory (a warp's lanes read different j).
// z2: the third word's step for n < 2^32 (ShortState), else the exact remainder.
struct BlockSteps {
    uint64_t zh[kMaxDim], zl[kMaxDim], z2[kMaxDim];
    __device__ __forceinline__ void set(int j, const DimConst &c, uint64_t n) {
        const LatticeStep st = lattice_step_of(c, n);
        zh[j] = st.fz_hi;
        zl[j] = st.fz_lo;
        z2[j] = n >> kShortBits ? st.remz : short_step_word(c, n);
    }
    __device__ __forceinline__ void start(int j, uint64_t i, const DimConst &c, uint64_t n,
                                          ShortState &s) const {
        lattice_state_at(i, c, n, s.f_hi, s.f_lo, s.f_2);
        if (!(n >> kShortBits)) s.f_2 = i * z2[j];
    }
    __device__ __forceinline__ void step(int j, uint64_t n, ShortState &s) const {
        if (n >> kShortBits) lattice_step(LatticeStep{zh[j], zl[j], z2[j]}, n, s.f_hi, s.f_lo, s.f_2);
        else s.step(zh[j], zl[j], z2[j]);
    }
};

// The published state of one warp: [buffer][][pair], the top words of two points or the words
// of one.
template <int TK>
struct WarpLattice {
    static constexpr int kWords = kTopWordOnly<TK> ? 1 : 2;
    uint64_t w[2][2][kPairs];
};

// A point's coordinates as eval_point reads them: from the warp's buffer or a thread's own.
struct SharedState {
    const uint64_t *w;   // this lane's stream in the buffer
    __device__ __forceinline__ uint64_t hi(int j) const { return w[j]; }
    __device__ __forceinline__ uint64_t lo(int j) const { return w[kPairs + j]; }
};
struct OwnState {
    const uint64_t *fhi, *flo;
    __device__ __forceinline__ uint64_t hi(int j) const { return fhi[j]; }
    __device__ __forceinline__ uint64_t lo(int j) const { return flo[j]; }
};

// The block's shifts in shared memory, D_kj 2^11 (the 53-bit shift in units of the lattice
// state's top word) as [j][k]: the lanes of a warp read consecutive words.  (Read from the
// caller's [k][j] rows through the read-only cache, a warp's load touched up to 20 lines.)
struct Shifts {
    const uint64_t *s;
    int m;
    __device__ __forceinline__ uint64_t operator()(int j) const { return s[j * m]; }
};

// The separable families' evaluation of NP points entirely in fixed point, coordinate and
// integrand form (no fit: the fit map needs x as a double).  Points share the loads of the
// shift and of the dimension's constants and the loop around them, and their integer chains
// interleave : osc d = 6 baker at n = 1,072,187, m = 32
// 520 -> 445 us, Gaussian d = 10 Korobov-3 at n = 10,560,653 16.29 -> 15.32 ms (two points;
// 48 registers and five blocks beat 64 and four).
template <int FAM, int TK, int R, int NP, class St>
__device__ __forceinline__ void eval_fixed(const Integral &p, const SeparableShared &fsh, Shifts dsh,
                                           double cd, const St (&st)[NP], double (&g)[NP]) {
    Weight W[NP];
    FamilyAcc<FAM> fa[NP];
#pragma unroll
    for (int u = 0; u < NP; ++u) fa[u].init_fixed(p.d);
    auto dim = [&](int j, auto norm) {
        const uint64_t D = dsh(j);
#pragma unroll
        for (int u = 0; u < NP; ++u)
            fa[u].add_fixed(j, transform_fixed<TK, R, true, decltype(norm)::value>(st[u].hi(j) + D, p.t, W[u]),
                            fsh);
    };
    if constexpr (TK == kTKorobovInt) {
        // pairs of dimensions: the weight's product is renormalized once a pair
        int j = 0;
        if (p.d & 1) dim(j++, std::true_type{});
#pragma unroll 1
        for (; j < p.d; j += 2) {
            dim(j, std::false_type{});
            dim(j + 1, std::true_type{});
        }
    } else {
#pragma unroll 1
        for (int j = 0; j < p.d; ++j) dim(j, std::true_type{});
    }
#pragma unroll
    for (int u = 0; u < NP; ++u) {
        if constexpr (kFxFinish<FAM>) {
            Fx f = fa[u].finish_fx(p.d, fsh);
            if constexpr (kIntKorobov<TK>) f = fx_mul(f, weight_fx<TK, R>(W[u], p.t, cd, p.d));
            g[u] = fx_to_double_sat(fx_norm(f));
        } else {
            g[u] = fa[u].finish_fixed(fsh) * weight_finish<TK, R>(W[u], p.t, cd, p.d);
        }
    }
}

// Whether the fixed-point form serves the integrand under the transform (uniform over the
// block).  The asymmetric map in FP64 keeps x relative near its ends, the integer one is absolute
// (~2^-57): a corner peak, or a C0 peak at w = 0, of large coefficients lives near x = 0 and needs
// sum c < 32 (S >= 58) there.  (A corner peak of d = 1 under Korobov<1,3> with c = 1e3, 1e6, 1e8
// was 1e-15, 1.5e-12, 2.7e-10 off on integers, 4e-16 in FP64; at c = 31 both 2e-16.)
template <int FAM, int TK>
__device__ __forceinline__ bool fixed_form_ok(const FixedForms &fx) {
    constexpr bool kSharp = TK == kTKorobovGen && (FAM == QMC_GENZ_CORNER_PEAK || FAM == QMC_GENZ_C0);
    return fx.ok && (!kSharp || fx.S >= 58);
}

// Most of eval_point's `extra` for the complex family: F's coefficients sum up to 16 |c0|
// (stage_feynman_full), so this is 2^-43 of c0.  (A fit of slope 56 over the orders 5 and 6, 172,032
// units, was 1.3e-14 off at d = 3.)
constexpr int kFeynRoom = 1 << 15;

// One evaluation of g at a point with lattice state `st`.
template <int FAM, int TK, int R, class St>
__device__ __forceinline__ void eval_point(const Integral &p, const FamilyShared<FAM> &fsh,
                                           const double *s_fit, const FitFixed *fit_fixed, bool use_fit,
                                           Shifts dsh, double cd, const St &st, double &g_re, double &g_im,
                                           unsigned long long &signfail) {
    Weight W;
    FamilyAcc<FAM> fa;
    constexpr bool kGen = TK == kTKorobovGen;
    if constexpr (kFixedTransform<TK> && kPolyFamily<FAM>) {
        // the polynomial families' fixed-point forms take the coordinates as x 2^64 from the
        // integer-pipe transform, through the integer fit map where there is one.  The asymmetric
        // map and the fit leave x absolute to a few units of 2^-kf and 2^-58, where in FP64 it is
        // relative near 0 and may be raised to any power: they serve where the polynomials are bounded
        // away from zero, or only factors, with room for it (extra: what the error, 4 and on average
        // 2 units, adds to a cubic, in units of 2^-62 of its bound)
        bool fixed = !use_fit || fit_fixed->ok;
        int extra = use_fit ? FitFixed::kErrorUnits : 0;
        if constexpr (kGen) extra += (use_fit ? fit_fixed->slope : 1) * (3 * 2) << (63 - p.t.kf);
        if constexpr (FAM == QMC_SECTOR) fixed = fixed && sector_fixed_ok(fsh.poly, p.d, extra);
        else fixed = fixed && feyn_fixed_ok(fsh.poly, p.d) && (!extra || (fsh.poly.feyn_full && extra <= kFeynRoom));
        if (fixed) {   // uniform over the block
            Weight V;
            Fx J;
            uint64_t X[8];
#pragma unroll 1
            for (int j = 0; j < p.d; ++j) X[j] = transform_fixed<TK, R>(st.hi(j) + dsh(j), p.t, V);
            if (!use_fit || fit_fixed->apply_all(X, p.d, &J)) {
                double wt;
                if (use_fit) {
                    if constexpr (kIntKorobov<TK>) J = fx_mul(J, weight_fx<TK, R>(V, p.t, cd, 0));
                    wt = fx_to_double(J);
                } else {
                    wt = weight_finish<TK, R>(V, p.t, cd);
                }
                if constexpr (FAM == QMC_SECTOR) {
                    g_re = sector_value_x(X, p.d, fsh.poly) * wt;
                    g_im = 0.0;
                } else {
                    feynman_value_x(X, p.d, fsh.poly, g_re, g_im, signfail);
                    g_re *= wt;
                    g_im *= wt;
                }
                return;
            }
        }
    }
    // the asymmetric map in FP64, relative near its ends
    bool rel = kGen && kPolyFamily<FAM>;
    if constexpr (kGen && kHasFixedForm<FAM>) rel = !fixed_form_ok<FAM, TK>(fsh.fx);
    fa.init(fsh);
#pragma unroll 1
    for (int j = 0; j < p.d; ++j) {
        Mapped mx;
        if (kGen && rel) {
            mx = apply_transform<QMC_T_KOROBOV>(fixed_to_double(st.hi(j) + dsh(j), st.lo(j), p.n), p.t, W);
        } else if constexpr (kIntKorobov<TK> && kPolyFamily<FAM>) {
            // the polynomial families use x itself: formed from x 2^64 by integer
            // operations instead of an FP64 conversion and reflection
            mx = Mapped{fixed_u64_to_double(transform_fixed<TK, R>(st.hi(j) + dsh(j), p.t, W), 64), false};
        } else if constexpr (kIntKorobov<TK>) {
            mx = korobov_int_x<TK, R>(st.hi(j) + dsh(j), p.t, W);
        } else {
            const double u = fixed_to_double(st.hi(j) + dsh(j), st.lo(j), p.n);
            mx = apply_transform<TK>(u, p.t, W);
        }
        if (use_fit) mx = Mapped{apply_fit(reflected(mx), s_fit + kFitStride * j, W.w), false};
        fa.add(j, mx, fsh);
    }
    const double wt = kGen && rel ? weight_finish<QMC_T_KOROBOV>(W, p.t, cd) : weight_finish<TK, R>(W, p.t, cd);
    fa.finish(p.d, fsh, g_re, g_im, signfail);
    g_re *= wt;
    if constexpr (FamilyAcc<FAM>::kComplex) g_im *= wt;
}

// A stream's running sums.  Two-level FP64 accumulation: blocks of kInner samples, then the
// block sums (rounding error ~ (kInner + L/kInner) ulp instead of L ulp).
struct StreamSum {
    double in_re = 0.0, in_im = 0.0, re = 0.0, im = 0.0;
    unsigned long long nonfinite = 0, signfail = 0;
    template <bool CPLX>
    __device__ __forceinline__ void add(double g_re, double g_im) {
        if (not_finite(g_re) || (CPLX && not_finite(g_im))) ++nonfinite;
        in_re += g_re;
        if constexpr (CPLX) in_im += g_im;
    }
    template <bool CPLX>
    __device__ __forceinline__ void flush() {
        re += in_re;
        in_re = 0.0;
        if constexpr (CPLX) {
            im += in_im;
            in_im = 0.0;
        }
    }
};

// The sums of one tile: this thread's stream covers points [i0, i0 + cnt) of the lattice,
// i0 = w0 + mine * L with w0 the first point of the warp's first stream.  eval(states, g_re,
// g_im, signfail) takes NP points at a time (one with a thread's own state).  kTail: an odd
// stream's last point by itself instead of as half of a pair.
template <bool CPLX, int NP, bool kTail, class Lat, class Eval>
__device__ __forceinline__ void run_stream(const Integral &p, const BlockSteps &steps,
                                           const WarpStreams &ws, Lat &lat, uint64_t w0, uint32_t cnt,
                                           StreamSum &acc, Eval &&eval) {
    const int d = p.d;
    const uint64_t n = p.n;
    const int stride = d | 1;   // pairs of a stream in the buffer: odd, no bank conflicts
    const int pairs = ws.count * d;
    const int lanes = __popc(ws.mask);   // 32 but in a ragged last warp
    if (pairs <= 2 * lanes && ws.count * stride <= kPairs) {
        // this lane's one or two pairs (stream, coordinate)
        const int lane = threadIdx.x & 31;
        struct Pair {
            ShortState f{0, 0, 0};
            int j = 0, at = 0;
            bool own = false;
        } a, b;
        auto start = [&](Pair &s, int e) {
            s.own = e < pairs;
            if (!s.own) return;
            const int st = e / d;
            s.j = e - st * d;
            s.at = st * stride + s.j;
            steps.start(s.j, w0 + (uint64_t)st * p.L, p.dc[s.j], n, s.f);
        };
        start(a, lane);
        start(b, lane + lanes);
        const uint32_t most = __reduce_max_sync(ws.mask, cnt);
        // points t .. t + N - 1
        auto points = [&](uint32_t t, auto count) {
            constexpr int N = decltype(count)::value;
            auto &buf = lat.w[(t / NP) & 1];
            auto publish = [&](Pair &s) {
                if (!s.own) return;
#pragma unroll
                for (int u = 0; u < N; ++u) {
                    buf[u][s.at] = s.f.f_hi;
                    if constexpr (NP == 1 && Lat::kWords == 2) buf[1][s.at] = s.f.f_lo;
                    steps.step(s.j, n, s.f);
                }
            };
            publish(a);
            if (pairs > lanes) publish(b);
            __syncwarp(ws.mask);
            if (t < cnt) {
                double g_re[N], g_im[N];
                SharedState st[N];
#pragma unroll
                for (int u = 0; u < N; ++u) st[u].w = &buf[u][ws.mine * stride];
                eval(st, g_re, g_im, acc.signfail);
                acc.template add<CPLX>(g_re[0], g_im[0]);
#pragma unroll
                for (int u = 1; u < N; ++u)
                    if (t + u < cnt) acc.template add<CPLX>(g_re[u], g_im[u]);
            }
            if (((t + N - 1) & (kInner - 1)) == kInner - 1) acc.template flush<CPLX>();
        };
        uint32_t t = 0;
        const uint32_t paired = kTail ? most / NP * NP : most;
#pragma unroll 1
        for (; t < paired; t += NP) points(t, std::integral_constant<int, NP>{});
        if constexpr (kTail)
            if (t < most) points(t, std::integral_constant<int, 1>{});
    } else {
        uint64_t fhi[kMaxDim], flo[kMaxDim], f2[kMaxDim];
        const uint64_t i0 = w0 + (uint64_t)ws.mine * p.L;
#pragma unroll 1
        for (int j = 0; j < d; ++j) {
            ShortState s;
            steps.start(j, i0, p.dc[j], n, s);
            fhi[j] = s.f_hi;
            flo[j] = s.f_lo;
            f2[j] = s.f_2;
        }
#pragma unroll 1
        for (uint32_t t = 0; t < cnt; ++t) {
            double g_re[1], g_im[1];
            const OwnState st[1] = {{fhi, flo}};
            eval(st, g_re, g_im, acc.signfail);
            acc.template add<CPLX>(g_re[0], g_im[0]);
            if ((t & (kInner - 1)) == kInner - 1) acc.template flush<CPLX>();
#pragma unroll 1
            for (int j = 0; j < d; ++j) {
                ShortState s{fhi[j], flo[j], f2[j]};
                steps.step(j, n, s);
                fhi[j] = s.f_hi;
                flo[j] = s.f_lo;
                f2[j] = s.f_2;
            }
        }
    }
    acc.template flush<CPLX>();
}

template <int FAM, int TK, int R>
__device__ __forceinline__ void stream_sums_r(const Integral &p, const FamilyShared<FAM> &fsh,
                                              const double *s_fit, const FitFixed *fit_fixed,
                                              bool use_fit, Shifts dsh, const BlockSteps &steps, const WarpStreams &ws,
                                              WarpLattice<TK> &lat, uint64_t w0, uint32_t cnt,
                                              StreamSum &acc) {
    constexpr bool kCplx = FamilyAcc<FAM>::kComplex;
    const double cd = p.cd;
    if constexpr (kFixedTransform<TK> && kHasFixedForm<FAM>) {
        if (!use_fit && fixed_form_ok<FAM, TK>(fsh.fx)) {   // uniform over the block
            // The tail of its own pays under Korobov<r,r> (streams of 9 points, the d = 4, n =
            // 108,863, m = 16 integral's: 75.8 -> 71.7 us); under baker and the asymmetric map
            // the second copy of the code cost 1 and 3 %.
            run_stream<false, 2, TK == kTKorobovInt>(p, steps, ws, lat, w0, cnt, acc,
                                 [&](auto &st, auto &g_re, auto &, unsigned long long &) {
                                     eval_fixed<FAM, TK, R>(p, fsh, dsh, cd, st, g_re);
                                 });
            return;
        }
    }
    run_stream<kCplx, 1, false>(p, steps, ws, lat, w0, cnt, acc,
                         [&](auto &st, auto &g_re, auto &g_im, unsigned long long &signfail) {
                             g_im[0] = 0.0;
                             eval_point<FAM, TK, R>(p, fsh, s_fit, fit_fixed, use_fit, dsh, cd, st[0],
                                                    g_re[0], g_im[0], signfail);
                         });
}

// The integer Korobov is compiled once per order r (uniform branch per tile) for the separable
// families, whose time it is; the polynomial families choose the order at each use.
template <int FAM, int TK, class... A>
__device__ __forceinline__ void stream_sums(const Integral &p, A &&...a) {
    if constexpr (TK == kTKorobovInt && !kPolyFamily<FAM>) {
        switch (p.t.r0) {
        case 1: stream_sums_r<FAM, TK, 1>(p, a...); return;
        case 2: stream_sums_r<FAM, TK, 2>(p, a...); return;
        case 3: stream_sums_r<FAM, TK, 3>(p, a...); return;
        case 4: stream_sums_r<FAM, TK, 4>(p, a...); return;
        case 5: stream_sums_r<FAM, TK, 5>(p, a...); return;
        default: stream_sums_r<FAM, TK, 6>(p, a...); return;
        }
    } else {
        stream_sums_r<FAM, TK, 0>(p, a...);
    }
}

// Per-shift tile partial: fixed-order compensated sum over the block's spb streams of
// shift k, written as (sum, compensation) to out_re[2k..] (and out_im).  Contains a block
// barrier; every thread of the block must call it.
template <bool CPLX>
__device__ __forceinline__ void tile_partial(const StreamSum &acc, double *s_red, int m, int spb,
                                             double *out_re, double *out_im) {
    const int tid = threadIdx.x;
    s_red[tid] = acc.re;
    if constexpr (CPLX) s_red[kSumsThreads + tid] = acc.im;
    __syncthreads();
    if (tid < m) {
        const int k = tid;
        double sr = 0.0, cr = 0.0, si = 0.0, ci = 0.0;
        for (int s = 0; s < spb; ++s) {
            neumaier_add(sr, cr, s_red[s * m + k]);
            if constexpr (CPLX) neumaier_add(si, ci, s_red[kSumsThreads + s * m + k]);
        }
        out_re[2 * k] = sr;
        out_re[2 * k + 1] = cr;
        if constexpr (CPLX) {
            out_im[2 * k] = si;
            out_im[2 * k + 1] = ci;
        }
    }
}

// Blocks per SM the register allocation must allow: five for the separable families (48
// registers; their throughput depends on hiding integer latency), three for the sector family
// (85 registers; d = 8, n = 1,072,187, m = 32: 4.55 ms with two blocks, 4.43 with three (4.53 since U's check), 9.0
// with the one the compiler leaves room for by itself), two for the complex family with the
// dimension compiled in (128 registers with a few spills; d = 5 at the same size: 23.3 ms with
// one, 19.1 with two) and one without (d = 8 with two blocks was 15 % slower).
template <int FAM>
constexpr int kSumsMinBlocks = FAM == QMC_FEYNMAN ? 2 : FAM == QMC_SECTOR ? 3 : 5;

// Dynamic shared memory: the shifts, [kMaxDim or d][m].  kOne: a launch of one integral that reads it
// in place, as kernel parameters, instead of a copy in shared memory.  For the FP64 Korobov map,
// whose run-time orders and coefficients are then uniform operands: a monomial of d = 6 at
// n = 108,863, m = 32 under the orders 0 takes 270 us instead of 347, under the orders 8 835 instead of
// 900.
template <int FAM, int TK, int MINB, bool kOne>
__global__ void __launch_bounds__(kSumsThreads, MINB)
    lattice_kernel(const __grid_constant__ LatticeLaunch lp) {
    extern __shared__ uint64_t s_dsh[];
    __shared__ FamilyShared<FAM> fsh;
    __shared__ double s_fit[kMaxDim * kFitStride];
    __shared__ double s_red[(FamilyAcc<FAM>::kComplex ? 2 : 1) * kSumsThreads];
    __shared__ WarpLattice<TK> s_lat[kSumsThreads / 32];
    __shared__ Integral s_item;
    __shared__ BlockSteps s_step;
    FitFixed *fit_fixed = nullptr;
    if constexpr (kFixedTransform<TK> && kPolyFamily<FAM>) {
        __shared__ FitFixed s_fitq;
        fit_fixed = &s_fitq;
    }
    __shared__ int s_q[2];   // by the parity of the search round
    constexpr bool kCplx = FamilyAcc<FAM>::kComplex;

    const int tid = threadIdx.x;
    const int m = lp.m, spb = lp.spb;
    const WarpStreams ws = warp_streams(m);
    if (lp.chain) asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    for (uint64_t tile = lp.first_tile + blockIdx.x; tile < lp.end_tile; tile += gridDim.x) {
        __syncthreads();   // the previous tile's shared data is no longer read
        const Integral *src = &lp.one;
        if (!kOne && lp.items) {
            // the integral whose tiles hold this one: in each round every thread looks at one of
            // `blockDim` equal parts of the prefix sums left (in small blocks several of 32), so
            // up to 256 integrals take one round of loads and 65,536 two.  (Every thread at its
            // share of all the sums, in one round: 65,536 integrals of 16 tiles 128 ms a batch,
            // 16,384 18.2; in rounds 60.5 and 15.1.)
            int lo = 0, hi = lp.count, step;
            for (int round = 0;; ++round) {
                const int parts = max((int)blockDim.x, 32);
                step = (hi - lo + parts - 1) / parts;
                for (int a = lo + tid * step; a < hi; a += blockDim.x * step)
                    if (lp.tile_begin[a] <= tile && tile < lp.tile_begin[min(a + step, hi)]) s_q[round & 1] = a;
                __syncthreads();
                lo = s_q[round & 1];
                hi = min(lo + step, hi);
                if (step == 1) break;
            }
            src = lp.items + lo;
        }
        for (int w = tid; !kOne && w < (int)(sizeof(Integral) / 8); w += blockDim.x)
            reinterpret_cast<uint64_t *>(&s_item)[w] = reinterpret_cast<const uint64_t *>(src)[w];
        if constexpr (kFixedTransform<TK> && kPolyFamily<FAM>)
            if (tid == 0) fit_fixed->ok = fit_fixed->slope = 1;
        __syncthreads();
        const Integral &it = kOne ? lp.one : s_item;
        const int d = it.d;
        for (int i = tid; i < m * d; i += blockDim.x) {
            const int k = i / d, j = i - k * d;
            s_dsh[j * m + k] = it.shifts[i] << 11;
        }
        for (int j = tid; j < d; j += blockDim.x) s_step.set(j, it.dc[j], it.n);
        stage_family<FAM, false>(it, fsh);
        prepare_fit(it.fit, d, s_fit);
        if constexpr (kFixedTransform<TK> && kPolyFamily<FAM>)
            for (int j = tid; it.fit && j < d; j += blockDim.x) fit_fixed->stage(it.fit, j);
        __syncthreads();
        if constexpr (kHasFixedForm<FAM>) {
            // the FP64 forms' subset-sum tables (256 FP64 sums per block), only when the
            // fixed-point form does not take every evaluation (uniform over the block)
            if (!(kFixedTransform<TK> && it.fit == nullptr && fixed_form_ok<FAM, TK>(fsh.fx))) {
                stage_subset_sums<FAM>(it, fsh);
                __syncthreads();
            }
        }
        const uint64_t local = tile - it.tile_begin;
        const uint64_t w0 = it.i_begin + (local * (uint64_t)spb + ws.first) * it.L;
        const uint64_t i0 = w0 + (uint64_t)ws.mine * it.L;
        uint32_t cnt = 0;
        if (i0 < it.i_end) cnt = it.i_end - i0 < it.L ? (uint32_t)(it.i_end - i0) : it.L;
        StreamSum acc;
        stream_sums<FAM, TK>(it, fsh, s_fit, (const FitFixed *)fit_fixed, it.fit != nullptr, Shifts{s_dsh + tid % m, m}, s_step, ws,
                             s_lat[tid >> 5], w0, cnt, acc);
        double *base = lp.partials + it.partial_off;
        tile_partial<kCplx>(acc, s_red, m, spb, base + 2 * (local * (uint64_t)m),
                            base + 2 * (it.tiles * (uint64_t)m) + 2 * (local * (uint64_t)m));
        if (lp.counters) {
            if (acc.nonfinite) atomicAdd(lp.counters + 2 * it.slot, acc.nonfinite);
            if (acc.signfail) atomicAdd(lp.counters + 2 * it.slot + 1, acc.signfail);
        }
    }
    // ends after the launch before it, whose end then follows from this one's
    if (lp.chain) asm volatile("griddepcontrol.wait;" ::: "memory");
}

}  // namespace qmc
