// qmc_fixed.cuh -- the symmetric Korobov map (Sec. 2.3, Eq. (korobov)) on the integer pipe.
//
// For Korobov<r,r> the map is phi(v) = v^(r+1) P(v) on v = min(x, 1 - x) in [0, 1/2]
// (phi(x) = 1 - phi(1 - x) above 1/2), with P(v) = sum_k A_k v^k,
// A_k = C (-1)^k binom(r,k) / (r+1+k), and the weight is C (v (1 - v))^r.  In w = 1 - v the
// polynomial has positive integer coefficients, so for r = 1..6 (compiled orders) the map
// is evaluated with unsigned 64-bit integer multiplies, r being a compile-time constant:
//
//   * v enters in 0.64 fixed point, V = v 2^64, straight from the top word X of the shifted
//     lattice fraction x: V = X (x < 1/2) or 2^64 - 1 - X, within 2^-64 of min(x, 1 - x).
//   * P is evaluated in w = 1 - v, where its coefficients are positive:
//       P(v) = C int_0^1 s^r (1 - v s)^r ds = sum_k binom(r+k, k) (1 - v)^k
//     (expand (1 - v s)^r = ((1 - s) + w s)^r and integrate the Beta integrals), e.g.
//     1 + 2w | 1 + 3w + 6w^2 | 1 + 4w + 10w^2 + 20w^3 | 1 + 5w + 15w^2 + 35w^3 + 70w^4.
//     Unsigned Estrin form in fixed point with F fractional bits, F the largest value with
//     P(1) 2^F = sum_k binom(r+k, k) 2^F < 2^64 (every partial sum is at most that for
//     w <= 1): coefficient pairs (c_2j + c_2j+1 w) by shifts and adds, times w^2j from
//     squarings; each product truncates by at most 3 units of 2^-F (F = 62, 60, 58, 57,
//     55, 53 for r = 1..6; the products drop their low partial products, see mulhi_trunc).
//     w^2 comes from v^2 by additions.  Exact-arithmetic checks of these integer steps give
//     the same worst phi error as Horner's scheme (2^-56.2 for r = 3) with one or two fewer
//     64-bit products per dimension (and no multiplies for the coefficients).
//   * phi = v^(r+1) P in 0.64 fixed point; the absolute error is below 2^-(61 - 1.7 r)
//     (2^-54.9 for r = 4, 2^-50.9 for r = 6: the power's truncations times
//     P <= binom(2r+1, r), and the truncations of the last product scaled by 2^(64 - F)).  The integrands
//     that accept a fixed-point coordinate take it as is; otherwise it is rounded to double.
//   * t = v (1 - v) = V - V^2 2^-64 in 0.64 fixed point enters the running product over
//     the dimensions, kept in the format Fx (a 64-bit mantissa, renormalized after each
//     factor, and an exponent), whose r-th power times C^d is rounded once to double: the
//     product keeps relative precision however small it becomes.  Each t is exact to
//     3 2^-64 absolutely, which moves the weight by less than 2^-58 of its largest value
//     C^d 4^(-rd); t itself is not normalized (its low bits are all it has), so a factor
//     t >= 2^-k costs the product about 2^-(62-k) relatively.
//
// GB300 runs ~2 FP64 fused multiply-adds per clock per SM but ~32x as many 32-bit integer
// multiply-adds, so the ~8 FP64 instructions per dimension of the FP64 form cost more than
// the ~60 integer instructions that replace them.
#pragma once
#include <cstdint>

#include "qmc_params.cuh"

namespace qmc {

// ---------------------------------------------------------------------------------------
// Compile-time coefficients of Korobov<r,r>.
__host__ __device__ constexpr double pow2_c(int e) {
    double x = 1.0;
    for (int i = 0; i < e; ++i) x *= 2.0;
    return x;
}
__host__ __device__ constexpr long long korobov_Pw(int r, int k) {   // binom(r+k, k)
    long long b = 1;
    for (int i = 1; i <= k; ++i) b = b * (r + i) / i;
    return b;
}
__host__ __device__ constexpr int korobov_F(int r) {   // fractional bits of P in w = 1 - v
    double S = 0.0;
    for (int k = 0; k <= r; ++k) S += (double)korobov_Pw(r, k);
    int F = 0;
    while (S * pow2_c(F + 1) < pow2_c(64)) ++F;
    return F;
}

// ---------------------------------------------------------------------------------------
// High word of a 64 x 64-bit product without the low x low partial product and the low
// halves of the cross products: a 32 x 32 -> 64-bit multiply, two 32-bit high multiplies
// and a 64-bit add.  The result is at most 2 below floor(a b / 2^64) (never above), which
// the fixed-point error bounds below include.
__device__ __forceinline__ uint64_t mulhi_trunc(uint64_t a, uint64_t b) {
    const uint32_t al = (uint32_t)a, ah = (uint32_t)(a >> 32);
    const uint32_t bl = (uint32_t)b, bh = (uint32_t)(b >> 32);
    return (uint64_t)ah * bh + __umulhi(ah, bl) + __umulhi(al, bh);
}

// The same for a square: the two cross products are equal, so one 32-bit high multiply
// doubled (bit-identical to mulhi_trunc(a, a), which the compiler does not fold).
__device__ __forceinline__ uint64_t sqhi_trunc(uint64_t a) {
    const uint32_t al = (uint32_t)a, ah = (uint32_t)(a >> 32);
    return (uint64_t)ah * ah + ((uint64_t)__umulhi(ah, al) << 1);
}

// Fixed point for polynomial work on the integer multiply pipe: a value v is held as the
// integer round(v 2^s) with one scale s per polynomial (signed for the complex family's
// tensors, unsigned for the real family's non-negative dense forms), a coordinate x in
// [0, 1] as the uint64 X = x 2^64.
//   c X / 2^64 for signed c: the unsigned high word of (c mod 2^64) X, minus X when c < 0.
__device__ __forceinline__ int64_t smulhi_x(int64_t c, uint64_t X) {
    const uint64_t h = mulhi_trunc((uint64_t)c, X);
    return (int64_t)(c < 0 ? h - X : h);
}

// ---------------------------------------------------------------------------------------
// value = m 2^(e - 64); m == 0 encodes zero.  Normalized: m >= 2^63.
struct Fx {
    uint64_t m;
    int e;
};

// v >= 0, zero or normal.
__device__ __forceinline__ Fx fx_of_double(double v) {
    const uint64_t b = (uint64_t)__double_as_longlong(v);
    return {b ? ((b << 11) | 0x8000000000000000ull) : 0ull, (int)(b >> 52) - 1022};
}

// Truncated product (relative error below 2^-61 for normalized inputs); exponents add.
__device__ __forceinline__ Fx fx_mul(Fx a, Fx b) { return {mulhi_trunc(a.m, b.m), a.e + b.e}; }
__device__ __forceinline__ Fx fx_sq(Fx a) { return {sqhi_trunc(a.m), 2 * a.e}; }

// Normalize a mantissa that is zero or >= 2^32 (shift 0..32; zero stays zero).
__device__ __forceinline__ Fx fx_norm(Fx a) {
    const int lz = __clz((unsigned)(a.m >> 32));
    return {a.m << lz, a.e - lz};
}

// Normalize any mantissa (zero stays zero).  Mantissas below 2^32 (a lattice coordinate
// within 2^-32 of 0 or 1) take the slower branch.
__device__ __forceinline__ Fx fx_norm_any(uint64_t m, int e) {
    const uint32_t hi = (uint32_t)(m >> 32);
    if (hi) {
        const int lz = __clz(hi);
        return {m << lz, e - lz};
    }
    const int lz = __clzll(m);   // 64 for zero
    return {m ? (m << (lz & 63)) : 0ull, e - lz};
}

// Round to the nearest double (ties to even on the truncated mantissa).  Zero, and values
// below the normal range, give 0.
__device__ __forceinline__ double fx_to_double(Fx a) {
    a = fx_norm_any(a.m, a.e);
    const int be = a.e + 1021;   // biased exponent minus one
    if (!a.m || be < 0) return 0.0;
    uint64_t mant = a.m >> 11;
    const uint64_t rb = (a.m >> 10) & 1u;
    const uint64_t sticky = a.m & 0x3FFull;
    mant += rb & ((sticky != 0) | (mant & 1u));
    // adding the mantissa with its leading one to (exponent - 1) << 52 carries correctly
    return __longlong_as_double((long long)(((uint64_t)be << 52) + mant));
}

// The same for a normalized (or zero) mantissa, with overflow to +infinity.
__device__ __forceinline__ double fx_to_double_sat(Fx a) {
    const int be = a.e + 1021;
    if (!a.m || be < 0) return 0.0;
    if (be > 2045) return __longlong_as_double(0x7FF0000000000000ll);
    uint64_t mant = a.m >> 11;
    const uint64_t rb = (a.m >> 10) & 1u;
    const uint64_t sticky = a.m & 0x3FFull;
    mant += rb & ((sticky != 0) | (mant & 1u));
    return __longlong_as_double((long long)(((uint64_t)be << 52) + mant));
}

// a^p for a normalized a and a runtime p >= 1 (binary powering from the top bit; the loop
// is uniform when p is).  Each product truncates by at most 2^-61 relatively.
__device__ __forceinline__ Fx fx_powi(Fx a, int p) {
    Fx r = a;
#pragma unroll 1
    for (int i = 30 - __clz(p); i >= 0; --i) {
        r = fx_norm(fx_sq(r));
        if ((p >> i) & 1) r = fx_norm(fx_mul(r, a));
    }
    return r;
}

// 2^127 / m for m in [2^63, 2^64), at most 2^-59 low: a single-precision estimate made slightly
// low, r0 = 2^63 / m 2^32 (1 - e) with 0 < e < 2^-20, and r0 (1 + e + e^2).  (The estimate, the
// conversion to single precision and two products err by less than 2^-21.6 in all.)
__device__ __forceinline__ uint64_t recip_fixed(uint64_t m) {
    const uint32_t mh = (uint32_t)(m >> 32), ml = (uint32_t)m;
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(__uint2float_rn(mh)));
    const uint32_t r0 = __float2uint_rz(r * (0x1p63f * (1.0f - 0x1p-21f)));   // below 2^32
    // e 2^63 < 2^43, less one for the dropped fraction, so that R never exceeds 2^127 / m
    const uint64_t E = 0x7FFFFFFFFFFFFFFFull - ((uint64_t)mh * r0 + __umulhi(ml, r0));
    const uint32_t e22 = (uint32_t)(E >> 20);                                  // e 2^43
    const uint64_t E2 = E + (((uint64_t)e22 * e22) >> 23);                     // (e + e^2) 2^63
    return ((uint64_t)r0 << 32) + (((uint64_t)r0 * (uint32_t)E2) >> 31) + ((uint64_t)r0 * (uint32_t)(E2 >> 32) << 1);
}

// 1/a for a normalized a = m 2^(e - 64), at most 2^-59 low (~25 instructions; two Newton steps
// with full 64-bit products, to 2^-61, took ~60).
__device__ __forceinline__ Fx fx_recip(Fx a) { return Fx{recip_fixed(a.m), 1 - a.e}; }

// x 2^-64 for a 0.64 fixed-point x, rounded to nearest.
__device__ __forceinline__ double fixed_to_double64(uint64_t x) {
    const long long b = __double_as_longlong(__ull2double_rn(x));
    return __longlong_as_double(b ? b - (64ll << 52) : 0ll);
}

// ---------------------------------------------------------------------------------------
// v^E 2^64 for V = v 2^64 and V2 = v^2 2^64 (E >= 2): products of squares, E - 1 roundings
// at most (each truncating by at most 3 units of 2^-64).
template <int E>
__device__ __forceinline__ uint64_t fixed_pow(uint64_t V, uint64_t V2) {
    static_assert(E >= 2, "power");
    if constexpr (E == 2) {
        return V2;
    } else if constexpr (E == 3) {
        return mulhi_trunc(V2, V);
    } else {
        const uint64_t h = fixed_pow<E / 2>(V, V2);
        const uint64_t sq = sqhi_trunc(h);
        if constexpr (E % 2) return mulhi_trunc(sq, V);
        else return sq;
    }
}

// x C for a compile-time constant C as shifts and adds (the integer-multiply pipe is the
// busier one in this kernel; the product must fit in 64 bits).
__host__ __device__ constexpr int ctz_c(uint64_t c) {
    int b = 0;
    while (!(c & 1)) {
        c >>= 1;
        ++b;
    }
    return b;
}
template <uint64_t C>
__device__ __forceinline__ uint64_t mul_const(uint64_t x) {
    if constexpr (C == 0) return 0;
    else return (x << ctz_c(C)) + mul_const<(C & (C - 1))>(x);
}

// The pair J of P's coefficients as (binom(R+2J, 2J) + binom(R+2J+1, 2J+1) w) 2^F, with
// ws = w 2^F (the second coefficient is 0 past k = R).
template <int R, int J>
__device__ __forceinline__ uint64_t korobov_pair(uint64_t ws) {
    constexpr int F = korobov_F(R);
    constexpr uint64_t c0 = (uint64_t)korobov_Pw(R, 2 * J) << F;
    constexpr uint64_t c1 = 2 * J + 1 <= R ? (uint64_t)korobov_Pw(R, 2 * J + 1) : 0ull;
    return c0 + mul_const<c1>(ws);
}

// P(w) 2^F = sum_k binom(R+k, k) w^k 2^F for Korobov<R,R>, W = w 2^64 (w = 1 - v), in
// Estrin's form: sum_J (c_2J + c_2J+1 w) w^2J.  The pairs need only shifts and adds, and
// w^2 = 1 - 2v + v^2 comes from V2 = v^2 2^64 by additions (2^64 - 2 - 2V + V2, within 3
// units of floor(W^2 2^-64); V < 2^63), so P costs 0 (R = 1), 1 (R = 2, 3), 3 (R = 4, 5)
// or 5 (R = 6) 64-bit high products against R in Horner's scheme, with the same error
// bound (every term is positive, every partial sum at most P(1) 2^F < 2^64).
template <int R>
__device__ __forceinline__ uint64_t korobov_P(uint64_t V, uint64_t V2) {
    constexpr int F = korobov_F(R);
    const uint64_t W = ~V;
    const uint64_t ws = W >> (64 - F);
    uint64_t P = korobov_pair<R, 0>(ws);
    if constexpr (R >= 2) {
        const uint64_t W2 = V2 - 2 * V - 2;
        P += mulhi_trunc(korobov_pair<R, 1>(ws), W2);
        if constexpr (R >= 4) {
            const uint64_t W4 = sqhi_trunc(W2);
            P += mulhi_trunc(korobov_pair<R, 2>(ws), W4);
            if constexpr (R >= 6) P += mulhi_trunc(korobov_pair<R, 3>(ws), mulhi_trunc(W4, W2));
        }
    }
    return P;
}

// phi(v) 2^64 for V = v 2^64 (v <= 1/2), and t = v (1 - v) folded into the normalized
// running product Wp.
template <int R>
__device__ __forceinline__ uint64_t korobov_phi_fixed(uint64_t V, Fx &Wp) {
    static_assert(R >= 1 && R <= kMaxKorobovInt, "integer Korobov order");
    constexpr int F = korobov_F(R);
    const uint64_t V2 = sqhi_trunc(V);
    // P in w = 1 - v (2^64 - 1 - V, within 2^-64 of (1 - v) 2^64)
    const uint64_t p = korobov_P<R>(V, V2);
    // v^(r+1) 2^64
    const uint64_t pw = fixed_pow<R + 1>(V, V2);
    // t = v - v^2 in 0.64 fixed point (<= 2^62), into the weight product as it is: its
    // leading zeros carry no information (t is exact to 3 2^-64 absolutely), and the
    // product, at least 2^31 for t >= 2^-32, is renormalized afterwards
    Wp = fx_norm(fx_mul(Wp, Fx{V - V2, 0}));
    return mulhi_trunc(pw, p) << (64 - F);
}

// The asymmetric map.  phi_(r0,r1)(u) = v^(r0+1) sum_(k <= r1) binom(r0+k, k) w^k for u <= 1/2
// (v = u, w = 1 - v: the same Beta integrals as above, the powers of s and 1 - s exchanged),
// and 1 - phi_(r1,r0)(1 - u) above.  The orders are those of the launch, so P runs in Horner's
// form over `deg` = max(r0, r1) products (the shorter half's coefficients are padded with
// zeros) and the power over as many; F = kf keeps binom(r0+r1+1, r1) 2^F below 2^64.  Returns
// phi 2^64 of this point's half (X above 1/2 means 1 - phi), and folds u into Wu, 1 - u into
// W1: the weight is C u^r0 (1-u)^r1, each product raised to its order once per evaluation.
// ~9 high products per dimension at (1, 3) against ~20 FP64 instructions of 17 SM cycles a
// warp each for the FP64 Horner form, which held corner peak, d = 8, n = 256,687, m = 20 at
// 1434 us (FP64 pipe 85 % busy).
__device__ __forceinline__ uint64_t korobov_gen_phi(uint64_t X, const TransformParams &t, Fx &Wu,
                                                    Fx &W1) {
    const bool lo = !(X >> 63);
    const uint64_t V = lo ? X : ~X, W = ~V;
    uint64_t P = lo ? t.KA[t.deg] : (uint64_t)t.KB[t.deg] << t.kf;
#pragma unroll 1
    for (int k = t.deg - 1; k >= 0; --k) P = mulhi_trunc(P, W) + (lo ? t.KA[k] : (uint64_t)t.KB[k] << t.kf);
    const int e = lo ? t.r0 : t.r1;   // v^(e + 1)
    uint64_t pw = V;
#pragma unroll 1
    for (int q = 1; q <= t.deg; ++q) {
        const uint64_t next = mulhi_trunc(pw, V);
        pw = q <= e ? next : pw;
    }
    Wu = fx_norm(fx_mul(Wu, Fx{X, 0}));
    W1 = fx_norm(fx_mul(W1, Fx{~X, 0}));
    return mulhi_trunc(pw, P) << (64 - t.kf);
}

// The same map for the separable families, which need phi absolutely but not relatively near 1:
// phi = u^(r0+1) sum_(k <= r1) binom(r0+k, k) (1 - u)^k holds on all of [0, 1], so there are no
// halves to choose between and r0 + r1 + 1 products instead of 2 max(r0, r1) + 1.  Every product
// truncates downwards, so phi stays below 1; the power is formed by itself at 2^-64 and meets P in
// the last product, the one power that truncates at 2^-kf.  On average phi is 1.7 units of 2^-54 low
// under the orders 5 and 6 (kf = 54; 0.04 at 1 and 3), where the FP64 form errs by 6 (0.7) either way;
// with P in the chain from the first power on it was 3.5 low, and a C0 or corner peak under the orders
// 5 and 6 up to four times as far off as in FP64.  (Setting the bits below 2^-kf would make up one
// more unit; at d = 8, n = 256,687, m = 20 it cost 2 %.)  kNorm as for korobov_odd_fixed.
template <bool kNorm>
__device__ __forceinline__ uint64_t korobov_gen_whole(uint64_t X, const TransformParams &t, Fx &Wu, Fx &W1) {
    const uint64_t W = ~X;
    const int r0 = t.r0, r1 = t.r1;
    uint64_t P = t.KA[r1];
#pragma unroll 1
    for (int k = r1 - 1; k >= 0; --k) P = mulhi_trunc(P, W) + t.KA[k];
    uint64_t pw = X;
#pragma unroll 1
    for (int q = 0; q < r0; ++q) pw = mulhi_trunc(pw, X);
    Wu = fx_mul(Wu, Fx{X, 0});
    W1 = fx_mul(W1, Fx{W, 0});
    if constexpr (kNorm) {
        Wu = fx_norm(Wu);
        W1 = fx_norm(W1);
    }
    return mulhi_trunc(pw, P) << (64 - t.kf);
}

// C^d Wu^r0 W1^r1; cdx = C^d as Fx.
__device__ __forceinline__ Fx korobov_gen_weight(Fx Wu, Fx W1, const TransformParams &t, Fx cdx) {
    return fx_norm(fx_mul(fx_norm(fx_mul(fx_powi(Wu, t.r0), fx_powi(W1, t.r1))), cdx));
}

// The same map as an odd function about 1/2, for the integrands that need x absolutely but not
// relatively near 0 (the separable families).  With s = 2 x - 1 and w = 1 - s^2 = 4 x (1 - x),
// phi' = C (w/4)^r integrates to
//   phi = (1 + s q(w)) / 2,  q = sum_(k <= r) binom(2k, k) (w/4)^k  (q = 1, 1/2 w, 3/8 w^2,
//   5/16 w^3, 35/128 w^4, ...: the series of (1 - w)^(-1/2), cut where phi' stops),
// so there is no half to reflect, the coefficients are positive, the linear ones are shifts, and
// the weight's factor w comes with the map at full precision.  13, 10, 13 and 15 32-bit
// multiplies per dimension with the weight for r = 1..4 (8, 14, 13 and 21 in the form above)
// and fewer shifts and adds.  kNorm = false leaves the weight's product unnormalized for one
// more factor: every second dimension is enough (the pair's product loses relative precision
// only where it is far below its largest value).  Gaussian d = 10 Korobov-3, n = 10,560,653,
// m = 32: 15.32 ms -> 15.25 with the odd form, 14.81 with the weight normalized once a pair.
// q is kept at 2^62, less 4 units so that |s| q stays below 1 whatever the truncations (without
// them s q could reach 1 and phi wrap); |phi error| < 2^-58 (r <= 4), 2^-57 (r = 6), against
// 2^-56 (r = 3) and 2^-51 (r = 6) above.
template <int R>
__device__ __forceinline__ uint64_t korobov_odd_q(uint64_t W) {   // W = w 2^64
    static_assert(R >= 1 && R <= kMaxKorobovInt, "integer Korobov order");
    const uint64_t p0 = (1ull << 62) - 4 + (W >> 3);
    if constexpr (R == 1) {
        return p0;
    } else {
        const uint64_t W2 = sqhi_trunc(W);
        if constexpr (R == 2) {
            return p0 + (W2 >> 4) + (W2 >> 5);
        } else {
            uint64_t p1 = (3ull << 59) + (W >> 4) + (W >> 6);
            if constexpr (R == 4) p1 += mulhi_trunc(W2, 35ull << 55);
            if constexpr (R >= 5) {
                uint64_t p2 = (35ull << 55) + mulhi_trunc(W, 63ull << 54);
                if constexpr (R == 6) p2 += mulhi_trunc(W2, 231ull << 52);
                p1 += mulhi_trunc(p2, W2);
            }
            return p0 + mulhi_trunc(p1, W2);
        }
    }
}

// phi 2^64 for X = x 2^64, and w folded into the normalized running product Wp.
template <int R, bool kNorm = true>
__device__ __forceinline__ uint64_t korobov_odd_fixed(uint64_t X, Fx &Wp) {
    const uint64_t low = (uint64_t)((int64_t)~X >> 63);   // all ones below 1/2
    const uint64_t A = (X << 1) ^ low;                    // |s| 2^64, at most one unit low
    const uint64_t W = ~sqhi_trunc(A);
    Wp = fx_mul(Wp, Fx{W, 0});
    if constexpr (kNorm) Wp = fx_norm(Wp);
    const uint64_t h = mulhi_trunc(A, korobov_odd_q<R>(W)) << 1;   // |s| q 2^63
    return (h ^ low) + 0x8000000000000000ull;
}

// Wp^E for a normalized Wp by binary powering.  Up to E = 4 the products stay unnormalized (at
// least 2^61 of 2^64): the few bits lost are below 2^-59 of the value, and the result is
// normalized once where it is used.
template <int E>
__device__ __forceinline__ Fx fx_pow(Fx Wp) {
    if constexpr (E == 1) {
        return Wp;
    } else {
        auto step = [](Fx v) { return E <= 4 ? v : fx_norm(v); };
        const Fx h = step(fx_pow<E / 2>(Wp));
        const Fx sq = step(fx_sq(h));
        if constexpr (E % 2) return step(fx_mul(sq, Wp));
        else return sq;
    }
}

// C^d (prod_j t_j)^r; cdx = C^d as Fx.  quarters: Wp holds prod_j 4 t_j over
// this many dimensions.
template <int R>
__device__ __forceinline__ Fx korobov_weight_fixed(Fx Wp, Fx cdx, int quarters = 0) {
    Fx w = fx_mul(fx_pow<R>(Wp), cdx);   // unnormalized, at least 2^59
    w.e -= 2 * R * quarters;
    return w;
}

}  // namespace qmc
