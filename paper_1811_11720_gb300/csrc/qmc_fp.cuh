// qmc_fp.cuh -- exact bit-level helpers that keep work off the FP64 pipe.
#pragma once
#include <cstdint>

namespace qmc {

// Non-negative double compare on the bit pattern.
__device__ __forceinline__ bool le_half(double u) {
    return (unsigned long long)__double_as_longlong(u) <= 0x3FE0000000000000ull;
}

// 1 - u for u in [1/2, 1], exact (Sterbenz), on the integer pipe.
__device__ __forceinline__ double one_minus_upper(double u) {
    uint64_t b = (uint64_t)__double_as_longlong(u);
    if (b >= 0x3FF0000000000000ull) return 0.0;             // u == 1
    uint64_t mant = (b & 0x000FFFFFFFFFFFFFull) | 0x0010000000000000ull;  // u = mant 2^-53
    uint64_t x = 0x0020000000000000ull - mant;               // 1 - u = x 2^-53, 1 <= x <= 2^52
    int lz = __clzll(x);                                     // >= 11
    return __longlong_as_double((long long)(((uint64_t)(1032 - lz) << 52) + (x << (lz - 11))));
}

// 2 y for y = 0 or a positive normal double, exact, on the integer pipe.
__device__ __forceinline__ double twice(double y) {
    uint64_t b = (uint64_t)__double_as_longlong(y);
    return __longlong_as_double((long long)(b ? b + 0x0010000000000000ull : 0ull));
}

// x^e for a small non-negative integer e (uniform across the warp): left-to-right binary
// powering, floor(log2 e) squarings plus one multiply per further set bit.
__device__ __forceinline__ double ipow_u(double x, int e) {
    if (e <= 0) return 1.0;
    const int top = 31 - __clz(e);
    double r = x;
#pragma unroll 1
    for (int b = top - 1; b >= 0; --b) {
        r *= r;
        if ((e >> b) & 1) r *= x;
    }
    return r;
}

// 1/a within 2^-52.9 of itself: the hardware's ~20-bit estimate r and one step of Chebyshev's
// iteration (third order: r - f/f' (1 + f f'' / (2 f'^2)) for f = 1/r - a, which is r (1 + e + e^2),
// e = 1 - a r), three FP64 instructions instead of a full division.  Outside the exponents where estimate and result are
// normal (zero, infinities and NaN among them) the division itself.
static __device__ __noinline__ double recip_any(double a) { return 1.0 / a; }
__device__ __forceinline__ bool mid_range(double a) {   // 2^-1020 <= |a| < 2^1020
    return ((uint32_t)__double2hiint(a) << 1 >> 21) - 3u < 2040u;
}
__device__ __forceinline__ double recip_cubic(double a) {
    if (!mid_range(a)) return recip_any(a);
    double r;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(a));
    const double e = fma(-a, r, 1.0);
    return fma(r, fma(e, e, e), r);
}

// 1/sqrt(a) for a > 0 likewise, f = y^-2 - a: y + y e (1/2 + 3/8 e), e = 1 - a y^2, five
// instructions, within 2^-52.3.
static __device__ __noinline__ double rsqrt_any(double a) { return rsqrt(a); }
__device__ __forceinline__ double rsqrt_cubic(double a) {
    if (!mid_range(a)) return rsqrt_any(a);
    double y;
    asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(a));
    const double e = fma(-(a * y), y, 1.0);
    return fma(y * e, fma(0.375, e, 0.5), y);
}

// Select between two doubles on the integer pipe.
__device__ __forceinline__ double sel(bool p, double a, double b) { return p ? a : b; }

}  // namespace qmc
