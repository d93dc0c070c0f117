// qmc_fitmap.cuh -- the PolySingular variance-reduction map (Sec. 2.4, Eq. (ISfit)) on the
// integer pipe, for the polynomial families with the coordinate in 0.64 fixed point.
//
// With b = -a1 > 0, v0 = (a0 - 1) / (a0 - x) and v1 = b / (x + b), both in (0, 1] on [0, 1],
//   p(x)  = |a2| x v0 + |a3| (1 + b) (1 - v1) + x (a4 + x (a5 + a6 x)),
//   p'(x) = |a2| a0/(a0 - 1) v0^2 + |a3| (1 + b)/b v1^2 + a4 + x (2 a5 + 3 a6 x),
// every factor bounded.  v0 and v1 are held at 2^62, p is formed at 2^58 (from coefficients at
// 2^60) and p' at 2^em with em from the sum of its coefficients; the Jacobian enters a
// normalized running product.  p's truncations, ~3.2 units of 2^-58 on average, are made up by
// three; what is left is within 4 units where x is small (7 elsewhere), where the FP64 form rounds
// x near 1 to 2^-53 before a0 - x divides by it, but is relative near 0 (see eval_point).
// ~230 integer instructions per dimension against 20 FP64 ones of 17 SM cycles a warp each,
// which kept fitted sector integrands FP64-bound: a batch of 256 (half of them fitted) took 62 ms
// and takes 50, the fitted d = 5 call with n = 108,863, m = 32 1090 us and takes 755.
//
// The form is taken when the coefficients are moderate (FitFixed::stage); a point that a map
// which is not monotone sends outside [0, 1], or where p' is not positive, is left to the FP64
// form (FitFixed::apply returns false).
#pragma once
#include <cstdint>

#include "qmc_fixed.cuh"
#include "qmc_params.cuh"

namespace qmc {

struct FitFixed {
    struct Dim {
        uint64_t a0, b;              // a0 2^(64 - k0), b 2^(64 - k1)
        uint64_t c0, cb;             // a0 - 1 and b, normalized mantissas
        uint64_t a2, a3b, k2, k3;    // |a2|, |a3| (1 + b) at 2^60; p' coefficients at 2^(em + 1)
        int64_t a4, a5, a6;          // at 2^60
        int64_t d4, d5, d6;          // a4, 2 a5, 3 a6 at 2^em
        int k0, k1, s0, s1, em;      // s: right shift of c R to v at 2^62, less the mantissa's lz
    } dim[kMaxDim];
    int ok;
    int slope;                       // p' is at most this in every dimension
    // what 4 units of 2^-58 in every coordinate add to a cubic, in units of 2^-62 of its bound
    static constexpr int kErrorUnits = 3 * 4 * 32;

    // Stages dimension j from fit[j][6] (one thread each; ok = slope = 1 and a barrier before, one after).
    __device__ __forceinline__ void stage(const double *fit, int j) {
        const double *a = fit + 6 * j;
        const double a0 = a[0], b = -a[1], a2 = fabs(a[2]), a3 = fabs(a[3]), a4 = a[4], a5 = a[5];
        const double a6 = 1.0 - a2 - a3 - a4 - a5;
        const double k2 = a2 * a0 / (a0 - 1.0), k3 = a3 * (1.0 + b) / b;
        const double M = k2 + k3 + fabs(a4) + 2.0 * fabs(a5) + 3.0 * fabs(a6);
        // p at 2^58 below 2^62, p' from coefficients of sum at most 64 (2^-56 of it is 2^-50)
        if (!(a0 >= 1.0005 && a0 < 1024.0 && b >= 0.0005 && b < 1023.0 && a2 + a3 * (1.0 + b) < 7.0 &&
              fabs(a4) + fabs(a5) + fabs(a6) < 7.0 && M < 64.0 && M > 0x1p-10)) {
            atomicAnd(&ok, 0);
            return;
        }
        atomicMax(&slope, (int)M + 1);
        Dim &o = dim[j];
        o.k0 = ilogb(a0) + 1;
        o.k1 = ilogb(1.0 + b) + 1;
        o.a0 = __double2ull_rn(ldexp(a0, 64 - o.k0));
        o.b = __double2ull_rn(ldexp(b, 64 - o.k1));
        const Fx c0 = fx_of_double(a0 - 1.0), cb = fx_of_double(b);
        o.c0 = c0.m;
        o.cb = cb.m;
        // v 2^62 = c R 2^-64 2^(ec - k + lz - 1) with c = m 2^(ec - 64)
        o.s0 = o.k0 - c0.e + 1;
        o.s1 = o.k1 - cb.e + 1;
        o.a2 = __double2ull_rn(ldexp(a2, 60));
        o.a3b = __double2ull_rn(ldexp(a3 * (1.0 + b), 60));
        o.a4 = llrint(ldexp(a4, 60));
        o.a5 = llrint(ldexp(a5, 60));
        o.a6 = llrint(ldexp(a6, 60));
        o.em = 61 - ilogb(M);
        o.k2 = __double2ull_rn(ldexp(k2, o.em + 1));
        o.k3 = __double2ull_rn(ldexp(k3, o.em + 1));
        o.d4 = llrint(ldexp(a4, o.em));
        o.d5 = llrint(ldexp(2.0 * a5, o.em));
        o.d6 = llrint(ldexp(3.0 * a6, o.em));
    }

    // X = x 2^64 to p(x) 2^64, with p' folded into the normalized product J.
    __device__ __forceinline__ static uint64_t ratio(uint64_t D, uint64_t c, int s) {
        const int lz = __clz((unsigned)(D >> 32));   // D >= 2^43
        return mulhi_trunc(c, recip_fixed(D << lz)) >> (s - lz);
    }
    __device__ __forceinline__ bool apply(uint64_t &X, int j, Fx &J) const {
        const Dim &o = dim[j];
        const uint64_t v0 = ratio(o.a0 - (X >> o.k0), o.c0, o.s0);
        const uint64_t v1 = ratio(o.b + (X >> o.k1), o.cb, o.s1);
        int64_t q = smulhi_x(smulhi_x(smulhi_x(o.a6, X) + o.a5, X) + o.a4, X) >> 2;
        q += (int64_t)(mulhi_trunc(mulhi_trunc(X, v0), o.a2) + mulhi_trunc((1ull << 62) - v1, o.a3b) + 3);
        const int64_t dp = smulhi_x(smulhi_x(o.d6, X) + o.d5, X) + o.d4 +
                           (int64_t)(mulhi_trunc(sqhi_trunc(v0) << 3, o.k2) + mulhi_trunc(sqhi_trunc(v1) << 3, o.k3));
        // within rounding of [0, 1], and p' not vanishing
        if (q < -(1ll << 20) || q > (1ll << 58) + (1ll << 20) || dp < (1ll << 40)) return false;
        J = fx_norm(fx_mul(J, fx_norm({(uint64_t)dp, 64 - o.em})));
        X = q <= 0 ? 0ull : q >= 1ll << 58 ? ~0ull : (uint64_t)q << 6;
        return true;
    }
    // All d dimensions; false when one of them is left to the FP64 form.  (A call of its own:
    // inlined beside the map of each dimension it cost the unfitted kernel its registers, 4.43 ->
    // 4.73 ms at d = 8, n = 1,072,187, m = 32.)
    __device__ __noinline__ bool apply_all(uint64_t *X, int d, Fx *J) const {
        Fx prod{0x8000000000000000ull, 1};
        bool inside = true;
#pragma unroll 1
        for (int j = 0; inside && j < d; ++j) inside = apply(X[j], j, prod);
        *J = prod;
        return inside;
    }
};

}  // namespace qmc
