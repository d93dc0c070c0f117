// qmc_lattice.cuh -- exact rank-1 lattice points on the integer pipe.
//
// A point coordinate of the shifted rank-1 lattice (Sec. 2.1, Eq. (lattice); Fig. 1) is
//     v = frac(r/n + Delta),  r = i z_j mod n,  Delta = D 2^-53  (D a 53-bit integer),
// and the library's contract is u = RN(v): the exact rational rounded once to the nearest
// double.  On GB300 the FP64 pipe is the scarce resource (~2 DFMA/clk/SM), while the
// integer pipe is ~30x wider, so the point itself never touches FP64:
//
//   * r/n is carried as a 128-bit fixed-point fraction F = floor(r 2^128 / n) plus the
//     exact remainder rem = r 2^128 mod n.  Stepping i -> i+1 adds the constants
//     Fz = floor(z 2^128 / n), remz = z 2^128 mod n with a carry from the remainder; the
//     wrap of r past n is the natural overflow of the 128-bit add (mod 2^128 is frac).
//   * The shift enters as D 2^75, i.e. D << 11 added to the high word (mod 2^64).
//   * v = (V + rem/n) 2^-128 with V = F + D 2^75 mod 2^128; rounding to 53 bits needs the
//     leading-zero count, a funnel shift, the round bit and a sticky bit (lower bits of V
//     or rem != 0).  When V's high word is zero (v < 2^-64, which needs r/n + Delta within
//     2^-64 of an integer) more quotient bits are produced from rem by long division.
//
// Everything here is exact integer arithmetic; the only floating-point object is the final
// bit pattern.
#pragma once
#include <cstdint>

namespace qmc {

struct DimConst {
    uint64_t fz_hi, fz_lo;  // floor(z 2^128 / n)
    uint64_t rq;            // the next 64 quotient bits, floor(remz 2^64 / n)
};

// What a step adds: F of one (or several) lattice steps and its exact remainder.
struct LatticeStep {
    uint64_t fz_hi, fz_lo, remz;
};
// remz = z 2^128 mod n: z 2^128 = F n + remz, so remz = -F n modulo 2^64, and remz < n < 2^63.
__device__ __forceinline__ LatticeStep lattice_step_of(const DimConst &c, uint64_t n) {
    return {c.fz_hi, c.fz_lo, 0 - c.fz_lo * n};
}

// Restoring division of (hi:lo) by n, requiring hi < n: quotient < 2^64.
__host__ __device__ inline void divmod_128_64(uint64_t hi, uint64_t lo, uint64_t n, uint64_t *q,
                                              uint64_t *r) {
    uint64_t quo = 0;
#pragma unroll 1
    for (int b = 0; b < 64; ++b) {
        uint64_t top = hi >> 63;
        hi = (hi << 1) | (lo >> 63);
        lo <<= 1;
        quo <<= 1;
        if (top || hi >= n) {
            hi -= n;
            quo |= 1;
        }
    }
    *q = quo;
    *r = hi;
}

// Lattice state of one coordinate at index i < 2^63: F(i) and rem(i) for r = i z mod n.
// F(i) = (i Fz + floor(i remz / n)) mod 2^128 and rem(i) = i remz mod n = -F(i) n mod 2^64.
// The quotient comes from the host's reciprocal word: with rq = floor(remz 2^64 / n),
// i remz / n - i rq / 2^64 lies in [0, i / 2^64), below 1, so q = floor(i rq / 2^64) is the
// exact quotient or one less, and the remainder it leaves lies in [0, 2n), which 64 bits
// hold for n < 2^63: one conditional correction, no division.  (Every stream of a lattice
// sum starts here; an FP64-assisted 128/64 division in its place cost ~30 FP64 warp
// instructions of ~17 SM cycles each per warp.)
__device__ __forceinline__ void lattice_state_at(uint64_t i, const DimConst &c, uint64_t n,
                                                 uint64_t &f_hi, uint64_t &f_lo,
                                                 uint64_t &rem) {
    const uint64_t lo = i * c.fz_lo;
    uint64_t add = __umul64hi(i, c.rq);
    uint64_t r = 0 - (lo + add) * n;
    if (r >= n) {
        r -= n;
        ++add;
    }
    rem = r;
    f_lo = lo + add;
    f_hi = __umul64hi(i, c.fz_lo) + i * c.fz_hi + (f_lo < lo);
}

// One lattice step i -> i+1.
__device__ __forceinline__ void lattice_step(const LatticeStep &c, uint64_t n, uint64_t &f_hi,
                                             uint64_t &f_lo, uint64_t &rem) {
    uint64_t r2 = rem + c.remz;             // < 2n < 2^64 for n < 2^63
    uint64_t carry = (r2 >= n) ? 1u : 0u;
    rem = carry ? r2 - n : r2;
    uint64_t lo = f_lo + c.fz_lo;
    uint64_t c1 = (lo < f_lo) ? 1u : 0u;
    uint64_t lo2 = lo + carry;
    uint64_t c2 = (lo2 < lo) ? 1u : 0u;
    f_lo = lo2;
    f_hi = f_hi + c.fz_hi + c1 + c2;
}

// The same step for n < 2^32: the fraction is carried to 192 bits, started with the third
// word i w mod 2^64 and stepped by one long addition of w = ceil(remz 2^64 / n), without an
// exact remainder.  After i steps the third word is high by less than i units.  So no carry out
// of it is missed, and none is spurious: that would take a true fraction of a unit of 2^-128,
// rem / n <= 1 - 1/n, above 1 - i / 2^64, and i < n < 2^32.  (Rounded down it would be low, and
// miss the carry wherever rem(i) = 0: at multiples of n's odd part, inside the lattice of an
// even n that is no power of two.)
constexpr int kShortBits = 32;
__device__ __forceinline__ uint64_t short_step_word(const DimConst &c, uint64_t n) {
    return c.rq + (c.rq * n != 0);   // remz 2^64 mod n = -rq n modulo 2^64
}
struct ShortState {
    uint64_t f_hi, f_lo, f_2;
    __device__ __forceinline__ void step(uint64_t z_hi, uint64_t z_lo, uint64_t z_2) {
        asm("add.cc.u64 %0, %0, %3; addc.cc.u64 %1, %1, %4; addc.u64 %2, %2, %5;"
            : "+l"(f_2), "+l"(f_lo), "+l"(f_hi)
            : "l"(z_2), "l"(z_lo), "l"(z_hi));
    }
};

// Round (vhi:vlo + rem/n) 2^-128 to the nearest double; general path for vhi == 0.
static __device__ __noinline__ double fixed_to_double_small(uint64_t vlo, uint64_t rem, uint64_t n) {
    if (vlo == 0 && rem == 0) return 0.0;
    // more bits: rem 2^64 = e n + rem2, so the value is (vlo 2^64 + e + rem2/n) 2^-192
    uint64_t e, rem2;
    divmod_128_64(rem, 0, n, &e, &rem2);
    uint64_t whi, wlo;
    int bexp;  // biased exponent minus one, see the fast path
    if (vlo != 0) {
        int lz = __clzll(vlo);
        whi = lz ? ((vlo << lz) | (e >> (64 - lz))) : vlo;
        wlo = lz ? (e << lz) : e;
        bexp = 957 - lz;   // value in [2^(-65-lz), 2^(-64-lz))
    } else {
        // v < 2^-128 cannot happen for n < 2^64 and a 53-bit shift (v >= 2^-53 / n);
        // kept total for any input
        if (e == 0) return 0.0;
        int lz = __clzll(e);
        whi = e << lz;
        wlo = 0;
        bexp = 893 - lz;   // value in [2^(-129-lz), 2^(-128-lz))
    }
    uint64_t mant = whi >> 11;
    uint64_t rb = (whi >> 10) & 1u;
    uint64_t sticky = (whi & 0x3FFull) | wlo | rem2;
    mant += rb & ((sticky != 0) | (mant & 1u));
    return __longlong_as_double((long long)(((uint64_t)bexp << 52) + mant));
}

// u = RN((V + rem/n) 2^-128) for V = (vhi:vlo), any point.
static __device__ __noinline__ double fixed_to_double_any(uint64_t vhi, uint64_t vlo, uint64_t n) {
    const uint64_t rem = 0 - vlo * n;   // F n = -rem modulo 2^64; the shift leaves F's low word
    if (vhi == 0) return fixed_to_double_small(vlo, rem, n);
    int lz = __clzll(vhi);
    uint64_t whi = lz ? ((vhi << lz) | (vlo >> (64 - lz))) : vhi;
    uint64_t wlo = lz ? (vlo << lz) : vlo;
    uint64_t mant = whi >> 11;                 // 53 bits, leading one at bit 52
    uint64_t rb = (whi >> 10) & 1u;
    uint64_t sticky = (whi & 0x3FFull) | wlo | rem;
    mant += rb & ((sticky != 0) | (mant & 1u));
    // value = mant 2^(-53-lz), biased exponent 1022 - lz; adding mant (implicit bit
    // included) to (exponent - 1) << 52 also handles the carry mant == 2^53.
    return __longlong_as_double((long long)(((uint64_t)(1021 - lz) << 52) + mant));
}

// The same.  A point v >= 2^-10 with bits below its top word (vlo != 0: all but ~2^-10 of
// them) is rounded from that word alone: it holds the 53 bits and the round bit, and what lies
// below is not zero.
__device__ __forceinline__ double fixed_to_double(uint64_t vhi, uint64_t vlo, uint64_t n) {
    const uint32_t top = (uint32_t)(vhi >> 32);
    if (top < 0x00400000u || !vlo) return fixed_to_double_any(vhi, vlo, n);
    const int lz = __clz(top);   // 0..9
    const uint32_t hi = __funnelshift_l((uint32_t)vhi, top, lz) ^ 0x80000000u;   // leading one off
    const uint32_t lo = ((uint32_t)vhi << lz) | 1u;                              // sticky
    const uint64_t m = ((uint64_t)hi << 32 | lo) + (0x3FFu + ((lo >> 11) & 1u));
    return __longlong_as_double((long long)((m >> 11) + ((uint64_t)(1022 - lz) << 52)));
}

}  // namespace qmc
