// ae_fixed.cuh -- fixed-point arithmetic of the terms zeta^2 / (p - lambda)^r.
//
// The FP64 pipe of this chip retires 2 lane-operations per clock and SM, the
// FP32 pipe 128, the integer multiply-add 32 x 32 + 64 bits 64 (measured), so
// an FP64 instruction costs as much as 32 wide integer multiply-adds.  A term
// is therefore formed with ONE FP64 subtraction D = fl(p - lambda) and
// integers from there on:
//   * the exact difference is known modulo 2^64 in units of 2^-106 (poles and
//     lambda are kept in that form too), which gives the rounding error of D
//     and lambda's own tail (tail_of);
//   * the reciprocal of D's significand starts from the 20-bit hardware seed;
//     its residual e = 1 - D r0 is exact in 64-bit arithmetic, and
//     r0 (1 + e + e^2) is good to |e|^3 <= 2^-57, typically 2^-61 (recip63);
//   * products keep the high 64 bits of 64 x 64 (mul_hi3, low cross terms
//     dropped: at most 3 units in the last place);
//   * sums are integers aligned to a bound on the whole sum: exact in any
//     order, so every team shape and every path gives the same bits.
// All values here are scaled by a power of two so that |p| < 1/2.
// The functions compile for the host too (the CPU tests check them against
// wide integers).
#pragma once
#include <stdint.h>
#include <string.h>

#ifdef __CUDACC__
#define AE_HD __host__ __device__ __forceinline__
#else
#define AE_HD static inline
#endif

namespace ae {

// unit of the modular representation: 2^-kFixFrac
constexpr int kFixFrac = 106;
// biased exponent of D below which its last place is too close to the unit
// (2^-45: the unit is then 2^-61 of D)
constexpr uint32_t kFixMinExp = 1023 - 45;
// exponents by which D may lie below lambda: its tail then stays below 2^22 last
// places
constexpr uint32_t kTailSpan = 20;

AE_HD uint64_t f64_bits(double x) {
#ifdef __CUDA_ARCH__
    return (uint64_t)__double_as_longlong(x);
#else
    uint64_t u;
    memcpy(&u, &x, 8);
    return u;
#endif
}

// a second representation, in units of 2^-140, takes the differences below
// kFixMinExp down to this exponent (unit 2^-61 of D again)
constexpr int kFixFrac2 = 140;
constexpr uint32_t kFixMinExp2 = kFixMinExp - 34;

// x modulo 2^64 in units of 2^-FRAC (bits below the unit dropped, towards -inf)
template <int FRAC = kFixFrac>
AE_HD uint64_t fix_mod(double x) {
    const uint64_t b = f64_bits(x);
    const int e = (int)((b >> 52) & 0x7ff);
    if (e == 0) return 0;                               // zero (or far below the unit)
    int64_t m = (int64_t)((b & 0xfffffffffffffull) | 0x10000000000000ull);
    if (b >> 63) m = -m;
    const int sh = e - 1075 + FRAC;
    if (sh >= 64) return 0;
    if (sh >= 0) return (uint64_t)m << sh;
    return sh <= -63 ? (uint64_t)(m >> 63) : (uint64_t)(m >> -sh);
}

// hi + lo in units of 2^(e - 63), e the exponent of hi > 0: lo is given in that
// unit, at most half of hi's last place (2^10; 2^9 below a power of two).  The top
// bit is 0 where a negative lo takes a power of two below itself (a spike of unit
// modulus, a product z * (1 / z)): the products need no leading 1, so the value
// stays as it is.  No carry: hi's significand is at most 2^64 - 2^11.
AE_HD uint64_t fix_mant(double hi, int64_t lo) {
    return (((f64_bits(hi) & 0xfffffffffffffull) | 0x10000000000000ull) << 11) + (uint64_t)lo;
}

// high 64 bits of a * b, at most 2 below the exact floor (on the device as one
// carry chain: 5 instructions, where the 64-bit adds take 8)
AE_HD uint64_t mul_hi3(uint64_t a, uint64_t b) {
    const uint32_t al = (uint32_t)a, ah = (uint32_t)(a >> 32);
    const uint32_t bl = (uint32_t)b, bh = (uint32_t)(b >> 32);
#ifdef __CUDA_ARCH__
    uint32_t lo, hi;
    asm("{\n\t.reg .u32 t, c;\n\t"
        "mul.hi.u32 t, %2, %5;\n\t"
        "mad.hi.cc.u32 t, %3, %4, t;\n\t"
        "addc.u32 c, 0, 0;\n\t"
        "mad.lo.cc.u32 %0, %3, %5, t;\n\t"
        "madc.hi.u32 %1, %3, %5, c;\n\t}"
        : "=&r"(lo), "=r"(hi)                        // (lo is written before the last reads)
        : "r"(al), "r"(ah), "r"(bl), "r"(bh));
    return ((uint64_t)hi << 32) | lo;
#endif
    const uint64_t t1 = (uint64_t)al * bh;
    const uint64_t t2 = (uint64_t)ah * bl;
    return (uint64_t)ah * bh + (t1 >> 32) + (t2 >> 32);
}

// The part of |p - lambda| beyond its rounded value D = (dh, dl), in 2^-7 of D's
// last place, rounded down.  T = P - L, the exact difference modulo 2^64.
template <int FRAC = kFixFrac>
AE_HD int tail_of(uint64_t T, uint32_t dh, uint32_t dl, uint32_t eb) {
    const uint64_t neg = (dh >> 31) ? ~0ull : 0ull;     // |difference|, one unit low if negative
    const uint64_t Dm = ((uint64_t)((dh & 0xfffffu) | 0x100000u) << 32) | dl;
    const int sh = (int)eb - (1075 - FRAC);
    const int64_t tail = (int64_t)((T ^ neg) - (Dm << (sh & 63)));
    return (int)(tail >> ((sh - 7) & 63));
}

// 2^63 / m for the significand m in [1, 2) of D = (dh, dl) with tail t (see
// tail_of), from the high word `seed` of an approximation of 1 / m.  CUBIC
// adds the e^3 term (one wide multiply more: sums take it, vector components,
// rounded to 53 bits, do not).
template <bool CUBIC>
AE_HD uint64_t recip63(uint32_t dh, uint32_t dl, int t, uint32_t seed) {
    const uint32_t Dmh = (dh & 0xfffffu) | 0x100000u;
    const uint32_t R0 = seed - 0x3fd00001u;             // 2^21 / m, below 2^21
    const uint32_t nR = 0u - (R0 << 8);
    // E = 2^81 (1 - (Dm + (t + 1/2) 2^-7) R0 / 2^73) mod 2^64; nR stands for
    // 2^32 - 2^8 R0, hence - dl
    const uint64_t w = (uint64_t)dl * nR;
    const uint32_t eh = Dmh * nR + (uint32_t)(w >> 32) - dl;
    const uint64_t E = (((uint64_t)eh << 32) | (uint32_t)w) +
                       (uint64_t)((int64_t)(2 * t + 1) * (int64_t)(int)(0u - R0));
    const int e32 = (int)(uint32_t)(E >> 32);            // e 2^49
    uint32_t sq = (uint32_t)((uint64_t)((int64_t)e32 * e32) >> 32);         // e^2 2^66
    if (CUBIC)                                                              // (e^2 + e^3) 2^66
        sq = (uint32_t)((uint64_t)((int64_t)e32 * (int64_t)(e32 + (int)(sq >> 17))) >> 32);
    const uint64_t C = E + (uint64_t)sq * 32768u;
    const uint64_t m0 = (uint64_t)(uint32_t)C * R0;
    const int64_t c = (int64_t)(int)(uint32_t)(C >> 32) * (int64_t)(int)R0 + (int64_t)(m0 >> 32);
    return ((uint64_t)(R0 << 10) << 32) + (uint64_t)(c >> 7);
}

// 2^124 / m for m in [0.87 2^62, 1.13 2^63), from R0 = 2^84 / m to less than one
// part in 2^21 (an FP32 reciprocal, rounded to an integer: 2^-21.2): with m R0 =
// 2^84 (1 + e) modulo 2^64 it is R0 (1 - e + e^2) to 2^-60 (e^3 < 2^-63; the last
// place is 2^-62 of 0.44 to 1.15).
AE_HD uint64_t recip62(uint64_t m, uint32_t R0) {
    const uint64_t w = (uint64_t)(uint32_t)m * R0;
    const uint32_t xh = (uint32_t)(m >> 32) * R0 + (uint32_t)(w >> 32);
    const uint64_t X = ((uint64_t)xh << 32) | (uint32_t)w;                  // e 2^84
    const uint32_t sq = (uint32_t)((uint64_t)((int64_t)(int)xh * (int)xh) >> 32);  // e^2 2^72
    const uint64_t C = X - (uint64_t)sq * 4096u;
    const uint64_t m0 = (uint64_t)(uint32_t)C * R0;
    const int64_t c = (int64_t)(int)(uint32_t)(C >> 32) * (int64_t)(int)R0 + (int64_t)(m0 >> 32);
    return ((uint64_t)(R0 << 8) << 32) - (uint64_t)(c >> 12);
}

}  // namespace ae
