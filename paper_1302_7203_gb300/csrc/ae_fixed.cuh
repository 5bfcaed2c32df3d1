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
// (2^-46: the unit is then 2^-60 of D)
constexpr uint32_t kFixMinExp = 1023 - 46;

AE_HD uint64_t f64_bits(double x) {
#ifdef __CUDA_ARCH__
    return (uint64_t)__double_as_longlong(x);
#else
    uint64_t u;
    memcpy(&u, &x, 8);
    return u;
#endif
}

// x modulo 2^64 in units of 2^-106 (bits below the unit dropped, towards -inf)
AE_HD uint64_t fix_mod(double x) {
    const uint64_t b = f64_bits(x);
    const int e = (int)((b >> 52) & 0x7ff);
    if (e == 0) return 0;                               // zero (or far below the unit)
    int64_t m = (int64_t)((b & 0xfffffffffffffull) | 0x10000000000000ull);
    if (b >> 63) m = -m;
    const int sh = e - 1075 + kFixFrac;
    if (sh >= 64) return 0;
    if (sh >= 0) return (uint64_t)m << sh;
    return sh <= -63 ? (uint64_t)(m >> 63) : (uint64_t)(m >> -sh);
}

// high 64 bits of a * b, at most 2 below the exact floor
AE_HD uint64_t mul_hi3(uint64_t a, uint64_t b) {
    const uint32_t al = (uint32_t)a, ah = (uint32_t)(a >> 32);
    const uint32_t bl = (uint32_t)b, bh = (uint32_t)(b >> 32);
    const uint64_t t1 = (uint64_t)al * bh;
    const uint64_t t2 = (uint64_t)ah * bl;
    return (uint64_t)ah * bh + (t1 >> 32) + (t2 >> 32);
}

// The part of |p - lambda| beyond its rounded value D = (dh, dl), in units of
// D's last place times 2^-23.  T = P - L, the exact difference modulo 2^64;
// the tail has to stay below 2^8 last places.
AE_HD int tail_of(uint64_t T, uint32_t dh, uint32_t dl, uint32_t eb) {
    const uint64_t neg = (dh >> 31) ? ~0ull : 0ull;     // |difference|, one unit low if negative
    const uint64_t Dm = ((uint64_t)((dh & 0xfffffu) | 0x100000u) << 32) | dl;
    const int sh = (int)eb - (1075 - kFixFrac);
    const uint64_t tail = (T ^ neg) - (Dm << (sh & 63));
    return (int)((tail << ((55 - sh) & 63)) >> 32);
}

// 2^63 / m for the significand m in [1, 2) of D = (dh, dl) with tail tl (see
// tail_of), from the high word `seed` of an approximation of 1 / m.  CUBIC
// adds the e^3 term (one wide multiply more: sums take it, vector components,
// rounded to 53 bits, do not).
template <bool CUBIC>
AE_HD uint64_t recip63(uint32_t dh, uint32_t dl, int tl, uint32_t seed) {
    const uint32_t Dmh = (dh & 0xfffffu) | 0x100000u;
    const uint32_t R0 = seed - 0x3fd00001u;             // 2^21 / m, below 2^21
    const uint32_t X = R0 << 10;
    const uint32_t nR = 0u - (R0 + R0);
    // E = 2^74 (1 - Dm R0 / 2^73) mod 2^64; nR stands for 2^32 - 2 R0, hence - dl
    const uint64_t w = (uint64_t)dl * nR;
    const uint32_t eh = Dmh * nR + (uint32_t)(w >> 32) - dl;
    const uint64_t E = ((uint64_t)eh << 32) | (uint32_t)w;
    const int corr = (int)(((int64_t)tl * (int64_t)(int)X) >> 32);
    const uint64_t C = E + (uint64_t)((int64_t)corr * -1);
    const int e32 = (int)(uint32_t)(C >> 26);            // e 2^48
    uint32_t sq = (uint32_t)((uint64_t)((int64_t)e32 * e32) >> 32);         // e^2 2^64
    if (CUBIC)                                                              // (e^2 + e^3) 2^64
        sq = (uint32_t)((uint64_t)((int64_t)e32 * (int64_t)(e32 + (int)(sq >> 16))) >> 32);
    const uint64_t C2 = C + (uint64_t)sq * 1024u;
    const uint64_t m0 = (uint64_t)(uint32_t)C2 * R0;
    return (((uint64_t)X << 32) | (m0 >> 32)) +
           (uint64_t)((int64_t)(int)(uint32_t)(C2 >> 32) * (int64_t)(int)R0);
}

}  // namespace ae
