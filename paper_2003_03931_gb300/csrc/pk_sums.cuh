// pk_sums.cuh -- sums of |delta~|^2 over a shell in integers.  A float32's square is a
// 48-bit product of mantissas; on one scale for a whole group of modes (the group's
// largest exponent) squares add up exactly, in three limbs of 21 bits that 32-bit
// shared-memory additions fill.  What is lost lies below 2^-(48 + SHIFT) of the group's
// largest square, where a float32 square would round every mode at 2^-24 of its own.
#pragma once

#include "common.cuh"

namespace pmpm {

PMPM_HD uint32_t float_bits(float x) {
#ifdef __CUDA_ARCH__
    return __float_as_uint(x);
#else
    union { float f; uint32_t u; } b;
    b.f = x;
    return b.u;
#endif
}

// x^2 in units of 2^(2 (emax - 150) - SHIFT), rounded: below 2^(48 + SHIFT) for an x of
// at most the exponent emax (0 .. 254, as stored).  0 for |x| < 2^-126.
template <int SHIFT>
PMPM_HD unsigned long long square_of(float x, int emax) {
    const uint32_t b = float_bits(x) & 0x7fffffffu;
    if (b < 0x00800000u) return 0;
    const uint32_t m = (b & 0x7fffffu) | 0x800000u;
    const unsigned long long p = (unsigned long long)m * m;
    const int sh = SHIFT - 2 * (emax - (int)(b >> 23));
    if (sh >= 0) return p << sh;
    return sh < -48 ? 0 : (p + (1ull << (-sh - 1))) >> -sh;
}

// An integer below 2^62 in limbs; 2048 of each fit 32 bits.
struct Limbs {
    uint32_t v[3];
};
PMPM_HD Limbs limbs_of(unsigned long long x) {
    return {{(uint32_t)x & 0x1fffffu, (uint32_t)(x >> 21) & 0x1fffffu, (uint32_t)(x >> 42)}};
}
// the sum of the squares that square_of<SHIFT> made
template <int SHIFT>
PMPM_HD double limbs_value(long long l0, long long l1, long long l2, int emax) {
    const double v = (double)(l0 + (l1 << 21)) + (double)l2 * 4398046511104.0;
    return ldexp(v, 2 * (emax - 150) - SHIFT);
}

}  // namespace pmpm
