// ic_noise.cuh -- the white noise of the initial conditions: SplitMix64 counters
// 2i and 2i + 1, Box-Muller in float64.
//
// FP64 and 64-bit conversions run at 1/64 of the FP32 rate on this part, and log,
// sqrt and cospi with the conversions came to about 70 such operations a value,
// half of the x pass.  Here integers take the numbers apart and tables leave short
// series (25 operations): 256^3 particles, x pass 2.24 -> 1.22 ms on a GB300.
//   -2 log u   u = f 2^-k, f in [3/4, 3/2); f c = 1 + r with c the table's 1/f of
//              the nearest 256th, |r| < 2^-9 (P. T. P. Tang, ACM TOMS 16, 1990):
//              2k log 2 + 2 log c - 2 log(1 + r).  c = 1 around f = 1, so that
//              nothing cancels where the logarithm vanishes
//   sqrt       one step for g = y / sqrt(y) and one for its remainder, from a float32 estimate
//   cos        of the nearest 512th of a turn and Taylor's series of the rest
// Errors against the formula in long double: 0.73 units of 2^-53 rms (0.76 by way of
// log, sqrt and cospi).
#pragma once

#include "common.cuh"

namespace pmpm {

constexpr int kLogSteps = 256, kCosSteps = 512, kExpSteps = 64;

// SplitMix64 output for counter j (Steele, Lea & Flood 2014)
PMPM_HD unsigned long long splitmix64(unsigned long long seed, unsigned long long j) {
    unsigned long long z = seed + (j + 1ull) * 0x9E3779B97F4A7C15ull;
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    return z ^ (z >> 31);
}

PMPM_HD double bits_double(unsigned long long b) {
#ifdef __CUDA_ARCH__
    return __longlong_as_double((long long)b);
#else
    double d;
    memcpy(&d, &b, 8);
    return d;
#endif
}
PMPM_HD unsigned long long double_bits(double d) {
#ifdef __CUDA_ARCH__
    return (unsigned long long)__double_as_longlong(d);
#else
    unsigned long long b;
    memcpy(&b, &d, 8);
    return b;
#endif
}
// leading zeros of a 64-bit number, not 0
PMPM_HD int lead_zeros(unsigned long long m) {
#ifdef __CUDA_ARCH__
    return __clzll((long long)m);
#else
    return __builtin_clzll(m);
#endif
}

// (double)k, |k| < 2^20, without a conversion
PMPM_HD double small_double(int k) {
    if (k == 0) return 0.0;
    const uint32_t a = (uint32_t)(k < 0 ? -k : k);
    const int e = 63 - lead_zeros(a);
    const uint32_t hi = ((1023u + e) << 20) | ((a << (20 - e)) & 0xfffffu) | (k < 0 ? 0x80000000u : 0u);
    return bits_double((unsigned long long)hi << 32);
}

// Two doubles, hi + lo, for the tables below (T. J. Dekker, Numer. Math. 18, 1971).
struct Pair {
    double hi, lo;
};
constexpr Pair pair_sum(double a, double b) {
    const double s = a + b, t = s - a;
    return {s, (a - (s - t)) + (b - t)};
}
constexpr Pair pair_product(double a, double b) {
    const double ca = 134217729.0 * a, cb = 134217729.0 * b;
    const double ah = ca - (ca - a), al = a - ah, bh = cb - (cb - b), bl = b - bh, p = a * b;
    return {p, ((ah * bh - p) + ah * bl + al * bh) + al * bl};
}
constexpr Pair operator+(Pair a, Pair b) {
    const Pair s = pair_sum(a.hi, b.hi);
    return pair_sum(s.hi, s.lo + (a.lo + b.lo));
}
constexpr Pair operator*(Pair a, Pair b) {
    const Pair p = pair_product(a.hi, b.hi);
    return pair_sum(p.hi, p.lo + (a.hi * b.lo + a.lo * b.hi));
}
constexpr Pair operator/(Pair a, double d) {
    const double q = a.hi / d;
    const Pair p = pair_product(q, d);
    return pair_sum(q, ((a.hi - p.hi) - p.lo + a.lo) / d);
}

// Made by the compiler, from series in Pairs.
struct alignas(16) NoiseTables {
    double lg[kLogSteps + 1][2] = {};   // c, 2 log c
    double cs[kCosSteps][4] = {};       // cos, what is left of it, sin
    double ex[kExpSteps][2] = {};       // 2k log 2, what is left of it
    constexpr NoiseTables() {
        // log((256 + i) / 256) is the sum of log((n + 1) / (n - 1)) = 2 (1/n + 1/(3 n^3) + ..), n = 511 + 2 i
        const Pair ln2 = {0.693147180559945309417232121458, 2.31904681384629961549e-17};
        Pair sum = {0.0, 0.0};
        for (int i = 0; i <= kLogSteps; ++i) {
            if (i > 0) {
                const double n = 2 * kLogSteps - 1 + 2 * i;
                Pair power = Pair{1.0, 0.0} / n, series = power;
                for (int k = 3; k < 15; k += 2) {
                    power = power / n / n;
                    series = series + power / k;
                }
                sum = sum + series + series;
            }
            const bool up = i >= kLogSteps / 2;   // c = 2 / .. there
            lg[i][0] = (up ? 2.0 : 1.0) * kLogSteps / (kLogSteps + i);
            // 2 log of the rounded c: its 1 + e part of the node's
            const Pair node = pair_product(lg[i][0], (double)(kLogSteps + i) / kLogSteps * (up ? 0.5 : 1.0));
            const double e = (node.hi - 1.0) + node.lo;
            const Pair log_c = up ? ln2 + Pair{-sum.hi, -sum.lo} + Pair{e, 0.0} : Pair{-sum.hi, -sum.lo} + Pair{e, 0.0};
            lg[i][1] = i == kLogSteps ? 0.0 : 2.0 * log_c.hi;
        }
        const Pair turn = {6.283185307179586476925286766559, 2.44929359829470635445e-16};
        for (int i = 0; i <= kCosSteps / 8; ++i) {
            const Pair x = turn * Pair{(double)i / kCosSteps, 0.0}, y = x * x;
            Pair c = {1.0, 0.0}, s = x, tc = c, ts = x;
            for (int k = 1; k < 15; ++k) {
                tc = tc * y / (-(2.0 * k - 1) * (2 * k));
                ts = ts * y / (-(2.0 * k) * (2 * k + 1));
                c = c + tc;
                s = s + ts;
            }
            // the eight angles of this cosine and sine
            constexpr int Q = kCosSteps / 4;
            for (int q = 0; q < 4; ++q) {
                put((q * Q + i) % kCosSteps, q, c, s);
                put((q * Q + Q - i) % kCosSteps, q, s, c);
            }
        }
        for (int k = 0; k < kExpSteps; ++k) {
            const Pair v = ln2 * Pair{2.0 * k, 0.0};
            ex[k][0] = v.hi;
            ex[k][1] = v.lo;
        }
    }
    // entry i: cos and sin of an angle of the first quadrant, turned by q quadrants
    constexpr void put(int i, int q, Pair c, Pair s) {
        const Pair a = q & 1 ? s : c, b = q & 1 ? c : s;
        const double ga = q == 1 || q == 2 ? -1.0 : 1.0, gb = q >= 2 ? -1.0 : 1.0;
        cs[i][0] = ga * a.hi;
        cs[i][1] = ga * a.lo;
        cs[i][2] = gb * b.hi;
    }
};

// -2 log((m + 1) / 2^53), m < 2^53
PMPM_HD double minus_two_log(unsigned long long m, const NoiseTables& t) {
    ++m;
    const int z = lead_zeros(m);   // 10 (m = 2^53) .. 63
    const unsigned long long frac = (m << z) >> 11 & 0xfffffffffffffull;   // of f = m / 2^(63 - z) in [1, 2)
    const int i = (int)((frac + (1ull << 43)) >> 44), up = i >= kLogSteps / 2;
    const double f = bits_double((unsigned long long)(1023 - up) << 52 | frac);
    const double r = fma(f, t.lg[i][0], -1.0);
    double p = fma(r, 1.0 / 3, -2.0 / 5);
    p = fma(r, p, 1.0 / 2);
    p = fma(r, p, -2.0 / 3);
    p = fma(r, p, 1.0);
    p = fma(r, p, -2.0);
    // u = f 2^-k
    const int k = z - 10 - up;
    return t.ex[k][0] + fma(r, p, t.lg[i][1] + t.ex[k][1]);
}

// sqrt(y), y = 0 or a float32's exponent
PMPM_HD double root(double y) {
    if (y == 0.0) return 0.0;
    // float32 of y's leading bits, and its inverse root as a double
    const unsigned long long b = double_bits(y);
    const uint32_t fb = (uint32_t)((b - (896ull << 52)) >> 29);
#ifdef __CUDA_ARCH__
    const uint32_t rb = __float_as_uint(rsqrtf(__uint_as_float(fb)));
#else
    float fy;
    memcpy(&fy, &fb, 4);
    fy = 1.0f / sqrtf(fy);
    uint32_t rb;
    memcpy(&rb, &fy, 4);
#endif
    const unsigned long long r64 = ((unsigned long long)rb << 29) + (896ull << 52);
    const double r = bits_double(r64), h = bits_double(r64 - (1ull << 52));   // 1 / sqrt(y) and half of it
    double g = y * r;
    g = fma(g, fma(-g, h, 0.5), g);
    return fma(fma(-g, g, y), h, g);
}

// cos(2 pi m / 2^53), m < 2^53
PMPM_HD double cos_turn(unsigned long long m, const NoiseTables& t) {
    constexpr double w = 6.283185307179586476925286766559;
    const unsigned long long a = m + (1ull << 43);
    const double* cs = t.cs[(a >> 44) & (kCosSteps - 1)];
    // the rest in turns, |x| <= 2^-10, exactly
    const double x = bits_double(0x3fe0000000000000ull | (a & ((1ull << 44) - 1))) - (0.5 + 0x1p-10), q = x * x;
    const double s = x * fma(q, fma(q, w * w * w * w * w / 120, -(w * w * w) / 6), w);
    const double c = q * fma(q, fma(q, -(w * w * w * w * w * w) / 720, w * w * w * w / 24), -(w * w) / 2);
    return cs[0] + fma(-cs[2], s, fma(cs[0], c, cs[1]));
}

// unit Gaussian of lattice point i
PMPM_HD double noise_at(unsigned long long seed, unsigned long long i, const NoiseTables& t) {
    return root(minus_two_log(splitmix64(seed, 2ull * i) >> 11, t)) * cos_turn(splitmix64(seed, 2ull * i + 1ull) >> 11, t);
}

}  // namespace pmpm
