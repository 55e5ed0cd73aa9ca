// pk_sums_check.cu -- the shell sums of pk_sums.cuh on the host against long double.
// Prints "name largest-error": of a group's sum, in units of 2^-53 of the sum, for
// modes of one size, of a million-fold range of sizes, and with zeros among them.
#include <math.h>
#include <stdio.h>

#include "../../paper_2003_03931_gb300/csrc/ic_noise.cuh"
#include "../../paper_2003_03931_gb300/csrc/pk_sums.cuh"

using namespace pmpm;

// `n` modes of amplitude range 2^-spread .. 1 times 2^top, each twice where `twice`
template <int SHIFT>
static long double off(unsigned long long seed, int n, int spread, int top, int zeros, int times) {
    long double want = 0;
    long long l[3] = {0, 0, 0};
    float x[2 * 2048];
    int emax = 0;
    for (int i = 0; i < 2 * n; ++i) {
        const unsigned long long r = splitmix64(seed, i);
        x[i] = ldexpf((float)((double)(long long)(r >> 8) * 0x1p-55 - 1.0), top - (int)(r % (spread + 1)));
        if (zeros && r % 3 == 0) x[i] = 0.f;
        const int e = (int)(float_bits(x[i]) >> 23 & 255u);
        emax = e > emax ? e : emax;
    }
    for (int i = 0; i < n; ++i) {
        const Limbs v = limbs_of((square_of<SHIFT>(x[2 * i], emax) + square_of<SHIFT>(x[2 * i + 1], emax)) << times);
        for (int e = 0; e < 3; ++e) {
            l[e] += v.v[e];
            if (l[e] >> 32) return INFINITY;   // a limb's 32 bits
        }
        want += ((long double)x[2 * i] * x[2 * i] + (long double)x[2 * i + 1] * x[2 * i + 1]) * (1 << times);
    }
    return fabsl(limbs_value<SHIFT>(l[0], l[1], l[2], emax) - want) / want * 0x1p53L;
}

int main() {
    long double one = 0, wide = 0, holes = 0, small = 0;
    for (int s = 0; s < 400; ++s) {
        const int n = s % 2 ? 2048 : 1 + s;
        one = fmaxl(one, off<12>(s, n, 0, s % 40 - 20, 0, s & 1));
        wide = fmaxl(wide, off<12>(s, n, 20, 3, 0, s & 1));
        holes = fmaxl(holes, off<12>(s, n, 2, -60, 1, s & 1));
        small = fmaxl(small, off<10>(s, 1 + s % 512, 2, 0, 0, 3));
    }
    printf("one %.3Lf\nwide %.3Lf\nholes %.3Lf\nsmall %.3Lf\n", one, wide, holes, small);
    return 0;
}
