// noise_check.cu -- the white noise of ic_noise.cuh on the host against its
// definition in long double.  Prints "name largest-error" in units of 2^-53.
#include <math.h>
#include <stdio.h>
#include <string.h>

#include "../../paper_2003_03931_gb300/csrc/ic_noise.cuh"

using namespace pmpm;

int main() {
    static constexpr NoiseTables t{};
    const long double turn = 6.283185307179586476925286766559L * 0x1p-53L;
    long double log_err = 0, root_err = 0, cos_err = 0, noise_err = 0;
    auto grow = [](long double& e, long double d) { e = fmaxl(e, fabsl(d) * 0x1p53L); };
    const unsigned long long top = (1ull << 53) - 1;
    for (long i = 0; i < 4000000; ++i) {
        unsigned long long m = splitmix64(7, i) >> 11, a = splitmix64(9, i) >> 11;
        if (i < 1000) m = i;                                     // the longest values
        else if (i < 2000) m = top - (i - 1000);                 // u up to 1
        else if (i < 1000000) m >>= i % 53;                      // every octave
        else if (i < 1100000) m = (i % 1024 << 43) - i % 3 & top;   // around the table's nodes and their middles
        if (i < 3000) a = ((unsigned long long)(i % 5) << 51) - 1 + i % 3 & top;   // quarter turns
        else if (i < 100000) a = (i % 1024 << 43) - i % 3 & top;
        const long double y = -2 * logl((long double)(m + 1) * 0x1p-53L), c = cosl(turn * a);
        const double yd = minus_two_log(m, t), g = root(yd), cd = cos_turn(a, t);
        if (m == top) grow(log_err, yd);
        else grow(log_err, (yd - y) / y);
        if (yd > 0) grow(root_err, (g - sqrtl((long double)yd)) / sqrtl((long double)yd));
        grow(cos_err, cd - c);
        grow(noise_err, g * cd - sqrtl(y) * c);
    }
    int wrong = 0;
    for (int k = -(1 << 20) + 1; k < 1 << 20; ++k) wrong += small_double(k) != (double)k;
    printf("log %.3Lf\nroot %.3Lf\ncos %.3Lf\nnoise %.3Lf\ndouble %d\n", log_err, root_err, cos_err, noise_err, wrong);
    return 0;
}
