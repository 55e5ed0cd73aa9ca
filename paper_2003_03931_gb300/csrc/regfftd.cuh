// regfftd.cuh -- the register transforms of regfft.cuh and the two-step passes
// of fftpass.cuh in float64, for the Zel'dovich fields.  FP64 runs at 1/64 of
// the FP32 rate on this part, so what counts is the number of operations: the
// fused multiply-add butterfly takes 6 for a twiddled pair of outputs, and the
// passes work on real fields (half the spectrum).
#pragma once

#include "regfft.cuh"

namespace pmpm {

// cos(2 pi j / 32) for any integer j (compile-time after unrolling)
__device__ __forceinline__ double cos32d(int j) {
    j &= 31;
    const int q = j >> 3, r = j & 7, idx = (q & 1) ? 8 - r : r;
    const double v = idx == 0 ? 1.0
                   : idx == 1 ? 0.98078528040323044913
                   : idx == 2 ? 0.92387953251128675613
                   : idx == 3 ? 0.83146961230254523708
                   : idx == 4 ? 0.70710678118654752440
                   : idx == 5 ? 0.55557023301960222474
                   : idx == 6 ? 0.38268343236508977173
                   : idx == 7 ? 0.19509032201612826785 : 0.0;
    return (q == 1 || q == 2) ? -v : v;
}

// (a, b) <- (a + w b, a - w b), w = exp(S 2 pi i j / 32); see twiddle_f
template <int S>
__device__ __forceinline__ void butterflyd(double2& a, double2& b, int j) {
    j &= 31;
    const double2 x = a, d = b;
    if (j == 0) {
        a = make_double2(x.x + d.x, x.y + d.y);
        b = make_double2(x.x - d.x, x.y - d.y);
        return;
    }
    if (j == 8) {   // w = S i
        a = make_double2(x.x - S * d.y, x.y + S * d.x);
        b = make_double2(x.x + S * d.y, x.y - S * d.x);
        return;
    }
    const double wr = cos32d(j), wi = S * cos32d(8 - j);
    double m;
    double2 u;
    if (fabs(wr) >= fabs(wi)) {
        const double t = wi / wr;
        m = wr;
        u = make_double2(d.x - t * d.y, d.y + t * d.x);
    } else {
        const double t = wr / wi;
        m = wi;
        u = make_double2(t * d.x - d.y, t * d.y + d.x);
    }
    a = make_double2(x.x + m * u.x, x.y + m * u.y);
    b = make_double2(x.x - m * u.x, x.y - m * u.y);
}

template <int N, int HALF, int S>
struct DitStaged {
    static __device__ __forceinline__ void run(double2 (&a)[N]) {
#pragma unroll
        for (int g = 0; g < N; g += 2 * HALF) {
#pragma unroll
            for (int k = 0; k < HALF; ++k) butterflyd<S>(a[g + k], a[g + k + HALF], k * (32 / (2 * HALF)));
        }
        DitStaged<N, 2 * HALF, S>::run(a);
    }
};
template <int N, int S>
struct DitStaged<N, N, S> {
    static __device__ __forceinline__ void run(double2 (&)[N]) {}
};
// a[bitrev(n)] = x[n] on entry, the N-point DFT (N up to 32) on return
template <int N, int S>
__device__ __forceinline__ void fft_ditd(double2 (&a)[N]) {
    DitStaged<N, 1, S>::run(a);
}

__device__ __forceinline__ double2 cmuld(double2 a, double2 w) {
    return make_double2(a.x * w.x - a.y * w.y, a.x * w.y + a.y * w.x);
}

constexpr int dlog2(int v) { return v <= 1 ? 0 : 1 + dlog2(v / 2); }

// A pass of n = N1 N2 points over a half-spectrum mesh (n/2 values along x): P
// pencils neighbouring in x per block, one step of a pencil a thread.
template <int N1, int N2>
struct PassD {
    static constexpr int n = N1 * N2, H = n / 2, L1 = dlog2(N1), L2 = dlog2(N2), LN = L1 + L2;
    static constexpr int kFit = 2048 / n < 4 ? 4 : 2048 / n, P = kFit < H ? kFit : H, LP = dlog2(P);
    static constexpr int kWide = P * (N1 > N2 ? N1 : N2), T = kWide < 32 ? 32 : (kWide > 256 ? 256 : kWide);
    static constexpr int RS = N2 + 1, PS = N1 * RS + 1;
    static constexpr size_t kBytes = sizeof(double2) * P * PS;
};

// N1-point step of item (p, n2) times W_n^(n2 k1) into the buffer, and the
// N2-point step of item (p, k1) from it (a[k2] at k = k1 + N1 k2)
template <int N1, int N2>
__device__ __forceinline__ void firstd(double2 (&a)[N1], double2* Y, int p, int n2, const double2* tw, int twsh) {
    using Q = PassD<N1, N2>;
    fft_ditd<N1, -1>(a);
    Y[p * Q::PS + n2] = a[0];
#pragma unroll
    for (int k1 = 1; k1 < N1; ++k1) Y[p * Q::PS + k1 * Q::RS + n2] = cmuld(a[k1], tw[(n2 * k1) << twsh]);
}
template <int N1, int N2>
__device__ __forceinline__ void secondd(double2 (&a)[N2], const double2* Y, int p, int k1) {
    using Q = PassD<N1, N2>;
#pragma unroll
    for (int n2 = 0; n2 < N2; ++n2) a[bitrev<Q::L2>(n2)] = Y[p * Q::PS + k1 * Q::RS + n2];
    fft_ditd<N2, -1>(a);
}
// inverse: N2-point step of item (p, k1) into the buffer, N1-point step of item
// (p, n2) from it (a[n1] at j = N2 n1 + n2)
template <int N1, int N2>
__device__ __forceinline__ void back_firstd(double2 (&a)[N2], double2* Y, int p, int k1, const double2* tw, int twsh) {
    using Q = PassD<N1, N2>;
    fft_ditd<N2, 1>(a);
    Y[p * Q::PS + k1 * Q::RS] = a[0];
#pragma unroll
    for (int n2 = 1; n2 < N2; ++n2) {
        const double2 w = tw[(n2 * k1) << twsh];
        Y[p * Q::PS + k1 * Q::RS + n2] = cmuld(a[n2], make_double2(w.x, -w.y));
    }
}
template <int N1, int N2>
__device__ __forceinline__ void back_secondd(double2 (&a)[N1], const double2* Y, int p, int n2) {
    using Q = PassD<N1, N2>;
#pragma unroll
    for (int k1 = 0; k1 < N1; ++k1) a[bitrev<Q::L1>(k1)] = Y[p * Q::PS + k1 * Q::RS + n2];
    fft_ditd<N1, 1>(a);
}

}  // namespace pmpm
