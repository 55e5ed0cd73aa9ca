// fftpass.cuh -- the two register steps of a mesh transform's pass along one
// axis, for kernels that fuse something into its ends (coarse.cu, power.cu).
//
// A pass of n = N1 N2 points per pencil takes two register transforms with one
// transpose through shared memory between (fft.cu).  With j = N2 n1 + n2 and
// k = k1 + N1 k2 the forward pass ends with all k2 of one k1 in a thread's
// registers, and that is where the inverse one begins.
#pragma once

#include "regfft.cuh"

namespace pmpm {

// The float32 nearest to d.  Two halves that float32 holds exactly and one
// multiply-add round it once; 64-bit conversions and FP64 run at 1/64 of the
// FP32 rate here (three per cell took 24 us for a 32^3 mesh on three SMs).
__device__ __forceinline__ float f32_of(long long d) {
    if (d >= (1ll << 40) || d < -(1ll << 40)) return __ll2float_rn(d);
    return __fmaf_rn((float)(int)(d >> 16), 65536.f, (float)((int)d & 0xffff));
}

// shared-memory add without a returned value
__device__ __forceinline__ void smem_red(uint32_t* p, uint32_t v) {
    asm volatile("red.shared.add.u32 [%0], %1;" ::"r"((unsigned)__cvta_generic_to_shared(p)), "r"(v) : "memory");
}

// |k| and sign (0 for k = 0) of a wavenumber index of an n-point axis
__device__ __forceinline__ void kfold(int k, int nc, int& a, float& sg) {
    if (k == 0) { a = 0; sg = 0.f; }
    else if (k <= nc / 2) { a = k; sg = 1.f; }
    else { a = nc - k; sg = -1.f; }
}

constexpr int kPassWidth = 256;
constexpr int clog2(int v) { return v <= 1 ? 0 : 1 + clog2(v / 2); }

template <int N1, int N2>
struct Pass {
    static constexpr int n = N1 * N2, L1 = clog2(N1), L2 = clog2(N2), LN = L1 + L2;
    // pencils of a block (32 at n = 32, 64 at 64 ... 16 at 256 and 512, 8 at 1024)
    static constexpr int P = n == 32 ? 32 : (n == 512 ? 16 : (4096 / n < 8 ? 8 : 4096 / n)), LP = clog2(P);
    static constexpr int RS = N2 + 1, PS = N1 * RS + 1;                    // see k_fft_pass_r
    static constexpr size_t kBytes = sizeof(float2) * P * PS;
};

__device__ __forceinline__ float2 cmulw(float2 a, float2 w) {
    return make_float2(a.x * w.x - a.y * w.y, a.x * w.y + a.y * w.x);
}

// N1-point step over n1 of item (p, n2), times W_n^(n2 k1), into the buffer
template <int N1, int N2>
__device__ __forceinline__ void pass_first(float2 (&a)[N1], float2* Y, int p, int n2, const float2* tw, int twsh) {
    using Q = Pass<N1, N2>;
    fft_dit<N1, -1>(a);
#pragma unroll
    for (int k1 = 0; k1 < N1; ++k1) Y[p * Q::PS + k1 * Q::RS + n2] = cmulw(a[k1], tw[(n2 * k1) << twsh]);
}
// and the N2-point step of item (p, k1) from it
template <int N1, int N2>
__device__ __forceinline__ void pass_second(float2 (&a)[N2], const float2* Y, int p, int k1) {
    using Q = Pass<N1, N2>;
#pragma unroll
    for (int n2 = 0; n2 < N2; ++n2) a[bitrev<Q::L2>(n2)] = Y[p * Q::PS + k1 * Q::RS + n2];
    fft_dit<N2, -1>(a);
}
// inverse: the N2-point step of item (p, k1) into the buffer
template <int N1, int N2>
__device__ __forceinline__ void back_first(float2 (&a)[N2], float2* Y, int p, int k1, const float2* tw, int twsh) {
    using Q = Pass<N1, N2>;
    fft_dit<N2, 1>(a);
#pragma unroll
    for (int n2 = 0; n2 < N2; ++n2) {
        const float2 w = tw[(n2 * k1) << twsh];
        Y[p * Q::PS + k1 * Q::RS + n2] = cmulw(a[n2], make_float2(w.x, -w.y));
    }
}
// and the N1-point step of item (p, n2): a[n1]
template <int N1, int N2>
__device__ __forceinline__ void back_second(float2 (&a)[N1], const float2* Y, int p, int n2) {
    using Q = Pass<N1, N2>;
#pragma unroll
    for (int k1 = 0; k1 < N1; ++k1) a[bitrev<Q::L1>(k1)] = Y[p * Q::PS + k1 * Q::RS + n2];
    fft_dit<N1, 1>(a);
}

}  // namespace pmpm
