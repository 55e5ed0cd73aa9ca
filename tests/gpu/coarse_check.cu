// coarse_check.cu -- the coarse force's fused passes (coarse.cu) against the general
// transforms (fft.cu) at every size, the ones whose boxes are too large for an oracle
// among them: a random integer density, a random kernel.  Prints "cells rms" lines, the
// rms difference of F_l over the rms of F_l.
#include <math.h>
#include <stdlib.h>

#include <vector>

#include "../../paper_2003_03931_gb300/csrc/coarse.cu"

namespace pmpm {

__global__ void k_fill(int64_t n, unsigned long long salt, long long mean, long long* rho) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        unsigned long long z = (i + salt) * 0x9E3779B97F4A7C15ull;
        z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
        rho[i] = mean + (long long)(z >> 34) - (1ll << 29);
    }
}
__global__ void k_kernel(int64_t n, float4* g) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        g[i] = make_float4(1e-9f * (float)(i % 101 + 1), 1e-9f * (float)(i % 89 + 1), 1e-9f * (float)(i % 97 + 1), 0.f);
}
__global__ void k_compare(int64_t n, const float* a, const float* b, double* sums) {
    double d = 0.0, r = 0.0;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        d += ((double)a[i] - b[i]) * ((double)a[i] - b[i]);
        r += (double)b[i] * b[i];
    }
    atomicAdd(&sums[0], d);
    atomicAdd(&sums[1], r);
}

template <int N1, int N2>
int check() {
    constexpr int nc = N1 * N2;
    Sim* const sp = new Sim();
    Sim& s = *sp;
    s.nc = s.fft_max = nc;
    s.ncells = (int64_t)nc * nc * nc;
    s.n = 8 * s.ncells;
    const int64_t h = nc / 2 + 1, C = s.ncells;
    std::vector<float2> tw(nc);
    for (int k = 0; k < nc; ++k)
        tw[k] = make_float2((float)cos(2 * M_PI * k / nc), (float)-sin(2 * M_PI * k / nc));
    float* kept = nullptr;
    double *sums = nullptr, out[2];
    if (cudaMalloc(&s.rho_c, 8 * C) || cudaMalloc(&s.cA, 8 * C) || cudaMalloc(&s.cB1, 8 * C) ||
        cudaMalloc(&s.cB2, 8 * C) || cudaMalloc(&s.Fl, 12 * C) || cudaMalloc(&kept, 12 * C) ||
        cudaMalloc(&s.green_coarse, 16 * h * h * h) || cudaMalloc(&s.tw_f, 8 * nc) || cudaMalloc(&sums, 16))
        return 1;
    cudaMemcpy(s.tw_f, tw.data(), 8 * nc, cudaMemcpyHostToDevice);
    cudaMemset(sums, 0, 16);
    const long long mean = 1ll << 30;
    k_fill<<<2048, 256>>>(C, nc, mean, s.rho_c);
    k_kernel<<<2048, 256>>>(h * h * h, s.green_coarse);
    float* const passes = s.Fl;
    launch_passes<N1, N2>(s, mean);
    s.Fl = kept;
    if (launch_kept(s, mean)) return 1;
    k_compare<<<2048, 256>>>(3 * C, passes, kept, sums);
    if (cudaMemcpy(out, sums, 16, cudaMemcpyDeviceToHost)) return 1;
    printf("%d %.3e\n", nc, out[1] > 0.0 ? sqrt(out[0] / out[1]) : 1.0);
    for (void* p : {(void*)s.rho_c, (void*)s.cA, (void*)s.cB1, (void*)s.cB2, (void*)passes, (void*)kept,
                    (void*)s.green_coarse, (void*)s.tw_f, (void*)sums})
        cudaFree(p);
    delete sp;
    return cudaGetLastError() != cudaSuccess;
}

}  // namespace pmpm

int main() {
    using namespace pmpm;
    fft_setup();
    coarse_setup();
    return check<8, 8>() || check<8, 16>() || check<16, 16>() || check<16, 32>() || check<32, 32>();
}
