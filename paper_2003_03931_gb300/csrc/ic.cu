// ic.cu -- Zel'dovich initial conditions (Sec. IV-A.2) for a power-law
// spectrum P(k) = k^slope exp(-(k/k_c)^2), in float64 on the device:
//   white noise (SplitMix64 counters 2i, 2i+1; Box-Muller) -> DFT ->
//   Psi~_d = i k_d / k^2 sqrt(P) w~ (k = 0 and Nyquist planes zeroed) ->
//   inverse DFT -> rms normalisation -> x = q + a Psi, p = a^(3/2) Psi (EdS; a^2 E f a Psi
//   in LambdaCDM) ->
//   Q = floor(64 x) mod (256 nc), p in float32 -> cell-ordered encode.
//
// The field is real, so the transforms keep kx < np/2 only (the amplitude is
// zero on the Nyquist planes), five passes of register transforms:
//   x      noise made in place of a load, two rows as one complex pencil
//   y
//   z      forward, times i k_d sqrt(P)/k^2 for the three components, back; the
//          rms of the displacement comes from the spectrum here (Parseval), so that
//          nothing waits for the fields
//   y      back, three components
//   x      back, two fields as one complex pencil, straight to codes and momenta
// FP64 bounds it: about 180 operations a particle at 1/64 of the FP32 rate.  On a
// GB300, 256^3 particles with their encode: 17.2 ms with complex radix-2 transforms
// and a pass per operation, 5.8 now (x with the noise 1.2, y 0.35, z 1.2, y back 1.1,
// x back 1.8); 7.4 with the library's logarithm and cosine and three fields through
// the inverse z transform.
#include "pmpm_impl.cuh"
#include "ic_noise.cuh"
#include "regfftd.cuh"

namespace pmpm {

namespace {

constexpr double kPi = 3.141592653589793238462643383279502884;

__device__ constexpr NoiseTables kNoise{};

// kf sqrt(P(k)) / k^2 (0 at k = 0), shared by the three displacement components.
// The amplitude depends on the mode only through m = nx^2 + ny^2 + nz^2
// (k^2 = kf^2 m): one table entry per m, so the float64 pow, exp and sqrt run
// 3 (np/2)^2 times instead of np^3 times.
__global__ void k_ic_amp_table(int mmax, int nf, double slope, double kc, double* __restrict__ tab) {
    const double kf = 2.0 * kPi / nf;
    for (int m = blockIdx.x * blockDim.x + threadIdx.x; m <= mmax; m += gridDim.x * blockDim.x) {
        double c = 0.0;
        if (m > 0) {
            const double k2 = kf * kf * (double)m;
            const double k = sqrt(k2);
            c = kf * (sqrt(pow(k, slope) * exp(-(k / kc) * (k / kc))) / k2);
        }
        tab[m] = 0.5 * c;   // the x pass gives twice the noise's spectrum
    }
}

// x: rows 2q and 2q + 1 of the noise as one complex pencil, then their spectra
// (kx < n/2) apart: 2 A = Z + conj Z', 2 B = -i (Z - conj Z') with Z' at -kx
template <int N1, int N2>
__global__ void __launch_bounds__(PassD<N1, N2>::T) k_ic_x(unsigned long long seed, double2* __restrict__ out,
                                                           const double2* __restrict__ tw, int twsh) {
    using Q = PassD<N1, N2>;
    constexpr int kZ = Q::n + 1;
    static_assert(kZ <= Q::PS, "");
    extern __shared__ __align__(16) unsigned char ic_smem[];
    double2* Y = reinterpret_cast<double2*>(ic_smem);
    const int64_t q0 = (int64_t)blockIdx.x * Q::P;
    for (int it = threadIdx.x; it < Q::P * N2; it += Q::T) {
        const int p = it >> Q::L2, n2 = it & (N2 - 1);
        const unsigned long long i = (unsigned long long)(2 * (q0 + p)) << Q::LN;
        double2 a[N1];
#pragma unroll 1
        for (int n1 = 0; n1 < N1; ++n1) {
            // (one copy of the noise's code; the values wait in the buffer's own places)
            const unsigned long long j = i + N2 * n1 + n2;
            Y[p * Q::PS + n1 * Q::RS + n2] = make_double2(noise_at(seed, j, kNoise), noise_at(seed, j + Q::n, kNoise));
        }
#pragma unroll
        for (int n1 = 0; n1 < N1; ++n1) a[bitrev<Q::L1>(n1)] = Y[p * Q::PS + n1 * Q::RS + n2];
        firstd<N1, N2>(a, Y, p, n2, tw, twsh);
    }
    __syncthreads();
    constexpr int kItems = (Q::P * N1 + Q::T - 1) / Q::T;
    double2 a[kItems][N2];
#pragma unroll
    for (int u = 0; u < kItems; ++u) {
        const int it = threadIdx.x + u * Q::T;
        if (it < Q::P * N1) secondd<N1, N2>(a[u], Y, it >> Q::L1, it & (N1 - 1));
    }
    __syncthreads();
#pragma unroll
    for (int u = 0; u < kItems; ++u) {
        const int it = threadIdx.x + u * Q::T, p = it >> Q::L1, k1 = it & (N1 - 1);
        if (it < Q::P * N1) {
#pragma unroll
            for (int k2 = 0; k2 < N2; ++k2) Y[p * Q::PS + k1 + N1 * k2] = a[u][k2];
        }
    }
    __syncthreads();
    for (int it = threadIdx.x; it < Q::P * Q::H; it += Q::T) {
        const int p = it / Q::H, k = it & (Q::H - 1);
        const double2 z = Y[p * Q::PS + k], w = Y[p * Q::PS + ((Q::n - k) & (Q::n - 1))];
        double2* row = out + (2 * (q0 + p)) * Q::H + k;
        row[0] = make_double2(z.x + w.x, z.y - w.y);
        row[Q::H] = make_double2(z.y + w.y, w.x - z.x);
    }
}

// y: pencils (kx, z), stride n/2; forward in place, back of component blockIdx.y from
// w (0; times ky: 1) or in place (2)
template <int N1, int N2, int S>
__global__ void __launch_bounds__(PassD<N1, N2>::T) k_ic_y(const double2* w, double2* field,
                                                           const double2* __restrict__ tw, int twsh) {
    using Q = PassD<N1, N2>;
    extern __shared__ __align__(16) unsigned char ic_smem[];
    double2* Y = reinterpret_cast<double2*>(ic_smem);
    const int64_t q0 = (int64_t)blockIdx.x * Q::P;
    const int64_t at = q0 / Q::H * ((int64_t)Q::H * Q::n) + q0 % Q::H;
    double2* data = field + (int64_t)blockIdx.y * Q::H * Q::n * Q::n + at;
    const double2* src = S > 0 && blockIdx.y < 2 ? w + at : data;
    if (S < 0) {
        for (int it = threadIdx.x; it < Q::P * N2; it += Q::T) {
            const int p = it & (Q::P - 1), n2 = it >> Q::LP;
            double2 a[N1];
#pragma unroll
            for (int n1 = 0; n1 < N1; ++n1) a[bitrev<Q::L1>(n1)] = src[p + (N2 * n1 + n2) * Q::H];
            firstd<N1, N2>(a, Y, p, n2, tw, twsh);
        }
        __syncthreads();
        for (int it = threadIdx.x; it < Q::P * N1; it += Q::T) {
            const int p = it & (Q::P - 1), k1 = it >> Q::LP;
            double2 a[N2];
            secondd<N1, N2>(a, Y, p, k1);
#pragma unroll
            for (int k2 = 0; k2 < N2; ++k2) data[p + (k1 + N1 * k2) * Q::H] = a[k2];
        }
    } else {
        for (int it = threadIdx.x; it < Q::P * N1; it += Q::T) {
            const int p = it & (Q::P - 1), k1 = it >> Q::LP;
            double2 a[N2];
#pragma unroll
            for (int k2 = 0; k2 < N2; ++k2) {
                const int k = k1 + N1 * k2;
                double2 v = src[p + k * Q::H];
                if (blockIdx.y == 1) {
                    const double c = small_double(k < Q::H ? k : k - Q::n);
                    v = make_double2(c * v.x, c * v.y);
                }
                a[bitrev<Q::L2>(k2)] = v;
            }
            back_firstd<N1, N2>(a, Y, p, k1, tw, twsh);
        }
        __syncthreads();
        for (int it = threadIdx.x; it < Q::P * N2; it += Q::T) {
            const int p = it & (Q::P - 1), n2 = it >> Q::LP;
            double2 a[N1];
            back_secondd<N1, N2>(a, Y, p, n2);
#pragma unroll
            for (int n1 = 0; n1 < N1; ++n1) data[p + (N2 * n1 + n2) * Q::H] = a[n1];
        }
    }
}

// z: forward, Psi~_d = i n_d tab w~ (zero on the Nyquist planes) and back.  kx and ky do
// not change along z: without them the x and the y component are one field, which
// takes w's place; the z component goes to `field`.  partial[block] = sum of |Psi~|^2
// over the whole spectrum (a kx > 0 counts for its mirror image), in a fixed order
template <int N1, int N2>
__global__ void __launch_bounds__(PassD<N1, N2>::T) k_ic_z(const double* __restrict__ tab,
                                                           double2* w, double2* __restrict__ field,
                                                           double* __restrict__ partial,
                                                           const double2* __restrict__ tw, int twsh) {
    using Q = PassD<N1, N2>;
    constexpr int64_t plane = (int64_t)Q::H * Q::n;
    constexpr int kItems = (Q::P * N1 + Q::T - 1) / Q::T;
    extern __shared__ __align__(16) unsigned char ic_smem[];
    double2* Y = reinterpret_cast<double2*>(ic_smem);
    __shared__ double sums[Q::T / 32];
    const int64_t q0 = (int64_t)blockIdx.x * Q::P;   // pencils (kx, ky)
    const int ky = (int)(q0 / Q::H), kx0 = (int)(q0 % Q::H);
    for (int it = threadIdx.x; it < Q::P * N2; it += Q::T) {
        const int p = it & (Q::P - 1), n2 = it >> Q::LP;
        double2 a[N1];
#pragma unroll
        for (int n1 = 0; n1 < N1; ++n1) a[bitrev<Q::L1>(n1)] = w[q0 + p + (N2 * n1 + n2) * plane];
        firstd<N1, N2>(a, Y, p, n2, tw, twsh);
    }
    __syncthreads();
    double2 a[kItems][N2];   // tab w~
    double energy = 0.0;
#pragma unroll
    for (int u = 0; u < kItems; ++u) {
        const int it = threadIdx.x + u * Q::T, p = it & (Q::P - 1), k1 = it >> Q::LP;
        if (it < Q::P * N1) {
            secondd<N1, N2>(a[u], Y, p, k1);
            const int kx = kx0 + p, ny = ky < Q::H ? ky : ky - Q::n, m0 = kx * kx + ny * ny;
            double e = 0.0;
#pragma unroll
            for (int k2 = 0; k2 < N2; ++k2) {
                const int kz = k1 + N1 * k2, nz = kz < Q::H ? kz : kz - Q::n, m = m0 + nz * nz;
                const double c = ky == Q::H || kz == Q::H ? 0.0 : tab[m];
                a[u][k2] = make_double2(c * a[u][k2].x, c * a[u][k2].y);
                e += small_double(m) * (a[u][k2].x * a[u][k2].x + a[u][k2].y * a[u][k2].y);
            }
            energy += kx == 0 ? e : 2.0 * e;
        }
    }
#pragma unroll 1
    for (int d = 0; d < 2; ++d) {
        __syncthreads();
#pragma unroll
        for (int u = 0; u < kItems; ++u) {
            const int it = threadIdx.x + u * Q::T, p = it & (Q::P - 1), k1 = it >> Q::LP;
            if (it < Q::P * N1) {
                double2 b[N2];
#pragma unroll
                for (int k2 = 0; k2 < N2; ++k2) {
                    b[bitrev<Q::L2>(k2)] = make_double2(-a[u][k2].y, a[u][k2].x);
                    if (d == 1) {   // (tab is 0 on the Nyquist plane)
                        const int kz = k1 + N1 * k2;
                        const double c = small_double(kz < Q::H ? kz : kz - Q::n);
                        b[bitrev<Q::L2>(k2)].x *= c;
                        b[bitrev<Q::L2>(k2)].y *= c;
                    }
                }
                back_firstd<N1, N2>(b, Y, p, k1, tw, twsh);
            }
        }
        __syncthreads();
        for (int it = threadIdx.x; it < Q::P * N2; it += Q::T) {
            const int p = it & (Q::P - 1), n2 = it >> Q::LP;
            double2 b[N1];
            back_secondd<N1, N2>(b, Y, p, n2);
#pragma unroll
            for (int n1 = 0; n1 < N1; ++n1) (d ? field : w)[q0 + p + (N2 * n1 + n2) * plane] = b[n1];
        }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) energy += __shfl_down_sync(0xffffffffu, energy, o);
    if ((threadIdx.x & 31) == 0) sums[threadIdx.x >> 5] = energy;
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int v = 1; v < Q::T / 32; ++v) energy += sums[v];
        partial[blockIdx.x] = energy;
    }
}

// displacement of the inverse transform's output, over its rms: what turns a value
// of the fields into a fine cell's displacement per unit scale factor.  By
// Parseval the mean square of the fields is sum |Psi~|^2 (of unnormalised
// transforms) over n^2; the 1/n of the inverse cancels.
__global__ void __launch_bounds__(256) k_ic_scale_sum(int nblk, double a_init, double rms_disp,
                                                      const double* __restrict__ partial, double* scale) {
    __shared__ double sh[256];
    double s = 0.0;
    for (int b = threadIdx.x; b < nblk; b += 256) s += partial[b];
    sh[threadIdx.x] = s;
    __syncthreads();
    for (int o = 128; o > 0; o >>= 1) {
        if ((int)threadIdx.x < o) sh[threadIdx.x] += sh[threadIdx.x + o];
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        const double rms = sqrt(sh[0]);   // of the unnormalised fields, times sqrt(n)
        *scale = rms > 0.0 ? rms_disp / (a_init * rms) : 0.0;
    }
}

struct IcOut {
    int64_t M;                  // position codes per side, a power of two
    double codes;               // displacement in codes per unit of scale psi
    double pfac;                // momentum likewise
    double half;                // code of lattice point l: (2 l + 1) half
    int32_t* Q;                 // [3][N]
    float* P;                   // [3][N]
};

// code and momentum of lattice coordinate l displaced by psi (scaled): the lattice
// code is an integer unless there are more than nc 2^(7 or 15) points a side
__device__ __forceinline__ void ic_put(const IcOut& o, int64_t i, int l, double psi, double fc, double fp, int64_t h) {
    const double t = fc * psi;
    const int64_t q = h > 0 ? (2 * (int64_t)l + 1) * h + __double2ll_rd(t)
                            : __double2ll_rd((double)(2 * l + 1) * o.half + t);
    o.Q[i] = (int32_t)(q & (o.M - 1));
    o.P[i] = (float)(fp * psi);
}

// x: back, two real fields as one complex pencil.  blockIdx.y = 0: components x and
// y of a row; 1: component z of two rows
template <int N1, int N2>
__global__ void __launch_bounds__(PassD<N1, N2>::T) k_ic_x_back(const double2* __restrict__ field, IcOut o,
                                                                const double* __restrict__ scale_p,
                                                                const double2* __restrict__ tw, int twsh) {
    using Q = PassD<N1, N2>;
    constexpr int64_t half_mesh = (int64_t)Q::H * Q::n * Q::n, N = 2 * half_mesh;
    extern __shared__ __align__(16) unsigned char ic_smem[];
    double2* Y = reinterpret_cast<double2*>(ic_smem);
    const int64_t q0 = (int64_t)blockIdx.x * Q::P;
    const bool z = blockIdx.y == 1;
    if (z && 2 * q0 >= (int64_t)Q::n * Q::n) return;
    const double2* X0 = z ? field + 2 * half_mesh : field;
    for (int it = threadIdx.x; it < Q::P * N1; it += Q::T) {
        const int p = it >> Q::L1, k1 = it & (N1 - 1);
        const double2* X = X0 + (z ? 2 * (q0 + p) : q0 + p) * Q::H;
        const double2* V = z ? X + Q::H : X + half_mesh;
        double2 a[N2];
#pragma unroll
        for (int k2 = 0; k2 < N2; ++k2) {
            const int k = k1 + N1 * k2;
            double2 r = make_double2(0.0, 0.0);
            if (k != Q::H) {
                const int kk = k < Q::H ? k : Q::n - k;
                const double2 x = X[kk], v = V[kk];
                // the x component's factor kx
                const double c = z ? 1.0 : small_double(kk);
                if (k == 0) r = make_double2(c * x.x, v.x);
                else if (k < Q::H) r = make_double2(c * x.x - v.y, c * x.y + v.x);
                else r = make_double2(c * x.x + v.y, v.x - c * x.y);
            }
            a[bitrev<Q::L2>(k2)] = r;
        }
        back_firstd<N1, N2>(a, Y, p, k1, tw, twsh);
    }
    __syncthreads();
    const double scale = *scale_p, fc = o.codes * scale, fp = o.pfac * scale;
    const int64_t h = o.half >= 1.0 ? (int64_t)o.half : 0;
    for (int it = threadIdx.x; it < Q::P * N2; it += Q::T) {
        const int p = it >> Q::L2, n2 = it & (N2 - 1);
        double2 a[N1];
        back_secondd<N1, N2>(a, Y, p, n2);
        const int64_t row = z ? 2 * (q0 + p) : q0 + p;
        const int ly = (int)(row & (Q::n - 1)), lz = (int)(row >> Q::LN);
#pragma unroll
        for (int n1 = 0; n1 < N1; ++n1) {
            const int j = N2 * n1 + n2;
            const int64_t i = (row << Q::LN) + j;
            if (z) {
                ic_put(o, 2 * N + i, lz, a[n1].x, fc, fp, h);
                ic_put(o, 2 * N + i + Q::n, (int)((row + 1) >> Q::LN), a[n1].y, fc, fp, h);
            } else {
                ic_put(o, i, j, a[n1].x, fc, fp, h);
                ic_put(o, N + i, ly, a[n1].y, fc, fp, h);
            }
        }
    }
}

template <int N1, int N2>
void ic_passes(Sim& s, uint64_t seed, double rms, const double* tab, double2* w, double2* field, double* partial,
               double* scale, const IcOut& out) {
    using Q = PassD<N1, N2>;
    if (Q::kBytes > 48 * 1024) {
        const auto smem = cudaFuncAttributeMaxDynamicSharedMemorySize;
        cudaFuncSetAttribute(k_ic_x<N1, N2>, smem, (int)Q::kBytes);
        cudaFuncSetAttribute(k_ic_y<N1, N2, -1>, smem, (int)Q::kBytes);
        cudaFuncSetAttribute(k_ic_z<N1, N2>, smem, (int)Q::kBytes);
        cudaFuncSetAttribute(k_ic_y<N1, N2, 1>, smem, (int)Q::kBytes);
        cudaFuncSetAttribute(k_ic_x_back<N1, N2>, smem, (int)Q::kBytes);
    }
    cudaStream_t st = s.stream;
    int twsh = 0;
    while ((Q::n << twsh) < s.fft_max) ++twsh;
    const unsigned rows = (unsigned)(Q::n * Q::n / Q::P), half = (unsigned)((int64_t)Q::H * Q::n / Q::P);
    k_ic_x<N1, N2><<<half, Q::T, Q::kBytes, st>>>(seed, w, s.tw_d, twsh);
    k_ic_y<N1, N2, -1><<<half, Q::T, Q::kBytes, st>>>(nullptr, w, s.tw_d, twsh);
    k_ic_z<N1, N2><<<half, Q::T, Q::kBytes, st>>>(tab, w, field + 2 * (s.n / 2), partial, s.tw_d, twsh);
    k_ic_scale_sum<<<1, 256, 0, st>>>((int)half, s.cfg.a_init, rms, partial, scale);
    k_ic_y<N1, N2, 1><<<dim3(half, 3), Q::T, Q::kBytes, st>>>(w, field, s.tw_d, twsh);
    k_ic_x_back<N1, N2><<<dim3(rows, 2), Q::T, Q::kBytes, st>>>(field, out, scale, s.tw_d, twsh);
    s.launches += 6;
}

__global__ void k_ic_scale(int nblk, int64_t n, double a_init, double rms_disp, const double* partial,
                           double* scale) {
    double s = 0.0;
    for (int d = 0; d < 3; ++d)
        for (int b = 0; b < nblk; ++b) s += partial[d * nblk + b];
    const double rms = sqrt(s / (double)n);
    *scale = rms > 0.0 ? rms_disp / (a_init * rms) : 0.0;
}

// float32 variants for low-memory sims: the same noise, spectrum and
// normalisation, one float2 work array (noise regenerated per component) and
// a float32 displacement field
__global__ void k_ic_noise_f(int64_t n, unsigned long long seed, float2* w) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x) {
        const unsigned long long z1 = splitmix64(seed, 2ull * i);
        const unsigned long long z2 = splitmix64(seed, 2ull * i + 1ull);
        const double u1 = ((double)(z1 >> 11) + 1.0) * 0x1p-53;
        const double u2 = (double)(z2 >> 11) * 0x1p-53;
        w[i] = make_float2((float)(sqrt(-2.0 * log(u1)) * cos(2.0 * kPi * u2)), 0.f);
    }
}
__global__ void k_ic_amplitude_f(int np, int nf, double slope, double kc, float* __restrict__ amp) {
    const int64_t n = (int64_t)np * np * np;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x) {
        const int ix = (int)(i % np), iy = (int)((i / np) % np), iz = (int)(i / ((int64_t)np * np));
        const int h = np / 2;
        const int nx = ix < h ? ix : ix - np, ny = iy < h ? iy : iy - np, nz = iz < h ? iz : iz - np;
        double c = 0.0;
        if (!(nx == -h || ny == -h || nz == -h) && (nx | ny | nz)) {
            const double kf = 2.0 * kPi / nf;
            const double kx = kf * nx, ky = kf * ny, kz = kf * nz;
            const double k2 = kx * kx + ky * ky + kz * kz;
            const double k = sqrt(k2);
            c = sqrt(pow(k, slope) * exp(-(k / kc) * (k / kc))) / k2;
        }
        amp[i] = (float)c;
    }
}
// in place: w = i k_d amp w
__global__ void k_ic_component_f(int np, int nf, int d, const float* __restrict__ amp, float2* w) {
    const int64_t n = (int64_t)np * np * np;
    const double kf = 2.0 * kPi / nf;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x) {
        const int ix = (int)(i % np), iy = (int)((i / np) % np), iz = (int)(i / ((int64_t)np * np));
        const int h = np / 2;
        const int nd = d == 0 ? (ix < h ? ix : ix - np) : (d == 1 ? (iy < h ? iy : iy - np)
                                                                  : (iz < h ? iz : iz - np));
        const double c = kf * nd * (double)amp[i];
        const float2 a = w[i];
        w[i] = make_float2((float)(-c * a.y), (float)(c * a.x));   // i c a
    }
}
__global__ void k_ic_store_f(int64_t n, int d, const float2* __restrict__ in, float* __restrict__ psi,
                             double* __restrict__ partial) {
    double acc = 0.0;
    const double inv_n = 1.0 / (double)n;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x) {
        const float v = (float)((double)in[i].x * inv_n);
        psi[d * n + i] = v;
        acc += (double)v * v;
    }
    __shared__ double sh[256];
    sh[threadIdx.x] = acc;
    __syncthreads();
    for (int o = 128; o > 0; o >>= 1) {
        if ((int)threadIdx.x < o) sh[threadIdx.x] += sh[threadIdx.x + o];
        __syncthreads();
    }
    if (threadIdx.x == 0) partial[d * gridDim.x + blockIdx.x] += sh[0];
}

}  // namespace

static int ic_zeldovich_lowmem(Sim& s, uint64_t seed, double slope, double kc, double rms) {
    const int np = s.np;
    const int64_t n = s.n;
    cudaStream_t st = s.stream;
    float2* w = s.ic_work;
    double* partial = s.ic_partial;
    const int nblk = 1024;
    cudaMemsetAsync(partial, 0, sizeof(double) * (3 * nblk + 1), st);
    int rc;
    // the amplitude lives in psi's last component until that component is stored
    float* amp = s.ic_psi + 2 * n;
    k_ic_amplitude_f<<<grid_for(n, 256), 256, 0, st>>>(np, s.nf, slope, kc, amp);
    for (int d = 0; d < 3; ++d) {
        k_ic_noise_f<<<grid_for(n, 256), 256, 0, st>>>(n, (unsigned long long)seed, w);
        if ((rc = fft3d<float>(s, w, np, -1))) return rc;
        k_ic_component_f<<<grid_for(n, 256), 256, 0, st>>>(np, s.nf, d, amp, w);
        if ((rc = fft3d<float>(s, w, np, 1))) return rc;
        k_ic_store_f<<<nblk, 256, 0, st>>>(n, d, w, s.ic_psi, partial);
    }
    double* scale = partial + 3 * nblk;
    k_ic_scale<<<1, 1, 0, st>>>(nblk, n, s.cfg.a_init, rms, partial, scale);
    s.launches += 3 * 3 + 2;
    if ((rc = check_launch(s, "ic"))) return rc;
    s.a = s.cfg.a_init;
    s.step = 0;
    set_device_step(s, 0);
    return encode_from_psi(s, scale);
}

int ic_zeldovich(Sim& s, uint64_t seed, double slope, double kc, double rms) {
    if (s.lowmem) return ic_zeldovich_lowmem(s, seed, slope, kc, rms);
    const int np = s.np;
    const int64_t n = s.n;
    cudaStream_t st = s.stream;
    // scratch: codes and momenta (24 n; before them the amplitude table and the
    // partial sums), the three half-spectrum fields (24 n), the noise's (8 n)
    double2* field = reinterpret_cast<double2*>(align_up(reinterpret_cast<uintptr_t>(s.Pn + 3 * n)));
    double2* w = field + 3 * (n / 2);
    const int mmax = 3 * (np / 2) * (np / 2);
    double* tab = reinterpret_cast<double*>(s.scratch);
    double* partial = tab + mmax + 1;   // at most n / 8 of them
    double* scale = s.ic_partial;
    k_ic_amp_table<<<grid_for(mmax + 1, 256), 256, 0, st>>>(mmax, s.nf, slope, kc, tab);
    s.launches++;
    const int64_t M = (int64_t)s.nc * (s.pb == 2 ? PosFmt<2>::kBins : PosFmt<1>::kBins);
    const double cpf = s.pb == 2 ? PosFmt<2>::kCodesPerFine : PosFmt<1>::kCodesPerFine;
    const IcOut out = {M, s.cfg.a_init * cpf, s.ic_pfac, (double)M / (2.0 * np), s.Qn, s.Pn};
    switch (np) {
        case 4: ic_passes<2, 2>(s, seed, rms, tab, w, field, partial, scale, out); break;
        case 8: ic_passes<2, 4>(s, seed, rms, tab, w, field, partial, scale, out); break;
        case 16: ic_passes<4, 4>(s, seed, rms, tab, w, field, partial, scale, out); break;
        case 32: ic_passes<4, 8>(s, seed, rms, tab, w, field, partial, scale, out); break;
        case 64: ic_passes<8, 8>(s, seed, rms, tab, w, field, partial, scale, out); break;
        case 128: ic_passes<8, 16>(s, seed, rms, tab, w, field, partial, scale, out); break;
        case 256: ic_passes<16, 16>(s, seed, rms, tab, w, field, partial, scale, out); break;
        case 512: ic_passes<32, 16>(s, seed, rms, tab, w, field, partial, scale, out); break;
        case 1024: ic_passes<32, 32>(s, seed, rms, tab, w, field, partial, scale, out); break;
        default: return set_error(s, PMPM_EINVAL, "initial conditions of %d particles a side", np);
    }
    const int rc = check_launch(s, "ic");
    if (rc) return rc;
    s.a = s.cfg.a_init;
    s.step = 0;
    set_device_step(s, 0);
    return encode_from_qp(s, false);
}

}  // namespace pmpm
