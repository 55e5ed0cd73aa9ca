// coarse.cu -- long-range force on the coarse mesh (Sec. II: the long-range
// part lives on a mesh four times coarser than the fine one; Eq. 1 with
// K~_l).
//
//  1. integer CIC of all particles on the nc^3 coarse mesh (int64, units
//     2^-27 per particle): one thread per cell sums its particles' weights on
//     the 27 surrounding nodes in 32-bit registers, an 8x8x4-cell brick
//     collects them in shared memory (64-bit sums kept as two 32-bit words)
//     and flushes one global atomic per touched node;
//  2. delta = rho - mean (float64 subtraction, float32 storage), 3-D FFT;
//  3. Green multiply: B1 = rho~ (K~_x + i K~_y), B2 = rho~ K~_z (K~ = -i S);
//  4. two inverse FFTs give F_x + i F_y and F_z.
// Meshes up to 16^3 fit one SM's shared memory: 2-4 are one launch
// (k_coarse_tiny).  32^3 cells take four launches of a warp a plane or row, larger
// meshes five passes over memory, the ends and the Green multiply fused into them.
#include "pmpm_impl.cuh"
#include "fftpass.cuh"

namespace pmpm {

namespace {

// One thread per coarse cell: the cell's particles reach only the 3^3 nodes
// around it, so their weights are summed in 27 registers and added to the
// brick's shared accumulator once per cell.  Bricks of 8 x 8 x 4 cells; boxes up to
// 16^3 cells take 4^3, four times the blocks (64 and not 16: 128^3 particles 158 us against
// 200 on a GB300, 32^3 11.5 both).  At 32^3 cells they lose, the more the denser: 64^3
// particles 15.9 us against 12.2, 128^3 54 against 31, 256^3 497 against 232.
template <int PB, int kBX, int kBY, int kBZ>
__global__ void __launch_bounds__(kBX * kBY * kBZ) k_coarse_deposit(int nc, const int32_t* counts,
                                                        const int64_t* offsets,
                                                        const uint8_t* m0,
                                                        const uint8_t* m1,
                                                        const uint8_t* m2,
                                                        unsigned long long* rho) {
    chain_begin();
    constexpr int kNX = kBX + 2, kNY = kBY + 2, kNZ = kBZ + 2;
    // the brick's node sums as 32-bit halves: a native 32-bit shared atomic on
    // the low word, and the high word counts its wraps (at most one per add)
    __shared__ uint32_t acc_lo[kNX * kNY * kNZ], acc_hi[kNX * kNY * kNZ];
    const int nbx = nc / kBX, nby = nc / kBY;
    const int bx = blockIdx.x % nbx, by = (blockIdx.x / nbx) % nby, bz = blockIdx.x / (nbx * nby);
    const int x0 = bx * kBX, y0 = by * kBY, z0 = bz * kBZ;
    for (int i = threadIdx.x; i < kNX * kNY * kNZ; i += blockDim.x) {
        acc_lo[i] = 0u;
        acc_hi[i] = 0u;
    }
    __syncthreads();
    const int lx = threadIdx.x % kBX, ly = (threadIdx.x / kBX) % kBY, lz = threadIdx.x / (kBX * kBY);
    const int cx = x0 + lx, cy = y0 + ly, cz = z0 + lz;
    const int64_t cell = cx + (int64_t)nc * (cy + (int64_t)nc * cz);
    const int64_t j0 = offsets[cell];
    const int cnt = counts[cell];
    // A particle's weight on one node is at most its whole mass, 2^27 units,
    // so 31 particles sum below 2^32: 32-bit accumulators (one multiply-add
    // per node), added to the brick every kChunk particles.
    constexpr int kChunk = 31;
    for (int q0 = 0; q0 < cnt; q0 += kChunk) {
        uint32_t a[27];
#pragma unroll
        for (int k = 0; k < 27; ++k) a[k] = 0u;
        const int qe = min(cnt, q0 + kChunk);
#pragma unroll 2
        for (int q = q0; q < qe; ++q) {
            const int64_t j = j0 + q;
            // per axis: weights of nodes c-1, c, c+1 (in 1/(2B)); the bins in the
            // lower half lie left of the cell centre
            constexpr int B = PosFmt<PB>::kBins;
            uint32_t w[3][3];
            const int mm[3] = {load_bin<PB>(m0, j), load_bin<PB>(m1, j), load_bin<PB>(m2, j)};
#pragma unroll
            for (int e = 0; e < 3; ++e) {
                const int s = 2 * mm[e] + 1 - B;     // offset from the centre, 1/(2B)
                w[e][0] = s < 0 ? (uint32_t)(-s) : 0u;
                w[e][1] = (uint32_t)(2 * B) - (uint32_t)(s < 0 ? -s : s);
                w[e][2] = s > 0 ? (uint32_t)s : 0u;
            }
#pragma unroll
            for (int kz = 0; kz < 3; ++kz)
#pragma unroll
                for (int ky = 0; ky < 3; ++ky) {
                    if (PB == 1) {
                        // 1-byte bins: products below 2^27
                        const uint32_t wyz = w[1][ky] * w[2][kz];
#pragma unroll
                        for (int kx = 0; kx < 3; ++kx) a[kx + 3 * (ky + 3 * kz)] += wyz * w[0][kx];
                    } else {
                        // 2-byte bins: the 2^-51 product rounded to the 2^-27 unit
                        const unsigned long long wyz = (unsigned long long)w[1][ky] * w[2][kz];
#pragma unroll
                        for (int kx = 0; kx < 3; ++kx)
                            a[kx + 3 * (ky + 3 * kz)] +=
                                (uint32_t)round_half_even_shift(wyz * w[0][kx], PosFmt<PB>::kRoundBits);
                    }
                }
        }
#pragma unroll
        for (int k = 0; k < 27; ++k) {
            if (!a[k]) continue;
            const int dx = k % 3, dy = (k / 3) % 3, dz = k / 9;
            const int i = (lx + dx) + kNX * ((ly + dy) + kNY * (lz + dz));
            const uint32_t old = atomicAdd(&acc_lo[i], a[k]);
            if (old + a[k] < old) atomicAdd(&acc_hi[i], 1u);
        }
    }
    __syncthreads();
    for (int i = threadIdx.x; i < kNX * kNY * kNZ; i += blockDim.x) {
        const unsigned long long v = ((unsigned long long)acc_hi[i] << 32) | acc_lo[i];
        if (!v) continue;
        const int ix = i % kNX, iy = (i / kNX) % kNY, iz = i / (kNX * kNY);
        const int gx = wrap(x0 - 1 + ix, nc), gy = wrap(y0 - 1 + iy, nc), gz = wrap(z0 - 1 + iz, nc);
        atomicAdd(&rho[gx + (int64_t)nc * (gy + (int64_t)nc * gz)], v);
    }
}

// fl32(rho - mean).  The mean, N 2^27 / nc^3 with powers of two, is an integer of
// at least 8, so the difference is exact in 64 bits.
__device__ __forceinline__ float delta_of(long long rho, long long mean) { return f32_of(rho - mean); }

// ------------------------------------------------------------ up to 16^3 cells
// The whole chain on a complex mesh in one CTA's shared memory: blockIdx.x = 0
// transforms back to F_x + i F_y, 1 to F_z, and both do the forward transform
// (as separate launches the chain is launch-bound: twelve take 68 us at 16^3 on
// a GB300, this one 13).  A thread holds a pencil; the radix-2 autosort stages,
// their twiddles, roundings and the order of the axes are those of fft.cu's
// k_fft_pass, so the two give the same bits.
__device__ __forceinline__ float2 cmul(float2 a, float2 b) {
    return make_float2(__fmaf_rn(a.x, b.x, -__fmul_rn(a.y, b.y)), __fmaf_rn(a.y, b.x, __fmul_rn(a.x, b.y)));
}

template <int N, int S>
__device__ __forceinline__ void autosort(float2 (&a)[N], const float2 (&tw)[N / 2]) {
#pragma unroll
    for (int Ns = 1; Ns < N; Ns *= 2) {
        float2 d[N];
#pragma unroll
        for (int j = 0; j < N / 2; ++j) {
            const int k = j & (Ns - 1), o = ((j - k) << 1) + k;
            float2 w = tw[k * (N / 2 / Ns)];
            if (S > 0) w.y = -w.y;
            const float2 v0 = a[j], v1 = cmul(a[j + N / 2], w);
            d[o] = make_float2(v0.x + v1.x, v0.y + v1.y);
            d[o + Ns] = make_float2(v0.x - v1.x, v0.y - v1.y);
        }
#pragma unroll
        for (int j = 0; j < N; ++j) a[j] = d[j];
    }
}

template <int N, int S>
__device__ __forceinline__ void tiny_pencil(float2* c, int stride, const float2 (&tw)[N / 2]) {
    float2 a[N];
#pragma unroll
    for (int k = 0; k < N; ++k) a[k] = c[k * stride];
    autosort<N, S>(a, tw);
#pragma unroll
    for (int k = 0; k < N; ++k) c[k * stride] = a[k];
}

// a (S_y - i S_x), or a (-i S_z)
__device__ __forceinline__ float2 green_times(float2 a, float4 g, float sx, float sy, float sz, bool xy) {
    const float Sx = sx * g.x, Sy = sy * g.y, Sz = sz * g.z;
    return xy ? make_float2(__fmaf_rn(a.x, Sy, __fmul_rn(a.y, Sx)), __fmaf_rn(a.y, Sy, -__fmul_rn(a.x, Sx)))
              : make_float2(a.y * Sz, -a.x * Sz);
}

template <int N>
__global__ void __launch_bounds__(N * N) k_coarse_tiny(long long mean, const long long* rho,
                                                       const float4* __restrict__ table, float* Fl,
                                                       const float2* __restrict__ twiddles, int twsh) {
    chain_wait();
    constexpr int P = N + 1, h = N / 2 + 1, cells = N * N * N;
    __shared__ float2 C[N * N * P];
    const int tid = threadIdx.x, x = tid % N, y = tid / N;   // (y, z) for the x pencils, (x, z) and (x, y)
    float2 tw[N / 2];
#pragma unroll
    for (int k = 0; k < N / 2; ++k) tw[k] = twiddles[k << twsh];
#pragma unroll 4
    for (int z = 0; z < N; ++z) C[(z * N + y) * P + x] = make_float2(delta_of(rho[z * N * N + tid], mean), 0.f);
    __syncthreads();
    tiny_pencil<N, -1>(C + tid * P, 1, tw);
    __syncthreads();
    tiny_pencil<N, -1>(C + y * N * P + x, P, tw);
    __syncthreads();
    float2 a[N];
    float2* const col = C + y * P + x;   // the z pencil of (x, y)
#pragma unroll
    for (int z = 0; z < N; ++z) a[z] = col[z * (N * P)];
    autosort<N, -1>(a, tw);
    int ax, ay;
    float sx, sy;
    kfold(x, N, ax, sx);
    kfold(y, N, ay, sy);
#pragma unroll
    for (int z = 0; z < N; ++z) {
        int az;
        float sz;
        kfold(z, N, az, sz);
        col[z * (N * P)] = green_times(a[z], table[(az * h + ay) * h + ax], sx, sy, sz, blockIdx.x == 0);
    }
    __syncthreads();
    tiny_pencil<N, 1>(C + tid * P, 1, tw);
    __syncthreads();
    tiny_pencil<N, 1>(C + y * N * P + x, P, tw);
    __syncthreads();
    // only now: the tile pass takes whole SMs, and its CTAs would keep other streams out
    chain_next();
#pragma unroll
    for (int z = 0; z < N; ++z) a[z] = col[z * (N * P)];
    autosort<N, 1>(a, tw);
#pragma unroll
    for (int z = 0; z < N; ++z) {
        if (blockIdx.x == 0) {
            Fl[z * N * N + tid] = a[z].x;
            Fl[cells + z * N * N + tid] = a[z].y;
        } else {
            Fl[2 * cells + z * N * N + tid] = a[z].x;
        }
    }
}

// ------------------------------------------------------------ 32^3 cells
// The same stages, twiddles and roundings (keeps_bits) in four launches: x and y of a
// plane by one warp, through registers and a plane of shared memory, z with the Green
// multiply, a pencil a thread, and both back.  Latency bounds it: one warp on an SM walks
// two pencils' 32 points in a row.  20 us on a GB300; twelve passes of fft.cu 69, the
// five fused passes of larger meshes, whose order of axes gives other bits, 14.
constexpr int kC32 = 32, kC32Plane = kC32 * kC32, kC32Cells = kC32 * kC32Plane, kC32Pitch = kC32 + 1;

// the 32-point twiddles of a table of 32 << twsh
__device__ __forceinline__ void c32_twiddles(const float2* __restrict__ twiddles, int twsh, float2 (&tw)[kC32 / 2]) {
#pragma unroll
    for (int k = 0; k < kC32 / 2; ++k) tw[k] = twiddles[k << twsh];
}

// x and y of plane blockIdx.x: of the density (S = -1) to A, or of A or B (by
// blockIdx.y), in place, back
template <int S>
__global__ void __launch_bounds__(kC32) k_coarse32_plane(long long mean, const long long* rho, float2* A, float2* B,
                                                         const float2* __restrict__ twiddles, int twsh) {
    chain_begin();
    __shared__ float2 C[kC32 * kC32Pitch];
    const int lane = threadIdx.x;
    const int64_t at = (int64_t)blockIdx.x * kC32Plane + lane;
    float2* const data = blockIdx.y ? B : A;
    float2 tw[kC32 / 2];
    c32_twiddles(twiddles, twsh, tw);
#pragma unroll 8
    for (int y = 0; y < kC32; ++y)
        C[y * kC32Pitch + lane] = S < 0 ? make_float2(delta_of(rho[at + y * kC32], mean), 0.f) : data[at + y * kC32];
    __syncwarp();
    tiny_pencil<kC32, S>(C + lane * kC32Pitch, 1, tw);
    __syncwarp();
    float2 a[kC32];
#pragma unroll
    for (int y = 0; y < kC32; ++y) a[y] = C[y * kC32Pitch + lane];
    autosort<kC32, S>(a, tw);
#pragma unroll
    for (int y = 0; y < kC32; ++y) data[at + y * kC32] = a[y];
}

// z: pencils (kx, ky = blockIdx.x); forward from A, Green multiply, to B1 (blockIdx.y = 0) or B2
__global__ void __launch_bounds__(kC32) k_coarse32_green(const float4* __restrict__ table, const float2* A, float2* B1,
                                                         float2* B2, const float2* __restrict__ twiddles, int twsh) {
    chain_begin();
    constexpr int h = kC32 / 2 + 1;
    const int x = threadIdx.x, y = blockIdx.x, at = y * kC32 + x;
    float2 tw[kC32 / 2], a[kC32];
    c32_twiddles(twiddles, twsh, tw);
#pragma unroll
    for (int z = 0; z < kC32; ++z) a[z] = A[z * kC32Plane + at];
    autosort<kC32, -1>(a, tw);
    int ax, ay;
    float sx, sy;
    kfold(x, kC32, ax, sx);
    kfold(y, kC32, ay, sy);
    float2* const out = blockIdx.y ? B2 : B1;
#pragma unroll
    for (int z = 0; z < kC32; ++z) {
        int az;
        float sz;
        kfold(z, kC32, az, sz);
        out[z * kC32Plane + at] = green_times(a[z], table[(az * h + ay) * h + ax], sx, sy, sz, blockIdx.y == 0);
    }
}

// z back: F_x + i F_y from B1 (blockIdx.y = 0), F_z from B2
__global__ void __launch_bounds__(kC32) k_coarse32_back(const float2* B1, const float2* B2, float* Fl,
                                                        const float2* __restrict__ twiddles, int twsh) {
    chain_wait();
    const int at = blockIdx.x * kC32 + threadIdx.x;
    const float2* const B = blockIdx.y ? B2 : B1;
    float2 tw[kC32 / 2], a[kC32];
    c32_twiddles(twiddles, twsh, tw);
#pragma unroll
    for (int z = 0; z < kC32; ++z) a[z] = B[z * kC32Plane + at];
    chain_next();   // (as in k_coarse_tiny)
    autosort<kC32, 1>(a, tw);
#pragma unroll
    for (int z = 0; z < kC32; ++z) {
        if (blockIdx.y == 0) {
            Fl[z * kC32Plane + at] = a[z].x;
            Fl[kC32Cells + z * kC32Plane + at] = a[z].y;
        } else {
            Fl[2 * kC32Cells + z * kC32Plane + at] = a[z].x;
        }
    }
}

// ------------------------------------------------------------ sparse boxes, 64^3 cells and more
// Density to delta, Green multiply and F_l around fft.cu's transforms, for boxes that
// keep their bits (keeps_bits): twelve launches, every pass through memory, 73 us at 64^3
// cells where the fused passes below take 41.
__global__ void __launch_bounds__(256) k_coarse_delta(int64_t ncells, long long mean, const long long* rho, float2* out) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < ncells; i += (int64_t)gridDim.x * blockDim.x)
        out[i] = make_float2(delta_of(rho[i], mean), 0.f);
}

__global__ void __launch_bounds__(256) k_coarse_green(int nc, const float4* table, const float2* A, float2* B1, float2* B2) {
    const int64_t ncells = (int64_t)nc * nc * nc, h = nc / 2 + 1;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < ncells; i += (int64_t)gridDim.x * blockDim.x) {
        int ax, ay, az;
        float sx, sy, sz;
        kfold((int)(i % nc), nc, ax, sx);
        kfold((int)((i / nc) % nc), nc, ay, sy);
        kfold((int)(i / ((int64_t)nc * nc)), nc, az, sz);
        const float4 g = table[(az * h + ay) * h + ax];
        const float2 a = A[i];
        B1[i] = green_times(a, g, sx, sy, sz, true);
        B2[i] = green_times(a, g, sx, sy, sz, false);
    }
}

__global__ void __launch_bounds__(256) k_coarse_extract(int64_t ncells, const float2* B1, const float2* B2, float* Fl) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < ncells; i += (int64_t)gridDim.x * blockDim.x) {
        const float2 b1 = B1[i];
        Fl[i] = b1.x;
        Fl[ncells + i] = b1.y;
        Fl[2 * ncells + i] = B2[i].x;
    }
}

// ------------------------------------------------------------ 64^3 cells and more
// Passes of n = N1 N2 points per pencil in two register steps with one
// transpose through shared memory (fft.cu).  With j = N2 n1 + n2 and
// k = k1 + N1 k2 the forward pass ends with all k2 of one k1 in a thread's
// registers, which is where the inverse one begins: the z pass transforms,
// multiplies and transforms back without another exchange.  116 bytes a cell
// over five launches against 212 over twelve: 64^3 cells 76 -> 41 us, 128^3
// 126 -> 75, 256^3 (HBM-bound) 709 -> 412.
// x: integer density rows -> delta -> spectrum
template <int N1, int N2>
__global__ void __launch_bounds__(kPassWidth) k_coarse_fwd_x(long long mean, const long long* rho,
                                                                 float2* out,
                                                                 const float2* __restrict__ tw, int twsh) {
    chain_begin();
    using Q = Pass<N1, N2>;
    extern __shared__ __align__(16) unsigned char pass_smem[];
    float2* Y = reinterpret_cast<float2*>(pass_smem);
    const int64_t q0 = (int64_t)blockIdx.x * Q::P;
    for (int it = threadIdx.x; it < Q::P * N2; it += kPassWidth) {
        const int p = it >> Q::L2, n2 = it & (N2 - 1);
        const long long* src = rho + ((q0 + p) << Q::LN) + n2;
        float2 a[N1];
#pragma unroll
        for (int n1 = 0; n1 < N1; ++n1)
            a[bitrev<Q::L1>(n1)] = make_float2(delta_of(src[N2 * n1], mean), 0.f);
        pass_first<N1, N2>(a, Y, p, n2, tw, twsh);
    }
    __syncthreads();
    for (int it = threadIdx.x; it < Q::P * N1; it += kPassWidth) {
        const int p = it >> Q::L1, k1 = it & (N1 - 1);
        float2 a[N2];
        pass_second<N1, N2>(a, Y, p, k1);
        float2* dst = out + ((q0 + p) << Q::LN) + k1;
#pragma unroll
        for (int k2 = 0; k2 < N2; ++k2) dst[N1 * k2] = a[k2];
    }
}

// y: in place, forward (S = -1) or back; blockIdx.y picks the array
template <int N1, int N2, int S>
__global__ void __launch_bounds__(kPassWidth) k_coarse_y(float2* d0, float2* d1, const float2* __restrict__ tw,
                                                             int twsh) {
    chain_begin();
    using Q = Pass<N1, N2>;
    extern __shared__ __align__(16) unsigned char pass_smem[];
    float2* Y = reinterpret_cast<float2*>(pass_smem);
    const int64_t q0 = (int64_t)blockIdx.x * Q::P;   // pencils (x, z), x fastest
    float2* data = (blockIdx.y ? d1 : d0) + ((q0 >> Q::LN) << (2 * Q::LN)) + (q0 & (Q::n - 1));
    if (S < 0) {
        for (int it = threadIdx.x; it < Q::P * N2; it += kPassWidth) {
            const int p = it & (Q::P - 1), n2 = it >> Q::LP;
            float2 a[N1];
#pragma unroll
            for (int n1 = 0; n1 < N1; ++n1) a[bitrev<Q::L1>(n1)] = data[p + ((N2 * n1 + n2) << Q::LN)];
            pass_first<N1, N2>(a, Y, p, n2, tw, twsh);
        }
        __syncthreads();
        for (int it = threadIdx.x; it < Q::P * N1; it += kPassWidth) {
            const int p = it & (Q::P - 1), k1 = it >> Q::LP;
            float2 a[N2];
            pass_second<N1, N2>(a, Y, p, k1);
#pragma unroll
            for (int k2 = 0; k2 < N2; ++k2) data[p + ((k1 + N1 * k2) << Q::LN)] = a[k2];
        }
    } else {
        for (int it = threadIdx.x; it < Q::P * N1; it += kPassWidth) {
            const int p = it & (Q::P - 1), k1 = it >> Q::LP;
            float2 a[N2];
#pragma unroll
            for (int k2 = 0; k2 < N2; ++k2) a[bitrev<Q::L2>(k2)] = data[p + ((k1 + N1 * k2) << Q::LN)];
            back_first<N1, N2>(a, Y, p, k1, tw, twsh);
        }
        __syncthreads();
        for (int it = threadIdx.x; it < Q::P * N2; it += kPassWidth) {
            const int p = it & (Q::P - 1), n2 = it >> Q::LP;
            float2 a[N1];
            back_second<N1, N2>(a, Y, p, n2);
#pragma unroll
            for (int n1 = 0; n1 < N1; ++n1) data[p + ((N2 * n1 + n2) << Q::LN)] = a[n1];
        }
    }
}

// z: forward, Green multiply and back for B1 and B2
template <int N1, int N2>
__global__ void __launch_bounds__(kPassWidth) k_coarse_z(const float4* __restrict__ table,
                                                             const float2* A, float2* B1,
                                                             float2* B2, const float2* __restrict__ tw,
                                                             int twsh) {
    chain_begin();
    using Q = Pass<N1, N2>;
    constexpr int64_t plane = (int64_t)Q::n * Q::n;
    constexpr int h = Q::n / 2 + 1;
    extern __shared__ __align__(16) unsigned char pass_smem[];
    float2* Y = reinterpret_cast<float2*>(pass_smem);
    float2* Z = Y + Q::P * Q::PS;
    const int64_t q0 = (int64_t)blockIdx.x * Q::P;   // pencils (kx, ky), kx fastest
    for (int it = threadIdx.x; it < Q::P * N2; it += kPassWidth) {
        const int p = it & (Q::P - 1), n2 = it >> Q::LP;
        float2 a[N1];
#pragma unroll
        for (int n1 = 0; n1 < N1; ++n1) a[bitrev<Q::L1>(n1)] = A[q0 + p + (N2 * n1 + n2) * plane];
        pass_first<N1, N2>(a, Y, p, n2, tw, twsh);
    }
    __syncthreads();
    const int ky = (int)(q0 >> Q::LN);   // a block's pencils share ky (P divides n)
    int ay;
    float sy;
    kfold(ky, Q::n, ay, sy);
#pragma unroll 1
    for (int b = 0; b < 2; ++b) {
        for (int it = threadIdx.x; it < Q::P * N1; it += kPassWidth) {
            const int p = it & (Q::P - 1), k1 = it >> Q::LP;
            int ax;
            float sx;
            kfold((int)(q0 & (Q::n - 1)) + p, Q::n, ax, sx);
            float2 a[N2];
            pass_second<N1, N2>(a, Y, p, k1);
            float2 w[N2];
#pragma unroll
            for (int k2 = 0; k2 < N2; ++k2) {
                int az;
                float sz;
                kfold(k1 + N1 * k2, Q::n, az, sz);
                const float4 g = table[((int64_t)az * h + ay) * h + ax];
                const float2 v = a[k2];
                float2 r;
                if (b == 0) {   // B1 = v (S_y - i S_x)
                    const float Sx = sx * g.x, Sy = sy * g.y;
                    r = make_float2(v.x * Sy + v.y * Sx, v.y * Sy - v.x * Sx);
                } else {        // B2 = -i S_z v
                    const float Sz = sz * g.z;
                    r = make_float2(v.y * Sz, -v.x * Sz);
                }
                w[bitrev<Q::L2>(k2)] = r;
            }
            back_first<N1, N2>(w, Z, p, k1, tw, twsh);
        }
        __syncthreads();
        float2* B = b == 0 ? B1 : B2;
        for (int it = threadIdx.x; it < Q::P * N2; it += kPassWidth) {
            const int p = it & (Q::P - 1), n2 = it >> Q::LP;
            float2 a[N1];
            back_second<N1, N2>(a, Z, p, n2);
#pragma unroll
            for (int n1 = 0; n1 < N1; ++n1) B[q0 + p + (N2 * n1 + n2) * plane] = a[n1];
        }
        if (b == 0) __syncthreads();
    }
}

// x: back to F_x + i F_y (blockIdx.y = 0) and F_z
template <int N1, int N2>
__global__ void __launch_bounds__(kPassWidth) k_coarse_inv_x(const float2* B1,
                                                                 const float2* B2,
                                                                 float* Fl,
                                                                 const float2* __restrict__ tw, int twsh) {
    chain_wait();
    using Q = Pass<N1, N2>;
    constexpr int64_t cells = (int64_t)Q::n * Q::n * Q::n;
    extern __shared__ __align__(16) unsigned char pass_smem[];
    float2* Y = reinterpret_cast<float2*>(pass_smem);
    const int64_t q0 = (int64_t)blockIdx.x * Q::P;
    const float2* B = blockIdx.y ? B2 : B1;
    for (int it = threadIdx.x; it < Q::P * N1; it += kPassWidth) {
        const int p = it >> Q::L1, k1 = it & (N1 - 1);
        const float2* src = B + ((q0 + p) << Q::LN) + k1;
        float2 a[N2];
#pragma unroll
        for (int k2 = 0; k2 < N2; ++k2) a[bitrev<Q::L2>(k2)] = src[N1 * k2];
        back_first<N1, N2>(a, Y, p, k1, tw, twsh);
    }
    __syncthreads();
    chain_next();
    for (int it = threadIdx.x; it < Q::P * N2; it += kPassWidth) {
        const int p = it >> Q::L2, n2 = it & (N2 - 1);
        float2 a[N1];
        back_second<N1, N2>(a, Y, p, n2);
        float* dst = Fl + ((q0 + p) << Q::LN) + n2;
        if (blockIdx.y) {
#pragma unroll
            for (int n1 = 0; n1 < N1; ++n1) dst[2 * cells + N2 * n1] = a[n1].x;
        } else {
#pragma unroll
            for (int n1 = 0; n1 < N1; ++n1) {
                dst[N2 * n1] = a[n1].x;
                dst[cells + N2 * n1] = a[n1].y;
            }
        }
    }
}

template <int N1, int N2>
void pass_setup() {
    using Q = Pass<N1, N2>;
    const int one = (int)Q::kBytes, two = 2 * one;
    cudaFuncSetAttribute(k_coarse_fwd_x<N1, N2>, cudaFuncAttributeMaxDynamicSharedMemorySize, one);
    cudaFuncSetAttribute(k_coarse_y<N1, N2, -1>, cudaFuncAttributeMaxDynamicSharedMemorySize, one);
    cudaFuncSetAttribute(k_coarse_y<N1, N2, 1>, cudaFuncAttributeMaxDynamicSharedMemorySize, one);
    cudaFuncSetAttribute(k_coarse_z<N1, N2>, cudaFuncAttributeMaxDynamicSharedMemorySize, two);
    cudaFuncSetAttribute(k_coarse_inv_x<N1, N2>, cudaFuncAttributeMaxDynamicSharedMemorySize, one);
}

template <int N>
void launch_tiny(Sim& s, long long mean) {
    int twsh = 0;
    while ((N << twsh) < s.fft_max) ++twsh;
    chain(s.chained, k_coarse_tiny<N>, 2, N * N, 0, s.stream, mean, s.rho_c, s.green_coarse, s.Fl, s.tw_f, twsh);
    s.launches++;
}
void launch_32(Sim& s, long long mean) {
    int twsh = 0;
    while ((kC32 << twsh) < s.fft_max) ++twsh;
    const dim3 both(kC32, 2);
    chain(s.chained, k_coarse32_plane<-1>, kC32, kC32, 0, s.stream, mean, s.rho_c, s.cA, s.cA, s.tw_f, twsh);
    chain(s.chained, k_coarse32_green, both, kC32, 0, s.stream, s.green_coarse, s.cA, s.cB1, s.cB2, s.tw_f, twsh);
    chain(s.chained, k_coarse32_plane<1>, both, kC32, 0, s.stream, 0, nullptr, s.cB1, s.cB2, s.tw_f, twsh);
    chain(s.chained, k_coarse32_back, both, kC32, 0, s.stream, s.cB1, s.cB2, s.Fl, s.tw_f, twsh);
    s.launches += 4;
}
int launch_kept(Sim& s, long long mean) {
    const int grid = grid_for(s.ncells, 256);
    k_coarse_delta<<<grid, 256, 0, s.stream>>>(s.ncells, mean, s.rho_c, s.cA);
    int rc = fft3d<float>(s, s.cA, s.nc, -1);
    if (rc) return rc;
    k_coarse_green<<<grid, 256, 0, s.stream>>>(s.nc, s.green_coarse, s.cA, s.cB1, s.cB2);
    if ((rc = fft3d<float>(s, s.cB1, s.nc, 1))) return rc;
    if ((rc = fft3d<float>(s, s.cB2, s.nc, 1))) return rc;
    k_coarse_extract<<<grid, 256, 0, s.stream>>>(s.ncells, s.cB1, s.cB2, s.Fl);
    s.launches += 3;
    return check_launch(s, "coarse force");
}
template <int N1, int N2>
void launch_passes(Sim& s, long long mean) {
    using Q = Pass<N1, N2>;
    const unsigned groups = (unsigned)((int64_t)Q::n * Q::n / Q::P);
    int twsh = 0;
    while ((Q::n << twsh) < s.fft_max) ++twsh;   // W_n^e = tw[e << twsh]
    const size_t sm = Q::kBytes;
    chain(s.chained, k_coarse_fwd_x<N1, N2>, groups, kPassWidth, sm, s.stream, mean, s.rho_c, s.cA, s.tw_f, twsh);
    chain(s.chained, k_coarse_y<N1, N2, -1>, groups, kPassWidth, sm, s.stream, s.cA, s.cA, s.tw_f, twsh);
    chain(s.chained, k_coarse_z<N1, N2>, groups, kPassWidth, 2 * sm, s.stream, s.green_coarse, s.cA, s.cB1, s.cB2, s.tw_f, twsh);
    chain(s.chained, k_coarse_y<N1, N2, 1>, dim3(groups, 2), kPassWidth, sm, s.stream, s.cB1, s.cB2, s.tw_f, twsh);
    chain(s.chained, k_coarse_inv_x<N1, N2>, dim3(groups, 2), kPassWidth, sm, s.stream, s.cB1, s.cB2, s.Fl, s.tw_f, twsh);
    s.launches += 5;
}

}  // namespace

int coarse_deposit(Sim& s, bool cleared) {
    if (!cleared) cudaMemsetAsync(s.rho_c, 0, sizeof(long long) * s.ncells, s.stream);
    const bool small = s.nc <= 16;
    const unsigned nb = (unsigned)(s.ncells / (small ? 64 : 256)), threads = small ? 64 : 256;
    auto k = s.pb == 2 ? (small ? k_coarse_deposit<2, 4, 4, 4> : k_coarse_deposit<2, 8, 8, 4>)
                       : (small ? k_coarse_deposit<1, 4, 4, 4> : k_coarse_deposit<1, 8, 8, 4>);
    chain(s.chained, k, nb, threads, 0, s.stream, s.nc, s.counts[s.cur], s.offsets[s.cur],
          m_stream(s, s.cur, 0), m_stream(s, s.cur, 1), m_stream(s, s.cur, 2),
          reinterpret_cast<unsigned long long*>(s.rho_c));
    s.launches++;
    return check_launch(s, "coarse deposit");
}

void coarse_setup() {
    pass_setup<8, 8>();
    pass_setup<8, 16>();
    pass_setup<16, 16>();
    pass_setup<16, 32>();
    pass_setup<32, 32>();
}

int coarse_force(Sim& s) {
    // N 2^27 / nc^3, all powers of two (N up to 2^36)
    const long long mean = s.n >= s.ncells ? (s.n / s.ncells) << 27 : (1ll << 27) / (s.ncells / s.n);
    if (s.nc > 32 && keeps_bits(s)) return launch_kept(s, mean);
    switch (s.nc) {
        case 8: launch_tiny<8>(s, mean); break;
        case 16: launch_tiny<16>(s, mean); break;
        case 32: launch_32(s, mean); break;
        case 64: launch_passes<8, 8>(s, mean); break;
        case 128: launch_passes<8, 16>(s, mean); break;
        case 256: launch_passes<16, 16>(s, mean); break;
        case 512: launch_passes<16, 32>(s, mean); break;
        case 1024: launch_passes<32, 32>(s, mean); break;
        default: return set_error(s, PMPM_EINVAL, "coarse mesh of %d cells a side", s.nc);
    }
    return check_launch(s, "coarse force");
}

}  // namespace pmpm
