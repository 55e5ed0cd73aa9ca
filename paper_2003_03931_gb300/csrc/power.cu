// power.cu -- power spectrum of the particle density (Sec. IV-D): CIC density
// on an nmesh^3 mesh (integer weights, exact), delta = rho/rho_bar - 1, DFT,
// P(k) = L^3 / nmesh^6 |delta~|^2 averaged in shells j = round(|n|).
//
//   deposit  one block per brick of cells sums its own nodes' weights in shared
//            memory from the brick's particles and those of the cells around it,
//            and writes delta: no search for a particle's cell, no atomics on the
//            mesh, no mesh to clear or to convert
//   x, y, z  register transforms (fftpass.cuh); the z pass adds |delta~|^2 to its
//            block's shells and writes nothing.  Up to 16^3 points one CTA does
//            all of it (k_pk_small).
//   shells   mean |k| and the number of modes follow from the mesh alone: modes counted
//            by |n|^2, one block a shell
// FP64 runs at 1/64 of the FP32 rate here, so squares and shell sums are integers
// (pk_sums.cuh) and only a block's totals become doubles.
//
// On a GB300: 256^3 particles on 512^3 points 10.5 -> 1.93 ms (a search per
// particle, 64-bit global atomics and three double shared atomics a mode before):
// deposit 0.51 (issue: the particles of 2.8 bricks are looked at), x 0.27, y 0.43, z with the
// shells 0.68 (exact squares 0.14 of it), of 0.8 ms for 40 bytes a point at the copy
// bandwidth; 32^3 on 32^3, without allocation, 118 -> 70 us.
#include "power.cuh"

#include <new>

#include "fftpass.cuh"
#include "pk_sums.cuh"

namespace pmpm {

namespace {

constexpr double kPi = 3.141592653589793238462643383279502884;

// Brick of cells by node spacing h = 2^LH fine cells (4 >> LH nodes a cell).
// SMALL (boxes up to 32^3 cells): 4^3 cells, so that 16^3 cells are 64 blocks of 16
// warps and not 8 of 8 (41 us a deposit of 32^3 particles then, 10 now).
template <int LH, bool SMALL>
struct Brick {
    static constexpr int R = 4 >> LH, CX = SMALL ? 4 : 8, CY = SMALL || LH == 0 ? 4 : 8, CZ = CY;
    static constexpr int NX = CX * R, NY = CY * R, NZ = CZ * R, kNodes = NX * NY * NZ;
    static constexpr int kThreads = SMALL ? 512 : 256;
    static constexpr size_t kBytes = 8 * (size_t)kNodes;
    // 8 cells of this many particles reach no node with 2^32 units
    static constexpr int kSafe = LH == 0 ? 255 : (LH == 1 ? 31 : 3);
};

// delta of a node whose weights sum to v.  For a power of two of particles (a sim's)
// all sizes are powers of two and it is (v - mean) scale for a mean of at least one
// unit, else v << shift - 1, exact up to one rounding; other particle counts
// (inv > 0) take v inv - 1 in float64.
struct PkMean {
    long long mean;
    int shift;
    float scale;
    double inv;
    __device__ __forceinline__ float delta(unsigned long long v) const {
        if (inv > 0.0) return (float)((double)v * inv - 1.0);
        return f32_of(((long long)v << shift) - mean) * scale;
    }
    // the same for v < 2^31 where narrow()
    __device__ __forceinline__ bool narrow() const { return inv <= 0.0 && shift == 0 && mean < (1ll << 31); }
    __device__ __forceinline__ float delta(uint32_t v) const { return __int2float_rn((int)(v - (uint32_t)mean)) * scale; }
};

// four nodes from i, a multiple of 4
__device__ __forceinline__ void put(float* out, int64_t i, float4 v) { *reinterpret_cast<float4*>(out + i) = v; }
__device__ __forceinline__ void put(float2* out, int64_t i, float4 v) {
    *reinterpret_cast<float4*>(out + i) = make_float4(v.x, 0.f, v.y, 0.f);
    *reinterpret_cast<float4*>(out + i + 2) = make_float4(v.z, 0.f, v.w, 0.f);
}

// the cells x0 - 1 .. of row (by, bz) around the brick, one per lane; never past
// the store, whatever the counts
__device__ __forceinline__ int pk_row(const PkStore& st, int64_t base, int x, bool live, int64_t& off) {
    off = 0;
    if (!live) return 0;
    const int64_t cell = base + wrap1(x, st.nc);
    off = st.offsets[cell];
    const int64_t c = st.counts[cell];
    return off < 0 || off >= st.n || c < 0 ? 0 : (int)(c < st.n - off ? c : st.n - off);
}

// Node sums are 64-bit, as 32-bit halves: where a cell holds enough particles the
// low word's wraps are counted in the high word.  A warp takes a row of cells (x
// fastest, CX + 2 of them), its particles 32 at a time; the cell of each comes from
// the row's prefix counts, one per lane.  2-byte products are rounded to the
// 1-byte unit (2U_1)^-3.  Cells of more than kPkCrowd particles are the whole block's, one
// after another, four particles a thread at a time: a warp would walk a row for as long as
// its fullest cell is (128^3 particles, 20000 of them in one cell: CROWD).
constexpr int kPkCrowd = 1024;
template <int PB>
struct PackedBins {
    using type = uint32_t;
};
template <>
struct PackedBins<2> {
    using type = unsigned long long;
};
template <int PB, int LH, bool SMALL, typename OUT>
__global__ void __launch_bounds__(Brick<LH, SMALL>::kThreads) k_pk_deposit(const PkStore st, PkMean mean,
                                                                           OUT* out) {
    chain_begin();
    using B = Brick<LH, SMALL>;
    using F = PosFmt<PB>;
    constexpr int U = F::kCodesPerFine << LH, W = 2 * U, T = B::kThreads;
    constexpr int LW = F::kFineWBits + LH, kRows = (B::CY + 2) * (B::CZ + 2);
    extern __shared__ __align__(16) uint32_t pk_smem[];
    uint32_t* const lo = pk_smem;
    uint32_t* const hi = pk_smem + B::kNodes;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nc = st.nc;
    const int nbx = nc / B::CX, nby = nc / B::CY;
    const int x0 = (int)(blockIdx.x % nbx) * B::CX, y0 = (int)(blockIdx.x / nbx % nby) * B::CY,
              z0 = (int)(blockIdx.x / (nbx * nby)) * B::CZ;
    auto row_base = [&](int row) {
        const int by = row % (B::CY + 2), bz = row / (B::CY + 2);
        return (int64_t)nc * (wrap1(y0 - 1 + by, nc) + (int64_t)nc * wrap1(z0 - 1 + bz, nc));
    };
    for (int i = tid; i < B::kNodes / 2; i += T) reinterpret_cast<uint4*>(pk_smem)[i] = make_uint4(0u, 0u, 0u, 0u);
    int most = 0;
    for (int row = warp; row < kRows; row += T / 32) {
        int64_t off;
        most = max(most, pk_row(st, row_base(row), x0 - 1 + lane, lane < B::CX + 2, off));
    }
    const bool safe = !__syncthreads_or(most > B::kSafe);
    // particle of cell (bx, by, bz) with bins m to its nodes
    auto cloud = [&](int bx, int by, int bz, const int (&m)[3]) {
        const int sx = (bx - 1) * 2 * F::kBins + 2 * m[0] + 1 - U;
        const int sy = (by - 1) * 2 * F::kBins + 2 * m[1] + 1 - U;
        const int sz = (bz - 1) * 2 * F::kBins + 2 * m[2] + 1 - U;
        const int ix = sx >> LW, iy = sy >> LW, iz = sz >> LW;
        if ((unsigned)(ix + 1) > (unsigned)B::NX || (unsigned)(iy + 1) > (unsigned)B::NY ||
            (unsigned)(iz + 1) > (unsigned)B::NZ)
            return;
        const int wx = sx & (W - 1), wy = sy & (W - 1), wz = sz & (W - 1);
#pragma unroll
        for (int c = 0; c < 8; ++c) {
            const int dx = c & 1, dy = (c >> 1) & 1, dz = c >> 2;
            const int x = ix + dx, y = iy + dy, z = iz + dz;
            const uint32_t w = cic_weight3<PB>(dx ? wx : W - wx, dy ? wy : W - wy, dz ? wz : W - wz);
            if ((unsigned)x < (unsigned)B::NX && (unsigned)y < (unsigned)B::NY && (unsigned)z < (unsigned)B::NZ) {
                const int i = x + B::NX * (y + B::NY * z);
                if (safe) {
                    smem_red(&lo[i], w);
                } else {
                    const uint32_t old = atomicAdd(&lo[i], w);
                    if (old + w < old) atomicAdd(&hi[i], 1u);
                }
            }
        }
    };
    for (int row = warp; row < kRows; row += T / 32) {
        const int by = row % (B::CY + 2), bz = row / (B::CY + 2);
        int64_t off;
        int cnt = pk_row(st, row_base(row), x0 - 1 + lane, lane < B::CX + 2, off);
        if (cnt > kPkCrowd) cnt = 0;
        int incl = cnt;
#pragma unroll
        for (int o = 1; o < 16; o <<= 1) {
            const int v = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += v;
        }
        const int pre = incl - cnt;
        const int64_t rel = off - pre;   // particle v of the row lies at rel[its cell] + v
        const int total = __shfl_sync(0xffffffffu, incl, B::CX + 1);
        for (int v0 = 0; v0 < total; v0 += 32) {
            const int v = v0 + lane;
            int bx = 0;
#pragma unroll
            for (int k = 1; k < B::CX + 2; ++k) bx += v >= __shfl_sync(0xffffffffu, pre, k) ? 1 : 0;
            const int64_t j = __shfl_sync(0xffffffffu, rel, bx) + v;
            if (v >= total) continue;
            const int m[3] = {load_bin<PB>(st.m[0], j), load_bin<PB>(st.m[1], j), load_bin<PB>(st.m[2], j)};
            cloud(bx, by, bz, m);
        }
    }
    if (__syncthreads_or(most > kPkCrowd)) {
        for (int row = 0; row < kRows; ++row) {
            int64_t off;
            const int cnt = pk_row(st, row_base(row), x0 - 1 + lane, lane < B::CX + 2, off);
            for (unsigned crowded = __ballot_sync(0xffffffffu, cnt > kPkCrowd); crowded; crowded &= crowded - 1u) {
                const int bx = __ffs(crowded) - 1;
                const unsigned n = __shfl_sync(0xffffffffu, cnt, bx);
                const int64_t at = __shfl_sync(0xffffffffu, off, bx);
                using Bins = typename PackedBins<PB>::type;
                constexpr int kAhead = PB == 1 ? 4 : 2;
#pragma unroll 1
                for (unsigned v0 = tid; v0 < n; v0 += kAhead * T) {
                    Bins p[kAhead];
#pragma unroll
                    for (int u = 0; u < kAhead; ++u) {
                        const int64_t j = at + min(v0 + u * T, n - 1);
                        p[u] = 0;
#pragma unroll
                        for (int e = 0; e < 3; ++e) p[u] |= (Bins)load_bin<PB>(st.m[e], j) << (8 * PB * e);
                    }
#pragma unroll 1
                    for (int u = 0; u < kAhead && v0 + u * T < n; ++u) {
                        const int m[3] = {(int)(p[0] & (F::kBins - 1)), (int)(p[0] >> 8 * PB & (F::kBins - 1)),
                                          (int)(p[0] >> 16 * PB)};
                        cloud(bx, row % (B::CY + 2), row / (B::CY + 2), m);
#pragma unroll
                        for (int k = 1; k < kAhead; ++k) p[k - 1] = p[k];
                    }
                }
            }
        }
    }
    __syncthreads();
    // four nodes a thread (NX and the mesh's side are multiples of 4); by 32-bit integers
    // where they hold the sums: half of the kernel's instructions were 64-bit ones here
    const int64_t nm = (int64_t)nc * B::R;
    const bool narrow = safe && mean.narrow();
    for (int q = tid; q < B::kNodes / 4; q += T) {
        const int x = 4 * q % B::NX, y = 4 * q / B::NX % B::NY, z = 4 * q / (B::NX * B::NY);
        const uint4 l = reinterpret_cast<const uint4*>(lo)[q];
        float4 d;
        if (narrow && (int)(l.x | l.y | l.z | l.w) >= 0) {
            d = make_float4(mean.delta(l.x), mean.delta(l.y), mean.delta(l.z), mean.delta(l.w));
        } else {
            const uint4 h = reinterpret_cast<const uint4*>(hi)[q];
            d = make_float4(mean.delta((unsigned long long)h.x << 32 | l.x), mean.delta((unsigned long long)h.y << 32 | l.y),
                            mean.delta((unsigned long long)h.z << 32 | l.z), mean.delta((unsigned long long)h.w << 32 | l.w));
        }
        put(out, (x0 * B::R + x) + nm * ((y0 * B::R + y) + nm * (int64_t)(z0 * B::R + z)), d);
    }
}

// ------------------------------------------------------------ shells
// A square root within two float32 steps, and what is made exact from it.
__device__ __forceinline__ float root(float v) {
    float r;
    asm("sqrt.approx.f32 %0, %1;" : "=f"(r) : "f"(v));
    return r;
}
// shell of a mode with |n|^2 = m: round(sqrt(m)), exact
__device__ __forceinline__ int shell_of(int m) {
    int j = (int)(root((float)m) + 0.5f);
    if (m > j * j + j) ++j;
    else if (m < j * j - j + 1) --j;
    return j;
}
__device__ __forceinline__ int isqrt(int v) {   // floor, v >= 0
    int r = (int)root((float)v);
    if (r * r > v) --r;
    else if ((r + 1) * (r + 1) <= v) ++r;
    return r;
}

// Modes of shell j of an nmesh^3 mesh by |n|^2: adds to hist[m - (j^2 - j + 1)], m up to
// j^2 + j, by the lanes of warp w of W.  Octant points (a, b, c), a <= b, with their
// multiplicities.  A root per m is left, 2 j of them, and not one per mode: in float64.
__device__ __forceinline__ void count_shell(int nmesh, int j, int w, int W, int lane, uint32_t* hist) {
    const int h = nmesh / 2, mlo = j * j - j + 1, mhi = j * j + j, side = min(h, j);
    for (int b = w; b <= side; b += W) {
        for (int a = lane; a <= b; a += 32) {
            const int m0 = a * a + b * b;
            if (m0 > mhi) break;
            const int mult = (a == 0 || a == h ? 1 : 2) * (b == 0 || b == h ? 1 : 2) * (a == b ? 1 : 2);
            const int c1 = min(h, isqrt(mhi - m0));
            int c0 = 0;
            if (m0 < mlo) {
                c0 = isqrt(mlo - m0);
                if (c0 * c0 < mlo - m0) ++c0;
            }
            for (int c = c0; c <= c1; ++c) smem_red(&hist[m0 + c * c - mlo], mult * (c == 0 || c == h ? 1 : 2));
        }
    }
}
template <typename V>
__device__ __forceinline__ V warp_sum(V v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// k and mode sums of shell j, by one block; hist: 2 j words of shared memory
__device__ __forceinline__ void block_shell(int nmesh, int nbins, int j, double kf, double* bins, uint32_t* hist) {
    __shared__ double shk[kPassWidth / 32];
    __shared__ int shm[kPassWidth / 32];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, mlo = j * j - j + 1;
    for (int i = tid; i < 2 * j; i += kPassWidth) hist[i] = 0u;
    __syncthreads();
    count_shell(nmesh, j, warp, kPassWidth / 32, lane, hist);
    __syncthreads();
    double k = 0.0;
    int modes = 0;
    for (int i = tid; i < 2 * j; i += kPassWidth) {
        k += (double)hist[i] * __dsqrt_rn((double)(mlo + i));
        modes += (int)hist[i];
    }
    k = warp_sum(k);
    modes = warp_sum(modes);
    if (lane == 0) {
        shk[warp] = k;
        shm[warp] = modes;
    }
    __syncthreads();
    if (tid == 0) {
        for (int w = 1; w < kPassWidth / 32; ++w) {
            k += shk[w];
            modes += shm[w];
        }
        bins[nbins + j - 1] = kf * k;
        bins[2 * nbins + j - 1] = (double)modes;
    }
    __syncthreads();
}

// for meshes whose shells are not the z pass's; nmesh words of shared memory
__global__ void __launch_bounds__(kPassWidth) k_pk_shells(int nmesh, int nbins, double kf, double* __restrict__ bins,
                                                          const uint32_t* __restrict__ err) {
    extern __shared__ uint32_t shell_smem[];
    if (blockIdx.x == 0 && threadIdx.x == 0) bins[3 * nbins] = (double)*err;
    block_shell(nmesh, nbins, blockIdx.x + 1, kf, bins, shell_smem);
}

// Adds an integer of up to 62 bits to a shell (pk_sums.cuh).
__device__ __forceinline__ void add_limbs(uint32_t* limb, int stride, unsigned long long x) {
    const Limbs l = limbs_of(x);
    if (l.v[0]) smem_red(limb, l.v[0]);
    if (l.v[1]) smem_red(limb + stride, l.v[1]);
    if (l.v[2]) smem_red(limb + 2 * stride, l.v[2]);
}

// ------------------------------------------------------------ transforms
// Complex passes over the real deltas, every mode beside its mirror image: their roundings
// are different ones, and a shell's mean takes both.  Two real planes as one complex
// plane through x and y, or half the spectrum, cost half the points (256^3 particles on 512^3
// points 1.36 ms and not 1.93) but give one of the two, and P(k) was up to sqrt(2) further off 64 bits
// (512^3 points on fresh initial conditions 9.4e-7 against 6.6e-7, median).
// x, from real deltas or in place; clears the sums that the z pass adds to
template <int N1, int N2, bool REAL>
__global__ void __launch_bounds__(kPassWidth) k_pk_x(const float* delta, float2* mesh, int nbins, double* bins,
                                                     const uint32_t* err, const float2* __restrict__ tw, int twsh) {
    chain_begin();
    using Q = Pass<N1, N2>;
    extern __shared__ __align__(16) unsigned char pass_smem[];
    float2* Y = reinterpret_cast<float2*>(pass_smem);
    if (blockIdx.x == 0) {
        for (int j = threadIdx.x; j < nbins; j += kPassWidth) bins[j] = 0.0;
        if (threadIdx.x == 0) bins[3 * nbins] = (double)*err;
    }
    const int64_t q0 = (int64_t)blockIdx.x * Q::P;
    for (int it = threadIdx.x; it < Q::P * N2; it += kPassWidth) {
        const int p = it >> Q::L2, n2 = it & (N2 - 1);
        const int64_t i = ((q0 + p) << Q::LN) + n2;
        float2 a[N1];
#pragma unroll
        for (int n1 = 0; n1 < N1; ++n1)
            a[bitrev<Q::L1>(n1)] = REAL ? make_float2(delta[i + N2 * n1], 0.f) : mesh[i + N2 * n1];
        pass_first<N1, N2>(a, Y, p, n2, tw, twsh);
    }
    __syncthreads();
    for (int it = threadIdx.x; it < Q::P * N1; it += kPassWidth) {
        const int p = it >> Q::L1, k1 = it & (N1 - 1);
        float2 a[N2];
        pass_second<N1, N2>(a, Y, p, k1);
        float2* dst = mesh + ((q0 + p) << Q::LN) + k1;
#pragma unroll
        for (int k2 = 0; k2 < N2; ++k2) dst[N1 * k2] = a[k2];
    }
}

template <int N1, int N2>
__global__ void __launch_bounds__(kPassWidth) k_pk_y(float2* mesh, const float2* __restrict__ tw, int twsh) {
    chain_begin();
    using Q = Pass<N1, N2>;
    extern __shared__ __align__(16) unsigned char pass_smem[];
    float2* Y = reinterpret_cast<float2*>(pass_smem);
    const int64_t q0 = (int64_t)blockIdx.x * Q::P;
    float2* data = mesh + ((q0 >> Q::LN) << (2 * Q::LN)) + (q0 & (Q::n - 1));
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
}

// Largest float (not negative) of the block, to every thread.
__device__ __forceinline__ float block_max(float v, float* sh) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
    if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = v;
    __syncthreads();
    v = sh[0];
    for (int w = 1; w < (int)(blockDim.x >> 5); ++w) v = fmaxf(v, sh[w]);
    return v;
}

// z, and the shells: the mesh's own sums first (a shell a block).  Blocks take groups of
// P pencils (one ky, P neighbouring kx) in turn and keep their shells in double
// precision, one owner thread each.  A shell takes at most 2 sqrt(2 j) + 1 modes of a
// pencil, so a limb's 2048 hold a group at every size.
template <int N1, int N2>
__global__ void __launch_bounds__(kPassWidth) k_pk_z(int nbins, double norm, double kf,
                                                     const float2* mesh,
                                                     double* bins, const float2* __restrict__ tw,
                                                     int twsh) {
    chain_begin();
    using Q = Pass<N1, N2>;
    constexpr int64_t plane = (int64_t)Q::n * Q::n;
    constexpr int h = Q::n / 2, kItems = (Q::P * N1 + kPassWidth - 1) / kPassWidth;
    constexpr int kGroups = (int)(plane / Q::P);
    extern __shared__ __align__(16) unsigned char pass_smem[];
    double* acc = reinterpret_cast<double*>(pass_smem);
    uint32_t* limb = reinterpret_cast<uint32_t*>(acc + h + 1);
    float* mx = reinterpret_cast<float*>(limb + 3 * (h + 1));
    float2* Y = reinterpret_cast<float2*>(mx + 33);   // 8-byte aligned: h + 1 is odd
    const int tid = threadIdx.x;
    for (int j = 1 + blockIdx.x; j <= nbins; j += gridDim.x) block_shell(Q::n, nbins, j, kf, bins, reinterpret_cast<uint32_t*>(Y));
    for (int j = tid; j <= h; j += kPassWidth) {
        acc[j] = 0.0;
        limb[j] = limb[h + 1 + j] = limb[2 * (h + 1) + j] = 0u;
    }
    for (int g = blockIdx.x; g < kGroups; g += gridDim.x) {
        const int64_t q0 = (int64_t)g * Q::P;
        const int ky = (int)(q0 >> Q::LN), kx0 = (int)(q0 & (Q::n - 1)), ny = ky < h ? ky : ky - Q::n;
        for (int it = tid; it < Q::P * N2; it += kPassWidth) {
            const int p = it & (Q::P - 1), n2 = it >> Q::LP;
            float2 a[N1];
#pragma unroll
            for (int n1 = 0; n1 < N1; ++n1) a[bitrev<Q::L1>(n1)] = mesh[q0 + p + (N2 * n1 + n2) * plane];
            pass_first<N1, N2>(a, Y, p, n2, tw, twsh);
        }
        __syncthreads();
        float2 a[kItems][N2];
        float big = 0.f;
#pragma unroll
        for (int u = 0; u < kItems; ++u) {
            const int it = tid + u * kPassWidth, p = it & (Q::P - 1), k1 = it >> Q::LP;
            if (it < Q::P * N1) {
                pass_second<N1, N2>(a[u], Y, p, k1);
#pragma unroll
                for (int k2 = 0; k2 < N2; ++k2) big = fmaxf(big, fmaxf(fabsf(a[u][k2].x), fabsf(a[u][k2].y)));
            }
        }
        const int emax = (int)(__float_as_uint(block_max(big, mx)) >> 23);
#pragma unroll
        for (int u = 0; u < kItems; ++u) {
            const int it = tid + u * kPassWidth, p = it & (Q::P - 1), k1 = it >> Q::LP;
            if (it < Q::P * N1) {
                const int kx = kx0 + p, nx = kx < h ? kx : kx - Q::n;
                const int m0 = nx * nx + ny * ny;
#pragma unroll
                for (int k2 = 0; k2 < N2; ++k2) {
                    const int kz = k1 + N1 * k2, nz = kz < h ? kz : kz - Q::n;
                    const int j = shell_of(m0 + nz * nz);
                    if (j >= 1 && j <= nbins)
                        add_limbs(limb + j, h + 1, square_of<13>(a[u][k2].x, emax) + square_of<13>(a[u][k2].y, emax));
                }
            }
        }
        __syncthreads();
        for (int j = tid; j <= nbins; j += kPassWidth) {
            uint32_t* l = limb + j;
            if (l[0] | l[h + 1] | l[2 * (h + 1)]) {
                acc[j] += limbs_value<13>(l[0], l[h + 1], l[2 * (h + 1)], emax);
                l[0] = l[h + 1] = l[2 * (h + 1)] = 0u;
            }
        }
        // (the next group's writes to limb and mx come after its own barrier)
    }
    for (int j = tid; j <= nbins; j += kPassWidth)
        if (j >= 1 && acc[j] != 0.0) atomicAdd(&bins[j - 1], norm * acc[j]);
}

// Up to 16^3 points: transforms, shells and the mesh's own sums in one CTA.  Real
// transforms along x with the kx = N/2 plane in the imaginary part of kx = 0; a mode with 0 < kx < N/2 stands for its mirror image too.
template <int N>
struct PkSmall {
    static constexpr int kH = N / 2, kP = kH + 1, kLog = N == 16 ? 4 : 3;
    static constexpr int kThreads = N * kH;
    static constexpr size_t kBytes = sizeof(float2) * N * N * kP;
};

template <int N>
__global__ void __launch_bounds__(PkSmall<N>::kThreads) k_pk_small(int nbins, double norm, double kf,
                                                                   const float* delta,
                                                                   double* bins,
                                                                   const uint32_t* err) {
    chain_begin();
    using M = PkSmall<N>;
    constexpr int H = M::kH, P = M::kP, T = M::kThreads, L = M::kLog;
    extern __shared__ __align__(16) unsigned char pass_smem[];
    float2* C = reinterpret_cast<float2*>(pass_smem);
    float* R = reinterpret_cast<float*>(pass_smem);
    __shared__ uint32_t limb[3][H][H + 1], hist[T / 32][N];
    __shared__ float mx[32];
    const int tid = threadIdx.x;
    if (tid == 0) bins[3 * nbins] = (double)*err;
    for (int i = tid; i < 3 * H * (H + 1); i += T) (&limb[0][0][0])[i] = 0u;
#pragma unroll 8
    for (int i = tid; i < N * N * N; i += T) R[(i >> L) * (2 * P) + (i & (N - 1))] = delta[i];
    __syncthreads();
    for (int r = tid; r < N * N; r += T) {
        float2* row = C + r * P;
        float x[N];
        float2 X[H + 1];
#pragma unroll
        for (int k = 0; k < H; ++k) {
            x[2 * k] = row[k].x;
            x[2 * k + 1] = row[k].y;
        }
        rfftx2<N, true>(x, X);
        row[0] = make_float2(X[0].x, X[H].x);
#pragma unroll
        for (int k = 1; k < H; ++k) row[k] = X[k];
    }
    __syncthreads();
    float2 a[N];
    {
        float2* col = C + (tid / H) * (N * P) + tid % H;   // along y: kx, z
#pragma unroll
        for (int k = 0; k < N; ++k) a[bitrev<L>(k)] = col[k * P];
        fft_dit<N, -1, true>(a);
#pragma unroll
        for (int k = 0; k < N; ++k) col[k * P] = a[k];
    }
    __syncthreads();
    const int kx = tid / N, ky = tid % N, ny = ky < H ? ky : ky - N;
    float2* col = C + ky * P + kx;
#pragma unroll
    for (int k = 0; k < N; ++k) a[bitrev<L>(k)] = col[k * (N * P)];
    fft_dit<N, -1, true>(a);
    if (kx == 0) {
#pragma unroll
        for (int k = 0; k < N; ++k) col[k * (N * P)] = a[k];
    }
    __syncthreads();
    // The modes at kz of this kx (they stand for their mirror images too), or for kx = 0
    // those of kx = 0 and N/2, times two: 2 A = Z + conj Z', 2 B = -i (Z - conj Z'), Z' at
    // (-ky, -kz)
    auto modes = [&](int k, float2& at0, float2& atH) {
        at0 = a[k];
        atH = make_float2(0.f, 0.f);
        if (kx == 0) {
            const float2 b = C[((N - ky) & (N - 1)) * P + ((N - k) & (N - 1)) * (N * P)];
            at0 = make_float2(a[k].x + b.x, a[k].y - b.y);
            atH = make_float2(a[k].x - b.x, a[k].y + b.y);
        }
    };
    float big = 0.f;
#pragma unroll
    for (int k = 0; k < N; ++k) {
        float2 v, w;
        modes(k, v, w);
        big = fmaxf(big, fmaxf(fmaxf(fabsf(v.x), fabsf(v.y)), fmaxf(fabsf(w.x), fabsf(w.y))));
    }
    // |delta~|^2 times 16 (rfftx2 doubles, and so does `modes` at kx = 0)
    const int emax = (int)(__float_as_uint(block_max(big, mx)) >> 23), times8 = kx == 0 ? 0 : 3;
#pragma unroll
    for (int k = 0; k < N; ++k) {
        float2 v, w;
        modes(k, v, w);
        const int nz = k < H ? k : k - N, m = kx * kx + ny * ny + nz * nz;
        const int j = shell_of(m);
        if (j >= 1 && j <= nbins)
            add_limbs(&limb[0][kx][j], H * (H + 1), (square_of<10>(v.x, emax) + square_of<10>(v.y, emax)) << times8);
        if (kx == 0) {
            const int i = shell_of(m + H * H);
            if (i <= nbins)
                add_limbs(&limb[0][0][i], H * (H + 1), square_of<10>(w.x, emax) + square_of<10>(w.y, emax));
        }
    }
    __syncthreads();
    // a warp per shell: its limbs over kx, and the mesh's own sums
    const int lane = tid & 31;
    for (int j = 1 + (tid >> 5); j <= nbins; j += T / 32) {
        long long s[3];
#pragma unroll
        for (int e = 0; e < 3; ++e) s[e] = warp_sum(lane < H ? (long long)limb[e][lane][j] : 0ll);
        uint32_t* const count = hist[tid >> 5];
        if (lane < N) count[lane] = 0u;
        __syncwarp();
        count_shell(N, j, 0, 1, lane, count);
        __syncwarp();
        const int m = j * j - j + 1 + lane, n = lane < 2 * j ? (int)count[lane] : 0;
        const double k = warp_sum((double)n * __dsqrt_rn((double)m));
        const int modes = warp_sum(n);
        __syncwarp();
        if (lane == 0) {
            bins[j - 1] = 0.0625 * norm * limbs_value<10>(s[0], s[1], s[2], emax);
            bins[nbins + j - 1] = kf * k;
            bins[2 * nbins + j - 1] = (double)modes;
        }
    }
}

// Meshes past 1024 points a side: the general transform (fft.cu) and one mode a
// thread.
__global__ void __launch_bounds__(kPassWidth) k_pk_modes(int nmesh, int nbins, double norm,
                                                         const float2* __restrict__ mesh, double* __restrict__ bins) {
    extern __shared__ double sb[];
    for (int i = threadIdx.x; i <= nbins; i += blockDim.x) sb[i] = 0.0;
    __syncthreads();
    const int64_t m3 = (int64_t)nmesh * nmesh * nmesh;
    const int h = nmesh / 2;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < m3; i += (int64_t)gridDim.x * blockDim.x) {
        const int ix = (int)(i % nmesh), iy = (int)((i / nmesh) % nmesh), iz = (int)(i / ((int64_t)nmesh * nmesh));
        const int nx = ix < h ? ix : ix - nmesh, ny = iy < h ? iy : iy - nmesh, nz = iz < h ? iz : iz - nmesh;
        const int j = shell_of(nx * nx + ny * ny + nz * nz);
        if (j < 1 || j > nbins) continue;
        const float2 v = mesh[i];
        atomicAdd(&sb[j], (double)v.x * v.x + (double)v.y * v.y);
    }
    __syncthreads();
    for (int i = 1 + threadIdx.x; i <= nbins; i += blockDim.x)
        if (sb[i] != 0.0) atomicAdd(&bins[i - 1], norm * sb[i]);
}

template <int PB, int LH, bool SMALL, typename OUT>
void launch_deposit(cudaStream_t stream, const PkStore& st, const PkMean& mean, OUT* out) {
    using B = Brick<LH, SMALL>;
    const unsigned nb = (unsigned)((st.nc / B::CX) * (st.nc / B::CY) * (st.nc / B::CZ));
    chain(st.chained, k_pk_deposit<PB, LH, SMALL, OUT>, nb, B::kThreads, B::kBytes, stream, st, mean, out);
}
template <int PB, bool SMALL, typename OUT>
void deposit_of(cudaStream_t stream, const PkStore& st, int lh, const PkMean& mean, OUT* out) {
    if (lh == 0) launch_deposit<PB, 0, SMALL>(stream, st, mean, out);
    else if (lh == 1) launch_deposit<PB, 1, SMALL>(stream, st, mean, out);
    else launch_deposit<PB, 2, SMALL>(stream, st, mean, out);
}
template <typename OUT>
void deposit(cudaStream_t stream, const PkStore& st, int lh, const PkMean& mean, OUT* out) {
    const bool small = st.nc <= 32;
    if (st.pb == 2 && small) deposit_of<2, true>(stream, st, lh, mean, out);
    else if (st.pb == 2) deposit_of<2, false>(stream, st, lh, mean, out);
    else if (small) deposit_of<1, true>(stream, st, lh, mean, out);
    else deposit_of<1, false>(stream, st, lh, mean, out);
}

template <int N1, int N2>
size_t z_bytes() {
    constexpr int h = Pass<N1, N2>::n / 2;
    return 20 * (size_t)(h + 1) + 4 * 33 + Pass<N1, N2>::kBytes;
}

template <int N1, int N2>
void launch_transforms(cudaStream_t stream, bool chained, int nbins, double norm, double kf, float2* mesh,
                       const float* delta, double* bins, const uint32_t* err, const float2* tw, int tw_n) {
    using Q = Pass<N1, N2>;
    const unsigned groups = (unsigned)((int64_t)Q::n * Q::n / Q::P);
    const bool ahead = chained && (int64_t)Q::n * Q::n * Q::n <= kChainCells;
    int twsh = 0;
    while ((Q::n << twsh) < tw_n) ++twsh;
    chain(ahead, delta ? k_pk_x<N1, N2, true> : k_pk_x<N1, N2, false>, groups, kPassWidth, Q::kBytes, stream, delta, mesh,
          nbins, bins, err, tw, twsh);
    chain(ahead, k_pk_y<N1, N2>, groups, kPassWidth, Q::kBytes, stream, mesh, tw, twsh);
    const unsigned gz = groups < 152 * 6 ? groups : 152 * 6;
    chain(ahead, k_pk_z<N1, N2>, gz, kPassWidth, z_bytes<N1, N2>(), stream, nbins, norm, kf, mesh, bins, tw, twsh);
}

template <int N>
void launch_small(cudaStream_t stream, bool chained, int nbins, double norm, double kf, const float* delta,
                  double* bins, const uint32_t* err) {
    using M = PkSmall<N>;
    chain(chained, k_pk_small<N>, 1, M::kThreads, M::kBytes, stream, nbins, norm, kf, delta, bins, err);
}

template <int N1, int N2>
void setup_transforms() {
    using Q = Pass<N1, N2>;
    const auto smem = cudaFuncAttributeMaxDynamicSharedMemorySize;
    cudaFuncSetAttribute(k_pk_x<N1, N2, true>, smem, (int)Q::kBytes);
    cudaFuncSetAttribute(k_pk_x<N1, N2, false>, smem, (int)Q::kBytes);
    cudaFuncSetAttribute(k_pk_y<N1, N2>, smem, (int)Q::kBytes);
    cudaFuncSetAttribute(k_pk_z<N1, N2>, smem, (int)z_bytes<N1, N2>());
}

}  // namespace

void pk_setup() {
    const auto smem = cudaFuncAttributeMaxDynamicSharedMemorySize;
    const int big = (int)Brick<0, false>::kBytes;
    cudaFuncSetAttribute(k_pk_deposit<1, 0, false, float>, smem, big);
    cudaFuncSetAttribute(k_pk_deposit<2, 0, false, float>, smem, big);
    cudaFuncSetAttribute(k_pk_deposit<1, 0, false, float2>, smem, big);
    cudaFuncSetAttribute(k_pk_deposit<2, 0, false, float2>, smem, big);
    setup_transforms<8, 8>();
    setup_transforms<8, 16>();
    setup_transforms<16, 16>();
    setup_transforms<16, 32>();
    setup_transforms<32, 32>();
}

cudaError_t pk_enqueue(cudaStream_t stream, const PkStore& st, int nmesh, int nbins, float2* mesh,
                       float* delta, double* bins, const uint32_t* err, const float2* tw, int tw_n, int64_t* launches) {
    const int64_t m3 = (int64_t)nmesh * nmesh * nmesh;
    int lh = 0;
    while ((nmesh << lh) < 4 * st.nc) ++lh;
    // the mean weight of a node, n (2U)^3 / nmesh^3
    const int64_t W = (int64_t)(2 * kCodesPerFine) << lh, w3 = W * W * W;
    PkMean mean = {1, 0, 1.f, 0.0};
    const __int128 total = (__int128)st.n * w3;
    if (st.n & (st.n - 1)) {
        mean.inv = (double)m3 / (double)total;
    } else if (total >= m3) {
        mean.mean = (long long)(total / m3);
        mean.scale = (float)(1.0 / (double)mean.mean);
    } else {
        while (((total << mean.shift)) < m3) ++mean.shift;
    }
    const double L = 4.0 * st.nc, norm = L * L * L / ((double)m3 * (double)m3), kf = 2.0 * kPi / L;
    const bool small = nmesh <= 16;
    float* real = small ? reinterpret_cast<float*>(mesh) : (nmesh <= 1024 ? delta : nullptr);
    if (real) deposit(stream, st, lh, mean, real);
    else deposit(stream, st, lh, mean, mesh);
    *launches += 1;
    if (small) {
        if (nmesh == 8) launch_small<8>(stream, st.chained, nbins, norm, kf, real, bins, err);
        else launch_small<16>(stream, st.chained, nbins, norm, kf, real, bins, err);
        *launches += 1;
        return cudaGetLastError();
    }
    *launches += 3;
    if (nmesh == 32) launch_transforms<4, 8>(stream, st.chained, nbins, norm, kf, mesh, real, bins, err, tw, tw_n);
    else if (nmesh == 64) launch_transforms<8, 8>(stream, st.chained, nbins, norm, kf, mesh, real, bins, err, tw, tw_n);
    else if (nmesh == 128) launch_transforms<8, 16>(stream, st.chained, nbins, norm, kf, mesh, real, bins, err, tw, tw_n);
    else if (nmesh == 256) launch_transforms<16, 16>(stream, st.chained, nbins, norm, kf, mesh, real, bins, err, tw, tw_n);
    else if (nmesh == 512) launch_transforms<16, 32>(stream, st.chained, nbins, norm, kf, mesh, real, bins, err, tw, tw_n);
    else if (nmesh == 1024) launch_transforms<32, 32>(stream, st.chained, nbins, norm, kf, mesh, real, bins, err, tw, tw_n);
    else {
        cudaMemsetAsync(bins, 0, sizeof(double) * nbins, stream);
        k_pk_shells<<<nbins, kPassWidth, sizeof(uint32_t) * nmesh, stream>>>(nmesh, nbins, kf, bins, err);
        const cudaError_t e = fft3d_float_raw(stream, mesh, nmesh, -1, tw, tw_n);
        if (e != cudaSuccess) return e;
        k_pk_modes<<<grid_for(m3, kPassWidth, 152 * 4), kPassWidth, sizeof(double) * (nbins + 1), stream>>>(
            nmesh, nbins, norm, mesh, bins);
        *launches += 1;
    }
    return cudaGetLastError();
}

int power_spectrum_enqueue(Sim& s, int nmesh, int nbins, double* host_bins, bool word) {
    if (nmesh < 2 || (nmesh & (nmesh - 1)) || nmesh > s.pk_max || s.nf % nmesh)
        return set_error(s, PMPM_EINVAL, "nmesh %d must be a power of two dividing %d, <= %d",
                         nmesh, s.nf, s.pk_max);
    if (nbins < 1 || nbins > nmesh / 2)
        return set_error(s, PMPM_EINVAL, "nbins %d must be in [1, nmesh/2]", nbins);
    if (nmesh < s.nc) return set_error(s, PMPM_EINVAL, "nmesh below nf/4 is not supported");
    const int64_t m3 = (int64_t)nmesh * nmesh * nmesh;
    float2* mesh = reinterpret_cast<float2*>(s.scratch);
    float* delta = reinterpret_cast<float*>(align_up(reinterpret_cast<uintptr_t>(mesh + m3)));   // (16 pk_max^3 + 512 bytes)
    const PkStore st = {s.nc, s.pb, s.n, s.offsets[s.cur], s.counts[s.cur],
                        {m_stream(s, s.cur, 0), m_stream(s, s.cur, 1), m_stream(s, s.cur, 2)}, s.chained};
    cudaError_t e = pk_enqueue(s.stream, st, nmesh, nbins, mesh, delta, s.pk_bins, s.err, s.tw_f, s.fft_max, &s.launches);
    if (e == cudaSuccess)
        e = cudaMemcpyAsync(host_bins, s.pk_bins, sizeof(double) * (3 * nbins + word), cudaMemcpyDeviceToHost, s.stream);
    if (e != cudaSuccess) return set_error(s, PMPM_ECUDA, "power spectrum: %s", cudaGetErrorString(e));
    return PMPM_OK;
}

void power_spectrum_finish(const double* hb, int nbins, double* k, double* pk, int64_t* nm) {
    for (int j = 0; j < nbins; ++j) {
        const double c = hb[2 * nbins + j];
        nm[j] = (int64_t)c;
        k[j] = c > 0 ? hb[nbins + j] / c : 0.0;
        pk[j] = c > 0 ? hb[j] / c : 0.0;
    }
}

int power_spectrum(Sim& s, int nmesh, int nbins, double* k, double* pk, int64_t* nm, bool* flagged) {
    double* hb = new (std::nothrow) double[3 * (size_t)(nbins > 0 ? nbins : 1) + 1];
    if (!hb) return set_error(s, PMPM_ENOMEM, "host bins");
    int rc = power_spectrum_enqueue(s, nmesh, nbins, hb, true);
    if (!rc) {
        const cudaError_t e = cudaStreamSynchronize(s.stream);
        if (e != cudaSuccess) rc = set_error(s, PMPM_ECUDA, "power spectrum: %s", cudaGetErrorString(e));
    }
    if (!rc) {
        power_spectrum_finish(hb, nbins, k, pk, nm);
        *flagged = hb[3 * nbins] != 0.0;
    }
    delete[] hb;
    return rc;
}

}  // namespace pmpm
