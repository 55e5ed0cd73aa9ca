// column.cu -- the short-range pass of a step: fine-mesh force of Sec. II on
// columns of tiles, with the force interpolation and, in step mode, the kick
// and the integer drift.
//
// The (x, y) plane is cut into the tiles of tile_core.cuh (4 or 5 coarse
// cells a side, grown by the 6-cell buffer to a 32 x 32 box of fine nodes).
// One CTA takes one tile's column and walks it along z, one coarse layer (4
// fine planes) at a time, over a segment of the box:
//   deposit   integer CIC of the layer's particles (tile and halo) on its planes
//   forward   2-D real transform of the 4 planes that are complete now
//   z sum     the kernel's z extent is 11 planes (|dz| < 6), so along z Eq. 1 is a
//             direct sum over 11 spectra per (kx, ky), three components at once
//   inverse   pruned 2-D transforms of the 4 new force planes
//   gather    all three force components, F_l, kick and drift of the layer three
//             below, whose planes are complete
// against a 32^3 box per tile (three transforms back along every axis): no
// plane is deposited or transformed twice along z, and the halo is 9 x 9 cells
// per layer of 5 x 5 instead of 9^3 per 5^3.
//
// What it keeps: the last 11 spectra per (kx, ky) and the 17 kernel values
// per (kx, ky) are private to one thread and wait in TMEM (56 of the 64 words
// per point, two points a thread), so that shared memory holds only 6 planes
// of density and 6 of each force component: 111 KB, two CTAs of 8 warps a SM
// whose barriers do not meet.  Register transforms take 128 registers a thread,
// so there is no room for a third.
//
// What bounds it: issue (49% of the slots, 16.5k warp instructions a layer, 6.3k of
// them floating point) and the waits between the three barriers of a layer and
// for the particles' bytes; memory moves 41 B a particle.  Short-range pass of a step on
// a GB300 against the 32^3-box tiles of one CTA a SM: 512^3 particles 35.5 -> 18.8 ms,
// 256^3 4.52 -> 2.52 ms, 128^3 598 -> 398 us; denser boxes, 256^3 on 64^3 cells 2.40 -> 1.87
// ms and 512^3 on 64^3, where every node is checked, 21.8 -> 15.0.  (keeps_bits: boxes that
// take tiles all the same.)
#include <algorithm>

#include "pmpm_impl.cuh"
#include "tile_core.cuh"

namespace pmpm {

namespace {

constexpr int kColThreads = 256;
constexpr int kColSlots = 6;                       // planes of a ring
// Rows of a plane are 34 words apart: 8-byte accesses down a column and along
// a row then both fall in distinct banks, and every address of a pencil is one
// base and a constant.
constexpr int kColPitch = 34;
constexpr int kColPlane = 32 * kColPitch;          // words of a force plane
// Density planes end in one row more.  A cloud that reaches one node over an
// edge of the box then writes to words that no transform reads (columns -1 and
// 32 are the two of the pitch, rows -1 and 32 that row), with no test per node.
constexpr int kColDens = (33 * kColPitch + 3) / 4 * 4;
constexpr int kColGuard = 36;                      // words before the first plane: its row -1
constexpr int kColOutMin = 18;                     // force nodes along an axis of the smaller tiles
constexpr int kColHalo = kHaloDim * kHaloDim;      // 81 halo cells of a layer
constexpr int kColOwn = kOwnDim * kOwnDim;         // 25 own cells of a layer
constexpr int kColTaps = 6;                        // |dz| = 0..5
constexpr int kColFlPlane = 3 * kFlWin * kFlWin;   // F_l window of one coarse plane
constexpr int kColMap = 1024;                      // halo particles whose cell is looked up by table
constexpr int kColMapLane = 16;                    // and those of a cell that one lane enters
// Deposit of a layer: the two warps that do not transform take the first 2 x 5
// groups of 32 particles, the other six 2 groups each (22 groups, 704 particles:
// a layer of 8 a cell holds 648); what is left goes to whichever warp is free.
constexpr int kColDepFree = 5, kColDepBusy = 2;
constexpr int kColDepStatic = 32 * (2 * kColDepFree + 6 * kColDepBusy);
constexpr int kTmemCols = 256;                     // of 512: two CTAs a SM
constexpr int kTmemPoint = 64;                     // words of one (kx, ky) point

// The halo cells of the layer about to be deposited.
struct ColHaloTab {
    int64_t off[kColHalo];     // particle v of the layer lies at off[its cell] + v
    int pre[kColHalo + 1];     // exclusive prefix of the cells' counts
    uint8_t map[kColMap];      // cell of the v-th particle
};
// The tile's own cells of a layer, likewise (a ring: they are gathered four
// layers later).
struct ColOwnTab {
    int64_t off[kColOwn];
    int pre[kColOwn + 1];
};

struct ColShared {
    uint32_t guard[kColGuard];
    uint32_t A[kColSlots * kColDens];           // density planes, then their spectra in place
    float2 O[3 * kColSlots * kColPlane / 2];    // force planes by component
    ColHaloTab halo;
    ColOwnTab own[8];
    float fl[4][kColFlPlane];                   // F_l window by coarse plane
    float Td[256];                              // velocity decode table of Eq. 3
    int cmax[4];                                // largest halo-cell count by layer
    int next, dep;                              // next particles to gather and to deposit
    uint32_t tmem;                              // TMEM address
};
static_assert(sizeof(ColShared) <= 113 * 1024, "two CTAs a SM");

struct ColParams {
    TileParams t;
    const float* table;    // [17][17][17]: 6 x taps, 6 y taps, 5 z taps of each (kx, |ky|)
    int lz;                // layers of a segment
};

// ring slot base + d, 0 <= d <= 6
__device__ __forceinline__ int slot6(int base, int d) {
    const int s = base + d;
    return s >= kColSlots ? s - kColSlots : s;
}
// complex (kx, row) of a plane; rows are ky or y
__device__ __forceinline__ int qidx(int kx, int row) { return row * (kColPitch / 2) + kx; }

// ------------------------------------------------------------------ TMEM
__device__ __forceinline__ void tmem_alloc(uint32_t* dst) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     (uint32_t)__cvta_generic_to_shared(dst)),
                 "r"(kTmemCols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
}
__device__ __forceinline__ void tmem_free(uint32_t addr) {
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(addr), "r"(kTmemCols));
}
// waits for this thread's loads; their registers are read only after it
template <int N>
__device__ __forceinline__ void tmem_wait_ld(float (&r)[N]) {
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
    for (int i = 0; i < N; ++i) asm volatile("" : "+f"(r[i]));
}
__device__ __forceinline__ void tmem_wait_st() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }
__device__ __forceinline__ void tmem_ld16(uint32_t a, float* r) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
                 : "=f"(r[0]), "=f"(r[1]), "=f"(r[2]), "=f"(r[3]), "=f"(r[4]), "=f"(r[5]), "=f"(r[6]), "=f"(r[7]), "=f"(r[8]), "=f"(r[9]), "=f"(r[10]), "=f"(r[11]), "=f"(r[12]), "=f"(r[13]), "=f"(r[14]), "=f"(r[15])
                 : "r"(a));
}
__device__ __forceinline__ void tmem_ld8(uint32_t a, float* r) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
                 : "=f"(r[0]), "=f"(r[1]), "=f"(r[2]), "=f"(r[3]), "=f"(r[4]), "=f"(r[5]), "=f"(r[6]), "=f"(r[7])
                 : "r"(a));
}
__device__ __forceinline__ void tmem_st16(uint32_t a, const float* r) {
    asm volatile("tcgen05.st.sync.aligned.32x32b.x16.b32 [%16], {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15};" ::"f"(r[0]), "f"(r[1]), "f"(r[2]), "f"(r[3]), "f"(r[4]), "f"(r[5]), "f"(r[6]), "f"(r[7]), "f"(r[8]), "f"(r[9]), "f"(r[10]), "f"(r[11]), "f"(r[12]), "f"(r[13]), "f"(r[14]), "f"(r[15]), "r"(a)
                 : "memory");
}
__device__ __forceinline__ void tmem_st4(uint32_t a, const float* r) {
    asm volatile("tcgen05.st.sync.aligned.32x32b.x4.b32 [%4], {%0,%1,%2,%3};" ::"f"(r[0]), "f"(r[1]), "f"(r[2]), "f"(r[3]), "r"(a)
                 : "memory");
}
__device__ __forceinline__ void tmem_st2(uint32_t a, const float* r) {
    asm volatile("tcgen05.st.sync.aligned.32x32b.x2.b32 [%2], {%0,%1};" ::"f"(r[0]), "f"(r[1]), "r"(a)
                 : "memory");
}

// ------------------------------------------------------------------ layer tables
// One warp; lane i < 27 holds cells 3 i .. 3 i + 2 of the 9 x 9 halo layer
// (row i / 3).  Loaded a phase before they are needed.
struct ColCells {
    int64_t st[3];
    int cnt[3];
};

__device__ __forceinline__ ColCells col_cells_load(int lane, const TileGeom& g, const TileParams& P, int layer) {
    ColCells c;
    const int by = lane / 3;
    const int hx = g.c1[0] - g.c0[0] + 4, hy = g.c1[1] - g.c0[1] + 4;
    const int cy = wrap1(g.c0[1] - 2 + by, P.nc), cz = wrap1(layer, P.nc);
#pragma unroll
    for (int e = 0; e < 3; ++e) {
        const int bx = 3 * (lane % 3) + e;
        c.st[e] = 0;
        c.cnt[e] = 0;
        if (lane < 27 && bx < hx && by < hy) {
            const int64_t cell = wrap1(g.c0[0] - 2 + bx, P.nc) + (int64_t)P.nc * (cy + (int64_t)P.nc * cz);
            c.st[e] = P.offsets[cell];
            c.cnt[e] = P.counts[cell];
        }
    }
    return c;
}

__device__ __forceinline__ int warp_incl(int lane, int v) {
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, v, o);
        if (lane >= o) v += y;
    }
    return v;
}

__device__ __forceinline__ void col_cells_store(int lane, const TileGeom& g, const ColCells& c, ColShared& S,
                                                int layer) {
    ColHaloTab& t = S.halo;
    ColOwnTab& w = S.own[layer & 7];
    const int sum = c.cnt[0] + c.cnt[1] + c.cnt[2];
    const int incl = warp_incl(lane, sum);
    const int from[3] = {incl - sum, incl - sum + c.cnt[0], incl - c.cnt[2]};
    int mx = max(c.cnt[0], max(c.cnt[1], c.cnt[2]));
    if (lane < 27) {
#pragma unroll
        for (int e = 0; e < 3; ++e) {
            t.off[3 * lane + e] = c.st[e] - from[e];
            t.pre[3 * lane + e] = from[e];
        }
        if (lane == 26) t.pre[kColHalo] = incl;
    }
    // the particles' cells: a lane enters its three cells' side by side, and the
    // warp what a crowded cell has beyond
    for (int q = 0; q < kColMapLane && __any_sync(0xffffffffu, q < mx); ++q) {
#pragma unroll
        for (int e = 0; e < 3; ++e)
            if (q < c.cnt[e] && from[e] + q < kColMap) t.map[from[e] + q] = (uint8_t)(3 * lane + e);
    }
#pragma unroll
    for (int e = 0; e < 3; ++e) {
        unsigned crowded = __ballot_sync(0xffffffffu, c.cnt[e] > kColMapLane && from[e] < kColMap);
        while (crowded) {
            const int src = __ffs(crowded) - 1;
            crowded &= crowded - 1u;
            const int f = __shfl_sync(0xffffffffu, from[e], src), n = __shfl_sync(0xffffffffu, c.cnt[e], src);
            for (int q = kColMapLane + lane; q < n && f + q < kColMap; q += 32) t.map[f + q] = (uint8_t)(3 * src + e);
        }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    if (lane == 0) S.cmax[layer & 3] = mx;
    __syncwarp();
    const int px = lane % kOwnDim, py = lane / kOwnDim;
    int n = 0;
    int64_t st = 0;
    if (lane < kColOwn && px < g.c1[0] - g.c0[0] && py < g.c1[1] - g.c0[1]) {
        const int h = (2 + px) + kHaloDim * (2 + py);
        n = t.pre[h + 1] - t.pre[h];
        st = t.off[h] + t.pre[h];
    }
    const int own = warp_incl(lane, n);
    if (lane < kColOwn) {
        w.pre[lane] = own - n;
        w.off[lane] = st - (own - n);
    }
    if (lane == kColOwn - 1) w.pre[kColOwn] = own;
}

// F_l on the 7 x 7 nodes around the tile of one coarse plane: five values a lane
__device__ __forceinline__ void col_fl_load(int lane, const TileGeom& g, const TileParams& P, int layer,
                                            float (&v)[5]) {
    const int64_t ncells = (int64_t)P.nc * P.nc * P.nc;
    const int z = wrap1(layer, P.nc);
#pragma unroll
    for (int k = 0; k < 5; ++k) {
        const int i = lane + 32 * k;
        v[k] = 0.f;
        if (i < kColFlPlane) {
            const int e = i / (kFlWin * kFlWin), w = i % (kFlWin * kFlWin);
            const int x = wrap1(g.c0[0] - 1 + w % kFlWin, P.nc), y = wrap1(g.c0[1] - 1 + w / kFlWin, P.nc);
            v[k] = P.Fl[e * ncells + x + P.nc * (y + (int64_t)P.nc * z)];
        }
    }
}
__device__ __forceinline__ void col_fl_store(int lane, const float (&v)[5], float* dst) {
#pragma unroll
    for (int k = 0; k < 5; ++k) {
        const int i = lane + 32 * k;
        if (i < kColFlPlane) dst[i] = v[k];
    }
}

// ------------------------------------------------------------------ deposit
// CIC of one particle of halo cell (bx, by) into the layer's six planes
// (slot `ab` is the lowest).  CHECK as in
// tile_core.cuh: a node can pass 2^32 only where a halo cell of this layer
// or the one below (the planes they share) holds more than 255 particles.
template <bool CHECK, int PB>
__device__ __forceinline__ void col_deposit_one(int bx, int by, const int (&m)[3], uint32_t* A, int ab,
                                                uint32_t* err) {
    using F = PosFmt<PB>;
    constexpr int W = F::kFineW;
    const int sx = W * (4 * bx - 2) + 2 * m[0] + 1 - F::kCodesPerFine;
    const int sy = W * (4 * by - 2) + 2 * m[1] + 1 - F::kCodesPerFine;
    const int sz = 2 * m[2] + 1 - F::kCodesPerFine + W;
    const int lx = sx >> F::kFineWBits, ly = sy >> F::kFineWBits, lz = sz >> F::kFineWBits;   // lz in 0..4
    const int wx = sx & (W - 1), wy = sy & (W - 1), wz = sz & (W - 1);
    if ((unsigned)(lx + 1) > 32u || (unsigned)(ly + 1) > 32u) return;   // misses the box
    const int o = ly * kColPitch + lx;
    uint32_t* const p0 = A + slot6(ab, lz) * kColDens + o;
    uint32_t* const p1 = A + slot6(ab, lz + 1) * kColDens + o;
#pragma unroll
    for (int c = 0; c < 8; ++c) {
        const int dx = c & 1, dy = (c >> 1) & 1, dz = c >> 2;
        const uint32_t w = cic_weight3<PB>(dx ? wx : W - wx, dy ? wy : W - wy, dz ? wz : W - wz);
        uint32_t* const p = (dz ? p1 : p0) + dx + kColPitch * dy;
        if (CHECK) {
            if (w == 0u || (unsigned)(lx + dx) >= 32u || (unsigned)(ly + dy) >= 32u) continue;
            const uint32_t old = smem_add_u32(p, w);
            if (old + w < old) flag_error(err, kErrFineOverflow);
        } else {
            smem_red_u32(p, w);
        }
    }
}

// halo cell and bins of a particle, packed: the cell in the top byte of hi
// (255: none)
template <int PB>
struct ColBins {
    uint32_t hi, lo;
};

// FIRST: v lies within the table of cells; total > 0.  (Searching the prefix for
// every particle instead took 8% more of the whole pass.)
template <bool FIRST, int PB>
__device__ __forceinline__ ColBins<PB> col_bins_load(int v, int total, const TileParams& P, const ColHaloTab& t) {
    static_assert(kColDepStatic <= kColMap, "");
    const int w = min(v, total - 1);
    const int b = FIRST || w < kColMap ? (int)t.map[w] : prefix_find_loop(t.pre, kColHalo, w);
    const int64_t j = t.off[b] + w;
    const uint32_t m0 = load_bin<PB>(P.m0, j), m1 = load_bin<PB>(P.m1, j), m2 = load_bin<PB>(P.m2, j);
    const uint32_t cell = v < total ? (uint32_t)b << 24 : 0xff000000u;
    if (PB == 1) return {cell | m2 << 16 | m1 << 8 | m0, 0u};
    return {cell | m2, m1 << 16 | m0};
}

template <bool CHECK, int PB>
__device__ __forceinline__ void col_deposit(ColBins<PB> r, uint32_t* A, int ab, uint32_t* err) {
    const int b = r.hi >> 24;
    const int m[3] = {(int)(PB == 1 ? r.hi & 255 : r.lo & 65535), (int)(PB == 1 ? r.hi >> 8 & 255 : r.lo >> 16),
                      (int)(PB == 1 ? r.hi >> 16 & 255 : r.hi & 65535)};
    if (b != 255) col_deposit_one<CHECK, PB>(b % kHaloDim, b / kHaloDim, m, A, ab, err);
}

// the whole layer 32 at a time with every node checked (rare)
template <int PB>
__device__ __noinline__ void col_deposit_checked(int warp, int lane, int total, const TileParams& P, ColShared& S,
                                                 int ab) {
    for (int v = 32 * warp + lane; v < total; v += kColThreads)
        col_deposit<true, PB>(col_bins_load<false, PB>(v, total, P, S.halo), S.A, ab, P.err);
}

// ------------------------------------------------------------------ forward
// In place: the real transform along x of one row (twice the spectrum, the
// kx = 16 value in the imaginary part of kx = 0) and the transform along y of
// one column.
__device__ __forceinline__ void col_fwd_x(uint32_t* row) {
    float x[32];
#pragma unroll
    for (int n = 0; n < 16; ++n) {
        const uint2 r = reinterpret_cast<const uint2*>(row)[n];
        x[2 * n] = u32_to_f32(r.x);
        x[2 * n + 1] = u32_to_f32(r.y);
    }
    float2 X[17];
    rfftx2<32, true>(x, X);
    float2* C = reinterpret_cast<float2*>(row);
    C[0] = make_float2(X[0].x, X[16].x);
#pragma unroll
    for (int k = 1; k < 16; ++k) C[k] = X[k];
}
__device__ __forceinline__ void col_fwd_y(float2* col) {
    float2 a[32];
#pragma unroll
    for (int k = 0; k < 32; ++k) a[bitrev<5>(k)] = col[qidx(0, k)];
    fft_dit<32, -1, true>(a);
#pragma unroll
    for (int k = 0; k < 32; ++k) col[qidx(0, k)] = a[k];
}

// ------------------------------------------------------------------ z sum
// Warp w owns kx = w and w + 8, lane l owns ky = l.  The packed column kx = 0
// (planes kx = 0 and 16) is unpacked first: lane l = 1..15 takes kx = 0, ky = l,
// lane 16 + l takes kx = 16, ky = l, and lanes 0 and 16 the two real values of
// ky = 0 and 16.  Every point then has its own 17 kernel values, and after the
// sum the column is packed again.
__device__ __forceinline__ float2 shfl2(float2 v, int src) {
    return make_float2(__shfl_sync(0xffffffffu, v.x, src), __shfl_sync(0xffffffffu, v.y, src));
}

// kernel values of one point as pairs (one per component of the complex
// value), into its TMEM words 22..55
__device__ __forceinline__ void col_taps_init(int kx, int ky, const float* __restrict__ table, uint32_t ta) {
    const int ay = kabs32(ky);
    int a = kx, b = ay, a2 = kx, b2 = ay;
    float sg = (ay == 0 || ay == 16) ? 0.f : ksgn32(ky);
    if (kx == 0) {
        if (ky > 16) { a = a2 = 16; b = b2 = ky - 16; sg = 1.f; }
        if (ky == 0 || ky == 16) a2 = 16;
    }
    float c[34];
#pragma unroll
    for (int d = 0; d < kColTaps; ++d) {
        const float x = kx == 0 ? 0.f : table[(d * kGreenS + a) * kGreenS + b];
        const float y = sg * table[((kColTaps + d) * kGreenS + a) * kGreenS + b];
        c[2 * d] = c[2 * d + 1] = x;
        c[2 * (kColTaps + d)] = c[2 * (kColTaps + d) + 1] = y;
    }
#pragma unroll
    for (int d = 0; d < kColTaps - 1; ++d) {
        c[24 + 2 * d] = table[((2 * kColTaps + d) * kGreenS + a) * kGreenS + b];
        c[25 + 2 * d] = table[((2 * kColTaps + d) * kGreenS + a2) * kGreenS + b2];
    }
    tmem_st2(ta + 22, c);
    tmem_st16(ta + 24, c + 2);
    tmem_st16(ta + 40, c + 18);
}

__device__ __forceinline__ float2 col_unpack(int lane, float2 Z) {
    const int k = lane & 15;
    const float2 a = shfl2(Z, k), b = shfl2(Z, (32 - k) & 31);
    if (k == 0) return Z;
    return lane < 16 ? make_float2(0.5f * (a.x + b.x), 0.5f * (a.y - b.y))
                     : make_float2(0.5f * (a.y + b.y), 0.5f * (b.x - a.x));
}

// A in lanes 1..15, B in lanes 17..31 (both Hermitian in ky) back to A + i B
// at ky = lane; lanes 0 and 16 hold the pair already
__device__ __forceinline__ float2 col_pack(int lane, float2 G) {
    const int k = lane < 16 ? lane : 32 - lane;
    const float2 a = shfl2(G, k), b = shfl2(G, (16 + k) & 31);
    if ((lane & 15) == 0) return G;
    return lane < 16 ? make_float2(a.x - b.y, a.y + b.x) : make_float2(a.x + b.y, b.x - a.y);
}

// a0, a1: the first and last two of the four new spectra; o0, o1: the planes of
// the four new force planes likewise
// The new spectra's places start again as density.
__device__ __forceinline__ void col_zsum(int warp, int lane, float2* a0, float2* a1, float2* o0, float2* o1,
                                         uint32_t tm, bool emit) {
    constexpr int kP = kColPlane / 2, kC = kColSlots * kP;
#pragma unroll 1
    for (int s = 0; s < 2; ++s) {
        const int kx = warp + 8 * s, i = qidx(kx, lane);
        const uint32_t ta = tm + kTmemPoint * s;
        float t[56];   // spectra of planes 4l-12 .. 4l-2, kernel values
        tmem_ld16(ta, t);
        tmem_ld16(ta + 16, t + 16);
        tmem_ld16(ta + 32, t + 32);
        tmem_ld8(ta + 48, t + 48);
        float2 z[4] = {a0[i], a0[kColDens / 2 + i], a1[i], a1[kColDens / 2 + i]};   // planes 4l-1 .. 4l+2
        a0[i] = a0[kColDens / 2 + i] = a1[i] = a1[kColDens / 2 + i] = make_float2(0.f, 0.f);
        if (kx == 0)
#pragma unroll
            for (int q = 0; q < 4; ++q) z[q] = col_unpack(lane, z[q]);
        tmem_wait_ld(t);
        auto at = [&](int k) { return k < 11 ? make_float2(t[2 * k], t[2 * k + 1]) : z[k - 11]; };
        if (emit) {
            auto tap = [&](int k) { return make_float2(t[22 + 2 * k], t[23 + 2 * k]); };
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const float2 v0 = at(q + 5);
                float2 gx = __fmul2_rn(tap(0), v0), gy = __fmul2_rn(tap(kColTaps), v0), gz;
#pragma unroll
                for (int d = 1; d < kColTaps; ++d) {
                    const float2 lo = at(q + 5 - d), hi = at(q + 5 + d);
                    const float2 e = __fadd2_rn(lo, hi);
                    const float2 o = __ffma2_rn(hi, make_float2(-1.f, -1.f), lo);
                    gx = __ffma2_rn(tap(d), e, gx);
                    gy = __ffma2_rn(tap(kColTaps + d), e, gy);
                    gz = d == 1 ? __fmul2_rn(tap(2 * kColTaps), o) : __ffma2_rn(tap(2 * kColTaps + d - 1), o, gz);
                }
                // The x and y kernels are odd in their own axis: times -i.  The
                // transform along x does that for all three (col_inv_x), so z
                // takes an i here.
                if (kx == 0) {
                    gx = make_float2(0.f, 0.f);
                    gy = col_pack(lane, make_float2(gy.y, -gy.x));
                    gy = make_float2(-gy.y, gy.x);
                    gz = col_pack(lane, gz);
                }
                float2* const o = (q < 2 ? o0 : o1) + (q & 1) * kP + i;
                o[0] = gx;
                o[kC] = gy;
                o[2 * kC] = make_float2(-gz.y, gz.x);
            }
        }
        float h[22];
#pragma unroll
        for (int k = 0; k < 11; ++k) {
            h[2 * k] = at(k + 4).x;
            h[2 * k + 1] = at(k + 4).y;
        }
        tmem_st16(ta, h);
        tmem_st4(ta + 16, h + 16);
        tmem_st2(ta + 20, h + 20);
    }
    tmem_wait_st();
}

// ------------------------------------------------------------------ inverse
// along y: one column of one plane, pruned to ny rows
__device__ __forceinline__ void col_inv_y(int ny, float2* col) {
    float2 a[32];
#pragma unroll
    for (int k = 0; k < 32; ++k) a[bitrev<5>(k)] = col[qidx(0, k)];
    fft_dit<32, 1, true>(a);
#pragma unroll
    for (int yo = 0; yo < kTileOut; ++yo)
        if (yo < kColOutMin || ny > kColOutMin) col[qidx(0, yo)] = a[yo + kBuffer - 1];
}

// times -i (col_zsum), then along x to real values: one row, pruned to nx columns
__device__ __forceinline__ void col_inv_x(int nx, float2* row) {
    float2 X[17];
    const float2 p0 = row[0];
    X[0] = make_float2(p0.y, 0.f);
    X[16] = make_float2(-p0.x, 0.f);
#pragma unroll
    for (int k = 1; k < 16; ++k) X[k] = make_float2(row[k].y, -row[k].x);
    float x[32];
    irfft32(X, x);
#pragma unroll
    for (int xo = 0; xo < kTileOut; xo += 2)
        if (xo < kColOutMin || nx > kColOutMin) row[xo >> 1] = make_float2(x[xo + kBuffer - 1], x[xo + kBuffer]);
}

// ------------------------------------------------------------------ gather
// One own particle: what it reads from global memory, loaded a phase before
// it is gathered.
struct ColOwn {
    int64_t j;       // storage index, -1: none
    int p;           // own cell
    int m[3], u[3];
    float vc[3];
};

template <int PB>
__device__ __forceinline__ void col_own_load(int v, int layer, const TileGeom& g, const TileParams& P,
                                             const ColShared& S, ColOwn& r) {
    const ColOwnTab& t = S.own[layer & 7];
    r.j = -1;
    if (v >= t.pre[kColOwn]) return;
    r.p = prefix_find<kColOwn>(t.pre, v);
    r.j = t.off[r.p] + v;
    r.m[0] = load_bin<PB>(P.m0, r.j);
    r.m[1] = load_bin<PB>(P.m1, r.j);
    r.m[2] = load_bin<PB>(P.m2, r.j);
    if (P.mode >= 1) {
        const int ncells = P.nc * P.nc * P.nc;   // at most 2^30
        const int cell = (g.c0[0] + r.p % kOwnDim) + P.nc * ((g.c0[1] + r.p / kOwnDim) + P.nc * wrap1(layer, P.nc));
        r.u[0] = P.u0[r.j];
        r.u[1] = P.u1[r.j];
        r.u[2] = P.u2[r.j];
#pragma unroll
        for (int e = 0; e < 3; ++e) r.vc[e] = (P.vc + (int64_t)e * ncells)[cell];
    }
}

// the drift of a component out of range: flagged, or several periods away
__device__ __noinline__ int col_drift_flagged(int code, float p, float drift, int M, uint32_t* err) {
    if (!(fabsf(p) < 1048576.f)) flag_error(err, p == p ? kErrMomentum : kErrNaN);
    return drift_code(code, p, drift, M, err);
}

// Its force: the three fine components with one set of weights, F_l from the
// window, then kick, drift and the new cell's sums as in tile_core.cuh.
template <bool LM, int PB>
__device__ __forceinline__ void col_gather(const ColOwn& r, int layer, const TileGeom& g, const TileParams& P,
                                           const ColShared& S, int ob, float sigma, float kick, float drift,
                                           unsigned long long& lo, unsigned long long& hi) {
    using F = PosFmt<PB>;
    constexpr int W = F::kFineW, CW = F::kCoarseW;
    const int64_t n = P.n;
    const int ncells = P.nc * P.nc * P.nc;   // at most 2^30
    const int M = P.nc * F::kBins, cz = wrap1(layer, P.nc);
    const float* Of = reinterpret_cast<const float*>(S.O);
    const int64_t j = r.j;
    const int px = r.p % kOwnDim, py = r.p / kOwnDim;
    const int (&m)[3] = r.m;
    {
        // long-range: the 2^3 coarse nodes around the particle
        float gc[3] = {0.f, 0.f, 0.f};
        {
            int i0[3], w1[3];
#pragma unroll
            for (int e = 0; e < 3; ++e) {
                const int s = 2 * m[e] + 1 - F::kBins;
                i0[e] = s >> F::kCoarseWBits;      // -1 or 0
                w1[e] = s & (CW - 1);
            }
            const int node = (px + 1 + i0[0]) + kFlWin * (py + 1 + i0[1]);
            const float* const f0 = S.fl[(layer + i0[2]) & 3] + node;
            const float* const f1 = S.fl[(layer + i0[2] + 1) & 3] + node;
            // 1-byte weights: exact products of two integers in float
            const float fx[2] = {(float)(CW - w1[0]), (float)w1[0]};
            const float fy[2] = {(float)(CW - w1[1]), (float)w1[1]};
            const float fz[2] = {(float)(CW - w1[2]), (float)w1[2]};
#pragma unroll
            for (int c = 0; c < 8; ++c) {
                const int dx = c & 1, dy = (c >> 1) & 1, dz = c >> 2;
                const float* fl = (dz ? f1 : f0) + dx + kFlWin * dy;
                const float w = PB == 1 ? (fx[dx] * fy[dy]) * fz[dz]
                                        : (float)cic_weight3<PB>(dx ? w1[0] : CW - w1[0], dy ? w1[1] : CW - w1[1],
                                                                 dz ? w1[2] : CW - w1[2]);
#pragma unroll
                for (int e = 0; e < 3; ++e) gc[e] += w * fl[e * kFlWin * kFlWin];
            }
        }
        // short-range: the 2^3 fine nodes
        float gf[3] = {0.f, 0.f, 0.f};
        {
            const int s0 = 4 * W * px + 2 * m[0] + 1 - F::kCodesPerFine + W;
            const int s1 = 4 * W * py + 2 * m[1] + 1 - F::kCodesPerFine + W;
            const int s2 = 2 * m[2] + 1 - F::kCodesPerFine + W;
            const int x = s0 >> F::kFineWBits, y = s1 >> F::kFineWBits, z = s2 >> F::kFineWBits;
            const int w1[3] = {s0 & (W - 1), s1 & (W - 1), s2 & (W - 1)};
            const float* const o0 = Of + slot6(ob, z) * kColPlane + y * kColPitch + x;
            const float* const o1 = Of + slot6(ob, z + 1) * kColPlane + y * kColPitch + x;
            const float fx[2] = {(float)(W - w1[0]), (float)w1[0]};
            const float fy[2] = {(float)(W - w1[1]), (float)w1[1]};
            const float fz[2] = {(float)(W - w1[2]), (float)w1[2]};
#pragma unroll
            for (int c = 0; c < 8; ++c) {
                const int dx = c & 1, dy = (c >> 1) & 1, dz = c >> 2;
                const float w = PB == 1 ? fx[dx] * (fy[dy] * fz[dz])
                                        : (float)cic_weight3<PB>(dx ? w1[0] : W - w1[0], dy ? w1[1] : W - w1[1],
                                                                 dz ? w1[2] : W - w1[2]);
                const float* o = (dz ? o1 : o0) + dx + kColPitch * dy;
#pragma unroll
                for (int e = 0; e < 3; ++e) gf[e] += w * o[e * kColSlots * kColPlane];
            }
        }
        float gval[3];
        // weights in units of 2^-21 and 2^-27; the forward transform along x doubles
#pragma unroll
        for (int e = 0; e < 3; ++e) gval[e] = gf[e] * 2.384185791015625e-07f + gc[e] * 7.450580596923828e-09f;
        if (P.mode == 0) {
#pragma unroll
            for (int e = 0; e < 3; ++e) P.G[e * n + j] = gval[e];
            return;
        }
        // drift_code of common.cuh with its checks put together: a particle that
        // leaves the range of any takes the slow path once
        int q[3];
        float pn[3], xq[3];
        bool ok = true;
        const int c[3] = {g.c0[0] + px, g.c0[1] + py, cz};
#pragma unroll
        for (int e = 0; e < 3; ++e) {
            pn[e] = fadd_rn(decode_momentum(r.vc[e], sigma, S.Td[r.u[e]]), fmul_rn(kick, gval[e]));
            xq[e] = fmul_rn(pn[e], drift);
            ok = ok && fabsf(pn[e]) < 1048576.f && fabsf(xq[e]) < 1.0e9f;
            const int to = c[e] * F::kBins + m[e] + __float2int_rd(fadd_rn(xq[e], 0.5f));
            q[e] = to < 0 ? to + M : (to >= M ? to - M : to);
        }
        ok = ok && (unsigned)q[0] < (unsigned)M && (unsigned)q[1] < (unsigned)M && (unsigned)q[2] < (unsigned)M;
        if (!ok) {
#pragma unroll
            for (int e = 0; e < 3; ++e) q[e] = col_drift_flagged(c[e] * F::kBins + m[e], pn[e], drift, M, P.err);
        }
        long long fx[3];
#pragma unroll
        for (int e = 0; e < 3; ++e) fx[e] = fabsf(pn[e]) < 1048576.f ? fix24_rn(pn[e]) : 0;
        const int key = (q[0] >> F::kShift) + P.nc * ((q[1] >> F::kShift) + P.nc * (q[2] >> F::kShift));
        gmem_add_i32(&P.counts_new[key], 1);
        // |fx| < 2^44: squares from 22-bit halves, three exact 64-bit sums
        unsigned long long s0 = 0, s1 = 0, s2 = 0;
#pragma unroll
        for (int e = 0; e < 3; ++e) {
            if (!LM) P.Qn[e * n + j] = q[e];
            P.Pn[e * n + j] = pn[e];
            gmem_add_u64(&(P.S + (int64_t)e * ncells)[key], (unsigned long long)fx[e]);
            const unsigned long long u = fx[e] < 0 ? (unsigned long long)(-fx[e]) : (unsigned long long)fx[e];
            const uint32_t ul = (uint32_t)u & 0x3fffffu, uh = (uint32_t)(u >> 22);
            s0 += (unsigned long long)ul * ul;
            s1 += (unsigned long long)ul * uh;
            s2 += (unsigned long long)uh * uh;
        }
        unsigned long long add = s0, up = (s1 >> 41) + (s2 >> 20);
        add += s1 << 23;
        up += add < s0 ? 1ull : 0ull;
        const unsigned long long t2 = add + (s2 << 44);
        up += t2 < add ? 1ull : 0ull;
        lo += t2;
        hi += up + (lo < t2 ? 1ull : 0ull);
    }
}

// Optional phase clocks (compiled only with -DPMPM_PHASE_CLOCKS): cycles of
// each warp from mark to mark, summed over the CTAs and layers of a launch
// (read back and cleared through pmpm_debug_phases).
#ifdef PMPM_PHASE_CLOCKS
constexpr int kMarks = 12;
__device__ unsigned long long g_phase[8 * kMarks];
#define PMPM_MARK(k)                                 \
    do {                                             \
        const long long now = clock64();             \
        phase[k] += now - last;                      \
        last = now;                                  \
    } while (0)
#else
#define PMPM_MARK(k) \
    do {             \
    } while (0)
#endif

// ------------------------------------------------------------------ the walk
template <bool LM, int PB>
__global__ void __launch_bounds__(kColThreads, 2) k_column(const ColParams CP) {
    chain_begin();
    extern __shared__ __align__(16) unsigned char col_smem[];
    ColShared& S = *reinterpret_cast<ColShared*>(col_smem);
    const TileParams& P = CP.t;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int col = blockIdx.x % (P.nt * P.nt), seg = blockIdx.x / (P.nt * P.nt);
    const TileGeom g = tile_geom(col, P.nc, P.nt);   // its z range is not used
    const int zs = seg * CP.lz, ze = min(P.nc, zs + CP.lz);
    const int nx = g.T[0] + 2, ny = g.T[1] + 2;      // 18 or 22
    const int rny = 65536 / ny + 1;
    const float sigma = *P.sigma;
    const float kick = P.mode >= 1 ? P.kd[0] : 0.f, drift = P.mode >= 1 ? P.kd[1] : 0.f;

    if (warp == 0) tmem_alloc(&S.tmem);
    S.Td[tid] = P.Tdec[tid];
    for (int i = tid; i < kColSlots * kColDens / 4; i += kColThreads)
        reinterpret_cast<uint4*>(S.A)[i] = make_uint4(0u, 0u, 0u, 0u);
    if (tid == 0) {
        S.cmax[(zs - 3) & 3] = 0;
        S.next = S.dep = 0;
    }
    __syncthreads();
    const uint32_t tm = S.tmem + ((uint32_t)(32 * (warp & 3)) << 16) + (uint32_t)(128 * (warp >> 2));
    for (int s = 0; s < 2; ++s) col_taps_init(warp + 8 * s, lane, CP.table, tm + kTmemPoint * s);
    tmem_wait_st();

    unsigned long long lo = 0, hi = 0;
    // ring slots of planes 4 l - 1 (density) and 4 l - 13 (force), always even; the
    // walk starts one layer early, with the deposit of layer zs - 2 alone
    int ab = 2, ob = 2;
#ifdef PMPM_PHASE_CLOCKS
    long long phase[kMarks] = {0}, last = clock64();
#endif
    // the 32 own particles that a warp gathers first: a layer of 8 a cell has
    // 6 full groups and a part of one, and warp 7 builds the tables
    const int chunk = warp < 2 ? 5 + warp : (warp < 4 ? 1 + warp : (warp < 7 ? warp - 4 : 7));
    ColOwn own;
    own.j = -1;
    // Layer l: its particles are deposited; planes 4l-1 .. 4l+2 are complete.
    for (int l = zs - 3; l <= ze + 2; ++l) {
        const bool fwd = l > zs - 3 && l <= ze + 1;   // the segment's planes end at 4 ze + 5
        const bool emit = fwd && l > zs;              // force planes 4l-7 .. 4l-4
        // A. forward transforms (4, then 2 warps), the tables of layer l + 1, F_l of
        //    coarse plane l - 1; force, kick and drift of layer l - 3
        float fl[5];
        if (warp < 4) {
            if (fwd) {
                col_fwd_x(S.A + slot6(ab, warp) * kColDens + lane * kColPitch);
                asm volatile("bar.sync 1, 128;" ::: "memory");
                if (warp < 2)
                    col_fwd_y(reinterpret_cast<float2*>(S.A + slot6(ab, 2 * warp + (lane >> 4)) * kColDens) +
                              (lane & 15));
            }
        } else if (warp == 7) {
            if (l <= ze) {
                const ColCells cells = col_cells_load(lane, g, P, l + 1);
                col_cells_store(lane, g, cells, S, l + 1);
            }
        } else if (warp == 6) {
            if (l >= zs && l <= ze + 1) col_fl_load(lane, g, P, l - 1, fl);
        }
        if (l - 3 >= zs) {
            const int total = S.own[(l - 3) & 7].pre[kColOwn];
            for (;;) {
                if (own.j >= 0) col_gather<LM, PB>(own, l - 3, g, P, S, ob, sigma, kick, drift, lo, hi);
                // more than a particle a thread: the rest, 32 at a time
                if (total <= kColThreads) break;
                int v = 0;
                if (lane == 0) v = atomicAdd(&S.next, 32);
                v = kColThreads + __shfl_sync(0xffffffffu, v, 0);
                if (v >= total) break;
                col_own_load<PB>(v + lane, l - 3, g, P, S, own);
            }
        }
        if (warp == 6 && l >= zs && l <= ze + 1) col_fl_store(lane, fl, S.fl[(l - 1) & 3]);
        PMPM_MARK(0);
        if (l > ze + 1) break;
        __syncthreads();
        PMPM_MARK(1);
        // B. the sum along z
        if (fwd) {
            float2* const C = reinterpret_cast<float2*>(S.A);
            col_zsum(warp, lane, C + ab * (kColDens / 2), C + slot6(ab, 2) * (kColDens / 2),
                     S.O + ob * (kColPlane / 2), S.O + slot6(ob, 2) * (kColPlane / 2), tm, emit);
        }
        if (tid == 0) S.next = S.dep = 0;
        PMPM_MARK(2);
        __syncthreads();
        PMPM_MARK(3);
        // C. inverse transforms, two warps a component, and deposit of layer l + 1, most of
        //    it by the other two; its first particles are loaded before the transforms
        const int total = l <= ze ? S.halo.pre[kColHalo] : 0;
        const bool check = max(S.cmax[(l + 1) & 3], S.cmax[l & 3]) > 255;
        const int ndep = warp < 6 ? kColDepBusy : kColDepFree;
        const int vdep = 32 * (warp < 6 ? 2 * kColDepFree + kColDepBusy * warp : kColDepFree * (warp - 6)) + lane;
        ColBins<PB> r[kColDepFree];
#pragma unroll
        for (int u = 0; u < kColDepFree; ++u) {
            r[u] = {0xff000000u, 0u};
            if (u < ndep && vdep - lane + 32 * u < total && !check)
                r[u] = col_bins_load<true, PB>(vdep + 32 * u, total, P, S.halo);
        }
        if (warp < 6) {
            if (emit) {
                float2* const W = S.O + (warp >> 1) * (kColSlots * kColPlane / 2);
                col_inv_y(ny, W + slot6(ob, (tid >> 4) & 3) * (kColPlane / 2) + (tid & 15));
                asm volatile("bar.sync %0, 64;" ::"r"(2 + (warp >> 1)) : "memory");
                PMPM_MARK(4);
                for (int w = tid & 63; w < 4 * ny; w += 64) {
                    const int q = w * rny >> 16;   // w / ny
                    col_inv_x(nx, W + slot6(ob, q) * (kColPlane / 2) + qidx(0, w - q * ny));
                }
                PMPM_MARK(5);
            }
        }
        PMPM_MARK(6);
        ab = slot6(ab, 4);
        ob = slot6(ob, 4);
        if (check) {
            col_deposit_checked<PB>(warp, lane, total, P, S, ab);
        } else {
            for (int u = 0;; ++u) {
                if (u < ndep) {
                    col_deposit<false, PB>(r[0], S.A, ab, P.err);
#pragma unroll
                    for (int k = 1; k < kColDepFree; ++k) r[k - 1] = r[k];
                    continue;
                }
                if (total <= kColDepStatic) break;
                int v = 0;
                if (lane == 0) v = atomicAdd(&S.dep, 32);
                v = kColDepStatic + __shfl_sync(0xffffffffu, v, 0);
                if (v >= total) break;
                r[0] = col_bins_load<false, PB>(v + lane, total, P, S.halo);
                u = ndep - 2;   // deposit it, then come back
            }
        }
        PMPM_MARK(7);
        if (l - 2 >= zs) col_own_load<PB>(32 * chunk + lane, l - 2, g, P, S, own);
        PMPM_MARK(8);
        __syncthreads();
        PMPM_MARK(9);
    }
#ifdef PMPM_PHASE_CLOCKS
    phase[10] = ze - zs + 5;
    if (lane == 0)
        for (int k = 0; k < kMarks; ++k) atomicAdd(&g_phase[warp * kMarks + k], (unsigned long long)phase[k]);
#endif
    __syncthreads();
    if (warp == 0) tmem_free(S.tmem);
    if (P.mode == 1) {
        // 128-bit sum of the new momenta's squares over the CTA
        unsigned long long* sh = reinterpret_cast<unsigned long long*>(S.O);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const unsigned long long l2 = __shfl_down_sync(0xffffffffu, lo, o);
            const unsigned long long h2 = __shfl_down_sync(0xffffffffu, hi, o);
            lo += l2;
            hi += h2 + (lo < l2 ? 1ull : 0ull);
        }
        if (lane == 0) {
            sh[2 * warp] = lo;
            sh[2 * warp + 1] = hi;
        }
        __syncthreads();
        if (tid == 0) {
            lo = 0;
            hi = 0;
            for (int w = 0; w < kColThreads / 32; ++w) {
                lo += sh[2 * w];
                hi += sh[2 * w + 1] + (lo < sh[2 * w] ? 1ull : 0ull);
            }
            add128_digits(P.d2, lo, hi);
        }
    }
}

}  // namespace

void column_setup() {
    const int bytes = (int)sizeof(ColShared);
    cudaFuncSetAttribute(k_column<false, 1>, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
    cudaFuncSetAttribute(k_column<false, 2>, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
    cudaFuncSetAttribute(k_column<true, 1>, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
}

// Layers of a segment.  A CTA walks lz layers and 5.5 more to fill its 11
// planes; a layer takes 16k cycles with two CTAs on the SM and 12k alone
// (measured), so the last 152 CTAs or fewer run at 0.74 of the time.  The
// shortest walk: 128^3 particles on 64^3 cells lz = 22 (404 us; 469 at 6, 407 at 11, 567 at
// 64), 256^3 on 128^3 64 (2.52 ms; 2.78 at 16, 2.58 at 43, 2.84 at 128), 512^3 on 256^3 256
// (18.8 ms; 19.7 at 43, 19.3 at 64).
//
// Where other boxes fill the SMs (sharers of them in all), the last CTAs of a pass cost
// nothing and what counts is the sum of all walks: longer ones, but none that would take
// 1.3 times as long alone.  Sixteen boxes of 32^3 to 128^3 particles 23.7 -> 22.5 ms; 400
// requests as they come at 1.5 times the capacity, p99 1.98 -> 1.85 s.  A captured step
// keeps the segments of the time of its capture (engines with graphs on); results do
// not depend on them.
static int column_layers(int nc, int nt, int sharers) {
    const auto ctas = [=](int lz) { return (int64_t)nt * nt * ((nc + lz - 1) / lz); };
    const auto alone = [=](int lz) {
        const int64_t n = ctas(lz), rest = n % 304;
        return ((double)(n / 304) + (rest == 0 ? 0.0 : (rest <= 152 ? 0.74 : 1.0))) * (lz + 5.5);
    };
    double least = 1e30, cost = 1e30;
    for (int lz = 1; lz <= nc; ++lz) least = std::min(least, alone(lz));
    int best = nc;
    for (int lz = 1; lz <= nc; ++lz) {
        if (alone(lz) > (sharers > 1 ? 1.3 : 1.0) * least) continue;
        const double c = alone(lz) + (sharers - 1) * (double)ctas(lz) / 304 * (lz + 5.5);
        if (c < cost) {
            cost = c;
            best = lz;
        }
    }
    return best;
}

void column_pass(cudaStream_t st, const TileParams& P, const float* table, bool lowmem, int pb, bool chained,
                 int sharers) {
    ColParams C;
    C.t = P;
    C.table = table;
    C.lz = column_layers(P.nc, P.nt, sharers);
    const unsigned grid = (unsigned)(P.nt * P.nt * ((P.nc + C.lz - 1) / C.lz));
    if (lowmem) chain(chained, k_column<true, 1>, grid, kColThreads, sizeof(ColShared), st, C);
    else if (pb == 2) chain(chained, k_column<false, 2>, grid, kColThreads, sizeof(ColShared), st, C);
    else chain(chained, k_column<false, 1>, grid, kColThreads, sizeof(ColShared), st, C);
}

}  // namespace pmpm

#ifdef PMPM_PHASE_CLOCKS
extern "C" int pmpm_debug_phases(unsigned long long* out, int n) {
    static const unsigned long long zero[8 * pmpm::kMarks] = {0};
    const cudaError_t e = cudaMemcpyFromSymbol(out, pmpm::g_phase, sizeof(unsigned long long) * n);
    return e ? (int)e : (int)cudaMemcpyToSymbol(pmpm::g_phase, zero, sizeof(zero));
}
#endif
