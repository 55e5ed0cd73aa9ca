// noalloc.cu -- a power spectrum entry point that allocates no device
// memory.  Its scratch (cell offsets, the density / spectrum mesh, shell sums
// and FFT twiddles) is one file-scope device array of fixed size, so the
// entry point serves boxes of at most kNaMaxNc coarse cells per side and
// meshes of at most kNaMaxMesh points per side.  The computation follows
// pmpm_power_spectrum step for step.
#include <mutex>

#include "power.cuh"

namespace pmpm {

namespace {

constexpr int kNaMaxNc = 64;
constexpr int kNaMaxMesh = 64;
constexpr int kNaMaxBins = kNaMaxMesh / 2;
constexpr int kNaMaxDevices = 64;
constexpr size_t kNaOffsetsBytes = 8 * ((size_t)kNaMaxNc * kNaMaxNc * kNaMaxNc + 1);
constexpr size_t kNaMeshBytes = 8 * (size_t)kNaMaxMesh * kNaMaxMesh * kNaMaxMesh;
constexpr size_t kNaBinsBytes = 8 * 3 * kNaMaxBins + 16;   // and the scan's error word, twice
constexpr size_t kNaTwBytes = 8 * kNaMaxMesh;
constexpr size_t kA = 256;
constexpr size_t kNaOffOffsets = 0;
constexpr size_t kNaOffMesh = (kNaOffOffsets + kNaOffsetsBytes + kA - 1) / kA * kA;
constexpr size_t kNaOffBins = (kNaOffMesh + kNaMeshBytes + kA - 1) / kA * kA;
constexpr size_t kNaOffTw = (kNaOffBins + kNaBinsBytes + kA - 1) / kA * kA;
constexpr size_t kNaOffSums = (kNaOffTw + kNaTwBytes + kA - 1) / kA * kA;
constexpr size_t kNaSumsBytes = 8 * (size_t)kNaMaxNc * kNaMaxNc * kNaMaxNc / 256;
constexpr size_t kNaBytes = (kNaOffSums + kNaSumsBytes + kA - 1) / kA * kA;   // about 4.2 MB

// Shared by every call on a device; it keeps the last call's contents.
static __device__ __align__(256) unsigned char g_noalloc_scratch[kNaBytes];

std::mutex g_na_lock;
unsigned char* g_na_ptr[kNaMaxDevices] = {nullptr};

__global__ void k_na_twiddles(int n, float2* tw) {
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= n) return;
    double sv, cv;
    sincospi(2.0 * (double)k / (double)n, &sv, &cv);
    tw[k] = make_float2((float)cv, (float)-sv);
}

char g_na_msg[256] = "";

int na_fail(int code, const char* msg) {
    snprintf(g_na_msg, sizeof(g_na_msg), "%s", msg);
    return code;
}

// One-time set-up on the current device: find the scratch array's device
// address and fill the twiddle table.  Runs on the first call per device.
int na_scratch(cudaStream_t st, unsigned char** out) {
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kNaMaxDevices)
        return na_fail(PMPM_ECUDA, "no usable CUDA device");
    std::lock_guard<std::mutex> lock(g_na_lock);
    if (!g_na_ptr[dev]) {
        void* p = nullptr;
        const cudaError_t e = cudaGetSymbolAddress(&p, g_noalloc_scratch);
        if (e != cudaSuccess || !p) {
            char m[200];
            snprintf(m, sizeof(m), "cudaGetSymbolAddress: %s", cudaGetErrorString(e));
            return na_fail(PMPM_ECUDA, m);
        }
        unsigned char* base = static_cast<unsigned char*>(p);
        pk_setup();
        k_na_twiddles<<<1, kNaMaxMesh, 0, st>>>(kNaMaxMesh, reinterpret_cast<float2*>(base + kNaOffTw));
        if (cudaGetLastError() != cudaSuccess || cudaStreamSynchronize(st) != cudaSuccess)
            return na_fail(PMPM_ECUDA, "scratch set-up failed");
        g_na_ptr[dev] = base;
    }
    *out = g_na_ptr[dev];
    return PMPM_OK;
}

}  // namespace
}  // namespace pmpm

using namespace pmpm;

extern "C" int pmpm_power_spectrum_noalloc(int32_t nc, int64_t n, const uint8_t* d_m0,
                                           const uint8_t* d_m1, const uint8_t* d_m2,
                                           const int32_t* d_counts, int32_t nmesh, int32_t nbins,
                                           double* k, double* pk, int64_t* nmodes,
                                           void* cuda_stream) {
    if (nc < 8 || nc > kNaMaxNc || (nc & (nc - 1)))
        return na_fail(PMPM_EINVAL, "nc must be a power of two in [8, 64] for the no-allocation entry point");
    const int nf = 4 * nc;
    if (nmesh < 4 || nmesh > kNaMaxMesh || (nmesh & (nmesh - 1)) || nf % nmesh)
        return na_fail(PMPM_EINVAL, "nmesh must be a power of two dividing 4*nc, at most 64");
    int lh = 0;
    while ((nmesh << lh) < nf) ++lh;
    if (lh > 2) return na_fail(PMPM_EINVAL, "nmesh below 4*nc/4 is not supported");
    if (nbins < 1 || nbins > nmesh / 2) return na_fail(PMPM_EINVAL, "nbins must be in [1, nmesh/2]");
    if (n < 1 || !d_m0 || !d_m1 || !d_m2 || !d_counts || !k || !pk || !nmodes)
        return na_fail(PMPM_EINVAL, "null pointer or empty store");
    cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
    unsigned char* base = nullptr;
    int rc = na_scratch(st, &base);
    if (rc) return rc;
    int64_t* offsets = reinterpret_cast<int64_t*>(base + kNaOffOffsets);
    double* bins = reinterpret_cast<double*>(base + kNaOffBins);
    uint32_t* err = reinterpret_cast<uint32_t*>(bins + 3 * kNaMaxBins + 1);
    const int64_t ncells = (int64_t)nc * nc * nc;
    int64_t launches = 0;
    cudaMemsetAsync(err, 0, 8, st);
    const bool chained = ncells <= kChainCells;
    scan_raw(st, chained, ncells, d_counts, reinterpret_cast<long long*>(base + kNaOffSums), offsets, n, err, &launches);
    const PkStore store = {nc, 1, n, offsets, d_counts, {d_m0, d_m1, d_m2}, chained};
    cudaError_t e = pk_enqueue(st, store, nmesh, nbins, reinterpret_cast<float2*>(base + kNaOffMesh), nullptr, bins, err,
                               reinterpret_cast<const float2*>(base + kNaOffTw), kNaMaxMesh, &launches);
    double hb[3 * kNaMaxBins + 1];
    if (e == cudaSuccess)
        e = cudaMemcpyAsync(hb, bins, sizeof(double) * (3 * nbins + 1), cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    if (e != cudaSuccess) return na_fail(PMPM_ECUDA, cudaGetErrorString(e));
    // counts that do not add up to n put particles in the wrong cells and the
    // mean density is wrong: refuse the result
    if (hb[3 * nbins] != 0.0) {
        long long total = -1;
        cudaMemcpyAsync(&total, offsets + ncells, sizeof(total), cudaMemcpyDeviceToHost, st);
        cudaStreamSynchronize(st);
        char m[160];
        snprintf(m, sizeof(m), "the counts add up to %lld, not n = %lld", total, (long long)n);
        return na_fail(PMPM_EINVAL, m);
    }
    power_spectrum_finish(hb, nbins, k, pk, nmodes);
    return PMPM_OK;
}

extern "C" const char* pmpm_noalloc_last_error(void) { return g_na_msg; }
