// power.cuh -- the power spectrum of a cell-ordered store on caller-supplied
// buffers (power.cu), shared by the two entry points.
#pragma once

#include "pmpm_impl.cuh"

namespace pmpm {

struct PkStore {
    int nc, pb;                  // coarse cells per side, bytes per position bin
    int64_t n;
    const int64_t* offsets;      // [nc^3 + 1]
    const int32_t* counts;       // [nc^3]
    const uint8_t* m[3];         // position bins, storage order
    bool chained;                // launches may overlap (chain())
};

// Enqueues P(k) sums of `st` on an nmesh^3 mesh (a power of two from nc to 4 nc,
// at least 8): bins[0..nbins) sum of P, then of |k|, then modes, per shell, then one
// double more: *err as the stream finds it.
// mesh: 8 nmesh^3 bytes; delta: 4 nmesh^3 bytes more, or null (nmesh up to 1024).
// tw: exp(-2 pi i k / tw_n), nmesh dividing tw_n.  launches: added to.
cudaError_t pk_enqueue(cudaStream_t stream, const PkStore& st, int nmesh, int nbins, float2* mesh,
                       float* delta, double* bins, const uint32_t* err, const float2* tw, int tw_n, int64_t* launches);
void pk_setup();

// offsets[0..nc^3] of `counts` (sort.cu); sums: kScanSums words
void scan_raw(cudaStream_t stream, bool chained, int64_t ncells, const int32_t* counts, long long* sums, int64_t* offsets,
              int64_t n, uint32_t* err, int64_t* launches);
// in place, forward or back, for sizes without a fused pass (fft.cu)
cudaError_t fft3d_float_raw(cudaStream_t st, float2* data, int n, int sign, const float2* tw, int tw_n);

}  // namespace pmpm
