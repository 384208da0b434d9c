// Launches and splits of the FP64 products of one to four columns (few_cols.cuh).
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>

#include "few_cols.cuh"
#include "internal.h"

namespace hdf {
namespace {

constexpr int kSMs = 152;
constexpr int kMaxPart = 1024;   // row chunks of U^T V

template <int C>
__global__ void __launch_bounds__(256) k_few_utv(const double* __restrict__ U, int64_t ldU, int64_t n, int64_t r,
                                                 const double* __restrict__ V, int64_t ldv, int64_t chunk,
                                                 int tx_log2, double* __restrict__ part) {
    const int64_t i0 = blockIdx.x * chunk;
    few::few_utv_block<C>(U, ldU, r, V, ldv, i0, min(n, i0 + chunk), blockIdx.y, tx_log2,
                          part + (int64_t)blockIdx.x * C * r);
}

template <int C, int R>
__global__ void __launch_bounds__(256) k_few_uw(const double* __restrict__ U, int64_t ldU, int64_t n, int64_t r,
                                                const double* __restrict__ W, double alpha,
                                                const double* __restrict__ B, int64_t ldb, double beta,
                                                double* __restrict__ Y, int64_t ldy, int ks_log2) {
    few::few_uw_block<C, R>(U, ldU, n, r, W, alpha, B, ldb, beta, Y, ldy, ks_log2, blockIdx.x);
}

// Threads across the columns of a U^T V block (a power of two, 32 .. 256).
int utv_tx_log2(int64_t r) {
    int l = 5;
    while (l < 8 && ((int64_t)2 << l) < r) ++l;
    return l;
}

}  // namespace

// Row chunks of U^T V: about 16 blocks per SM (four waves of four) when the rows allow it, at
// least 16 rows per thread, and partial sums of at most 1/16 of U's own bytes once there are
// enough rows for the chip.  5,000 x 35,048: 18 chunks; 2,000 x 456: 125 chunks.
void few_utv_split(int64_t n, int64_t r, int c, int64_t* chunk, int* nchunk) {
    const int l = utv_tx_log2(r);
    const int64_t cols = (r + (2 << l) - 1) / (2 << l), ty = 256 >> l;
    int64_t k = std::max<int64_t>(1, 16 * kSMs / cols);
    k = std::min<int64_t>({k, (n + 16 * ty - 1) / (16 * ty), (int64_t)kMaxPart});
    const int64_t fill = std::max<int64_t>(1, 2 * kSMs / cols);          // two blocks per SM
    k = std::max<int64_t>(std::min(k, fill), std::min<int64_t>(k, n / (16 * (int64_t)c)));
    *chunk = (n + k - 1) / k;
    *nchunk = (int)((n + *chunk - 1) / *chunk);
}

hdf_status few_utv(const double* U, int64_t ldU, int64_t n, int64_t r, const double* V, int64_t ldv, int c,
                   int64_t chunk, int nchunk, double* part, cudaStream_t st) {
    const int l = utv_tx_log2(r);
    const dim3 g((unsigned)nchunk, (unsigned)((r + (2 << l) - 1) / (2 << l)));
    HDF_COUNT_LAUNCH();
    switch (c) {
        case 1: k_few_utv<1><<<g, 256, 0, st>>>(U, ldU, n, r, V, ldv, chunk, l, part); break;
        case 2: k_few_utv<2><<<g, 256, 0, st>>>(U, ldU, n, r, V, ldv, chunk, l, part); break;
        case 3: k_few_utv<3><<<g, 256, 0, st>>>(U, ldU, n, r, V, ldv, chunk, l, part); break;
        case 4: k_few_utv<4><<<g, 256, 0, st>>>(U, ldU, n, r, V, ldv, chunk, l, part); break;
        default: return fail(HDF_EINVAL, "few_utv: 1 <= c <= 4");
    }
    HDF_CUDA(cudaGetLastError());
    return HDF_OK;
}

hdf_status few_uw(const double* U, int64_t ldU, int64_t n, int64_t r, const double* W, int c, double alpha,
                  const double* B, int64_t ldb, double beta, double* Y, int64_t ldy, cudaStream_t st) {
    const int R = c <= 2 ? 8 : 4;
    // warps per row group: split the columns until the chip has about 16 warps per SM, at least
    // two 64-column steps per warp
    const int64_t groups = (n + R - 1) / R;
    int l = 0;
    while (l < 3 && (groups << l) < 16 * kSMs && r > ((int64_t)128 << l)) ++l;
    const int64_t per = 8 >> l;
    const unsigned g = (unsigned)((groups + per - 1) / per);
    HDF_COUNT_LAUNCH();
    switch (c) {
        case 1: k_few_uw<1, 8><<<g, 256, 0, st>>>(U, ldU, n, r, W, alpha, B, ldb, beta, Y, ldy, l); break;
        case 2: k_few_uw<2, 8><<<g, 256, 0, st>>>(U, ldU, n, r, W, alpha, B, ldb, beta, Y, ldy, l); break;
        case 3: k_few_uw<3, 4><<<g, 256, 0, st>>>(U, ldU, n, r, W, alpha, B, ldb, beta, Y, ldy, l); break;
        case 4: k_few_uw<4, 4><<<g, 256, 0, st>>>(U, ldU, n, r, W, alpha, B, ldb, beta, Y, ldy, l); break;
        default: return fail(HDF_EINVAL, "few_uw: 1 <= c <= 4");
    }
    HDF_CUDA(cudaGetLastError());
    return HDF_OK;
}

}  // namespace hdf
