// K~V of FP64 factors for one to four columns: streaming products on the FP64 pipe (block bodies,
// launched by few_cols.cu and, over the sets of a batch, by batched.cu).
//
// What bounds them.  An FP64 multiply-add per column and 8-byte entry of U: at one column the
// FP64 pipe (2 multiply-adds per clock and SM) takes 16 bytes of U per clock and SM, 0.7 of the
// copy bandwidth, so both kernels have to keep memory and the pipe busy at once and must not
// spend FP64 operations on anything else (a warp-wide FP64 add costs as much as 32 entries).
// The register-tiled kernels of the wider blocks (k_utv_tile, k_uw_tile) put 128-256 rows or
// columns and a 2,048-row chunk on one block, which leaves most of the chip idle at the small
// sizes: 5,000 points x 35,048 columns, one column, U W on 20 blocks 7.90 ms, U^T V 0.52 ms;
// 2,000 points x 456 columns 0.063 ms and, on 2 blocks, 0.255 ms.  Here: 0.46, 0.31, 0.008 and
// 0.010 ms; at 100,000 x 10,680 U^T V 1.79 ms (4.8 TB/s, the pipe's rate at one column) and U W
// 1.91 ms, 3.50 and 3.81 ms at two columns.
#pragma once
#include <cuda_runtime.h>

#include <cstdint>

namespace hdf {
namespace few {

constexpr int kVTile = 256;      // rows of V staged per tile of U^T V

// part_chunk[j r + a] = sum over i0 <= i < i1 of U[i, a] V[i + j ldv] by one 256-thread block.  A thread owns
// two neighbouring columns (one 16-byte load per row, 8 rows in flight); tx_log2 threads span the
// columns of a block, the remaining threads split its rows and are added in shared memory.
template <int C>
__device__ __forceinline__ void few_utv_block(const double* __restrict__ U, int64_t ldU, int64_t r,
                                              const double* __restrict__ V, int64_t ldv, int64_t i0, int64_t i1,
                                              int64_t colblk, int tx_log2, double* __restrict__ part_chunk) {
    __shared__ double Vs[C][kVTile];
    __shared__ double red[256 * 2 * C];
    const int t = threadIdx.x;
    const int TX = 1 << tx_log2, TY = 256 >> tx_log2;
    const int tx = t & (TX - 1), ty = t >> tx_log2;
    const int64_t a = 2 * (colblk * TX + tx);
    const bool act = a < r;
    const double* Ua = U + (act ? a : 0);
    double acc[C][2];
#pragma unroll
    for (int j = 0; j < C; ++j) acc[j][0] = acc[j][1] = 0.0;
    for (int64_t t0 = i0; t0 < i1; t0 += kVTile) {
        const int cnt = (int)min((int64_t)kVTile, i1 - t0);
        __syncthreads();
        if (t < cnt) {
#pragma unroll
            for (int j = 0; j < C; ++j) Vs[j][t] = V[t0 + t + (int64_t)j * ldv];
        }
        __syncthreads();
        if (act) {
            const double* Ut = Ua + t0 * ldU;
#pragma unroll 8
            for (int k = ty; k < cnt; k += TY) {
                const double2 u = __ldcs(reinterpret_cast<const double2*>(Ut + (int64_t)k * ldU));
#pragma unroll
                for (int j = 0; j < C; ++j) {
                    acc[j][0] = fma(u.x, Vs[j][k], acc[j][0]);
                    acc[j][1] = fma(u.y, Vs[j][k], acc[j][1]);
                }
            }
        }
    }
    if (TY > 1) {
#pragma unroll
        for (int j = 0; j < C; ++j) {
            red[(2 * j) * 256 + t] = acc[j][0];
            red[(2 * j + 1) * 256 + t] = acc[j][1];
        }
        __syncthreads();
        if (ty == 0) {
            for (int y = 1; y < TY; ++y)
#pragma unroll
                for (int j = 0; j < C; ++j) {
                    acc[j][0] += red[(2 * j) * 256 + y * TX + tx];
                    acc[j][1] += red[(2 * j + 1) * 256 + y * TX + tx];
                }
        }
    }
    if (act && ty == 0) {
#pragma unroll
        for (int j = 0; j < C; ++j)
            *reinterpret_cast<double2*>(part_chunk + (int64_t)j * r + a) =
                make_double2(acc[j][0], acc[j][1]);
    }
}

// Y[i + j ldy] = alpha sum_a U[i, a] W[a C + j] + beta B[i + j ldb].  A warp owns R rows (so that
// one load of W serves R rows) and every KS-th 64-column step of them; lane l takes two columns
// of a step.  The R row sums leave the warp by a halving butterfly (R - 1 + log2(32 / R) FP64 adds
// per column instead of 5 R), and the KS warps of a row group are added in shared memory.
template <int C, int R>
__device__ __forceinline__ void few_uw_block(const double* __restrict__ U, int64_t ldU, int64_t n, int64_t r,
                                             const double* __restrict__ W, double alpha, const double* __restrict__ B,
                                             int64_t ldb, double beta, double* __restrict__ Y, int64_t ldy, int ks_log2,
                                             int64_t blk) {
    __shared__ double red[8][R * C];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int KS = 1 << ks_log2, G = 8 >> ks_log2;            // warps per row group, row groups per block
    const int grp = warp >> ks_log2, ks = warp & (KS - 1);
    const int64_t row0 = (blk * G + grp) * R;
    const double* Ur[R];
#pragma unroll
    for (int q = 0; q < R; ++q) Ur[q] = U + min(row0 + q, n - 1) * ldU;
    double acc[C][R];
#pragma unroll
    for (int j = 0; j < C; ++j)
#pragma unroll
        for (int q = 0; q < R; ++q) acc[j][q] = 0.0;
    for (int64_t a = 2 * (ks * 32 + lane); a < r; a += 64 * KS) {
        double2 u[R];
#pragma unroll
        for (int q = 0; q < R; ++q) u[q] = __ldcs(reinterpret_cast<const double2*>(Ur[q] + a));
        double w[2 * C];
#pragma unroll
        for (int j = 0; j < C; ++j) {
            const double2 v = *reinterpret_cast<const double2*>(W + a * C + 2 * j);
            w[2 * j] = v.x;
            w[2 * j + 1] = v.y;
        }
#pragma unroll
        for (int j = 0; j < C; ++j)
#pragma unroll
            for (int q = 0; q < R; ++q) acc[j][q] = fma(u[q].y, w[C + j], fma(u[q].x, w[j], acc[j][q]));
    }
#pragma unroll
    for (int j = 0; j < C; ++j) {
        int o = 16;
#pragma unroll
        for (int h = R / 2; h >= 1; h /= 2, o /= 2) {
#pragma unroll
            for (int k = 0; k < h; ++k) {
                const bool up = (lane & o) != 0;
                const double send = up ? acc[j][k] : acc[j][k + h];
                const double keep = up ? acc[j][k + h] : acc[j][k];
                acc[j][k] = keep + __shfl_xor_sync(0xffffffffu, send, o);
            }
        }
        for (; o >= 1; o /= 2) acc[j][0] += __shfl_xor_sync(0xffffffffu, acc[j][0], o);
        // lane l now holds the row whose bits, from the top, are the top log2(R) bits of l
        if ((lane & (32 / R - 1)) == 0) red[warp][(lane / (32 / R)) * C + j] = acc[j][0];
    }
    __syncthreads();
    const int e = threadIdx.x;
    if (e < G * R * C) {
        const int g = e / (R * C), q = (e / C) % R, j = e % C;
        double s = 0.0;
        for (int k = 0; k < KS; ++k) s += red[g * KS + k][q * C + j];
        const int64_t i = (blk * G + g) * R + q;
        if (i < n) {
            double out = alpha * s;
            if (B) out += beta * B[i + (int64_t)j * ldb];
            Y[i + (int64_t)j * ldy] = out;
        }
    }
}

}  // namespace few
}  // namespace hdf
