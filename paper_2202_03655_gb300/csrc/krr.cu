// Kernel ridge regression of Sec. 4.2 on the device: k-means clustering (Lloyd's iteration),
// the operator K^ (HDF factors of the diagonal blocks through the batched factorization, exact
// off-diagonal blocks evaluated on the fly), the block-diagonal preconditioner (inverses of the
// exact lambda I + K_{C_i C_i}) and preconditioned conjugate gradients for Eq. (opt).
// Declarations and argument contracts are in include/hdf.h.
#include <cuda_runtime.h>

#include <algorithm>
#include <chrono>
#include <cmath>
#include <cstring>
#include <functional>
#include <memory>
#include <string>
#include <vector>

#include "../../include/hdf.h"
#include "cg_state.h"
#include "hdf_kernels.cuh"
#include "internal.h"
#include "planner.h"

using namespace hdf;

namespace {

double wall_ms() {
    return std::chrono::duration<double, std::milli>(std::chrono::steady_clock::now().time_since_epoch()).count();
}

int blocks_for(int64_t work, int per_block, int cap) {
    const int64_t g = (work + per_block - 1) / per_block;
    return (int)std::max<int64_t>(1, std::min<int64_t>(g, cap));
}

// ------------------------------------------------------------------------- k-means
// Assignment step: label = nearest centre (squared distance summed over coordinates in order,
// the lowest index on ties); counts the points whose label changed.
__global__ void k_km_assign(const double* __restrict__ x, int64_t n, int d, int k, const double* __restrict__ C,
                            int* __restrict__ labels, int* __restrict__ changes) {
    extern __shared__ double Cs[];
    for (int e = threadIdx.x; e < k * d; e += blockDim.x) Cs[e] = C[e];
    __syncthreads();
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i >= n) return;
    double xi[dev::kMaxD];
    for (int j = 0; j < d; ++j) xi[j] = x[i * d + j];
    double best = INFINITY;
    int bc = 0;
    for (int c = 0; c < k; ++c) {
        double s = 0.0;
        for (int j = 0; j < d; ++j) { const double t = xi[j] - Cs[c * d + j]; s += t * t; }
        if (s < best) { best = s; bc = c; }
    }
    if (labels[i] != bc) { atomicAdd(changes, 1); labels[i] = bc; }
}

// Update step, first stage: block b sums the coordinates (and counts) of its chunks' points per
// cluster: part[(b k + c) (d + 1) + j], j = d the count.  A chunk (kKmChunk points) is staged in shared
// memory with its labels; warp w takes the clusters w, w + 8, ... and adds their points with fixed-order
// sums, from the second chunk on to what it has stored before (clusters without points in a chunk are
// passed over).  Bound by the passes over the staged labels (k chunk / 8 per warp) and the FP64 adds; 128
// points per chunk, so that a few thousand points fill the chip: with 2,048 points per block and a
// block-wide tree per cluster and coordinate it took 0.49 ms at 13,760 points, d = 8, 30 clusters (7
// blocks); now 0.010 ms.  At most kKmBlocks blocks, a block then taking several chunks: the sums stay
// below 512 k (d + 1) doubles whatever n is, and one warp per cluster can add them.
constexpr int kKmChunk = 128, kKmBlocks = 512;
__global__ void __launch_bounds__(256) k_km_partial(const double* __restrict__ x, int64_t n, int d, int k,
                                                    const int* __restrict__ labels, int64_t chunks,
                                                    double* __restrict__ part) {
    __shared__ double xs[kKmChunk * dev::kMaxD];
    __shared__ int ls[kKmChunk];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t first = blockIdx.x * chunks * kKmChunk, end = min(n, first + chunks * kKmChunk);
    for (int64_t i0 = first; i0 < end; i0 += kKmChunk) {
        const int cnt = (int)min((int64_t)kKmChunk, end - i0);
        if (i0 > first) __syncthreads();
        for (int e = threadIdx.x; e < cnt * d; e += blockDim.x) xs[e] = x[i0 * d + e];
        for (int e = threadIdx.x; e < kKmChunk; e += blockDim.x) ls[e] = e < cnt ? labels[i0 + e] : -1;
        __syncthreads();
        for (int c = warp; c < k; c += 8) {
            double* out = part + ((int64_t)blockIdx.x * k + c) * (d + 1);
            unsigned m[kKmChunk / 32], any = 0;
#pragma unroll
            for (int q = 0; q < kKmChunk / 32; ++q) any |= m[q] = __ballot_sync(0xffffffffu, ls[32 * q + lane] == c);
            if (i0 > first && !any) continue;
            // lane j <= d adds coordinate j (or 1) of the cluster's points in order
            double acc = i0 > first && lane <= d ? out[lane] : 0.0;
#pragma unroll
            for (int q = 0; q < kKmChunk / 32; ++q)
                for (unsigned w = m[q]; w; w &= w - 1) {
                    const int e = 32 * q + __ffs(w) - 1;
                    if (lane < d) acc += xs[e * d + lane];
                    else if (lane == d) acc += 1.0;
                }
            if (lane <= d) out[lane] = acc;
        }
    }
}

// Update step, second stage: centre c = mean of its points (one warp per cluster; lanes take the
// blocks in turn, then a fixed butterfly); a centre without points stays where it is.
__global__ void k_km_finish(const double* __restrict__ part, int G, int k, int d, double* __restrict__ C) {
    const int c = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
    if (c >= k) return;
    double s[dev::kMaxD + 1];
#pragma unroll
    for (int j = 0; j <= dev::kMaxD; ++j) s[j] = 0.0;
    for (int b = lane; b < G; b += 32)
#pragma unroll
        for (int j = 0; j <= dev::kMaxD; ++j)
            if (j <= d) s[j] += part[((int64_t)b * k + c) * (d + 1) + j];
#pragma unroll
    for (int j = 0; j <= dev::kMaxD; ++j)
        for (int o = 16; o > 0; o >>= 1) s[j] += __shfl_xor_sync(0xffffffffu, s[j], o);
    double count = 0.0;
#pragma unroll
    for (int j = 0; j <= dev::kMaxD; ++j)
        if (j == d) count = s[j];
    if (lane == 0 && count > 0.0)
#pragma unroll
        for (int j = 0; j < dev::kMaxD; ++j)
            if (j < d) C[c * d + j] = s[j] / count;
}

__global__ void k_gather_rows(const double* __restrict__ x, int d, const int64_t* __restrict__ idx, int64_t m,
                              double* __restrict__ out) {
    const int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (e >= m * d) return;
    const int64_t r = e / d;
    out[e] = x[idx[r] * d + (e % d)];
}

// --------------------------------------------------------- direct kernel evaluation
constexpr int kDkRows = 128;     // rows (outputs) per block
constexpr int kDkTile = 128;     // columns staged per tile

// part[s m + i] = sum over columns j of split s of k(|a_i - b_j|) w_j, skipping j with
// cb[j] == ca[i] when ca is given (the off-diagonal blocks of K^).  Coordinates are FP32 copies
// shifted by a common point and the kernel values k_ij are FP32 (one fixed, exactly symmetric
// matrix); w_j = w_hi + w_lo as two FP32 numbers, each product k_ij w_hi formed exactly (fma)
// and the sums of one tile kept as FP32 pairs (TwoSum), so that the product is linear in w to
// about 1e-14 -- conjugate gradients need the same linear operator in every iteration.  Tiles
// are added in FP64 in column order.
template <int DD>
__global__ void __launch_bounds__(kDkRows) k_direct_kernel(const float* __restrict__ a, int64_t m,
                                                          const float* __restrict__ b, int64_t n, int kernel,
                                                          float inv_ell, const double* __restrict__ w,
                                                          const int* __restrict__ ca, const int* __restrict__ cb,
                                                          int64_t split, double* __restrict__ part) {
    constexpr int U = 4;                         // independent accumulators (pairs in flight)
    __shared__ float bs[kDkTile][DD];
    __shared__ float ws[kDkTile], wl[kDkTile];
    __shared__ int cs[kDkTile];
    const int64_t i = blockIdx.x * (int64_t)kDkRows + threadIdx.x;
    const bool act = i < m;
    float ai[DD];
#pragma unroll
    for (int j = 0; j < DD; ++j) ai[j] = act ? a[i * DD + j] : 0.f;
    const int myc = (ca && act) ? ca[i] : -1;
    const int64_t j0 = blockIdx.y * split, j1 = min(n, j0 + split);
    double acc = 0.0;
    for (int64_t t0 = j0; t0 < j1; t0 += kDkTile) {
        const int nt = (int)min((int64_t)kDkTile, j1 - t0);
        __syncthreads();
        for (int e = threadIdx.x; e < kDkTile * DD; e += blockDim.x) {
            const int r = e / DD, q = e % DD;
            bs[r][q] = (r < nt) ? b[(t0 + r) * DD + q] : 0.f;
        }
        for (int r = threadIdx.x; r < kDkTile; r += blockDim.x) {
            const double wv = (r < nt) ? w[t0 + r] : 0.0;
            const float hi = (float)wv;
            ws[r] = hi;
            wl[r] = (float)(wv - (double)hi);
            cs[r] = (r < nt && cb) ? cb[t0 + r] : -2;        // rows past the tile carry w = 0
        }
        __syncthreads();
        float sh_[U], sl_[U];                    // tile sums as unevaluated FP32 pairs
#pragma unroll
        for (int u = 0; u < U; ++u) sh_[u] = sl_[u] = 0.f;
        const int ntu = (nt + U - 1) / U * U;    // the padded tail adds exact zeros (w = 0, k <= 1)
        for (int r0 = 0; r0 < ntu; r0 += U) {
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const int r = r0 + u;
                float s = 0.f;
#pragma unroll
                for (int q = 0; q < DD; ++q) { const float t = ai[q] - bs[r][q]; s = fmaf(t, t, s); }
                float kv = dev::kernel_value_f(kernel, sqrtf(s), inv_ell);
                kv = (cs[r] == myc) ? 0.f : kv;
                const float p = kv * ws[r];
                const float e = fmaf(kv, wl[r], fmaf(kv, ws[r], -p));    // exact error of p, plus k w_lo
                float t1, t2;
                dev::two_sum(sh_[u], p, t1, t2);
                sh_[u] = t1;
                sl_[u] += t2 + e;
            }
        }
#pragma unroll
        for (int u = 0; u < U; ++u) acc += (double)sh_[u] + (double)sl_[u];
    }
    if (act) part[blockIdx.y * m + i] = acc;
}

// Launch of k_direct_kernel for the dimension d.
void launch_direct(int d, dim3 g, cudaStream_t st, const float* a, int64_t m, const float* b, int64_t n, int kernel,
                   float inv_ell, const double* w, const int* ca, const int* cb, int64_t split, double* part) {
#define HDF_DK(DD)                                                                                         \
    case DD:                                                                                               \
        k_direct_kernel<DD><<<g, kDkRows, 0, st>>>(a, m, b, n, kernel, inv_ell, w, ca, cb, split, part);   \
        break;
    switch (d) { HDF_DK(1) HDF_DK(2) HDF_DK(3) HDF_DK(4) HDF_DK(5) HDF_DK(6) HDF_DK(7) HDF_DK(8) }
#undef HDF_DK
}

// The off-diagonal blocks of K^ stored once, each pair {i, j} in one place: tiles of kTI points i and
// kTJ points j that meet j < i, tile (ib, jb) as [j][i] at index 2 ib (ib + 1) + jb, jb < 4 (ib + 1); the
// FP32 value that k_direct_kernel forms for the pair, zero within a cluster, for j >= i and in the
// padding.  A conjugate-gradient solve applies the same matrix hundreds of times, and forming a value
// (d differences, a square root, an exponential) costs several times the bytes of reading it: 13,760
// points, d = 8, one product 0.43 ms evaluated, 0.12 ms from the full matrix,
// 0.095 from these tiles; 0.19 ms to store them.
constexpr int kTI = 512, kTJ = 128, kTPart = kTI + kTJ;
static __host__ __device__ int64_t off_tiles(int64_t n) {
    const int64_t nb = (n + kTI - 1) / kTI;
    return 2 * nb * (nb + 1);
}
// The tile at index t.
__device__ __forceinline__ void off_tile(int64_t t, int64_t& ib, int64_t& jb) {
    ib = (int64_t)((sqrt(1.0 + 2.0 * (double)t) - 1.0) * 0.5);
    while (2 * ib * (ib + 1) > t) --ib;
    while (2 * (ib + 1) * (ib + 2) <= t) ++ib;
    jb = t - 2 * ib * (ib + 1);
}
template <int DD>
__global__ void __launch_bounds__(128) k_off_store(const float* __restrict__ a, int64_t n, int kernel, float inv_ell,
                                                   const int* __restrict__ cl, float* __restrict__ M) {
    __shared__ float bs[kTJ][DD];
    __shared__ int cs[kTJ];
    int64_t ib, jb;
    off_tile(blockIdx.x, ib, jb);
    const int64_t j0 = jb * kTJ, i = ib * kTI + 4 * threadIdx.x;
    const int nt = (int)max((int64_t)0, min((int64_t)kTJ, n - j0));
    for (int e = threadIdx.x; e < nt * DD; e += 128) bs[e / DD][e % DD] = a[j0 * DD + e];
    for (int e = threadIdx.x; e < nt; e += 128) cs[e] = cl[j0 + e];
    __syncthreads();
    float ai[4][DD];
    int ci[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
        const int64_t q = min(i + u, n - 1);
#pragma unroll
        for (int e = 0; e < DD; ++e) ai[u][e] = a[q * DD + e];
        ci[u] = i + u < n ? cl[q] : -1;
    }
    float* Mt = M + (int64_t)blockIdx.x * kTI * kTJ + 4 * threadIdx.x;
    for (int r = 0; r < kTJ; ++r) {
        float kv[4] = {0.f, 0.f, 0.f, 0.f};
        if (r < nt && j0 + r < i + 3) {
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                float s = 0.f;
#pragma unroll
                for (int q = 0; q < DD; ++q) { const float t = ai[u][q] - bs[r][q]; s = fmaf(t, t, s); }
                kv[u] = dev::kernel_value_f(kernel, sqrtf(s), inv_ell);
                if (ci[u] == cs[r] || ci[u] < 0 || j0 + r >= i + u) kv[u] = 0.f;
            }
        }
        *reinterpret_cast<float4*>(Mt + r * kTI) = make_float4(kv[0], kv[1], kv[2], kv[3]);
    }
}
void launch_off_store(int d, cudaStream_t st, const float* a, int64_t n, int kernel, float inv_ell, const int* cl,
                      float* M) {
    const unsigned g = (unsigned)off_tiles(n);
#define HDF_OS(DD) case DD: k_off_store<DD><<<g, 128, 0, st>>>(a, n, kernel, inv_ell, cl, M); break;
    switch (d) { HDF_OS(1) HDF_OS(2) HDF_OS(3) HDF_OS(4) HDF_OS(5) HDF_OS(6) HDF_OS(7) HDF_OS(8) }
#undef HDF_OS
}

// Two FP32 operations per instruction, each rounded to nearest on its own.
typedef unsigned long long F2;
__device__ __forceinline__ F2 add2(F2 a, F2 b) { F2 d; asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b)); return d; }
__device__ __forceinline__ F2 sub2(F2 a, F2 b) { F2 d; asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b)); return d; }
__device__ __forceinline__ F2 mul2(F2 a, F2 b) { F2 d; asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b)); return d; }
__device__ __forceinline__ F2 fma2(F2 a, F2 b, F2 c) {
    F2 d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}
// (sh, sl) += k (wh + wl), k exact: p = k wh with its exact error, TwoSum into sh, the rest into sl;
// nwh = -wh.
__device__ __forceinline__ void dot_step2(F2 k, F2 wh, F2 nwh, F2 wl, F2& sh, F2& sl) {
    const F2 np = mul2(k, nwh);                               // -p
    const F2 e = fma2(k, wl, fma2(k, wh, np));
    const F2 s = sub2(sh, np), bb = sub2(s, sh);
    const F2 t = sub2(sub2(sh, sub2(s, bb)), add2(np, bb));   // (sh - (s - bb)) + (p - bb)
    sh = s;
    sl = add2(sl, add2(t, e));
}
// The sum of two pairs.
__device__ __forceinline__ void pair_add(float& h, float& l, float h2, float l2) {
    float s, e;
    dev::two_sum(h, h2, s, e);
    h = s;
    l += e + l2;
}

// Both halves of the product by the tiles: part[t kTPart + i'] = sum_j M[j][i] w_j over the tile's j, and
// part[t kTPart + kTI + j'] = sum_i M[j][i] w_i over its i.  Every entry is read once and used for both,
// with exact products and FP32-pair sums (in the order of the tile, the same on every run), two
// entries per instruction.  A warp takes 32 j, a lane four consecutive i of each 128; the j sums
// are reduced over the lanes eight at a time, halving their number with each exchange, the i sums over
// the four warps.  A lane copies the entries that it will use itself, kPieceJ j's ahead, into its own
// shared memory (with register loads at 12 warps per SM the warps waited for memory 40% of the time,
// 107 us).  Bound by the read of M (57 us at 13,760 points) and the FP32 pipe (11 operations per entry
// and side, 58 us).
constexpr int kPieceJ = 4, kPieces = 32 / kPieceJ;                 // j's per copy, copies per warp and tile
constexpr size_t kOffSmem = 4 * 2 * (size_t)kPieceJ * kTI * sizeof(float);
__global__ void __launch_bounds__(128, 2) k_off_apply(const float* __restrict__ M, int64_t n, int64_t ntiles,
                                                      const double* __restrict__ w, double* __restrict__ part) {
    extern __shared__ __align__(16) float4 ring[];                 // [warp][2][kPieceJ][4][lane]
    __shared__ __align__(16) float wih[kTI], win[kTI], wil[kTI];   // w_i = hi + lo, and -hi
    __shared__ __align__(16) float4 wj[kTJ];                       // (hi, hi, -hi, -hi)
    __shared__ __align__(16) float2 wjl[kTJ];                      // (lo, lo)
    __shared__ float2 red[4][kTI];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    float4* mine = ring + (size_t)warp * 2 * kPieceJ * 128 + lane;
    auto copy = [&](int64_t t, int p) {
        if (t < ntiles) {
            const float* src = M + t * kTI * kTJ + (int64_t)(32 * warp + kPieceJ * p) * kTI + 4 * lane;
            const uint32_t dst = (uint32_t)__cvta_generic_to_shared(mine + (p & 1) * kPieceJ * 128);
#pragma unroll
            for (int e = 0; e < 4 * kPieceJ; ++e)
                asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst + 512u * e), "l"(src + 128 * e) : "memory");
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    copy(blockIdx.x, 0);
    for (int64_t t = blockIdx.x; t < ntiles; t += gridDim.x) {
        int64_t ib, jb;
        off_tile(t, ib, jb);
        __syncthreads();                                           // the previous tile's w and sums are used up
        for (int e = threadIdx.x; e < kTI + kTJ; e += 128) {
            const int64_t q = e < kTI ? ib * kTI + e : jb * kTJ + (e - kTI);
            const double v = q < n ? w[q] : 0.0;
            const float hi = (float)v, lo = (float)(v - (double)hi);
            if (e < kTI) {
                wih[e] = hi; win[e] = -hi; wil[e] = lo;
            } else {
                wj[e - kTI] = make_float4(hi, hi, -hi, -hi);
                wjl[e - kTI] = make_float2(lo, lo);
            }
        }
        __syncthreads();
        double* out = part + t * kTPart;
        F2 hI[4][2], lI[4][2];
#pragma unroll
        for (int k = 0; k < 4; ++k)
#pragma unroll
            for (int u = 0; u < 2; ++u) hI[k][u] = lI[k][u] = 0ull;
#pragma unroll 1
        for (int g = 0; g < 4; ++g) {
            F2 hJ[8], lJ[8];
#pragma unroll
            for (int q = 0; q < 8; ++q) hJ[q] = lJ[q] = 0ull;
#pragma unroll
            for (int s = 0; s < 8 / kPieceJ; ++s) {
                const int p = 8 / kPieceJ * g + s;
                copy(p + 1 < kPieces ? t : t + gridDim.x, (p + 1) % kPieces);
                asm volatile("cp.async.wait_group 1;" ::: "memory");
                const float4* st = mine + (s & 1) * kPieceJ * 128;
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    const ulonglong2 ih = *reinterpret_cast<const ulonglong2*>(wih + 128 * k + 4 * lane);
                    const ulonglong2 in = *reinterpret_cast<const ulonglong2*>(win + 128 * k + 4 * lane);
                    const ulonglong2 il = *reinterpret_cast<const ulonglong2*>(wil + 128 * k + 4 * lane);
#pragma unroll
                    for (int q = 0; q < kPieceJ; ++q) {
                        const int j = 32 * warp + kPieceJ * p + q, o = kPieceJ * s + q;
                        const ulonglong2 jh = *reinterpret_cast<const ulonglong2*>(&wj[j]);
                        const F2 jl = *reinterpret_cast<const F2*>(&wjl[j]);
                        const ulonglong2 mm = *reinterpret_cast<const ulonglong2*>(st + (4 * q + k) * 32);
                        dot_step2(mm.x, jh.x, jh.y, jl, hI[k][0], lI[k][0]);
                        dot_step2(mm.y, jh.x, jh.y, jl, hI[k][1], lI[k][1]);
                        dot_step2(mm.x, ih.x, in.x, il.x, hJ[o], lJ[o]);
                        dot_step2(mm.y, ih.y, in.y, il.y, hJ[o], lJ[o]);
                    }
                }
            }
            float H[8], L[8];
#pragma unroll
            for (int q = 0; q < 8; ++q) {
                const float2 h = *reinterpret_cast<const float2*>(&hJ[q]), l = *reinterpret_cast<const float2*>(&lJ[q]);
                H[q] = h.x;
                L[q] = l.x;
                pair_add(H[q], L[q], h.y, l.y);
            }
#pragma unroll
            for (int o = 16, c = 4; o >= 4; o >>= 1, c >>= 1) {
                const bool up = lane & o;
#pragma unroll
                for (int q = 0; q < c; ++q) {
                    const float sh = up ? H[q] : H[q + c], sl = up ? L[q] : L[q + c];
                    const float rh = __shfl_xor_sync(0xffffffffu, sh, o), rl = __shfl_xor_sync(0xffffffffu, sl, o);
                    if (up) { H[q] = H[q + c]; L[q] = L[q + c]; }
                    pair_add(H[q], L[q], rh, rl);
                }
            }
#pragma unroll
            for (int o = 2; o >= 1; o >>= 1) {
                const float rh = __shfl_xor_sync(0xffffffffu, H[0], o), rl = __shfl_xor_sync(0xffffffffu, L[0], o);
                pair_add(H[0], L[0], rh, rl);
            }
            const int q = ((lane >> 4) & 1) * 4 + ((lane >> 3) & 1) * 2 + ((lane >> 2) & 1);
            if ((lane & 3) == 0) out[kTI + 32 * warp + 8 * g + q] = (double)H[0] + (double)L[0];
        }
#pragma unroll
        for (int k = 0; k < 4; ++k)
#pragma unroll
            for (int u = 0; u < 2; ++u) {
                const float2 h = *reinterpret_cast<const float2*>(&hI[k][u]), l = *reinterpret_cast<const float2*>(&lI[k][u]);
                red[warp][128 * k + 4 * lane + 2 * u] = make_float2(h.x, l.x);
                red[warp][128 * k + 4 * lane + 2 * u + 1] = make_float2(h.y, l.y);
            }
        __syncthreads();
        for (int e = threadIdx.x; e < kTI; e += 128) {
            float2 s = red[0][e];
#pragma unroll
            for (int v = 1; v < 4; ++v) pair_add(s.x, s.y, red[v][e].x, red[v][e].y);
            out[e] = (double)s.x + (double)s.y;
        }
    }
    asm volatile("cp.async.wait_group 0;" ::: "memory");
}

// Row i's partial sums: of the tiles (SYM), else of the S column splits; for the threads ty of eight
// that share the row.
template <bool SYM>
__device__ __forceinline__ double part_sum(const double* __restrict__ part, int S, int64_t n, int64_t i, int ty) {
    double s = 0.0;
    if (SYM) {
        const int64_t ib = i / kTI, jb = i / kTJ, nb = (n + kTI - 1) / kTI;
        const int ni = (int)(4 * (ib + 1)), nt = ni + (int)(nb - ib);
#pragma unroll 4
        for (int t = ty; t < nt; t += 8) {
            const int64_t b = ib + (t - ni);
            s += part[t < ni ? (2 * ib * (ib + 1) + t) * kTPart + i % kTI : (2 * b * (b + 1) + jb) * kTPart + kTI + i % kTJ];
        }
    } else {
#pragma unroll 4
        for (int t = ty; t < S; t += 8) s += part[t * n + i];
    }
    return s;
}

// out[i] = alpha v[i] + (add ? add[i] : 0) + the partial sums of row i; 32 rows by 8 parts a block.
template <bool SYM>
__global__ void __launch_bounds__(256) k_direct_finish(const double* __restrict__ part, int S, int64_t m, double alpha,
                                                       const double* __restrict__ v, const double* __restrict__ add,
                                                       double* __restrict__ out) {
    __shared__ double sh[8][32];
    const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
    const int64_t i = blockIdx.x * (int64_t)32 + tx;
    sh[ty][tx] = i < m ? part_sum<SYM>(part, S, m, i, ty) : 0.0;
    __syncthreads();
    if (ty || i >= m) return;
    double s = (v ? alpha * v[i] : 0.0) + (add ? add[i] : 0.0);
#pragma unroll
    for (int t = 0; t < 8; ++t) s += sh[t][tx];
    out[i] = s;
}

// FP32 copy of row-major points shifted by the point o (FP64 differences first).
__global__ void k_shift_f32(const double* __restrict__ x, int64_t n, int d, const double* __restrict__ o,
                            float* __restrict__ out) {
    const int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (e >= n * d) return;
    out[e] = (float)(x[e] - o[e % d]);
}

// Column splits for the direct kernel: enough blocks to fill the GPU a few times.
int64_t direct_split(int64_t m, int64_t n, int* S) {
    const int64_t rb = (m + kDkRows - 1) / kDkRows;
    int64_t s = std::max<int64_t>(1, std::min<int64_t>((4 * 152 + rb - 1) / rb, (n + kDkTile - 1) / kDkTile));
    s = std::min<int64_t>(s, 64);
    int64_t split = (n + s - 1) / s;
    split = ((split + kDkTile - 1) / kDkTile) * kDkTile;
    *S = (int)std::max<int64_t>(1, (n + split - 1) / split);
    return split;
}

// ---------------------------------------------------------------- vector kernels
__global__ void k_gather_vec(const double* __restrict__ v, const int64_t* __restrict__ perm, int64_t n,
                             double* __restrict__ out) {
    const int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (p < n) out[p] = v[perm[p]];
}

__global__ void k_scatter_vec(const double* __restrict__ v, const int64_t* __restrict__ perm, int64_t n,
                              double* __restrict__ out) {
    const int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (p < n) out[perm[p]] = v[p];
}

__global__ void k_to_f32(const double* __restrict__ v, int64_t n, float* __restrict__ out) {
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i < n) out[i] = (float)v[i];
}

__global__ void k_to_f64(const float* __restrict__ v, int64_t n, double* __restrict__ out) {
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i < n) out[i] = (double)v[i];
}

// ----------------------------------------------- conjugate gradients on the device
// One iteration is a fixed chain of kernels; its scalars live in CgState (cg_state.h), so that the
// host reads the state only every few iterations.  At 13,760 points an iteration went from 0.85 ms
// (0.43 the off-diagonal blocks, 0.57 + 0.11 the HDF blocks partly hidden, two host round trips) to
// 0.16 ms.  Kernels of an iteration after the last return at once, so iterations enqueued past the end
// change nothing.  Every block adds the partial sums of a dot product itself, in the same fixed order.

// Sum of m values v[stride e + off] by a 256-thread block, the same on every block and thread.
__device__ __forceinline__ double block_total(const double* __restrict__ v, int m, int stride, int off, double* sh) {
    double s = 0.0;
    for (int e = threadIdx.x; e < m; e += 256) s += v[(int64_t)stride * e + off];
    return dev::block_sum_256(s, sh);
}

// nb = |r|, rz[0] = r . z from the partial sums (2 per block) of k_block_gemv.
__global__ void __launch_bounds__(256) k_cg_init(const double* __restrict__ part, int m, double rtol, CgState* S) {
    __shared__ double sh[256];
    const double rz = block_total(part, m, 2, 0, sh), bb = block_total(part, m, 2, 1, sh);
    if (threadIdx.x == 0) {
        S->rz[0] = rz; S->rz[1] = 0.0;
        S->nb = sqrt(bb); S->rtol = rtol;
        S->res = bb > 0.0 ? 1.0 : 0.0;
        S->it = 0; S->bad = 0;
        S->last = bb > 0.0 ? kCgRunning : 0;
    }
}

// q = lambda p + add + the partial sums, and the part of p . q of the block's 32 rows.  Eight threads
// share a row's parts (13,760 points: 18 us with one thread per row, 12 so).
template <bool SYM>
__global__ void __launch_bounds__(256) k_cg_finish(const double* __restrict__ part, int nsplit, int64_t n, double lam,
                                                   const double* __restrict__ p, const double* __restrict__ add,
                                                   double* __restrict__ q, double* __restrict__ dot,
                                                   int it, const CgState* __restrict__ S) {
    __shared__ double sh[8][32];
    if (cg_past_end(S->last, it)) return;
    const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
    const int64_t i = blockIdx.x * (int64_t)32 + tx;
    sh[ty][tx] = i < n ? part_sum<SYM>(part, nsplit, n, i, ty) : 0.0;
    __syncthreads();
    if (ty) return;
    double d = 0.0;
    if (i < n) {
        double s = lam * p[i] + add[i];
#pragma unroll
        for (int t = 0; t < 8; ++t) s += sh[t][tx];
        q[i] = s;
        d = p[i] * s;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) d += __shfl_xor_sync(0xffffffffu, d, o);
    if (tx == 0) dot[blockIdx.x] = d;
}

// alpha = rz / (p . q); x += alpha p; r -= alpha q.
__global__ void __launch_bounds__(256) k_cg_step(double* __restrict__ x, double* __restrict__ r,
                                                 const double* __restrict__ p, const double* __restrict__ q, int64_t n,
                                                 const double* __restrict__ dot, int m, int it, CgState* S) {
    __shared__ double sh[256];
    if (cg_past_end(S->last, it)) return;
    const double pq = block_total(dot, m, 1, 0, sh);
    if (!(pq > 0.0)) {
        if (blockIdx.x == 0 && threadIdx.x == 0) { S->bad = 1; S->it = it; S->last = it; }
        return;
    }
    const double alpha = S->rz[(it - 1) & 1] / pq;
    const int64_t i = blockIdx.x * (int64_t)256 + threadIdx.x;
    if (i >= n) return;
    x[i] += alpha * p[i];
    r[i] -= alpha * q[i];
}

// Residual check; beta = rz_new / rz; p = z + beta p.  dot: (r . z, r . r) of every gemv block.
__global__ void __launch_bounds__(256) k_cg_dir(double* __restrict__ p, const double* __restrict__ z, int64_t n,
                                                const double* __restrict__ dot, int m, int it, CgState* S) {
    __shared__ double sh[256];
    if (cg_past_end(S->last, it)) return;
    const double rz = block_total(dot, m, 2, 0, sh), rr = block_total(dot, m, 2, 1, sh);
    const double res = sqrt(rr) / S->nb;
    const bool end = res <= S->rtol;
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        S->res = res;
        S->it = it;
        S->rz[it & 1] = rz;
        if (end) S->last = it;
    }
    const int64_t i = blockIdx.x * (int64_t)256 + threadIdx.x;
    if (!end && i < n) p[i] = z[i] + rz / S->rz[(it - 1) & 1] * p[i];
}

// ------------------------------------------------------------------- preconditioner
// Dense lambda I + K_{C_c C_c} of every cluster (exact kernel, FP64) into the packed array:
// block c at ioff[c], n_c x n_c row-major; one thread per entry.
__global__ void k_block_matrices(const double* __restrict__ xp, int d, const int64_t* __restrict__ offs,
                                 const int64_t* __restrict__ ioff, int nclus, int kernel, double ell, double lam,
                                 double* __restrict__ out) {
    const int c = blockIdx.y;
    const int64_t a0 = offs[c], nc = offs[c + 1] - a0;
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < nc * nc; e += (int64_t)gridDim.x * blockDim.x) {
        const int64_t i = e / nc, j = e % nc;
        double s = 0.0;
        for (int q = 0; q < d; ++q) { const double t = xp[(a0 + i) * d + q] - xp[(a0 + j) * d + q]; s += t * t; }
        out[ioff[c] + e] = dev::kernel_value(kernel, sqrt(s), ell) + (i == j ? lam : 0.0);
    }
}

// z = M r: one warp per row of the block-diagonal inverse (packed as above), four loads in flight
// per lane (13,760 rows of about 660 entries 31 us, of which the FP64 pipe takes 20; two rows per warp
// 31, four 36).  With dot (and an iteration that is not past the end): (r . z, r . r) of the block's
// rows as well.
__global__ void __launch_bounds__(256) k_block_gemv(const double* __restrict__ inv, const int64_t* __restrict__ offs,
                                                    const int64_t* __restrict__ ioff, const int* __restrict__ cl,
                                                    int64_t n, const double* __restrict__ r, double* __restrict__ z,
                                                    double* __restrict__ dot, int it, const CgState* __restrict__ S) {
    __shared__ double sh[2][8];
    if (S && cg_past_end(S->last, it)) return;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t row = blockIdx.x * (int64_t)8 + warp;
    double s = 0.0, rv = 0.0;
    if (row < n) {
        const int c = cl[row];
        const int64_t a0 = offs[c], nc = offs[c + 1] - a0, i = row - a0;
        const double* M = inv + ioff[c] + i * nc;
        const double* rc = r + a0;
        rv = r[row];
#pragma unroll 4
        for (int64_t j = lane; j < nc; j += 32) s = fma(__ldcs(M + j), rc[j], s);
        for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
        if (lane == 0) z[row] = s;
    }
    if (!dot) return;
    if (lane == 0) { sh[0][warp] = row < n ? rv * s : 0.0; sh[1][warp] = rv * rv; }
    __syncthreads();
    if (threadIdx.x < 2) {
        double t = 0.0;
        for (int q = 0; q < 8; ++q) t += sh[threadIdx.x][q];
        dot[2 * (int64_t)blockIdx.x + threadIdx.x] = t;
    }
}

// --------------------------------------- block preconditioner: batched SPD inverse (FP64)
// A_c = lambda I + K_{C_c C_c} of every cluster c (packed row-major n_c x n_c at ioff[c]) is
// inverted on the device in 64 x 64 tiles, all clusters side by side (blockIdx.y = cluster):
//   Cholesky A = L L^T, right-looking, per panel j: the diagonal tile is factored in shared
//   memory and its inverse D_j = L_jj^-1 kept; L_ij = A_ij D_j^T for the tiles below; the
//   trailing lower tiles A_ik -= L_ij L_kj^T;
//   W = L^-1: W_ii = D_i, W_ij = -D_i sum_{j <= k < i} L_ik W_kj, panel by panel on a second stream
//   beside the factorization, whose diagonal tiles leave most SMs idle;
//   A^-1 = W^T W, both triangles written.
// A non-positive pivot sets *bad (the host reports HDF_ESINGULAR).
constexpr int kST = 64;                 // tile edge
constexpr int kSP = kST + 1;            // shared row stride (doubles)

struct SpdArgs {
    double* A;                          // packed blocks (overwritten by L in the lower tiles)
    double* W;                          // packed blocks: L^-1 (lower tiles), then A^-1 is written to A
    double* D;                          // per cluster: nb_c diagonal-tile inverses, 64 x 64 each
    const int64_t* offs;                // cluster c: rows offs[c] .. offs[c + 1]
    const int64_t* ioff;                // packed offsets of the blocks
    const int64_t* doff;                // offsets of the diagonal-tile inverses
    int* bad;
};

__device__ __forceinline__ int64_t spd_n(const SpdArgs& P, int c) { return P.offs[c + 1] - P.offs[c]; }

// tile (bi, bj) of the n x n row-major M -> s (kST x kSP), zeros outside the matrix
__device__ __forceinline__ void spd_load(const double* M, int64_t n, int bi, int bj, double* s) {
    for (int e = threadIdx.x; e < kST * kST; e += blockDim.x) {
        const int r = e / kST, q = e % kST;
        const int64_t gr = (int64_t)bi * kST + r, gc = (int64_t)bj * kST + q;
        s[r * kSP + q] = (gr < n && gc < n) ? M[gr * n + gc] : 0.0;
    }
}
__device__ __forceinline__ void spd_store(double* M, int64_t n, int bi, int bj, const double* s, bool transpose) {
    for (int e = threadIdx.x; e < kST * kST; e += blockDim.x) {
        const int r = e / kST, q = e % kST;
        const int64_t gr = (int64_t)bi * kST + r, gc = (int64_t)bj * kST + q;
        if (gr < n && gc < n) {
            if (transpose) M[gc * n + gr] = s[r * kSP + q];
            else M[gr * n + gc] = s[r * kSP + q];
        }
    }
}
// acc (4 x 4 per thread, 256 threads: rows 4 ty.., columns 4 tx..) += X Y^T or X Y (tiles in shared)
template <bool YT>
__device__ __forceinline__ void spd_mma(const double* X, const double* Y, double acc[4][4]) {
    const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
    for (int m = 0; m < kST; ++m) {
        double xv[4], yv[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) xv[i] = X[(4 * ty + i) * kSP + m];
#pragma unroll
        for (int j = 0; j < 4; ++j) yv[j] = YT ? Y[(4 * tx + j) * kSP + m] : Y[m * kSP + 4 * tx + j];
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int j = 0; j < 4; ++j) acc[i][j] = fma(xv[i], yv[j], acc[i][j]);
    }
}

// Panel j, step 1: factor the diagonal tile in shared memory, write L_jj to A, D_j = L_jj^-1.
__global__ void __launch_bounds__(256) k_spd_potrf(SpdArgs P, int j) {
    extern __shared__ double sh[];
    const int c = blockIdx.y;
    const int64_t n = spd_n(P, c);
    if ((int64_t)j * kST >= n) return;
    const int t = (int)min((int64_t)kST, n - (int64_t)j * kST);
    double* A = P.A + P.ioff[c];
    double* S = sh;                       // the tile
    double* X = sh + kST * kSP;           // its inverse
    spd_load(A, n, j, j, S);
    __syncthreads();
    for (int k = 0; k < t; ++k) {
        if (threadIdx.x == 0) {
            const double piv = S[k * kSP + k];
            if (!(piv > 0.0)) { atomicExch(P.bad, 1); S[k * kSP + k] = 1.0; }
            else S[k * kSP + k] = sqrt(piv);
        }
        __syncthreads();
        const double dk = S[k * kSP + k];
        for (int r = k + 1 + threadIdx.x; r < t; r += blockDim.x) S[r * kSP + k] /= dk;
        __syncthreads();
        // trailing lower triangle: S[r][q] -= S[r][k] S[q][k], k < q <= r < t
        const int m = t - k - 1;
        for (int e = threadIdx.x; e < m * m; e += blockDim.x) {
            const int r = k + 1 + e / m, q = k + 1 + e % m;
            if (q <= r) S[r * kSP + q] -= S[r * kSP + k] * S[q * kSP + k];
        }
        __syncthreads();
    }
    // zero the strict upper triangle and the padding, so that the tile is exactly L_jj
    for (int e = threadIdx.x; e < kST * kST; e += blockDim.x) {
        const int r = e / kST, q = e % kST;
        if (q > r || r >= t) S[r * kSP + q] = (r == q && r >= t) ? 1.0 : 0.0;
    }
    __syncthreads();
    // X = L^-1, column q by thread q: X[r][q] = (delta_rq - sum_{q <= m < r} L[r][m] X[m][q]) / L[r][r]
    if (threadIdx.x < kST) {
        const int q = threadIdx.x;
        for (int r = 0; r < kST; ++r) {
            if (r < q) { X[r * kSP + q] = 0.0; continue; }
            double v = (r == q) ? 1.0 : 0.0;
            for (int m = q; m < r; ++m) v -= S[r * kSP + m] * X[m * kSP + q];
            X[r * kSP + q] = v / S[r * kSP + r];
        }
    }
    __syncthreads();
    spd_store(A, n, j, j, S, false);
    double* D = P.D + P.doff[c] + (int64_t)j * kST * kST;
    for (int e = threadIdx.x; e < kST * kST; e += blockDim.x) D[e] = X[(e / kST) * kSP + e % kST];
}

// Panel j, step 2: L_ij = A_ij D_j^T for the tiles below the diagonal (blockIdx.x = i - j - 1).
__global__ void __launch_bounds__(256) k_spd_trsm(SpdArgs P, int j) {
    extern __shared__ double sh[];
    const int c = blockIdx.y;
    const int64_t n = spd_n(P, c);
    const int i = j + 1 + blockIdx.x;
    if ((int64_t)i * kST >= n) return;
    double* A = P.A + P.ioff[c];
    const double* D = P.D + P.doff[c] + (int64_t)j * kST * kST;
    double* Xs = sh;
    double* Ds = sh + kST * kSP;
    spd_load(A, n, i, j, Xs);
    for (int e = threadIdx.x; e < kST * kST; e += blockDim.x) Ds[(e / kST) * kSP + e % kST] = D[e];
    __syncthreads();
    double acc[4][4] = {};
    spd_mma<true>(Xs, Ds, acc);
    __syncthreads();
    const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
        for (int b2 = 0; b2 < 4; ++b2) Xs[(4 * ty + a) * kSP + 4 * tx + b2] = acc[a][b2];
    __syncthreads();
    spd_store(A, n, i, j, Xs, false);
}

// Panel j, step 3: A_ik -= L_ij L_kj^T for j < k <= i (blockIdx.x enumerates the pairs).
__global__ void __launch_bounds__(256) k_spd_update(SpdArgs P, int j) {
    extern __shared__ double sh[];
    const int c = blockIdx.y;
    const int64_t n = spd_n(P, c);
    // pair index -> (i, k) with 0 <= kk <= ii, i = j + 1 + ii, k = j + 1 + kk
    const int e = blockIdx.x;
    int ii = (int)((sqrt(8.0 * e + 1.0) - 1.0) / 2.0);
    while ((ii + 1) * (ii + 2) / 2 <= e) ++ii;
    while (ii * (ii + 1) / 2 > e) --ii;
    const int kk = e - ii * (ii + 1) / 2;
    const int i = j + 1 + ii, k = j + 1 + kk;
    if ((int64_t)i * kST >= n) return;
    double* A = P.A + P.ioff[c];
    double* Li = sh;
    double* Lk = sh + kST * kSP;
    double* Cs = sh + 2 * kST * kSP;
    spd_load(A, n, i, j, Li);
    spd_load(A, n, k, j, Lk);
    spd_load(A, n, i, k, Cs);
    __syncthreads();
    double acc[4][4] = {};
    spd_mma<true>(Li, Lk, acc);
    const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
        for (int b2 = 0; b2 < 4; ++b2) Cs[(4 * ty + a) * kSP + 4 * tx + b2] -= acc[a][b2];
    __syncthreads();
    spd_store(A, n, i, k, Cs, false);
}

// W = L^-1 by columns of L: row k is finished, W_kk = D_k, W_kj = -D_k S_kj (blockIdx.x = j <= k), and
// then every S_ij below takes its term, S_ij += L_ik W_kj.  A tile product is 64^3 multiplications and
// additions at two per clock and SM, 68 us; with the sum over k inside one block the last rows of the
// largest cluster kept 16 blocks busy for 1.3 ms each (1,088 rows: 12.6 ms in all).
__global__ void __launch_bounds__(256) k_spd_wrow(SpdArgs P, int k) {
    extern __shared__ double sh[];
    const int c = blockIdx.y;
    const int64_t n = spd_n(P, c);
    const int j = blockIdx.x;
    if ((int64_t)k * kST >= n) return;
    double* W = P.W + P.ioff[c];
    const double* D = P.D + P.doff[c] + (int64_t)k * kST * kST;
    double* X = sh;
    double* Y = sh + kST * kSP;
    const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
    for (int e = threadIdx.x; e < kST * kST; e += blockDim.x) X[(e / kST) * kSP + e % kST] = D[e];
    if (j < k) {
        spd_load(W, n, k, j, Y);
        __syncthreads();
        double out[4][4] = {};
        spd_mma<false>(X, Y, out);
        __syncthreads();
#pragma unroll
        for (int a = 0; a < 4; ++a)
#pragma unroll
            for (int b = 0; b < 4; ++b) X[(4 * ty + a) * kSP + 4 * tx + b] = -out[a][b];
    }
    __syncthreads();
    spd_store(W, n, k, j, X, false);
}
// The terms of row k; blockIdx.x enumerates (i > k, j <= k).
__global__ void __launch_bounds__(256) k_spd_wupdate(SpdArgs P, int k) {
    extern __shared__ double sh[];
    const int c = blockIdx.y;
    const int64_t n = spd_n(P, c);
    const int i = k + 1 + (int)blockIdx.x / (k + 1), j = (int)blockIdx.x % (k + 1);
    if ((int64_t)i * kST >= n) return;
    const double* A = P.A + P.ioff[c];
    double* W = P.W + P.ioff[c];
    double* X = sh;
    double* Y = sh + kST * kSP;
    double* Z = sh + 2 * kST * kSP;
    const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
    spd_load(A, n, i, k, X);
    spd_load(W, n, k, j, Y);
    if (j < k) spd_load(W, n, i, j, Z);          // S_ik starts at zero
    __syncthreads();
    double acc[4][4];
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
        for (int b = 0; b < 4; ++b) acc[a][b] = j < k ? Z[(4 * ty + a) * kSP + 4 * tx + b] : 0.0;
    spd_mma<false>(X, Y, acc);
    __syncthreads();
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
        for (int b = 0; b < 4; ++b) Z[(4 * ty + a) * kSP + 4 * tx + b] = acc[a][b];
    __syncthreads();
    spd_store(W, n, i, j, Z, false);
}

// A^-1 = W^T W: tile (i, j), j <= i (blockIdx.x enumerates the pairs) = sum_{k >= i} W_ki^T W_kj,
// written to (i, j) and, transposed, to (j, i).
__global__ void __launch_bounds__(256) k_spd_wtw(SpdArgs P) {
    extern __shared__ double sh[];
    const int c = blockIdx.y;
    const int64_t n = spd_n(P, c);
    const int nb = (int)((n + kST - 1) / kST);
    const int e = blockIdx.x;
    int i = (int)((sqrt(8.0 * e + 1.0) - 1.0) / 2.0);
    while ((i + 1) * (i + 2) / 2 <= e) ++i;
    while (i * (i + 1) / 2 > e) --i;
    const int j = e - i * (i + 1) / 2;
    if (i >= nb) return;
    const double* W = P.W + P.ioff[c];
    double* A = P.A + P.ioff[c];
    double* X = sh;
    double* Y = sh + kST * kSP;
    const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
    double acc[4][4] = {};
    for (int k = i; k < nb; ++k) {
        // X = W_ki^T (transposed on load), Y = W_kj
        for (int q = threadIdx.x; q < kST * kST; q += blockDim.x) {
            const int r = q / kST, s2 = q % kST;
            const int64_t gr = (int64_t)k * kST + r, gc = (int64_t)i * kST + s2;
            X[s2 * kSP + r] = (gr < n && gc < n) ? W[gr * n + gc] : 0.0;
        }
        spd_load(W, n, k, j, Y);
        __syncthreads();
        spd_mma<false>(X, Y, acc);
        __syncthreads();
    }
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
        for (int b2 = 0; b2 < 4; ++b2) X[(4 * ty + a) * kSP + 4 * tx + b2] = acc[a][b2];
    __syncthreads();
    spd_store(A, n, i, j, X, false);
    if (i != j) spd_store(A, n, i, j, X, true);
}

}  // namespace

struct hdf_krr {
    int64_t n = 0;
    int d = 0, nclus = 0, prec = 0, kernel = 0;
    double ell = 0.0, lam = 0.0;
    std::vector<int64_t> offs, ioff;
    DevBuf perm, xp, xp32, cl, doffs, dioff, inv;
    hdf_batch* batch = nullptr;
    DevBuf vb, yb, hd, part, dotp;       // work: bulk-typed vectors, HDF result, direct-kernel partials
    DevBuf koff;                         // the stored off-diagonal blocks (none: evaluated per product)
    DevBuf cgst;                         // CgState of the running solve
    CgState* cgh = nullptr;              // two pinned copies for the host
    cudaEvent_t cgev[2] = {nullptr, nullptr};
    cudaStream_t side = nullptr;         // the off-diagonal blocks beside the HDF blocks
    cudaEvent_t fork = nullptr, join = nullptr;
    int S = 1;
    int64_t split = 0;
    double t_build = 0.0, t_precond = 0.0;
    ~hdf_krr() {
        if (batch) hdf_batch_free(batch);
        if (cgh) cudaFreeHost(cgh);
        for (cudaEvent_t e : {cgev[0], cgev[1], fork, join}) if (e) cudaEventDestroy(e);
        if (side) cudaStreamDestroy(side);
    }
};

namespace {

// Bytes that the device can still hand out: free ones and those that the default pool keeps unused.
size_t device_room() {
    size_t free = 0, total = 0;
    if (cudaMemGetInfo(&free, &total) != cudaSuccess) { cudaGetLastError(); return 0; }
    int dev = 0;
    cudaMemPool_t pool;
    uint64_t reserved = 0, used = 0;
    if (cudaGetDevice(&dev) == cudaSuccess && cudaDeviceGetDefaultMemPool(&pool, dev) == cudaSuccess &&
        cudaMemPoolGetAttribute(pool, cudaMemPoolAttrReservedMemCurrent, &reserved) == cudaSuccess &&
        cudaMemPoolGetAttribute(pool, cudaMemPoolAttrUsedMemCurrent, &used) == cudaSuccess)
        free += reserved - used;
    cudaGetLastError();
    return free;
}

// The off-diagonal blocks times vp into K->part.
hdf_status apply_off(hdf_krr* K, const double* vp, cudaStream_t st) {
    const int64_t n = K->n;
    HDF_COUNT_LAUNCH();
    if (K->koff.p) {
        int dv = 0, nsm = 0;
        HDF_CUDA(cudaGetDevice(&dv));
        HDF_CUDA(cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dv));
        HDF_CUDA(cudaFuncSetAttribute(k_off_apply, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kOffSmem));
        const int64_t tiles = off_tiles(n);
        k_off_apply<<<(unsigned)std::min<int64_t>(tiles, 2 * nsm), 128, kOffSmem, st>>>(K->koff.as<float>(), n, tiles, vp,
                                                                                       K->part.as<double>());
    } else {
        dim3 g((unsigned)((n + kDkRows - 1) / kDkRows), (unsigned)K->S);
        launch_direct(K->d, g, st, K->xp32.as<float>(), n, K->xp32.as<float>(), n, K->kernel, (float)(1.0 / K->ell),
                      vp, K->cl.as<int>(), K->cl.as<int>(), K->split, K->part.as<double>());
    }
    HDF_CUDA(cudaGetLastError());
    return HDF_OK;
}

// The diagonal blocks (HDF) times vp into K->hd.
hdf_status apply_diag(hdf_krr* K, const double* vp, cudaStream_t st) {
    const int64_t n = K->n;
    if (K->prec != HDF_FP32)
        return hdf_batch_matvec(K->batch, vp, n, 1, K->hd.p, n, reinterpret_cast<hdf_stream>(st));
    const int gb = blocks_for(n, 256, 1 << 30);
    HDF_COUNT_LAUNCH();
    k_to_f32<<<gb, 256, 0, st>>>(vp, n, K->vb.as<float>());
    if (hdf_status s = hdf_batch_matvec(K->batch, K->vb.p, n, 1, K->yb.p, n, reinterpret_cast<hdf_stream>(st)); s != HDF_OK)
        return s;
    HDF_COUNT_LAUNCH();
    k_to_f64<<<gb, 256, 0, st>>>(K->yb.as<float>(), n, K->hd.as<double>());
    HDF_CUDA(cudaGetLastError());
    return HDF_OK;
}

// The parts of K^ vp in cluster order (vp FP64, length n): the HDF blocks into K->hd, the partial sums
// of the off-diagonal blocks into K->part, side by side (the HDF blocks' two kernels wait for memory
// most of their 24 us at 13,760 points, the off-diagonal one for the FP32 pipe: 383 iterations 9 ms
// less than one after the other).
hdf_status apply_parts(hdf_krr* K, const double* vp, cudaStream_t st) {
    HDF_CUDA(cudaEventRecord(K->fork, st));
    HDF_CUDA(cudaStreamWaitEvent(K->side, K->fork, 0));
    const hdf_status so = apply_off(K, vp, K->side);
    const hdf_status sd = so == HDF_OK ? apply_diag(K, vp, st) : so;
    HDF_CUDA(cudaEventRecord(K->join, K->side));
    HDF_CUDA(cudaStreamWaitEvent(st, K->join, 0));
    return sd;
}

// tp = lambda vp + K^ vp in cluster order (vp, tp length n, FP64, device)
hdf_status apply_perm(hdf_krr* K, const double* vp, double* tp, cudaStream_t st) {
    if (hdf_status s = apply_parts(K, vp, st); s != HDF_OK) return s;
    HDF_COUNT_LAUNCH();
    auto finish = K->koff.p ? k_direct_finish<true> : k_direct_finish<false>;
    finish<<<blocks_for(K->n, 32, 1 << 30), 256, 0, st>>>(K->part.as<double>(), K->S, K->n, K->lam, vp,
                                                         K->hd.as<double>(), tp);
    HDF_CUDA(cudaGetLastError());
    return HDF_OK;
}

hdf_status precond_perm(hdf_krr* K, const double* rp, double* zp, cudaStream_t st, double* dot = nullptr,
                        int it = 0, const CgState* S = nullptr) {
    HDF_COUNT_LAUNCH();
    k_block_gemv<<<(unsigned)((K->n + 7) / 8), 256, 0, st>>>(K->inv.as<double>(), K->doffs.as<int64_t>(),
                                                             K->dioff.as<int64_t>(), K->cl.as<int>(), K->n, rp, zp, dot,
                                                             it, S);
    HDF_CUDA(cudaGetLastError());
    return HDF_OK;
}

}  // namespace

extern "C" {

hdf_status hdf_kmeans(const double* x_dev, int64_t n, int d, int k, const int64_t* init_host, int max_iter,
                      int* labels_dev, double* centres_dev, int* iterations, hdf_stream stream) {
    if (!x_dev || !init_host || !labels_dev || n < 1 || d < 1 || d > HDF_MAX_D || k < 1 || k > n ||
        (int64_t)k * d > 6144 || max_iter < 1)
        return fail(HDF_EINVAL, "hdf_kmeans: bad argument (1 <= k <= n, k d <= 6144, 1 <= d <= 8)");
    for (int c = 0; c < k; ++c)
        if (init_host[c] < 0 || init_host[c] >= n) return fail(HDF_EINVAL, "hdf_kmeans: initial index out of range");
    cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
    DevBuf C, idx, part, chg;
    HDF_CUDA(C.alloc_on(sizeof(double) * k * d, st));
    HDF_CUDA(idx.alloc_on(sizeof(int64_t) * k, st));
    HDF_CUDA(cudaMemcpyAsync(idx.p, init_host, sizeof(int64_t) * k, cudaMemcpyHostToDevice, st));
    HDF_COUNT_LAUNCH();
    k_gather_rows<<<blocks_for((int64_t)k * d, 256, 1 << 30), 256, 0, st>>>(x_dev, d, idx.as<int64_t>(), k,
                                                                           C.as<double>());
    HDF_CUDA(cudaMemsetAsync(labels_dev, 0xff, sizeof(int) * n, st));      // -1: every label changes first
    const int64_t chunks = (n + (int64_t)kKmBlocks * kKmChunk - 1) / ((int64_t)kKmBlocks * kKmChunk);   // of a block
    const int G = (int)((n + chunks * kKmChunk - 1) / (chunks * kKmChunk));
    HDF_CUDA(part.alloc_on(sizeof(double) * (size_t)G * k * (d + 1), st));
    HDF_CUDA(chg.alloc_on(sizeof(int), st));
    int it = 0;
    for (it = 1; it <= max_iter; ++it) {
        HDF_CUDA(cudaMemsetAsync(chg.p, 0, sizeof(int), st));
        HDF_COUNT_LAUNCH();
        k_km_assign<<<blocks_for(n, 256, 1 << 30), 256, sizeof(double) * k * d, st>>>(x_dev, n, d, k, C.as<double>(),
                                                                                     labels_dev, chg.as<int>());
        HDF_CUDA(cudaGetLastError());
        int changes = 0;
        HDF_CUDA(cudaMemcpyAsync(&changes, chg.p, sizeof(int), cudaMemcpyDeviceToHost, st));
        HDF_CUDA(cudaStreamSynchronize(st));
        if (changes == 0 && it > 1) break;
        HDF_COUNT_LAUNCH();
        k_km_partial<<<G, 256, 0, st>>>(x_dev, n, d, k, labels_dev, chunks, part.as<double>());
        HDF_COUNT_LAUNCH();
        k_km_finish<<<(k + 3) / 4, 128, 0, st>>>(part.as<double>(), G, k, d, C.as<double>());
        HDF_CUDA(cudaGetLastError());
    }
    if (it > max_iter) it = max_iter;
    if (centres_dev) HDF_CUDA(cudaMemcpyAsync(centres_dev, C.p, sizeof(double) * k * d, cudaMemcpyDeviceToDevice, st));
    HDF_CUDA(cudaStreamSynchronize(st));
    if (iterations) *iterations = it;
    return HDF_OK;
}

hdf_status hdf_kernel_matvec(const double* xq_dev, int64_t m, const double* x_dev, int64_t n, int d,
                             hdf_kernel kernel, double lengthscale, const double* w_dev, double* out_dev,
                             hdf_stream stream) {
    if (!xq_dev || !x_dev || !w_dev || !out_dev || m < 1 || n < 1 || d < 1 || d > HDF_MAX_D || kernel < 0 ||
        kernel > 3 || !(lengthscale > 0))
        return fail(HDF_EINVAL, "hdf_kernel_matvec: bad argument");
    cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
    DevBuf a, b, part;
    HDF_CUDA(a.alloc_on(sizeof(float) * m * d, st));
    HDF_CUDA(b.alloc_on(sizeof(float) * n * d, st));
    HDF_COUNT_LAUNCH();
    k_shift_f32<<<blocks_for(m * d, 256, 1 << 30), 256, 0, st>>>(xq_dev, m, d, x_dev, a.as<float>());
    HDF_COUNT_LAUNCH();
    k_shift_f32<<<blocks_for(n * d, 256, 1 << 30), 256, 0, st>>>(x_dev, n, d, x_dev, b.as<float>());
    int S = 1;
    const int64_t split = direct_split(m, n, &S);
    HDF_CUDA(part.alloc_on(sizeof(double) * (size_t)S * m, st));
    dim3 g((unsigned)((m + kDkRows - 1) / kDkRows), (unsigned)S);
    HDF_COUNT_LAUNCH();
    launch_direct(d, g, st, a.as<float>(), m, b.as<float>(), n, kernel, (float)(1.0 / lengthscale), w_dev, nullptr,
                  nullptr, split, part.as<double>());
    HDF_COUNT_LAUNCH();
    k_direct_finish<false><<<blocks_for(m, 32, 1 << 30), 256, 0, st>>>(part.as<double>(), S, m, 0.0, nullptr, nullptr,
                                                                 out_dev);
    HDF_CUDA(cudaGetLastError());
    return HDF_OK;
}

hdf_status hdf_krr_build(const double* x_dev, int64_t n, int d, const int* labels_dev, hdf_kernel kernel,
                         double lengthscale, double lambda, double tol, hdf_precision prec, const hdf_options* opt,
                         hdf_stream stream, hdf_krr** out) {
    if (out) *out = nullptr;
    if (!x_dev || !labels_dev || !out || n < 1 || d < 3 || d > HDF_MAX_D || kernel < 0 || kernel > 3 ||
        !(lengthscale > 0) || !(lambda > 0) || !(tol > 0 && tol < 1) || (prec != HDF_FP64 && prec != HDF_FP32))
        return fail(HDF_EINVAL, "hdf_krr_build: bad argument");
    cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
    const double t0 = wall_ms();
    // clusters in label order (empty labels dropped), points permuted cluster by cluster
    std::vector<int> lab(n);
    HDF_CUDA(cudaMemcpyAsync(lab.data(), labels_dev, sizeof(int) * n, cudaMemcpyDeviceToHost, st));
    HDF_CUDA(cudaStreamSynchronize(st));
    int lmax = -1;
    for (int64_t i = 0; i < n; ++i) {
        if (lab[i] < 0) return fail(HDF_EINVAL, "hdf_krr_build: negative label");
        lmax = std::max(lmax, lab[i]);
    }
    std::vector<int64_t> cnt((size_t)lmax + 1, 0);
    for (int64_t i = 0; i < n; ++i) cnt[lab[i]]++;
    std::vector<int> remap((size_t)lmax + 1, -1);
    // the locals below (work space of both streams and the guard that waits for them) go before the model
    std::unique_ptr<hdf_krr> model(new hdf_krr());
    hdf_krr* K = model.get();
    K->n = n; K->d = d; K->prec = prec; K->kernel = kernel; K->ell = lengthscale; K->lam = lambda;
    K->offs.push_back(0);
    for (int c = 0; c <= lmax; ++c)
        if (cnt[c] > 0) { remap[c] = (int)K->offs.size() - 1; K->offs.push_back(K->offs.back() + cnt[c]); }
    K->nclus = (int)K->offs.size() - 1;
    std::vector<int64_t> perm(n), pos(K->offs.begin(), K->offs.end() - 1);
    std::vector<int> clp(n);
    for (int64_t i = 0; i < n; ++i) {
        const int c = remap[lab[i]];
        perm[pos[c]] = i;
        clp[pos[c]++] = c;
    }
    hdf_status s = HDF_OK;
    HDF_CUDA(K->perm.alloc(sizeof(int64_t) * n));
    HDF_CUDA(K->xp.alloc(sizeof(double) * n * d));
    HDF_CUDA(K->xp32.alloc(sizeof(float) * n * d));
    HDF_CUDA(K->cl.alloc(sizeof(int) * n));
    HDF_CUDA(K->doffs.alloc(sizeof(int64_t) * K->offs.size()));
    HDF_CUDA(cudaMemcpyAsync(K->perm.p, perm.data(), sizeof(int64_t) * n, cudaMemcpyHostToDevice, st));
    HDF_CUDA(cudaMemcpyAsync(K->cl.p, clp.data(), sizeof(int) * n, cudaMemcpyHostToDevice, st));
    HDF_CUDA(cudaMemcpyAsync(K->doffs.p, K->offs.data(), sizeof(int64_t) * K->offs.size(), cudaMemcpyHostToDevice, st));
    HDF_COUNT_LAUNCH();
    k_gather_rows<<<blocks_for(n * d, 256, 1 << 30), 256, 0, st>>>(x_dev, d, K->perm.as<int64_t>(), n, K->xp.as<double>());
    HDF_COUNT_LAUNCH();
    k_shift_f32<<<blocks_for(n * d, 256, 1 << 30), 256, 0, st>>>(K->xp.as<double>(), n, d, K->xp.as<double>(),
                                                                 K->xp32.as<float>());
    HDF_CUDA(cudaGetLastError());
    // HDF factors of the diagonal blocks: one batched build over the clusters
    std::vector<double> ells(K->nclus, lengthscale);
    s = hdf_build_batched(K->nclus, K->offs.data(), K->xp.as<double>(), d, kernel, ells.data(), tol, prec, opt, stream,
                          &K->batch);
    if (s != HDF_OK && s != HDF_ETOL_UNREACHABLE) return s;
    const hdf_status build_status = s;
    K->t_build = wall_ms() - t0;
    // block preconditioner: exact blocks, inverted on the device (Cholesky, FP64)
    const double t1 = wall_ms();
    K->ioff.assign(K->nclus + 1, 0);
    for (int c = 0; c < K->nclus; ++c) {
        const int64_t nc = K->offs[c + 1] - K->offs[c];
        K->ioff[c + 1] = K->ioff[c] + nc * nc;
    }
    if (K->ioff.back() > ((int64_t)1 << 28))
        return fail(HDF_ETOOBIG, "hdf_krr_build: sum of squared cluster sizes > 2^28 (block preconditioner)");
    HDF_CUDA(K->dioff.alloc(sizeof(int64_t) * K->ioff.size()));
    HDF_CUDA(cudaMemcpyAsync(K->dioff.p, K->ioff.data(), sizeof(int64_t) * K->ioff.size(), cudaMemcpyHostToDevice, st));
    HDF_CUDA(K->inv.alloc(sizeof(double) * std::max<int64_t>(1, K->ioff.back())));
    {
        int64_t nmax = 0;
        for (int c = 0; c < K->nclus; ++c) nmax = std::max(nmax, K->offs[c + 1] - K->offs[c]);
        dim3 g((unsigned)blocks_for(nmax * nmax, 256, 4096), (unsigned)K->nclus);
        HDF_COUNT_LAUNCH();
        k_block_matrices<<<g, 256, 0, st>>>(K->xp.as<double>(), d, K->doffs.as<int64_t>(), K->dioff.as<int64_t>(),
                                            K->nclus, kernel, lengthscale, lambda, K->inv.as<double>());
        HDF_CUDA(cudaGetLastError());
    }
    for (cudaEvent_t* e : {&K->cgev[0], &K->cgev[1], &K->fork, &K->join})
        HDF_CUDA(cudaEventCreateWithFlags(e, cudaEventDisableTiming));
    HDF_CUDA(cudaStreamCreateWithFlags(&K->side, cudaStreamNonBlocking));
    {
        // invert every block on the device (batched tiles; see k_spd_potrf and its siblings)
        int nbmax = 0;
        std::vector<int64_t> doff(K->nclus + 1, 0);
        for (int c = 0; c < K->nclus; ++c) {
            const int nb = (int)((K->offs[c + 1] - K->offs[c] + kST - 1) / kST);
            nbmax = std::max(nbmax, nb);
            doff[c + 1] = doff[c] + (int64_t)nb * kST * kST;
        }
        DevBuf W, D, ddoff, bad;
        struct SideDone { cudaStream_t s; ~SideDone() { cudaStreamSynchronize(s); } } side_done{K->side};   // before W goes
        HDF_CUDA(W.alloc_on(sizeof(double) * std::max<int64_t>(1, K->ioff.back()), st));
        HDF_CUDA(D.alloc_on(sizeof(double) * std::max<int64_t>(1, doff.back()), st));
        HDF_CUDA(ddoff.alloc_on(sizeof(int64_t) * doff.size(), st));
        HDF_CUDA(bad.alloc_on(sizeof(int), st));
        HDF_CUDA(cudaMemcpyAsync(ddoff.p, doff.data(), sizeof(int64_t) * doff.size(), cudaMemcpyHostToDevice, st));
        HDF_CUDA(cudaMemsetAsync(bad.p, 0, sizeof(int), st));
        SpdArgs P{K->inv.as<double>(), W.as<double>(), D.as<double>(), K->doffs.as<int64_t>(),
                  K->dioff.as<int64_t>(), ddoff.as<int64_t>(), bad.as<int>()};
        const int tile = (int)(sizeof(double) * kST * kSP);
        HDF_CUDA(cudaFuncSetAttribute(k_spd_potrf, cudaFuncAttributeMaxDynamicSharedMemorySize, 2 * tile));
        HDF_CUDA(cudaFuncSetAttribute(k_spd_trsm, cudaFuncAttributeMaxDynamicSharedMemorySize, 2 * tile));
        HDF_CUDA(cudaFuncSetAttribute(k_spd_update, cudaFuncAttributeMaxDynamicSharedMemorySize, 3 * tile));
        HDF_CUDA(cudaFuncSetAttribute(k_spd_wrow, cudaFuncAttributeMaxDynamicSharedMemorySize, 2 * tile));
        HDF_CUDA(cudaFuncSetAttribute(k_spd_wupdate, cudaFuncAttributeMaxDynamicSharedMemorySize, 3 * tile));
        HDF_CUDA(cudaFuncSetAttribute(k_spd_wtw, cudaFuncAttributeMaxDynamicSharedMemorySize, 2 * tile));
        const unsigned ncl = (unsigned)K->nclus;
        for (int j = 0; j < nbmax; ++j) {
            HDF_COUNT_LAUNCH();
            k_spd_potrf<<<dim3(1, ncl), 256, 2 * tile, st>>>(P, j);
            const int nt = nbmax - j - 1;
            if (nt > 0) {
                HDF_COUNT_LAUNCH();
                k_spd_trsm<<<dim3((unsigned)nt, ncl), 256, 2 * tile, st>>>(P, j);
            }
            HDF_CUDA(cudaEventRecord(K->fork, st));
            HDF_CUDA(cudaStreamWaitEvent(K->side, K->fork, 0));
            HDF_COUNT_LAUNCH();
            k_spd_wrow<<<dim3((unsigned)(j + 1), ncl), 256, 2 * tile, K->side>>>(P, j);
            if (nt > 0) {
                HDF_COUNT_LAUNCH();
                k_spd_wupdate<<<dim3((unsigned)(nt * (j + 1)), ncl), 256, 3 * tile, K->side>>>(P, j);
                HDF_COUNT_LAUNCH();
                k_spd_update<<<dim3((unsigned)(nt * (nt + 1) / 2), ncl), 256, 3 * tile, st>>>(P, j);
            }
        }
        HDF_CUDA(cudaEventRecord(K->join, K->side));
        HDF_CUDA(cudaStreamWaitEvent(st, K->join, 0));
        HDF_COUNT_LAUNCH();
        k_spd_wtw<<<dim3((unsigned)(nbmax * (nbmax + 1) / 2), ncl), 256, 2 * tile, st>>>(P);
        HDF_CUDA(cudaGetLastError());
        int hbad = 0;
        HDF_CUDA(cudaMemcpyAsync(&hbad, bad.p, sizeof(int), cudaMemcpyDeviceToHost, st));
        HDF_CUDA(cudaStreamSynchronize(st));
        if (hbad) return fail(HDF_ESINGULAR, "hdf_krr_build: a block lambda I + K_cc is not positive definite");
    }
    // work space
    HDF_CUDA(K->hd.alloc(sizeof(double) * n));
    HDF_CUDA(K->dotp.alloc(sizeof(double) * 2 * (size_t)((n + 7) / 8)));
    HDF_CUDA(K->cgst.alloc(sizeof(CgState)));
    HDF_CUDA(cudaMallocHost(reinterpret_cast<void**>(&K->cgh), 2 * sizeof(CgState)));
    if (prec == HDF_FP32) {
        HDF_CUDA(K->vb.alloc(sizeof(float) * n));
        HDF_CUDA(K->yb.alloc(sizeof(float) * n));
    }
    // The off-diagonal blocks are stored while they take at most 8 GiB (65,000 points) and the device has
    // room for them, their partial sums and kSpare besides; else every product evaluates them.  They come
    // last, so that nothing else fails for their sake.
    constexpr size_t kSpare = (size_t)512 << 20;
    const size_t kbytes = sizeof(float) * (size_t)off_tiles(n) * kTI * kTJ;
    const size_t pbytes = sizeof(double) * (size_t)off_tiles(n) * kTPart;
    const bool stored = kbytes <= ((size_t)8 << 30) && device_room() >= kbytes + pbytes + kSpare &&
                        K->part.alloc(pbytes) == cudaSuccess && K->koff.alloc_on(kbytes, st) == cudaSuccess;
    if (stored) {
        HDF_COUNT_LAUNCH();
        launch_off_store(d, st, K->xp32.as<float>(), n, kernel, (float)(1.0 / lengthscale), K->cl.as<int>(),
                         K->koff.as<float>());
        HDF_CUDA(cudaGetLastError());
    } else {
        cudaGetLastError();
        K->split = direct_split(n, n, &K->S);
        HDF_CUDA(K->part.alloc(sizeof(double) * (size_t)K->S * n));
    }
    HDF_CUDA(cudaStreamSynchronize(st));
    K->t_precond = wall_ms() - t1;
    *out = model.release();
    return build_status;
}

hdf_status hdf_krr_apply(hdf_krr* K, const double* v_dev, double* out_dev, hdf_stream stream) {
    if (!K || !v_dev || !out_dev) return fail(HDF_EINVAL, "hdf_krr_apply: null argument");
    cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
    DevBuf vp, tp;
    HDF_CUDA(vp.alloc_on(sizeof(double) * K->n, st));
    HDF_CUDA(tp.alloc_on(sizeof(double) * K->n, st));
    const int gb = blocks_for(K->n, 256, 1 << 30);
    HDF_COUNT_LAUNCH();
    k_gather_vec<<<gb, 256, 0, st>>>(v_dev, K->perm.as<int64_t>(), K->n, vp.as<double>());
    if (hdf_status s = apply_perm(K, vp.as<double>(), tp.as<double>(), st); s != HDF_OK) return s;
    HDF_COUNT_LAUNCH();
    k_scatter_vec<<<gb, 256, 0, st>>>(tp.as<double>(), K->perm.as<int64_t>(), K->n, out_dev);
    HDF_CUDA(cudaGetLastError());
    return HDF_OK;
}

hdf_status hdf_krr_precond(hdf_krr* K, const double* r_dev, double* z_dev, hdf_stream stream) {
    if (!K || !r_dev || !z_dev) return fail(HDF_EINVAL, "hdf_krr_precond: null argument");
    cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
    DevBuf rp, zp;
    HDF_CUDA(rp.alloc_on(sizeof(double) * K->n, st));
    HDF_CUDA(zp.alloc_on(sizeof(double) * K->n, st));
    const int gb = blocks_for(K->n, 256, 1 << 30);
    HDF_COUNT_LAUNCH();
    k_gather_vec<<<gb, 256, 0, st>>>(r_dev, K->perm.as<int64_t>(), K->n, rp.as<double>());
    if (hdf_status s = precond_perm(K, rp.as<double>(), zp.as<double>(), st); s != HDF_OK) return s;
    HDF_COUNT_LAUNCH();
    k_scatter_vec<<<gb, 256, 0, st>>>(zp.as<double>(), K->perm.as<int64_t>(), K->n, z_dev);
    HDF_CUDA(cudaGetLastError());
    return HDF_OK;
}

hdf_status hdf_krr_solve(hdf_krr* K, const double* y_dev, double rtol, int max_iter, double* w_dev, int* iterations,
                         double* relres, hdf_stream stream) {
    if (!K || !y_dev || !w_dev || !(rtol > 0) || max_iter < 1) return fail(HDF_EINVAL, "hdf_krr_solve: bad argument");
    cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
    const int64_t n = K->n;
    DevBuf buf;
    HDF_CUDA(buf.alloc_on(sizeof(double) * 5 * n, st));
    double *x = buf.as<double>(), *r = x + n, *z = r + n, *p = z + n, *q = p + n;
    const int gb = blocks_for(n, 256, 1 << 30);
    HDF_CUDA(cudaMemsetAsync(x, 0, sizeof(double) * n, st));
    HDF_COUNT_LAUNCH();
    k_gather_vec<<<gb, 256, 0, st>>>(y_dev, K->perm.as<int64_t>(), n, r);
    CgState* S = K->cgst.as<CgState>();
    double* dot = K->dotp.as<double>();
    const int mgemv = (int)((n + 7) / 8), gf = blocks_for(n, 32, 1 << 30);
    auto finish = K->koff.p ? k_cg_finish<true> : k_cg_finish<false>;
    if (hdf_status s = precond_perm(K, r, z, st, dot); s != HDF_OK) return s;
    HDF_CUDA(cudaMemcpyAsync(p, z, sizeof(double) * n, cudaMemcpyDeviceToDevice, st));
    HDF_COUNT_LAUNCH();
    k_cg_init<<<1, 256, 0, st>>>(dot, mgemv, rtol, S);
    HDF_CUDA(cudaGetLastError());
    // the host looks at the state of kPoll iterations ago while the next kPoll are enqueued
    constexpr int kPoll = 4;
    int polls = 0;
    bool done = false;
    auto poll = [&]() -> hdf_status {
        HDF_CUDA(cudaMemcpyAsync(&K->cgh[polls & 1], S, sizeof(CgState), cudaMemcpyDeviceToHost, st));
        HDF_CUDA(cudaEventRecord(K->cgev[polls & 1], st));
        if (polls > 0) {
            HDF_CUDA(cudaEventSynchronize(K->cgev[(polls - 1) & 1]));
            done = K->cgh[(polls - 1) & 1].last != kCgRunning;
        }
        ++polls;
        return HDF_OK;
    };
    for (int it = 1; it <= max_iter && !done; ++it) {
        if (it % kPoll == 1)
            if (hdf_status s = poll(); s != HDF_OK) return s;
        if (done) break;
        if (hdf_status s = apply_parts(K, p, st); s != HDF_OK) return s;
        HDF_COUNT_LAUNCH();
        finish<<<gf, 256, 0, st>>>(K->part.as<double>(), K->S, n, K->lam, p, K->hd.as<double>(), q, dot, it, S);
        HDF_COUNT_LAUNCH();
        k_cg_step<<<gb, 256, 0, st>>>(x, r, p, q, n, dot, gf, it, S);
        HDF_CUDA(cudaGetLastError());
        if (hdf_status s = precond_perm(K, r, z, st, dot, it, S); s != HDF_OK) return s;
        HDF_COUNT_LAUNCH();
        k_cg_dir<<<gb, 256, 0, st>>>(p, z, n, dot, mgemv, it, S);
        HDF_CUDA(cudaGetLastError());
    }
    HDF_CUDA(cudaMemcpyAsync(&K->cgh[0], S, sizeof(CgState), cudaMemcpyDeviceToHost, st));
    HDF_CUDA(cudaStreamSynchronize(st));
    if (K->cgh[0].bad) return fail(HDF_ESINGULAR, "hdf_krr_solve: the operator is not positive definite");
    const int it = K->cgh[0].it;
    const double res = K->cgh[0].res;
    HDF_COUNT_LAUNCH();
    k_scatter_vec<<<gb, 256, 0, st>>>(x, K->perm.as<int64_t>(), n, w_dev);
    HDF_CUDA(cudaGetLastError());
    HDF_CUDA(cudaStreamSynchronize(st));
    if (iterations) *iterations = it;
    if (relres) *relres = res;
    return (res <= rtol) ? HDF_OK : fail(HDF_ETOL_UNREACHABLE, "hdf_krr_solve: max_iter reached before rtol");
}

hdf_status hdf_krr_info(const hdf_krr* K, int* nclusters, int64_t* rank_total, double* t_ms) {
    if (!K) return fail(HDF_EINVAL, "hdf_krr_info: null argument");
    if (nclusters) *nclusters = K->nclus;
    if (rank_total) {
        int64_t tot = 0;
        for (int c = 0; c < K->nclus; ++c) {
            hdf_info I;
            if (hdf_status s = hdf_batch_info(K->batch, c, &I); s != HDF_OK) return s;
            tot += I.rank;
        }
        *rank_total = tot;
    }
    if (t_ms) { t_ms[0] = K->t_build; t_ms[1] = K->t_precond; }
    return HDF_OK;
}

void hdf_krr_free(hdf_krr* K) {
    if (!K) return;
    cudaDeviceSynchronize();
    K->koff.st = nullptr;            // nothing reads it any more: back to the pool on the legacy stream
    delete K;
}

}  // extern "C"
