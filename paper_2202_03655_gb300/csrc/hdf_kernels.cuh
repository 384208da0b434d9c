// Device kernels of the HDF factorization for sm_103a.
//
// Layout in HBM (all row-major unless stated):
//   x   n x d FP64 points (input, caller-owned)
//   F   n x ldF radial factors F[i, (k,s)] = f_{k,s}(|x'_i|)   (bulk type T)
//   U   n x ldU factor, column (k, s, h) = F[i, (k,s)] * Y_k^h(x_hat_i)   (bulk type T)
//   V,Y column-major n x c blocks (caller-owned)
// Every reduction over points is two-stage (per-block partials, then a fixed-order
// sum), so results do not depend on scheduling.
#pragma once
#include <cstdint>
#include <cuda_runtime.h>

namespace hdf {
namespace dev {

constexpr int kMaxD = 8;

struct Center {
    double c[kMaxD];
};

// ----------------------------------------------------------------- kernel values
__device__ __forceinline__ double kernel_value(int kernel, double r, double ell) {
    const double z = fabs(r) / ell;
    switch (kernel) {
        case 0: return exp(-0.5 * z * z);
        case 1: return 1.0 / (1.0 + z * z);
        case 2: { const double s = 1.7320508075688772 * z; return (1.0 + s) * exp(-s); }
        default: { const double s = 2.23606797749979 * z; return (1.0 + s + s * s / 3.0) * exp(-s); }
    }
}

// The same kernels in FP32 (r >= 0, inv_ell = 1 / l); values <= 1.
__device__ __forceinline__ float kernel_value_f(int kernel, float r, float inv_ell) {
    const float z = r * inv_ell;
    switch (kernel) {
        case 0: return expf(-0.5f * z * z);
        case 1: return 1.0f / (1.0f + z * z);
        case 2: { const float s = 1.7320508f * z; return (1.0f + s) * expf(-s); }
        default: { const float s = 2.2360680f * z; return (1.0f + s + s * s * (1.0f / 3.0f)) * expf(-s); }
    }
}

// Deterministic tree sum of one double per thread over the block (blockDim = 256).
__device__ __forceinline__ double block_sum_256(double v, double* sh) {
    sh[threadIdx.x] = v;
    __syncthreads();
    for (int s = 128; s > 0; s >>= 1) {
        if (threadIdx.x < s) sh[threadIdx.x] += sh[threadIdx.x + s];
        __syncthreads();
    }
    const double out = sh[0];
    __syncthreads();
    return out;
}

// ------------------------------------------------------------- A0: centre, radius
// part[b*d + j] = sum over the block's chunk of x[i, j].
static __global__ void k_sum_partial(const double* __restrict__ x, int64_t n, int d, int64_t chunk,
                              double* __restrict__ part) {
    __shared__ double sh[256];
    const int64_t i0 = blockIdx.x * chunk, i1 = min(n, i0 + chunk);
    double acc[kMaxD];
#pragma unroll
    for (int j = 0; j < kMaxD; ++j) acc[j] = 0.0;
    for (int64_t i = i0 + threadIdx.x; i < i1; i += blockDim.x)
        for (int j = 0; j < d; ++j) acc[j] += x[i * d + j];
    for (int j = 0; j < d; ++j) {
        const double s = block_sum_256(acc[j], sh);
        if (threadIdx.x == 0) part[blockIdx.x * d + j] = s;
    }
}

// part[b] = max over the block's chunk of |x_i - c|^2.
static __global__ void k_maxnorm_partial(const double* __restrict__ x, int64_t n, int d, int64_t chunk,
                                  Center c, double* __restrict__ part) {
    __shared__ double sh[256];
    const int64_t i0 = blockIdx.x * chunk, i1 = min(n, i0 + chunk);
    double m = 0.0;
    for (int64_t i = i0 + threadIdx.x; i < i1; i += blockDim.x) {
        double s = 0.0;
        for (int j = 0; j < d; ++j) { const double y = x[i * d + j] - c.c[j]; s += y * y; }
        m = fmax(m, s);
    }
    sh[threadIdx.x] = m;
    __syncthreads();
    for (int s = 128; s > 0; s >>= 1) {
        if (threadIdx.x < s) sh[threadIdx.x] = fmax(sh[threadIdx.x], sh[threadIdx.x + s]);
        __syncthreads();
    }
    if (threadIdx.x == 0) part[blockIdx.x] = sh[0];
}

// Mean-square kernel value over the subsample idx(t) = floor(t n / m), t < m:
// part[t] = sum_u k(|x_idx(t) - x_idx(u)|)^2.
static __global__ void k_mu2_rows(const double* __restrict__ x, int64_t n, int d, int m, int kernel,
                           double ell, double* __restrict__ part) {
    __shared__ double sh[256];
    const int t = blockIdx.x;
    const int64_t i = ((int64_t)t * n) / m;
    double xi[kMaxD];
    for (int j = 0; j < d; ++j) xi[j] = x[i * d + j];
    double acc = 0.0;
    for (int u = threadIdx.x; u < m; u += blockDim.x) {
        const int64_t jj = ((int64_t)u * n) / m;
        double s = 0.0;
        for (int j = 0; j < d; ++j) { const double y = xi[j] - x[jj * d + j]; s += y * y; }
        const double kv = kernel_value(kernel, sqrt(s), ell);
        acc += kv * kv;
    }
    const double tot = block_sum_256(acc, sh);
    if (threadIdx.x == 0) part[t] = tot;
}

// Cross-pair version for K(X, Y): part[t] = sum_u k(|x_ix(t) - y_iy(u)|)^2 over the strided
// subsamples ix(t) = floor(t m / mx), t < mx, of X and iy(u) = floor(u n / my), u < my, of Y.
static __global__ void k_mu2_cross(const double* __restrict__ x, int64_t m, int mx, const double* __restrict__ y,
                                   int64_t n, int my, int d, int kernel, double ell, double* __restrict__ part) {
    __shared__ double sh[256];
    const int t = blockIdx.x;
    const int64_t i = ((int64_t)t * m) / mx;
    double xi[kMaxD];
    for (int j = 0; j < d; ++j) xi[j] = x[i * d + j];
    double acc = 0.0;
    for (int u = threadIdx.x; u < my; u += blockDim.x) {
        const int64_t jj = ((int64_t)u * n) / my;
        double s = 0.0;
        for (int j = 0; j < d; ++j) { const double z = xi[j] - y[jj * d + j]; s += z * z; }
        const double kv = kernel_value(kernel, sqrt(s), ell);
        acc += kv * kv;
    }
    const double tot = block_sum_256(acc, sh);
    if (threadIdx.x == 0) part[t] = tot;
}

// ----------------------------------------------------- A3: radial-basis Gram matrices
// B0[l] = T_l(u), l <= L and B1[l] = rho T_l(u), l < L, u = 8 rho^2 - 1, rho = |x - c|/(2R).
// part[b][q] (q < npairs) = sum_i B0[l] B0[l'] and part[b][npairs + q] = sum_i rho^2 T_l T_l'
// over the block's chunk, for the pairs (l, l') = pairs[q], l <= l'.
constexpr int kGramTile = 64;
constexpr int kGramMaxQ = 9;     // ceil(npairs / 256) for L <= 64

static __global__ void __launch_bounds__(256) k_radial_gram(const double* __restrict__ x, int64_t n, int d,
                                                     int64_t chunk, Center c, double inv2R, int L,
                                                     const uint16_t* __restrict__ pairs, int npairs,
                                                     double* __restrict__ part) {
    extern __shared__ double smem[];
    const int LP1 = L + 1;
    double* Ts = smem;                          // [kGramTile][LP1]
    double* r2 = smem + kGramTile * LP1;        // [kGramTile]
    const int64_t i0 = blockIdx.x * chunk, i1 = min(n, i0 + chunk);
    double a0[kGramMaxQ], a1[kGramMaxQ];
#pragma unroll
    for (int q = 0; q < kGramMaxQ; ++q) { a0[q] = 0.0; a1[q] = 0.0; }
    for (int64_t t0 = i0; t0 < i1; t0 += kGramTile) {
        const int cnt = (int)min((int64_t)kGramTile, i1 - t0);
        if (threadIdx.x < kGramTile) {
            const int p = threadIdx.x;
            double* T = Ts + p * LP1;
            if (p < cnt) {
                const int64_t i = t0 + p;
                double s = 0.0;
                for (int j = 0; j < d; ++j) { const double y = (x[i * d + j] - c.c[j]) * inv2R; s += y * y; }
                const double u = 8.0 * s - 1.0;
                r2[p] = s;
                T[0] = 1.0;
                if (L >= 1) T[1] = u;
                for (int l = 2; l <= L; ++l) T[l] = 2.0 * u * T[l - 1] - T[l - 2];
            } else {
                r2[p] = 0.0;
                for (int l = 0; l <= L; ++l) T[l] = 0.0;
            }
        }
        __syncthreads();
#pragma unroll
        for (int q = 0; q < kGramMaxQ; ++q) {
            const int pi = threadIdx.x + 256 * q;
            if (pi < npairs) {
                const int l = pairs[2 * pi], lp = pairs[2 * pi + 1];
                double s0 = 0.0, s1 = 0.0;
                for (int p = 0; p < cnt; ++p) {
                    const double v = Ts[p * LP1 + l] * Ts[p * LP1 + lp];
                    s0 += v;
                    s1 += v * r2[p];
                }
                a0[q] += s0;
                a1[q] += s1;
            }
        }
        __syncthreads();
    }
#pragma unroll
    for (int q = 0; q < kGramMaxQ; ++q) {
        const int pi = threadIdx.x + 256 * q;
        if (pi < npairs) {
            part[(int64_t)blockIdx.x * 2 * npairs + pi] = a0[q];
            part[(int64_t)blockIdx.x * 2 * npairs + npairs + pi] = a1[q];
        }
    }
}

// Chebyshev moments of the radial data: part[b][j] = sum over the block's chunk of T_j(u_i),
// u_i = 8 rho_i^2 - 1, j < nmom.  The radial-basis Gram matrices follow from them exactly
// (T_l T_l' = (T_{l+l'} + T_{|l-l'|}) / 2 and u T_j = (T_{j+1} + T_{|j-1|}) / 2), so the Gram
// costs O(n L) instead of O(n L^2).
// Every tile's values pass through shared memory and are added by groups of nmom threads (thread =
// moment, groups splitting the tile's points), since one group alone leaves most of a block idle at
// small degrees; blocks take few points (moment_blocks), so that a few thousand points reach many
// SMs.  100,000 points, 66 moments, FP64: 0.90 ms on 13 blocks, 0.037 ms here; 10,000,000 points, 18
// moments, double-float: 1.16 ms with one group, 0.53 ms here.
constexpr int kMomTile = 64;
constexpr int kMomTileDf = 256;

// Blocks for n points in tiles of `tile`: one tile each up to four blocks per SM.
inline int moment_blocks(int64_t n, int tile) {
    const int64_t t = (n + tile - 1) / tile;
    return (int)(t < 4 * 152 ? (t > 1 ? t : 1) : 4 * 152);
}

// Sum over the groups of a block (v of thread group * nmom + l) for the threads l < nmom, in order.
__device__ __forceinline__ double moment_groups(double v, int nmom, double* sh) {
    const int G = blockDim.x / nmom;
    __syncthreads();
    sh[threadIdx.x] = v;
    __syncthreads();
    double s = v;
    if ((int)threadIdx.x < nmom)
        for (int g = 1; g < G; ++g) s += sh[g * nmom + threadIdx.x];
    return s;
}

static __global__ void __launch_bounds__(256) k_radial_moments(const double* __restrict__ x, int64_t n, int d,
                                                               int64_t chunk, Center c, double inv2R, int nmom,
                                                               double* __restrict__ part) {
    extern __shared__ double smem[];
    __shared__ double sh[256];
    double* Ts = smem;                          // [kMomTile][nmom]
    const int64_t i0 = blockIdx.x * chunk, i1 = min(n, i0 + chunk);
    const int G = 256 / nmom, grp = threadIdx.x / nmom, l = threadIdx.x % nmom;
    double acc = 0.0;
    for (int64_t t0 = i0; t0 < i1; t0 += kMomTile) {
        const int cnt = (int)min((int64_t)kMomTile, i1 - t0);
        if (threadIdx.x < cnt) {
            const int p = threadIdx.x;
            double* T = Ts + p * nmom;
            const int64_t i = t0 + p;
            double s = 0.0;
            for (int j = 0; j < d; ++j) { const double y = (x[i * d + j] - c.c[j]) * inv2R; s += y * y; }
            const double u = 8.0 * s - 1.0;
            T[0] = 1.0;
            if (nmom > 1) T[1] = u;
            for (int q = 2; q < nmom; ++q) T[q] = 2.0 * u * T[q - 1] - T[q - 2];
        }
        __syncthreads();
        if (grp < G) {
            double s = 0.0;
            for (int p = grp; p < cnt; p += G) s += Ts[p * nmom + l];
            acc += s;
        }
        __syncthreads();
    }
    const double tot = moment_groups(acc, nmom, sh);
    if (threadIdx.x < nmom) part[(int64_t)blockIdx.x * nmom + threadIdx.x] = tot;
}

// out[j] = sum_b part[b * ncols + j]: one block per column, fixed-order tree.
static __global__ void __launch_bounds__(256) k_reduce_cols(const double* __restrict__ part, int nblk, int64_t ncols,
                              double* __restrict__ out) {
    __shared__ double sh[256];
    double s = 0.0;
    for (int b = threadIdx.x; b < nblk; b += 256) s += part[(int64_t)b * ncols + blockIdx.x];
    const double tot = block_sum_256(s, sh);
    if (threadIdx.x == 0) out[blockIdx.x] = tot;
}

__host__ __device__ inline size_t align16(size_t b) { return (b + 15) & ~size_t(15); }

// ------------------------------------------------------------- A5a: radial factors
// Per point: B_par (FP64) -> Q_par = B_par Qmat_par (FP64, the orthonormalised radial basis
// of Eq. svd) -> F[i, col] = sum_l Q_par(col)[l] Wt[l, col] (type T).  Tiles of 32 points.
constexpr int kFTile = 32;

struct RFParams {
    const double* x; int64_t n; int d; Center c; double inv2R; int L;
    const double* Qm0; int nb0, m0;
    const double* Qm1; int nb1, m1;
    const float2* QC; int mtp;   // FP32 factors: [Qm0 | Qm1] as (hi, lo) float pairs, (L+1) x mtp
    int kopt;                    // FP32 factors in the batched build: outputs per Q unit
    int tiles;                   // FP32 factors, single build: tiles between two barriers
    int stage_wt;                // FP32 factors: copy Wt into shared memory
    const void* Wt; const uint8_t* colpar; int nF;
    void* F; int64_t ldF;
};

// Dynamic shared memory of one radial tile, in bytes.
__host__ __device__ inline size_t radialF_smem(int L, int m0, int m1, size_t tsize) {
    return sizeof(double) * (kFTile * (L + 1) + kFTile) + tsize * (size_t)(m0 + m1) * kFTile;
}

// Compensated FP32 arithmetic for the radial basis of FP32 factors.  Q = B Qmat cancels (Qmat
// grows like the inverse square root of the smallest kept Gram eigenvalue), so a plain FP32
// sum is not enough; FP64 is, but runs at a small fraction of the FP32 rate on this GPU.  The
// basis values and Qmat are carried as unevaluated (hi, lo) float pairs (about 48 bits) and the
// dot product uses error-free transformations: TwoProd by fma (Dekker/Kahan) and TwoSum
// (Knuth), the "Dot2" scheme of Ogita, Rump and Oishi (SIAM J. Sci. Comput. 26, 2005), whose
// result is as accurate as a sum in twice the working precision.
__device__ __forceinline__ void two_sum(float a, float b, float& s, float& e) {
    s = a + b;
    const float bb = s - a;
    e = (a - (s - bb)) + (b - bb);
}

// One Dot2 step: (sh, c) accumulates a * (bh + bl), a = (hi, lo).
__device__ __forceinline__ void dot2_step(float2 a, float bh, float bl, float& sh, float& c) {
    const float ph = a.x * bh;
    float pe = fmaf(a.x, bh, -ph);
    pe = fmaf(a.x, bl, fmaf(a.y, bh, pe));
    float s2, es;
    two_sum(sh, ph, s2, es);
    sh = s2;
    c += es + pe;
}

// FP32 factors (k_radial_F_df), one tile of kFTile points in three parts:
//   basis: u = 8 rho^2 - 1 and T_l(u) by the FP64 recurrence, split into (hi, lo) float pairs;
//   Q:     Q[o][p] = sum_l T_l(u_p) Qmat[l][o] by Dot2 against QC, the combined even | odd Qmat as
//          float pairs ((L+1) x mtp, odd columns zero in row L, mtp a multiple of 8), times rho
//          for the odd outputs;
//   F:     F[p][col] = sum_l Q[par(col) block + l][p] Wt[l][col] in FP32.
// The basis of the next tiles and the Q of the current ones are units of one warp each, as are then the
// columns of F (k_radial_F_df).
__device__ __forceinline__ void fast_two_sum(float a, float b, float& s, float& e) {
    s = a + b;
    e = b - (s - a);
}

// Chebyshev moments for FP32 factors: sum over the points [i0, i1) of T_l(u), l < nmom,
// u = 8 rho^2 - 1, by one 256-thread block.  Each thread runs one point's recurrence in
// double-float arithmetic (FP32 pairs; FP64 runs at a small fraction of the FP32 rate here),
// the values pass through shared memory (Tsm: 256 rows of nmom + 1 float2, an odd stride that
// keeps the 8-byte accesses conflict-free), groups of nmom threads add moment l over their share of
// the tile with error-free sums, and the tile and group sums are added in FP64.  Thread l < nmom
// returns moment l.
__device__ __forceinline__ double moments_df_range(const double* __restrict__ x, int d, const double* cc,
                                                   double inv2R, int nmom, int64_t i0, int64_t i1, float2* Tsm) {
    const int S = nmom + 1;
    const int G = 256 / nmom, grp = threadIdx.x / nmom, l0 = threadIdx.x % nmom;
    double acc = 0.0;
    for (int64_t t0 = i0; t0 < i1; t0 += kMomTileDf) {
        const int cnt = (int)min((int64_t)256, i1 - t0);
        const int p = threadIdx.x;
        if (p < cnt) {
            float2* T = Tsm + p * S;
            const int64_t i = t0 + p;
            double s = 0.0;
            for (int j = 0; j < d; ++j) { const double y = (x[i * d + j] - cc[j]) * inv2R; s += y * y; }
            const double u = 8.0 * s - 1.0;
            const float uh = (float)u, ul = (float)(u - (double)uh);
            const float u2h = 2.f * uh, u2l = 2.f * ul;
            float ah = 1.f, al = 0.f, bh = uh, bl = ul;
            T[0] = make_float2(1.f, 0.f);
            if (nmom > 1) T[1] = make_float2(uh, ul);
            for (int l = 2; l < nmom; ++l) {
                const float ph = u2h * bh;
                float pl = fmaf(u2h, bh, -ph);
                pl = fmaf(u2h, bl, fmaf(u2l, bh, pl));
                float sh, se;
                two_sum(ph, -ah, sh, se);
                se += pl - al;
                float th, tl;
                fast_two_sum(sh, se, th, tl);
                T[l] = make_float2(th, tl);
                ah = bh; al = bl;
                bh = th; bl = tl;
            }
        }
        __syncthreads();
        if (grp < G) {
            float mh = 0.f, ml = 0.f;
            for (int q = grp; q < cnt; q += G) {
                const float2 v = Tsm[q * S + l0];
                float sh, se;
                two_sum(mh, v.x, sh, se);
                se += ml + v.y;
                fast_two_sum(sh, se, mh, ml);
            }
            acc += (double)mh + (double)ml;
        }
        __syncthreads();
    }
    return moment_groups(acc, nmom, reinterpret_cast<double*>(Tsm));
}

// Drop-in for k_radial_moments (same part layout) for FP32 factors.
static __global__ void __launch_bounds__(256) k_radial_moments_df(const double* __restrict__ x, int64_t n, int d,
                                                                  int64_t chunk, Center c, double inv2R, int nmom,
                                                                  double* __restrict__ part) {
    extern __shared__ float2 tsm_raw[];
    const int64_t i0 = blockIdx.x * chunk, i1 = min(n, i0 + chunk);
    const double v = moments_df_range(x, d, c.c, inv2R, nmom, i0, i1, tsm_raw);
    if (threadIdx.x < nmom) part[(int64_t)blockIdx.x * nmom + threadIdx.x] = v;
}

// Basis values of one point in double-float arithmetic (FP32 pairs, about 48 bits): u and rho
// from FP64 coordinates (a few FP64 operations), then T_l(u) = 2 u T_{l-1} - T_{l-2} with
// error-free products and sums; the recurrence is stable on [-1, 1].
__device__ __forceinline__ void radialF_df_basis(const RFParams& P, int64_t t0, int p, float2* Ts, float* rh) {
    const int LP1 = P.L + 1;
    const int cnt = (int)min((int64_t)kFTile, P.n - t0);
    float2* Tp = Ts + p * LP1;
    double s = 0.0;
    if (p < cnt) {
        const int64_t i = t0 + p;
        for (int j = 0; j < P.d; ++j) { const double y = (P.x[i * P.d + j] - P.c.c[j]) * P.inv2R; s += y * y; }
    }
    const double u = 8.0 * s - 1.0;
    rh[p] = sqrtf((float)s);
    const float uh = (float)u, ul = (float)(u - (double)uh);
    const float u2h = 2.f * uh, u2l = 2.f * ul;                     // 2u, exact
    float ah = 1.f, al = 0.f, bh = uh, bl = ul;                       // T_{l-2}, T_{l-1}
    Tp[0] = make_float2(1.f, 0.f);
    if (P.L >= 1) Tp[1] = make_float2(uh, ul);
    for (int l = 2; l <= P.L; ++l) {
        // (ph, pl) = 2u * T_{l-1}
        const float ph = u2h * bh;
        float pl = fmaf(u2h, bh, -ph);
        pl = fmaf(u2h, bl, fmaf(u2l, bh, pl));
        // T_l = (ph, pl) - T_{l-2}
        float sh, se;
        two_sum(ph, -ah, sh, se);
        se += pl - al;
        float th, tl;
        fast_two_sum(sh, se, th, tl);
        Tp[l] = make_float2(th, tl);
        ah = bh; al = bl;
        bh = th; bl = tl;
    }
}

// The Q and F parts as units of one warp, which the warps of a CTA take from a counter: the parts
// of several tiles run between two barriers, so that no warp waits for the one with the most work.
// Q unit: lane = point of the tile, kOpt outputs from o0 (each basis value read from shared memory
// serves kOpt outputs, one 16-byte load brings two outputs).
template <int kOpt>
__device__ __forceinline__ void radialF_df_q(const RFParams& P, const float2* Ts, const float* rh, const float2* QC,
                                             float* Qs, int o0, int lane) {
    const int LP1 = P.L + 1, mt = P.m0 + P.m1;
    const float2* Tp = Ts + lane * LP1;
    float sh[kOpt], c[kOpt];
#pragma unroll
    for (int j = 0; j < kOpt; ++j) { sh[j] = 0.f; c[j] = 0.f; }
#pragma unroll 2
    for (int l = 0; l < LP1; ++l) {
        const float2 a = Tp[l];
        const float4* qr = reinterpret_cast<const float4*>(QC + (size_t)l * P.mtp + o0);
#pragma unroll
        for (int j2 = 0; j2 < kOpt / 2; ++j2) {
            const float4 b = qr[j2];
            dot2_step(a, b.x, b.y, sh[2 * j2], c[2 * j2]);
            dot2_step(a, b.z, b.w, sh[2 * j2 + 1], c[2 * j2 + 1]);
        }
    }
#pragma unroll
    for (int j = 0; j < kOpt; ++j) {
        const int o = o0 + j;
        if (o < mt) {
            float q = sh[j] + c[j];
            if (o >= P.m0) q *= rh[lane];
            Qs[o * kFTile + lane] = q;
        }
    }
}

// F unit: lane = column, 32 columns from col0; Wt from shared memory (Ws, max(m0, m1) x nF) when
// staged.
__device__ __forceinline__ void radialF_df_f(const RFParams& P, int64_t t0, const float* Qs, const float* Ws, int col0,
                                             int lane) {
    const int cnt = (int)min((int64_t)kFTile, P.n - t0);
    float* F = reinterpret_cast<float*>(P.F);
    const int col = col0 + lane;
    if (col >= P.ldF) return;
    if (col >= P.nF) {                           // row padding: zeros, so that sectors are whole
#pragma unroll
        for (int p = 0; p < kFTile; ++p)
            if (p < cnt) F[(t0 + p) * P.ldF + col] = 0.f;
        return;
    }
    const int par = P.colpar[col];
    const int ob = par ? P.m0 : 0, mp = par ? P.m1 : P.m0;
    float acc[kFTile];
#pragma unroll
    for (int p = 0; p < kFTile; ++p) acc[p] = 0.f;
    for (int l = 0; l < mp; ++l) {
        const float w = Ws[(int64_t)l * P.nF + col];
        const float4* q4 = reinterpret_cast<const float4*>(Qs + (ob + l) * kFTile);
#pragma unroll
        for (int p4 = 0; p4 < kFTile / 4; ++p4) {
            const float4 v = q4[p4];
            acc[4 * p4 + 0] += v.x * w;
            acc[4 * p4 + 1] += v.y * w;
            acc[4 * p4 + 2] += v.z * w;
            acc[4 * p4 + 3] += v.w * w;
        }
    }
#pragma unroll
    for (int p = 0; p < kFTile; ++p)
        if (p < cnt) F[(t0 + p) * P.ldF + col] = acc[p];
}

// The next unit of a warp from a shared counter.
__device__ __forceinline__ int next_unit(int* counter, int lane) {
    int u = 0;
    if (lane == 0) u = atomicAdd(counter, 1);
    return __shfl_sync(0xffffffffu, u, 0);
}

// Radial factors of the points [t0, t0 + kFTile): block-wide, ends with a barrier.
template <typename T>
__device__ __forceinline__ void radialF_tile(const RFParams& P, int64_t t0, unsigned char* smem_raw) {
    const int LP1 = P.L + 1;
    double* Ts = reinterpret_cast<double*>(smem_raw);            // [kFTile][LP1]
    double* rh = Ts + kFTile * LP1;                              // [kFTile]
    T* Qs = reinterpret_cast<T*>(rh + kFTile);                   // [m0 + m1][kFTile]
    const T* Wt = reinterpret_cast<const T*>(P.Wt);
    T* F = reinterpret_cast<T*>(P.F);
    const int cnt = (int)min((int64_t)kFTile, P.n - t0);
    if (threadIdx.x < kFTile) {
        const int p = threadIdx.x;
        double* Tp = Ts + p * LP1;
        double s = 0.0;
        if (p < cnt) {
            const int64_t i = t0 + p;
            for (int j = 0; j < P.d; ++j) { const double y = (P.x[i * P.d + j] - P.c.c[j]) * P.inv2R; s += y * y; }
        }
        const double u = 8.0 * s - 1.0;
        rh[p] = sqrt(s);
        Tp[0] = 1.0;
        if (P.L >= 1) Tp[1] = u;
        for (int l = 2; l <= P.L; ++l) Tp[l] = 2.0 * u * Tp[l - 1] - Tp[l - 2];
    }
    __syncthreads();
    const int mt = P.m0 + P.m1;
    for (int idx = threadIdx.x; idx < mt * kFTile; idx += blockDim.x) {
        const int o = idx / kFTile, p = idx % kFTile;
        const double* Tp = Ts + p * LP1;
        double q = 0.0;
        if (o < P.m0) {
            for (int l = 0; l < P.nb0; ++l) q += Tp[l] * P.Qm0[l * P.m0 + o];
        } else {
            const int oo = o - P.m0;
            for (int l = 0; l < P.nb1; ++l) q += Tp[l] * P.Qm1[l * P.m1 + oo];
            q *= rh[p];
        }
        Qs[o * kFTile + p] = (T)q;
    }
    __syncthreads();
    for (int col = threadIdx.x; col < P.nF; col += blockDim.x) {
        const int par = P.colpar[col];
        const int ob = par ? P.m0 : 0, mp = par ? P.m1 : P.m0;
        T acc[kFTile];
#pragma unroll
        for (int p = 0; p < kFTile; ++p) acc[p] = (T)0;
        for (int l = 0; l < mp; ++l) {
            const T w = Wt[(int64_t)l * P.nF + col];
            const T* q = Qs + (ob + l) * kFTile;
#pragma unroll
            for (int p = 0; p < kFTile; ++p) acc[p] += q[p] * w;
        }
#pragma unroll
        for (int p = 0; p < kFTile; ++p)
            if (p < cnt) F[(t0 + p) * P.ldF + col] = acc[p];
    }
    __syncthreads();
}

// Per point: B_par (FP64) -> Q_par = B_par Qmat_par (FP64, the orthonormalised radial basis
// of Eq. svd) -> F[i, col] = sum_l Q_par(col)[l] Wt[l, col] (type T).  Tiles of 32 points.
template <typename T>
__global__ void __launch_bounds__(256) k_radial_F(RFParams P) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int64_t ntiles = (P.n + kFTile - 1) / kFTile;
    for (int64_t tile = blockIdx.x; tile < ntiles; tile += gridDim.x) radialF_tile<T>(P, tile * kFTile, smem_raw);
}

// Shared memory of k_radial_F_df: QC, Wt (when staged), two buffers of basis values and one of Q for
// each of `tiles` tiles.
__host__ __device__ inline size_t radialF_df_basis_bytes(int L) {
    return align16(sizeof(float2) * kFTile * (L + 1) + sizeof(float) * kFTile);
}
__host__ __device__ inline size_t radialF_df_smem(int L, int m0, int m1, int mtp, int nF, bool stage_wt, int tiles) {
    const int mmax = m0 > m1 ? m0 : m1;
    return align16(sizeof(float2) * (size_t)(L + 1) * mtp) +
           (stage_wt ? align16(sizeof(float) * (size_t)mmax * nF) : 0) +
           tiles * (2 * radialF_df_basis_bytes(L) + sizeof(float) * (size_t)(m0 + m1) * kFTile);
}

// Outputs per Q unit (2, 4 or 8) for mt outputs of `tiles` tiles over `warps` warps: the fewest
// outputs per warp after rounding, larger groups on ties (fewer shared loads per output).
__host__ __device__ inline int radialF_df_kopt(int mt, int tiles, int warps) {
    int best = 8, cost = 1 << 30;
    for (int k = 8; k >= 2; k /= 2) {
        const int units = tiles * ((mt + k - 1) / k);
        const int c = ((units + warps - 1) / warps) * k;
        if (c < cost) { cost = c; best = k; }
    }
    return best;
}

// FP32 factors, one CTA of kRfThreads per SM, P.tiles tiles of kFTile points between two barriers:
// the basis of the CTA's next tiles and the Q units of the current ones, then the F units, warps
// taking units from a counter.  QC (and Wt when P.stage_wt) are staged per CTA.  Bound by the FP32
// issue of the Dot2 products; with one tile between barriers (warp 0 forming the next basis, the
// others a fixed share of Q) the warps waited for one another half of the time: 1,000,000 points,
// L = 32 2.57 -> 2.45 ms, 500,000 points, d = 4, L = 14 0.44 -> 0.23.
constexpr int kRfThreads = 512;
template <int KOPT>
static __global__ void __launch_bounds__(kRfThreads, 1) k_radial_F_df(RFParams P) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ int counter[2];
    const int LP1 = P.L + 1, mt = P.m0 + P.m1, NT = P.tiles;
    const int mmax = P.m0 > P.m1 ? P.m0 : P.m1;
    const int lane = threadIdx.x & 31;
    unsigned char* sp = smem_raw;
    float2* QC = reinterpret_cast<float2*>(sp);
    sp += align16(sizeof(float2) * (size_t)LP1 * P.mtp);
    const float* Ws = reinterpret_cast<const float*>(P.Wt);
    if (P.stage_wt) {
        float* w = reinterpret_cast<float*>(sp);
        for (int t = threadIdx.x; t < mmax * P.nF; t += blockDim.x) w[t] = reinterpret_cast<const float*>(P.Wt)[t];
        Ws = w;
        sp += align16(sizeof(float) * (size_t)mmax * P.nF);
    }
    const size_t bb = radialF_df_basis_bytes(P.L);
    unsigned char* basis = sp;                   // [2][NT]
    float* Qs = reinterpret_cast<float*>(sp + 2 * NT * bb);
    auto Tb = [&](int buf, int q) { return reinterpret_cast<float2*>(basis + (buf * NT + q) * bb); };
    for (int t = threadIdx.x; t < LP1 * P.mtp; t += blockDim.x) QC[t] = P.QC[t];
    const int64_t ntiles = (P.n + kFTile - 1) / kFTile;
    const int64_t nsup = (ntiles + NT - 1) / NT;
    auto form_basis = [&](int64_t sup, int q, int buf) {
        const int64_t t0 = (sup * NT + q) * kFTile;
        float2* T = Tb(buf, q);
        radialF_df_basis(P, t0, lane, T, reinterpret_cast<float*>(T + kFTile * LP1));
    };
    if (threadIdx.x < 2) counter[threadIdx.x] = 0;
    if (blockIdx.x < nsup && (int)(threadIdx.x >> 5) < NT) form_basis(blockIdx.x, threadIdx.x >> 5, 0);
    __syncthreads();
    const int groups = (mt + KOPT - 1) / KOPT, fgroups = (int)((P.ldF + 31) / 32);
    int cur = 0;
    for (int64_t sup = blockIdx.x; sup < nsup; sup += gridDim.x, cur ^= 1) {
        const int64_t nxt = sup + gridDim.x;
        const int nt = (int)min((int64_t)NT, ntiles - sup * NT);
        const int nb = nxt < nsup ? (int)min((int64_t)NT, ntiles - nxt * NT) : 0;
        for (int u = next_unit(&counter[0], lane); u < nb + nt * groups; u = next_unit(&counter[0], lane)) {
            if (u < nb) {
                form_basis(nxt, u, cur ^ 1);
            } else {
                const int q = (u - nb) / groups, g = (u - nb) % groups;
                const float2* T = Tb(cur, q);
                radialF_df_q<KOPT>(P, T, reinterpret_cast<const float*>(T + kFTile * LP1), QC,
                                   Qs + (size_t)q * mt * kFTile, g * KOPT, lane);
            }
        }
        __syncthreads();
        if (threadIdx.x == 0) counter[0] = 0;    // every warp is past its last unit; read again after the barrier below
        for (int u = next_unit(&counter[1], lane); u < nt * fgroups; u = next_unit(&counter[1], lane)) {
            const int q = u / fgroups, g = u % fgroups;
            radialF_df_f(P, (sup * NT + q) * kFTile, Qs + (size_t)q * mt * kFTile, Ws, 32 * g, lane);
        }
        __syncthreads();
        if (threadIdx.x == 0) counter[1] = 0;    // likewise, before the next F units' barrier
    }
}

// ------------------------------------------------------- A5b: harmonics and U writer
// One warp per point.  Solid-harmonic form of the real hyperspherical harmonics:
//   Y = prod_j P_j(|mu_{j+1}|, mu_j - |mu_{j+1}|) * N_phi * {Re|Im} (x0 + i x1)^{|mu_{d-2}|},
//   P_j(m, n) = s_n r_j^n C_n^{m + alpha_j}(x_{D_j} / r_j),  D_j = d-1-j, r_j^2 = sum_{i<=D_j} x_i^2,
// a polynomial in (x_{D_j}, r_j^2) from the normalised three-term recurrence (coefA/coefB).
// Per-warp shared: level tables, trig powers, Y for all used harmonics, the point's F row.
template <typename T> struct Vec16;                      // columns per 16 bytes
template <> struct Vec16<float> { typedef float4 type; static constexpr int w = 4; };
template <> struct Vec16<double> { typedef double2 type; static constexpr int w = 2; };

// How a warp gets a harmonic: looked up in the point's slots (all harmonics formed first), formed
// per column from G and the prefix levels, or from a table of every level and the trigonometric
// factors (only where the first two do not leave eight warps per SM).
enum UWMode { kSlots = 0, kProducts = 1, kChains = 2 };
// Column descriptors: read from global memory by 16-byte chunk, the same staged in shared memory, or
// one word per column in shared memory.
enum UWDesc { kGlobal = 0, kChunks = 1, kColumns = 2 };

struct UWParams {
    const double* x; int64_t n; int d; Center c; double inv2R;
    int L;                     // highest harmonic degree with kept columns
    int tri;                   // (L+1)(L+2)/2
    const int16_t* chains;     // nH x cstride: level offsets, trig index, zero padding
    int nH, cstride;
    const int32_t* ychain;     // nYp padded harmonic slots -> chain (-1: padding)
    int nYp;
    const int32_t* gbase;      // d = 3: slot of (k, m = 0)
    const uint32_t* ydesc; int yw;   // d >= 4: per slot, factors of the harmonic (see make_tables)
    const uint32_t* qdesc;     // ldU / VW chunks, two words each (see make_tables)
    int nF;
    const void* F; int64_t ldF;
    void* U; int64_t ldU;
    const void* coefA; const void* coefB;   // (d-2) x tri, type T
    int per_warp;              // shared elements (type T) per warp (an equal part per group of lanes)
    int tab_bytes;             // bytes of index tables staged in shared memory (0: read from global)
};

// The index tables the U writer reads for every point (global, or staged in shared memory).
template <int N> struct Count { static constexpr int value = N; };

struct UWTabs {
    const uint32_t* qdesc;     // two words per chunk (see make_tables)
    const uint32_t* cdesc;     // kColumns: one word per column
    const int16_t* chains;     // kChains
    const int32_t* ychain;
    const int32_t* gbase;      // kSlots, d = 3
    const uint32_t* ydesc;     // kSlots and kProducts, d >= 4
};

// Bytes of the staged index tables: the column descriptors, and (kSlots) gbase or ydesc, (kChains)
// chains and ychain; the kernel lays them out in this order, each 16-byte aligned.  kProducts
// reads ydesc from global memory.
__host__ __device__ inline size_t uwriter_tab_bytes(int64_t ldU, int vw, int nH, int cstride, int nYp, int levels, int L,
                                                    int yw, int mode, int desc) {
    if (desc == kGlobal) return 0;
    const size_t q = desc == kColumns ? align16(sizeof(uint32_t) * ldU) : align16(sizeof(uint32_t) * 2 * (ldU / vw));
    if (mode == kSlots)
        return q + (levels == 1 ? align16(sizeof(int32_t) * (size_t)(L + 1)) : align16(sizeof(uint32_t) * (size_t)yw * nYp));
    if (mode == kProducts) return q;
    return q + align16(sizeof(int16_t) * (size_t)nH * cstride) + align16(sizeof(int32_t) * (size_t)nYp);
}

// Elements of a warp's G table (d >= 4: (L + 1)^2 and a zero; d = 3 writes the slots directly).
__host__ __device__ inline int uwriter_g_size(int levels, int L) { return levels == 1 ? 0 : (L + 1) * (L + 1) + 1; }

// Shared elements (type T) per warp of the U writer (a multiple of 16 bytes).
__host__ __device__ inline int uwriter_per_warp(int levels, int tri, int L, int nYp, int nF, int mode) {
    const int harm = mode == kChains ? levels * tri + 2 * L + 1
                                     : (mode == kSlots ? nYp : 0) + (levels - 1) * tri + uwriter_g_size(levels, L);
    return (harm + nF + 1 + 3) & ~3;
}

// This lane's centre coordinate (compile-time indices: the centre stays in registers).
__device__ __forceinline__ double lane_centre(const Center& cen, int lane) {
    double cj = cen.c[0];
#pragma unroll
    for (int j = 1; j < kMaxD; ++j) cj = (lane == j) ? cen.c[j] : cj;
    return cj;
}

// A group of GL lanes (32, 16 or 8) forms one point's row; `lane` is the lane within the group.

// Direction x_hat of point i: differences in FP64, normalisation in the bulk precision T; the
// zero vector gets e_0.  Lane j forms coordinate j (x_lane: loaded ahead by the caller; cj: its
// centre) and the warp shares it by shuffles, since an FP64 instruction holds the pipe for 16 cycles
// whatever its active lanes.  xh is indexed with compile-time indices only (loops over kMaxD with
// the dimension as a predicate), so that it stays in registers.
template <typename T, int GL>
__device__ __forceinline__ void point_direction(const double* __restrict__ x, int d, double cj, double inv2R, int64_t i,
                                                int lane, bool have_x, double x_lane, T* xh) {
    T s = (T)0;
    const T xt = (T)((lane < d) ? ((have_x ? x_lane : x[i * d + lane]) - cj) * inv2R : 0.0);
#pragma unroll
    for (int j = 0; j < kMaxD; ++j) {
        if (sizeof(T) == 4 || j < d) {
            xh[j] = __shfl_sync(0xffffffffu, xt, j, GL);          // zero for j >= d
            s += xh[j] * xh[j];
        } else {
            xh[j] = (T)0;
        }
    }
    if (s > (T)0) {
        const T inv = (T)1 / sqrt(s);
#pragma unroll
        for (int j = 0; j < kMaxD; ++j)
            if (sizeof(T) == 4 || j < d) xh[j] *= inv;
    } else {
#pragma unroll
        for (int j = 0; j < kMaxD; ++j) xh[j] = (j == 0) ? (T)1 : (T)0;
    }
}

// Level table j (j < levels) of the normalised three-term recurrences, lanes over mu'.
template <typename T, int GL>
__device__ __forceinline__ void level_table(const T* xh, int d, int j, int L, int tri, const T* cA, const T* cB, T* tb,
                                            int lane) {
    const int D = d - 1 - j;
    T q = (T)0, z = (T)0;
#pragma unroll
    for (int m = 0; m < kMaxD; ++m) {
        if (m <= D) q += xh[m] * xh[m];
        if (m == D) z = xh[m];
    }
    const T qq = q;
    const T* A = cA + j * tri;
    const T* B = cB + j * tri;
    for (int mu = lane; mu <= L; mu += GL) {
        const int o = mu * (L + 1) - mu * (mu - 1) / 2;
        const int nmax = L - mu;
        T pm2 = A[o];
        tb[o] = pm2;
        if (nmax >= 1) {
            T pm1 = A[o + 1] * z;
            tb[o + 1] = pm1;
            for (int nn = 2; nn <= nmax; ++nn) {
                const T pn = A[o + nn] * z * pm1 - B[o + nn] * qq * pm2;
                tb[o + nn] = pn;
                pm2 = pm1;
                pm1 = pn;
            }
        }
    }
}

// Powers (x0 + i x1)^m for the exponents m = lane, lane + GL, .. <= L of a group's lanes.  FP64: a scan
// of products over the lanes, five steps at most, then a factor per GL exponents; binary powering
// takes a product and a square per step and an FP64 instruction holds its pipe for 16 cycles (200,000
// points, d = 3, rank 66 with this and the shared direction: 1.39 -> 1.08 ms).  FP32: binary
// powering (the scan's shuffles made rows 2 to 5% slower).
template <typename T, int GL> struct TrigPowers {
    T x0, x1, re, im, sr, si;
    __device__ __forceinline__ TrigPowers(T a, T b, int L, int lane) : x0(a), x1(b) {
        if constexpr (sizeof(T) == 8) {
            re = lane ? a : (T)1;
            im = lane ? b : (T)0;
#pragma unroll
            for (int off = 1; off < GL; off <<= 1) {
                if (off > L) break;
                const T ur = __shfl_up_sync(0xffffffffu, re, off, GL), ui = __shfl_up_sync(0xffffffffu, im, off, GL);
                const T t = re * ur - im * ui, v = re * ui + im * ur;
                if (lane >= off) { re = t; im = v; }
            }
            if (L >= GL) {
                const T r = __shfl_sync(0xffffffffu, re, GL - 1, GL), i = __shfl_sync(0xffffffffu, im, GL - 1, GL);
                sr = r * a - i * b;
                si = r * b + i * a;
            }
        }
    }
    // the power m; FP64: called for m = lane, lane + GL, .. in turn
    __device__ __forceinline__ void get(int m, T& rr, T& ri) {
        if constexpr (sizeof(T) == 8) {
            if (m >= GL) { const T t = re * sr - im * si; im = re * si + im * sr; re = t; }
            rr = re;
            ri = im;
        } else {
            T br = x0, bi = x1;
            rr = (T)1;
            ri = (T)0;
            for (int e = m; e; e >>= 1) {
                if (e & 1) { const T t = rr * br - ri * bi; ri = rr * bi + ri * br; rr = t; }
                const T t = br * br - bi * bi;
                bi = (T)2 * br * bi;
                br = t;
            }
        }
    }
};

// The direction of point i, then the level tables (levels x tri, lanes over mu') and the
// trigonometric powers (x0 + i x1)^mu times the normalisers (2L+1, index L + mu), written by one
// warp into its shared tbl and trig.
template <typename T>
__device__ __forceinline__ void point_harmonic_tables(const double* __restrict__ x, int d, double cj,
                                                      double inv2R, int L, int tri, const T* cA, const T* cB,
                                                      T* tbl, T* trig, int64_t i, int lane, bool have_x = false,
                                                      double x_lane = 0.0) {
    const int levels = d - 2;
    T xh[kMaxD];
    point_direction<T, 32>(x, d, cj, inv2R, i, lane, have_x, x_lane, xh);
    for (int j = 0; j < levels; ++j) level_table<T, 32>(xh, d, j, L, tri, cA, cB, tbl + j * tri, lane);
    TrigPowers<T, 32> pw(xh[0], xh[1], L, lane);
    for (int mu = lane; mu <= L; mu += 32) {
        T rr, ri;
        pw.get(mu, rr, ri);
        if (mu == 0) {
            trig[L] = (T)0.3989422804014327;             // 1/sqrt(2 pi)
        } else {
            trig[L + mu] = rr * (T)0.5641895835477563;   // 1/sqrt(pi)
            trig[L - mu] = ri * (T)0.5641895835477563;
        }
    }
}

// The harmonic of slot y (d >= 4): G[g] times its prefix.
template <typename T>
__device__ __forceinline__ T slot_product(const uint32_t* ydesc, uint32_t y, int levels, const T* Pl, const T* G) {
    if (levels <= 4) {
        const uint2 w = *reinterpret_cast<const uint2*>(ydesc + 2 * (size_t)y);
        T v = G[w.x & 0xffffu] * Pl[w.x >> 16];
        if (levels >= 3) v *= Pl[w.y & 0xffffu];
        if (levels >= 4) v *= Pl[w.y >> 16];
        return v;
    }
    const uint4 w = *reinterpret_cast<const uint4*>(ydesc + 4 * (size_t)y);
    T v = G[w.x & 0xffffu] * Pl[w.x >> 16] * Pl[w.y & 0xffffu] * Pl[w.y >> 16] * Pl[w.z & 0xffffu];
    if (levels >= 6) v *= Pl[w.z >> 16];
    return v;
}

// All harmonics of point i into the warp's slots Ys.  Lane m runs the last level's recurrence and
// multiplies each value by the trigonometric factors +-m at once: in d = 3 these are the harmonics
// and go to their slots, for d >= 4 they form G, and slot y is G[g] times its prefix (the tables Pl of the
// levels before the last).  With a table of every level, one of the trigonometric factors and a
// pass over the chains (two or more index words and as many factors per harmonic), the harmonics
// took more than half of the instructions of a row at some hundred columns.  slots = false stops at
// the prefix levels and G.
template <typename T, int GL>
__device__ __forceinline__ void point_harmonics(const double* __restrict__ x, int d, double cj, double inv2R, int L,
                                                int tri, const T* cA, const T* cB, const int32_t* gbase,
                                                const uint32_t* ydesc, int nYp, T* Ys, T* Pl, T* G, int64_t i, int lane,
                                                bool have_x, double x_lane, bool slots) {
    const int levels = d - 2;
    T xh[kMaxD];
    point_direction<T, GL>(x, d, cj, inv2R, i, lane, have_x, x_lane, xh);
    for (int j = 0; j < levels - 1; ++j) level_table<T, GL>(xh, d, j, L, tri, cA, cB, Pl + j * tri, lane);
    const T z = xh[2], qq = xh[0] * xh[0] + xh[1] * xh[1] + xh[2] * xh[2];
    const T* A = cA + (levels - 1) * tri;
    const T* B = cB + (levels - 1) * tri;
    TrigPowers<T, GL> pw(xh[0], xh[1], L, lane);
    for (int m = lane; m <= L; m += GL) {
        T rr, ri;
        pw.get(m, rr, ri);
        rr *= m == 0 ? (T)0.3989422804014327 : (T)0.5641895835477563;    // 1/sqrt(2 pi), 1/sqrt(pi)
        ri *= (T)0.5641895835477563;
        const T* a = A + m * (L + 1) - m * (m - 1) / 2 - m;              // indexed by mu = m + n
        const T* b = B + (a - A);
        auto put = [&](int mu, T v) {
            if (levels == 1) {
                const int g = gbase[mu];
                if (g >= 0) {
                    Ys[g + m] = v * rr;
                    if (m > 0) Ys[g - m] = v * ri;
                }
            } else {
                T* g = G + mu * (mu + 1);
                g[m] = v * rr;
                if (m > 0) g[-m] = v * ri;
            }
        };
        T p2 = a[m];
        put(m, p2);
        if (m == L) continue;
        T p1 = a[m + 1] * z;
        put(m + 1, p1);
#pragma unroll 2
        for (int mu = m + 2; mu <= L; ++mu) {
            const T v = a[mu] * z * p1 - b[mu] * qq * p2;
            put(mu, v);
            p2 = p1;
            p1 = v;
        }
    }
    if (levels == 1 || !slots) return;
    __syncwarp();
    for (int y = lane; y < nYp; y += GL) Ys[y] = slot_product<T>(ydesc, y, levels, Pl, G);
}

// One point's U row, executed by one warp.  cA/cB: level recurrences in shared memory;
// base: this warp's shared area (P.per_warp elements, 16-byte aligned), laid out as [harmonic
// slots (kSlots)] [level tables but the last] [G] [radial factors], or (kChains) [level tables] [trig
// powers] [radial factors].  Column c is one radial factor times one harmonic.  With slots a lane
// writes a 16-byte chunk of the row, whose two descriptor words name the one or two (k, s) blocks it
// meets; otherwise lane l forms the columns l, l + 32, .. (consecutive words of the tables).  Slots
// with a column per lane measured 6.88 -> 7.55 ms at 1,000,000 x 10,680 (d = 3) and 3 to 7% less at
// d = 4, rank 1,000 to 5,000.
// The radial-factor slots of a warp's shared area (nF + 1, the last one zero).
template <typename T>
__device__ __forceinline__ T* uwriter_fs(const UWParams& P, int mode, T* base) {
    const int levels = P.d - 2;
    return base + (mode == kChains ? levels * P.tri + 2 * P.L + 1
                                   : (mode == kSlots ? P.nYp : 0) + (levels - 1) * P.tri + uwriter_g_size(levels, P.L));
}

// Radial factors and coordinate of one point loaded into registers one point ahead of use (FP32
// factors with nF <= GL kPfF): lane l holds F[i, l + GL k] and x[i, l] (l < d), so that their
// global-memory latency passes while the previous row is written.
constexpr int kPfF = 16;
template <typename T> struct PointPre { T f[kPfF]; double x; };
template <typename T, int GL>
__device__ __forceinline__ void point_prefetch(const UWParams& P, int64_t i, int lane, PointPre<T>& pp) {
    const T* Fg = reinterpret_cast<const T*>(P.F) + i * P.ldF;
#pragma unroll
    for (int k = 0; k < kPfF; ++k) {
        if (GL * k >= P.nF) break;
        const int f = lane + GL * k;
        pp.f[k] = (f < P.nF) ? Fg[f] : (T)0;
    }
    pp.x = (lane < P.d) ? P.x[i * P.d + lane] : 0.0;
}
template <typename T, int GL>
__device__ __forceinline__ void point_stage_f(const UWParams& P, const PointPre<T>& pp, T* Fs, int lane) {
#pragma unroll
    for (int k = 0; k < kPfF; ++k) {
        if (GL * k >= P.nF) break;
        const int f = lane + GL * k;
        if (f < P.nF) Fs[f] = pp.f[k];
    }
}

// Descriptor of column c, F index << 20 | slot, from the two words of its 16-byte chunk.
template <int VW>
__device__ __forceinline__ uint32_t uwriter_column(const uint32_t* qdesc, int64_t c) {
    const int64_t q = c / VW;
    const uint32_t u = (uint32_t)(c % VW);
    const uint32_t w0 = qdesc[2 * q], e = (w0 >> 18) & 3u;
    if (e == 0 || u < e) return (w0 & 0xFFF00000u) | ((w0 & 0x3FFFFu) + u);
    const uint32_t w1 = qdesc[2 * q + 1];
    return (w1 & 0xFFF00000u) | ((w1 & 0xFFFFFu) + u - e);
}

template <typename T, int MODE, int DESC, int GL>
__device__ __forceinline__ void uwriter_point(const UWParams& P, const UWTabs& X, double cj, int64_t i, bool valid,
                                              const T* cA, const T* cB, T* base, int lane, bool staged = false, double x_lane = 0.0) {
    const int levels = P.d - 2;
    T* Ys = base;                                            // nYp (kSlots)
    T* Pl = base + (MODE == kSlots ? P.nYp : 0);             // (levels - 1) * tri
    T* G = Pl + (levels - 1) * P.tri;
    T* tbl = base;                                           // kChains: levels * tri, then 2L+1 trig, index L + mu
    T* trig = tbl + levels * P.tri;
    T* Fs = uwriter_fs<T>(P, MODE, base);                    // nF + 1
    const T* Fg = reinterpret_cast<const T*>(P.F);
    if (MODE != kChains)
        point_harmonics<T, GL>(P.x, P.d, cj, P.inv2R, P.L, P.tri, cA, cB, X.gbase, X.ydesc, P.nYp, Ys, Pl, G, i, lane,
                           staged, x_lane, MODE == kSlots);
    else
        point_harmonic_tables<T>(P.x, P.d, cj, P.inv2R, P.L, P.tri, cA, cB, tbl, trig, i, lane, staged, x_lane);
    // this point's radial factors (staged: already in Fs, written by the caller)
    if (!staged) {
        for (int f = lane; f < P.nF; f += GL) Fs[f] = Fg[i * P.ldF + f];
        if (lane == 0) Fs[P.nF] = (T)0;
    }
    __syncwarp();
    auto column = [&](int64_t c) -> T {
        const uint32_t w = DESC == kColumns ? X.cdesc[c] : uwriter_column<Vec16<T>::w>(X.qdesc, c);
        const T f = Fs[w >> 20];
        const uint32_t y = w & 0xFFFFFu;
        if constexpr (MODE == kProducts) return f * slot_product<T>(X.ydesc, y, levels, Pl, G);
        const int ch = X.ychain[y];
        if (ch < 0) return (T)0;
        const int16_t* q = X.chains + (int64_t)ch * P.cstride;
        T h = trig[P.L + q[levels]];
        for (int j = 0; j < levels; ++j) h *= tbl[j * P.tri + q[j]];
        return f * h;
    };
    T* row = reinterpret_cast<T*>(P.U) + i * P.ldU;
    if constexpr (MODE == kSlots) {
        // a 16-byte chunk per lane, four (FP64: two) in flight: one or two runs of consecutive slots, in
        // one branch-free form (e = 0 reads as e = VW; the second word of a whole chunk names valid
        // slots and is never selected), so that the lanes of a warp do not diverge
        typedef typename Vec16<T>::type VT;
        constexpr int VW = Vec16<T>::w, NQ = VW;
        auto chunk = [&](int64_t q) {
            const uint2 w = *reinterpret_cast<const uint2*>(X.qdesc + 2 * q);
            const uint32_t e = (w.x >> 18) & 3u, ea = e ? e : (uint32_t)VW;
            const T fa = Fs[w.x >> 20], fb = Fs[w.y >> 20];
            const uint32_t ya = w.x & 0x3FFFFu, yb = (w.y & 0xFFFFFu) - ea;
            T v[VW];
            v[0] = fa * Ys[ya];
#pragma unroll
            for (int u = 1; u < VW; ++u) {
                const bool a = (uint32_t)u < ea;
                v[u] = (a ? fa : fb) * Ys[a ? ya + u : yb + u];
            }
            VT out;
            if constexpr (VW == 4) { out.x = v[0]; out.y = v[1]; out.z = v[2]; out.w = v[3]; }
            else { out.x = v[0]; out.y = v[1]; }
            return out;
        };
        VT* rq = reinterpret_cast<VT*>(row);
        const int64_t nq = valid ? P.ldU / VW : 0;
        int64_t q = lane;
        auto batch = [&](auto cnt) {
            constexpr int N = decltype(cnt)::value;
            VT o[N];
#pragma unroll
            for (int f = 0; f < N; ++f) o[f] = chunk(q + GL * f);
#pragma unroll
            for (int f = 0; f < N; ++f) rq[q + GL * f] = o[f];
            q += GL * N;
        };
        while (q + GL * (NQ - 1) < nq) batch(Count<NQ>());
        if (NQ > 2 && q + GL < nq) batch(Count<2>());
        while (q < nq) batch(Count<1>());
        __syncwarp();
        return;
    }
    constexpr int NF = 4;                                    // columns in flight per lane
    int64_t c = lane;
    for (; c + 32 * (NF - 1) < P.ldU; c += 32 * NF) {
        T o[NF];
#pragma unroll
        for (int f = 0; f < NF; ++f) o[f] = column(c + 32 * f);
#pragma unroll
        for (int f = 0; f < NF; ++f) row[c + 32 * f] = o[f];
    }
    for (; c < P.ldU; c += 32) row[c] = column(c);
    __syncwarp();
}

// Zeroes a warp's harmonic slots and G's last entry once (padding slots of d = 3 and that entry are
// never written afterwards).
template <typename T, int MODE, int GL>
__device__ __forceinline__ void uwriter_zero_slots(const UWParams& P, T* base, int lane) {
    if (MODE == kSlots)
        for (int g = lane; g < P.nYp; g += GL) base[g] = (T)0;
    if (MODE != kChains && P.d > 3 && lane == 0) uwriter_fs<T>(P, MODE, base)[-1] = (T)0;
    __syncwarp();
}

// Stages a set's coefficient tables (cA, cB: 2 levels tri elements) and, from `tp` on, its index
// tables (uwriter_tab_bytes) into shared memory; the caller synchronises.
template <typename T, int MODE, int DESC>
__device__ __forceinline__ UWTabs uwriter_stage(const UWParams& P, T* cA, unsigned char* tp) {
    const int levels = P.d - 2;
    T* cB = cA + levels * P.tri;
    for (int idx = threadIdx.x; idx < levels * P.tri; idx += blockDim.x) {
        cA[idx] = reinterpret_cast<const T*>(P.coefA)[idx];
        cB[idx] = reinterpret_cast<const T*>(P.coefB)[idx];
    }
    UWTabs X{P.qdesc, nullptr, P.chains, P.ychain, P.gbase, P.ydesc};
    if constexpr (DESC != kGlobal) {
        // staged in shared memory (a compile-time choice, so that the table reads compile to
        // shared-memory loads)
        uint32_t* q = reinterpret_cast<uint32_t*>(tp);
        if constexpr (DESC == kColumns) {
            for (int64_t k = threadIdx.x; k < P.ldU; k += blockDim.x) q[k] = uwriter_column<Vec16<T>::w>(P.qdesc, k);
            X.cdesc = q;
            tp += align16(sizeof(uint32_t) * P.ldU);
        } else {
            const int64_t nw = 2 * (P.ldU / Vec16<T>::w);
            for (int64_t k = threadIdx.x; k < nw; k += blockDim.x) q[k] = P.qdesc[k];
            X.qdesc = q;
            tp += align16(sizeof(uint32_t) * nw);
        }
        if (MODE == kSlots && levels == 1) {
            int32_t* gb = reinterpret_cast<int32_t*>(tp);
            for (int k = threadIdx.x; k <= P.L; k += blockDim.x) gb[k] = P.gbase[k];
            X.gbase = gb;
        } else if (MODE == kSlots) {
            uint32_t* yd = reinterpret_cast<uint32_t*>(tp);
            for (int k = threadIdx.x; k < P.yw * P.nYp; k += blockDim.x) yd[k] = P.ydesc[k];
            X.ydesc = yd;
        } else if (MODE == kChains) {
            int16_t* ch = reinterpret_cast<int16_t*>(tp);
            for (int64_t k = threadIdx.x; k < (int64_t)P.nH * P.cstride; k += blockDim.x) ch[k] = P.chains[k];
            tp += align16(sizeof(int16_t) * (size_t)P.nH * P.cstride);
            X.chains = ch;
            int32_t* yc = reinterpret_cast<int32_t*>(tp);
            for (int k = threadIdx.x; k < P.nYp; k += blockDim.x) yc[k] = P.ychain[k];
            X.ychain = yc;
        }
    }
    return X;
}

// The rows of a warp, 32 / GL points at a time, GL lanes each: points i, i + 1, .. (one per group), then
// i + step, .., below end.  wbase: the warp's area, an equal part per group.  PF: the next point's
// radial factors and coordinate travel in registers during this row (nF <= GL kPfF).  Groups of 16 or
// 8 lanes are for degrees below 16 or 8, where the rest of the warp has no recurrence of its own and
// a warp's instructions, bound by their issue, serve two or four points: 200,000 points, d = 3, FP32 rank
// 322 0.182 -> 0.106 ms, FP64 rank 66 1.08 -> 0.30 and rank 490 1.83 -> 1.03.
template <typename T, int MODE, bool PF, int DESC, int GL>
__device__ __forceinline__ void uwriter_rows(const UWParams& P, const UWTabs& X, const T* cA, const T* cB, T* wbase,
                                             int64_t i, int64_t step, int64_t end) {
    const int lane = threadIdx.x & (GL - 1), group = (threadIdx.x & 31) / GL;
    T* base = wbase + (size_t)group * (P.per_warp / (32 / GL));
    uwriter_zero_slots<T, MODE, GL>(P, base, lane);
    const double cj = lane_centre(P.c, lane);
    if constexpr (PF) {
        T* Fs = uwriter_fs<T>(P, MODE, base);
        if (lane == 0) Fs[P.nF] = (T)0;
        PointPre<T> pp;
        if (i < end) point_prefetch<T, GL>(P, min(i + group, end - 1), lane, pp);
        for (; i < end; i += step) {
            point_stage_f<T, GL>(P, pp, Fs, lane);
            const double xl = pp.x;
            if (i + step < end) point_prefetch<T, GL>(P, min(i + step + group, end - 1), lane, pp);
            uwriter_point<T, MODE, DESC, GL>(P, X, cj, min(i + group, end - 1), i + group < end, cA, cB, base, lane, true, xl);
        }
    } else {
        for (; i < end; i += step)
            uwriter_point<T, MODE, DESC, GL>(P, X, cj, min(i + group, end - 1), i + group < end, cA, cB, base, lane);
    }
}

// Shared memory: [nwarps x per_warp elements][cA][cB][staged index tables (tab_bytes)].
template <typename T>
__device__ __forceinline__ unsigned char* uwriter_tabs_at(const UWParams& P, unsigned char* smem, int nwarps) {
    return smem + align16(sizeof(T) * ((size_t)nwarps * P.per_warp + 2 * (size_t)(P.d - 2) * P.tri));
}

template <typename T, int MODE, bool PF, int DESC, int GL>
__global__ void __launch_bounds__(1024) k_uwriter(UWParams P) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
    T* base = reinterpret_cast<T*>(smem_raw) + (size_t)warp * P.per_warp;
    T* cA = reinterpret_cast<T*>(smem_raw) + (size_t)nwarps * P.per_warp;
    const UWTabs X = uwriter_stage<T, MODE, DESC>(P, cA, uwriter_tabs_at<T>(P, smem_raw, nwarps));
    __syncthreads();
    constexpr int G = 32 / GL;
    uwriter_rows<T, MODE, PF, DESC, GL>(P, X, cA, cA + (P.d - 2) * P.tri, base,
                                        ((int64_t)blockIdx.x * nwarps + warp) * G, (int64_t)gridDim.x * nwarps * G, P.n);
}

// --------------------------------------------------------------------- A7: matvec
// Register-tiled GEMMs on the CUDA cores.  CT = padded column count of the V block (c <= CT).
// U^T V: a block owns 128 (256 when CT = 1) columns of U and a chunk of rows; each thread
// keeps a TA x TJ tile of the product.  Partials per chunk are summed in FP64 afterwards.
template <int CT> struct UtvShape {
    static constexpr int AB = (CT == 1) ? 256 : 128;                       // columns per block
    static constexpr int TA = (CT >= 8) ? 4 : (CT == 4 ? 2 : 1);            // columns per thread
    static constexpr int TJ = (CT * (AB / TA)) / 256;                       // V columns per thread
};
constexpr int kKT = 32;     // rows (k) per shared tile

template <typename T, int N> struct VecLd;
template <typename T> struct VecLd<T, 1> { static __device__ __forceinline__ void ld(const T* p, T* o) { o[0] = p[0]; } };
template <typename T> struct VecLd<T, 2> {
    static __device__ __forceinline__ void ld(const T* p, T* o) { o[0] = p[0]; o[1] = p[1]; }
};
template <> struct VecLd<float, 4> {
    static __device__ __forceinline__ void ld(const float* p, float* o) {
        const float4 v = *reinterpret_cast<const float4*>(p); o[0] = v.x; o[1] = v.y; o[2] = v.z; o[3] = v.w;
    }
};
template <> struct VecLd<double, 4> {
    static __device__ __forceinline__ void ld(const double* p, double* o) {
        const double2 a = *reinterpret_cast<const double2*>(p), b = *reinterpret_cast<const double2*>(p + 2);
        o[0] = a.x; o[1] = a.y; o[2] = b.x; o[3] = b.y;
    }
};
template <> struct VecLd<float, 8> {
    static __device__ __forceinline__ void ld(const float* p, float* o) { VecLd<float, 4>::ld(p, o); VecLd<float, 4>::ld(p + 4, o + 4); }
};
template <> struct VecLd<double, 8> {
    static __device__ __forceinline__ void ld(const double* p, double* o) { VecLd<double, 4>::ld(p, o); VecLd<double, 4>::ld(p + 4, o + 4); }
};

// part_chunk[j * r + a] = sum_{i0 <= i < i1} U[i, a] V[i + j ldv] for the columns [a0, a0 + AB).
template <typename T, int CT>
__device__ __forceinline__ void utv_tile_body(const T* __restrict__ U, int64_t ldU, int64_t r,
                                              const T* __restrict__ V, int64_t ldv, int c, int64_t i0, int64_t i1,
                                              int64_t a0, double* __restrict__ part_chunk,
                                              T (*Us)[UtvShape<CT>::AB], T (*Vs)[CT]) {
    using S = UtvShape<CT>;
    const int t = threadIdx.x;
    const int tx = t % (S::AB / S::TA), ty = t / (S::AB / S::TA);
    T acc[S::TA][S::TJ];
#pragma unroll
    for (int p = 0; p < S::TA; ++p)
#pragma unroll
        for (int q = 0; q < S::TJ; ++q) acc[p][q] = (T)0;
    for (int64_t k0 = i0; k0 < i1; k0 += kKT) {
        // U tile: kKT rows x AB columns, row segments are contiguous
        for (int e = t; e < kKT * S::AB; e += 256) {
            const int kk = e / S::AB, aa = e % S::AB;
            const int64_t i = k0 + kk, a = a0 + aa;
            Us[kk][aa] = (i < i1 && a < ldU) ? U[i * ldU + a] : (T)0;
        }
        // V tile: kKT rows x CT columns (column-major source: coalesced along rows)
        for (int e = t; e < kKT * CT; e += 256) {
            const int kk = e % kKT, j = e / kKT;
            const int64_t i = k0 + kk;
            Vs[kk][j] = (i < i1 && j < c) ? V[i + (int64_t)j * ldv] : (T)0;
        }
        __syncthreads();
#pragma unroll 8
        for (int kk = 0; kk < kKT; ++kk) {
            T ua[S::TA], vj[S::TJ];
            VecLd<T, S::TA>::ld(&Us[kk][tx * S::TA], ua);
            VecLd<T, S::TJ>::ld(&Vs[kk][ty * S::TJ], vj);
#pragma unroll
            for (int p = 0; p < S::TA; ++p)
#pragma unroll
                for (int q = 0; q < S::TJ; ++q) acc[p][q] += ua[p] * vj[q];
        }
        __syncthreads();
    }
#pragma unroll
    for (int p = 0; p < S::TA; ++p) {
        const int64_t a = a0 + tx * S::TA + p;
#pragma unroll
        for (int q = 0; q < S::TJ; ++q) {
            const int j = ty * S::TJ + q;
            if (a < r && j < c) part_chunk[(int64_t)j * r + a] = (double)acc[p][q];
        }
    }
}

// part[(chunk * c + j) * r + a] = sum_{i in chunk} U[i, a] V[i + j ldv]
template <typename T, int CT>
__global__ void __launch_bounds__(256) k_utv_tile(const T* __restrict__ U, int64_t ldU, int64_t n, int64_t r,
                                                  const T* __restrict__ V, int64_t ldv, int c, int64_t chunk,
                                                  double* __restrict__ part) {
    __shared__ __align__(16) T Us[kKT][UtvShape<CT>::AB];
    __shared__ __align__(16) T Vs[kKT][CT];
    const int64_t i0 = blockIdx.x * chunk, i1 = min(n, i0 + chunk);
    utv_tile_body<T, CT>(U, ldU, r, V, ldv, c, i0, i1, blockIdx.y * (int64_t)UtvShape<CT>::AB,
                         part + (int64_t)blockIdx.x * c * r, Us, Vs);
}

// W[a * c + j] = scale_a * sum_chunk part[(chunk * c + j) * r + a]; scale = S[a] or 1.  Launched by
// launch_reduce_scale: 32 neighbouring columns a per block (whole 128- or 256-byte lines of a
// slice) by 8 threads that split the chunks, added in shared memory in a fixed order.  Bound by
// the read of the slices; the earlier form (one thread per (a, j), neighbouring threads r apart
// in a slice) took 0.33 ms for the slices of 10,680 x 64.
constexpr int kRedA = 32, kRedB = 8;
template <typename T, typename P>
__global__ void __launch_bounds__(kRedA * kRedB) k_reduce_scale(const P* __restrict__ part, int nchunk, int64_t r,
                                                                int c, const T* __restrict__ S, T* __restrict__ W,
                                                                double* __restrict__ Wd) {
    __shared__ double sh[kRedB][kRedA];
    const int tx = threadIdx.x % kRedA, ty = threadIdx.x / kRedA;
    const int64_t a = blockIdx.x * (int64_t)kRedA + tx;
    const int j = blockIdx.y;
    double s = 0.0;
    if (a < r) {
#pragma unroll 4
        for (int b = ty; b < nchunk; b += kRedB) s += (double)part[((int64_t)b * c + j) * r + a];
    }
    sh[ty][tx] = s;
    __syncthreads();
    if (ty != 0 || a >= r) return;
#pragma unroll
    for (int y = 1; y < kRedB; ++y) s += sh[y][tx];
    if (S) s *= (double)S[a];
    if (W) W[a * c + j] = (T)s;
    if (Wd) Wd[a * c + j] = s;
}
// The same for few chunks, where the form above leaves most of its threads without one and writes single
// elements c apart: a thread per (a, j), neighbouring threads along j.  262,152 x 16, one FP32 slice 110 ->
// 45 us, 16 of them 376 -> 280; 32,776 x 64, one FP64 slice 53 -> 14.
template <typename T, typename P>
__global__ void __launch_bounds__(256) k_reduce_scale_flat(const P* __restrict__ part, int nchunk, int64_t r, int c,
                                                           const T* __restrict__ S, T* __restrict__ W,
                                                           double* __restrict__ Wd) {
    const int64_t idx = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (idx >= r * c) return;
    const int64_t a = idx / c;
    const int j = (int)(idx % c);
    double s = 0.0;
    for (int b = 0; b < nchunk; ++b) s += (double)part[((int64_t)b * c + j) * r + a];
    if (S) s *= (double)S[a];
    if (W) W[idx] = (T)s;
    if (Wd) Wd[idx] = s;
}
// The same for few chunks and wide blocks, whose reads r apart would cost the lines of a slice more than
// once: 32 columns a by 32 columns j through shared memory, written in runs along j.  262,152 x 64, one
// FP32 slice 143 us (161 by a thread per (a, j), 475 with the chunks split), 16 FP64 slices 576 (1,749, 1,007).
template <typename T, typename P>
__global__ void __launch_bounds__(256) k_reduce_scale_tile(const P* __restrict__ part, int nchunk, int64_t r, int c,
                                                           const T* __restrict__ S, T* __restrict__ W,
                                                           double* __restrict__ Wd) {
    __shared__ double sh[32][33];
    const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
    const int64_t a0 = blockIdx.x * 32ll;
    const int j0 = blockIdx.y * 32;
    const int64_t a = a0 + tx;
    if (a < r) {
        const double scale = S ? (double)S[a] : 1.0;
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int j = j0 + ty + 8 * q;
            if (j < c) {
                double s = 0.0;
                for (int b = 0; b < nchunk; ++b) s += (double)part[((int64_t)b * c + j) * r + a];
                sh[ty + 8 * q][tx] = s * scale;
            }
        }
    }
    __syncthreads();
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const int64_t o = a0 + ty + 8 * q;
        const int j = j0 + tx;
        if (o < r && j < c) {
            const double s = sh[tx][ty + 8 * q];
            if (W) W[o * c + j] = (T)s;
            if (Wd) Wd[o * c + j] = s;
        }
    }
}
template <typename T, typename P>
void launch_reduce_scale(const P* part, int nchunk, int64_t r, int c, const T* S, T* W, double* Wd, cudaStream_t st) {
    // Few chunks: at 16 the flat form is still ahead (8,200 x 33, FP32 24 us against 28; at 32 40 and 45, at
    // 520 x 64 12 and 12); below 32,768 results it has too few threads (2,056 x 8, 16 slices 10 against 8).
    if (nchunk <= 16 && r * c >= 32768) {
        if (c < 48) {
            k_reduce_scale_flat<T, P><<<(unsigned)((r * c + 255) / 256), 256, 0, st>>>(part, nchunk, r, c, S, W, Wd);
        } else {
            const dim3 g((unsigned)((r + 31) / 32), (unsigned)((c + 31) / 32));
            k_reduce_scale_tile<T, P><<<g, 256, 0, st>>>(part, nchunk, r, c, S, W, Wd);
        }
        return;
    }
    const dim3 g((unsigned)((r + kRedA - 1) / kRedA), (unsigned)c);
    k_reduce_scale<T, P><<<g, kRedA * kRedB, 0, st>>>(part, nchunk, r, c, S, W, Wd);
}

// Y[i + j ldy] = alpha * sum_a U[i, a] W[a * c + j] + beta * B[i + j ldb].
// A block owns RB rows and all CT columns; each thread keeps a TM x TN tile.
template <int CT> struct UwShape {
    static constexpr int RB = (CT == 1) ? 256 : 128;
    static constexpr int TM = (CT == 64) ? 8 : (CT >= 8 ? 4 : (CT == 4 ? 2 : 1));
    static constexpr int TN = (CT * (RB / TM)) / 256;
};

constexpr int kUwPad = 4;

// Rows [m0, m0 + RB) of Y = alpha U W + beta B.
template <typename T, int CT>
__device__ __forceinline__ void uw_tile_body(const T* __restrict__ U, int64_t ldU, int64_t n, int64_t r,
                                             const T* __restrict__ W, int c, T alpha, const T* __restrict__ B,
                                             int64_t ldb, T beta, T* __restrict__ Y, int64_t ldy, int64_t m0,
                                             T (*Us)[UwShape<CT>::RB + kUwPad], T (*Ws)[CT]) {
    using S = UwShape<CT>;
    const int t = threadIdx.x;
    const int tx = t % (S::RB / S::TM), ty = t / (S::RB / S::TM);
    T acc[S::TM][S::TN];
#pragma unroll
    for (int p = 0; p < S::TM; ++p)
#pragma unroll
        for (int q = 0; q < S::TN; ++q) acc[p][q] = (T)0;
    for (int64_t k0 = 0; k0 < r; k0 += kKT) {
        for (int e = t; e < kKT * S::RB; e += 256) {
            const int mm = e / kKT, kk = e % kKT;            // consecutive threads walk one row
            const int64_t i = m0 + mm, a = k0 + kk;
            Us[kk][mm] = (i < n && a < r) ? U[i * ldU + a] : (T)0;
        }
        for (int e = t; e < kKT * CT; e += 256) {
            const int kk = e / CT, j = e % CT;
            const int64_t a = k0 + kk;
            Ws[kk][j] = (a < r && j < c) ? W[a * c + j] : (T)0;
        }
        __syncthreads();
#pragma unroll 8
        for (int kk = 0; kk < kKT; ++kk) {
            T um[S::TM], wn[S::TN];
            VecLd<T, S::TM>::ld(&Us[kk][tx * S::TM], um);
            VecLd<T, S::TN>::ld(&Ws[kk][ty * S::TN], wn);
#pragma unroll
            for (int p = 0; p < S::TM; ++p)
#pragma unroll
                for (int q = 0; q < S::TN; ++q) acc[p][q] += um[p] * wn[q];
        }
        __syncthreads();
    }
#pragma unroll
    for (int q = 0; q < S::TN; ++q) {
        const int j = ty * S::TN + q;
        if (j >= c) continue;
#pragma unroll
        for (int p = 0; p < S::TM; ++p) {
            const int64_t i = m0 + tx * S::TM + p;
            if (i < n) {
                T out = alpha * acc[p][q];
                if (B) out += beta * B[i + (int64_t)j * ldb];
                Y[i + (int64_t)j * ldy] = out;
            }
        }
    }
}

template <typename T, int CT>
__global__ void __launch_bounds__(256) k_uw_tile(const T* __restrict__ U, int64_t ldU, int64_t n, int64_t r,
                                                 const T* __restrict__ W, int c, T alpha,
                                                 const T* __restrict__ B, int64_t ldb, T beta,
                                                 T* __restrict__ Y, int64_t ldy) {
    __shared__ __align__(16) T Us[kKT][UwShape<CT>::RB + kUwPad];
    __shared__ __align__(16) T Ws[kKT][CT];
    uw_tile_body<T, CT>(U, ldU, n, r, W, c, alpha, B, ldb, beta, Y, ldy, blockIdx.x * (int64_t)UwShape<CT>::RB,
                        Us, Ws);
}

// ----------------------------------------------------------------- A6: Gram U^T U
// G[a, b] for the 64 x 64 tile (blockIdx.x, blockIdx.y), b-tile >= a-tile; FP64 output.
template <typename T>
__global__ void __launch_bounds__(256) k_gram(const T* __restrict__ U, int64_t ldU, int64_t n, int64_t r,
                                              double* __restrict__ G) {
    if (blockIdx.y < blockIdx.x) return;
    __shared__ T As[16][64 + 1], Bs[16][64 + 1];
    const int tx = threadIdx.x % 16, ty = threadIdx.x / 16;
    const int64_t a0 = blockIdx.x * 64, b0 = blockIdx.y * 64;
    double acc[4][4] = {};
    for (int64_t i0 = 0; i0 < n; i0 += 16) {
        for (int idx = threadIdx.x; idx < 16 * 64; idx += 256) {
            const int rr = idx / 64, cc = idx % 64;
            const int64_t i = i0 + rr;
            As[rr][cc] = (i < n && a0 + cc < r) ? U[i * ldU + a0 + cc] : (T)0;
            Bs[rr][cc] = (i < n && b0 + cc < r) ? U[i * ldU + b0 + cc] : (T)0;
        }
        __syncthreads();
#pragma unroll
        for (int rr = 0; rr < 16; ++rr) {
            T av[4], bv[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) { av[q] = As[rr][ty * 4 + q]; bv[q] = Bs[rr][tx * 4 + q]; }
#pragma unroll
            for (int q = 0; q < 4; ++q)
#pragma unroll
                for (int w = 0; w < 4; ++w) acc[q][w] += (double)(av[q] * bv[w]);
        }
        __syncthreads();
    }
#pragma unroll
    for (int q = 0; q < 4; ++q)
#pragma unroll
        for (int w = 0; w < 4; ++w) {
            const int64_t a = a0 + ty * 4 + q, b = b0 + tx * 4 + w;
            if (a < r && b < r) { G[a * r + b] = acc[q][w]; G[b * r + a] = acc[q][w]; }
        }
}

// Y = alpha * X + beta * Y on column-major blocks (used by the solve's refinement).
template <typename T>
__global__ void k_axpby(int64_t n, int c, T alpha, const T* __restrict__ X, int64_t ldx, T beta,
                        T* __restrict__ Y, int64_t ldy) {
    const int64_t idx = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (idx >= n * c) return;
    const int64_t i = idx % n, j = idx / n;
    Y[i + j * ldy] = alpha * X[i + j * ldx] + beta * Y[i + j * ldy];
}

}  // namespace dev
}  // namespace hdf
