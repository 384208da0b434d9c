// The core of the Woodbury solve without pivoting, and the substitutions of both factorizations.
//
// C = lambda S^-1 + U^T U (r x r, FP64).  With the columns of positive S first (set P) and the
// negative ones after them (set N), C_PP = lambda S_P^-1 + G_PP is positive definite, and the Schur
// complement C_NN - C_NP C_PP^-1 C_PN = -lambda (|S_N|^-1 - U_N^T A_P^-1 U_N), A_P = lambda I +
// U_P S_P U_P^T, is negative definite exactly when lambda I + K~ is positive definite
// (Sherman-Morrison-Woodbury applied to P, then to N).  So for the systems of Eq. (opt) C = L J L^T
// with J = +1 on P and -1 on N exists and is as stable as two Cholesky factorizations: like
// Cholesky it does not depend on the diagonal scaling S, and no pivot has to be searched.  A pivot
// of the wrong sign says that lambda I + K~ is indefinite; then the pivoted LU of lu.cu runs.
//
// Factorization (right-looking, panels of NB = 64): the diagonal tile and its inverse in one CTA,
// the panel below it as a product with that inverse, and the trailing update C_ik -= L_ij J L_kj^T
// on the tensor cores by the exact integer slices of tc_f64.cuh (K = 64 is one block of them); all
// on the device, no host round trip per panel.  What bounds it: the chain of diagonal tiles (FP64
// pipe of one SM) and launches.  At r = 2,104: 4.8 ms, of
// it 33 x 80 us for the diagonal tiles and 33 x 47 us for the updates; the pivoted LU with host
// panels took 26.6 ms.
//
// Substitutions L y = P z, U x = y (U = J L^T, stored in the upper triangle; or the LU factors): one
// cooperative kernel.  A CTA owns whole 64-row blocks; a block waits for each solved block before
// it (a flag in global memory), subtracts its 64 x 64 product, multiplies by the inverse of its
// diagonal tile and publishes the result, so a step of the chain is two small products and one
// flag instead of two launches, one of them a 64-step substitution by a single CTA: 0.41 ms for one
// column at r = 2,104, 13 ms before.  Where the blocks leave CTAs over, several chains run side by side,
// each with a group of the columns: 64 columns at r = 69, solve with kept factors 0.68 -> 0.24 ms.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <vector>

#include "internal.h"

namespace hdf {
namespace ldl {

constexpr int NB = 64;
constexpr int PT = 576;                       // threads of k_ldl_diag: 528 2 x 2 blocks of the lower triangle
constexpr int kCheck = 16;                    // panels between two looks at the pivot signs
constexpr long long kWaitCycles = 4000000000ll;   // limit of a wait on another CTA's block, about 2 s

// C = P (G + diag(lambda / S)) P^T, with 1 on the diagonal of padding columns (S = 0).
__global__ void k_core_perm(const double* __restrict__ G, const double* __restrict__ Spad, const int* __restrict__ perm,
                            double lambda, int64_t r, double* __restrict__ C) {
    const int64_t idx = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (idx >= r * r) return;
    const int64_t a = idx / r, b = idx % r, pa = perm[a];
    double v = G[pa * r + perm[b]];
    if (a == b) v += (Spad[pa] != 0.0) ? lambda / Spad[pa] : 1.0;
    C[idx] = v;
}

// Diagonal tile at k0 (w x w): L with L J L^T = tile into the lower triangle, D = L^-1 (64 x 64,
// identity beyond w).  Thread = one 2 x 2 block v of the lower triangle, rows descending with the
// thread index so that finished rows free whole warps.  Step k: the owners publish column k of
// the tile (rows >= k) and row k of the inverse (columns < k) in one array raw; with il = 1 / l_kk
// f[c] = raw[c] il (f[k] = il) is L's column times J_k and the finished row of the inverse at
// once, and every entry below row k takes v[r][c] += g[r] f[c], g = -J_k f: the tile's trailing update
// for c > k, the inverse's for c <= k (v[r][k] starts from zero).  *bad is set by a pivot whose
// sign is not J_k.
__global__ void __launch_bounds__(PT) k_ldl_diag(double* __restrict__ C, int64_t r, int64_t k0, int w,
                                                 const double* __restrict__ sg, double* __restrict__ D,
                                                 int* __restrict__ bad) {
    __shared__ double raw[2][NB], f[NB], g[NB];
    const int t = threadIdx.x;
    const int u = 527 - t;
    int bi = u >= 0 ? (int)((sqrtf(8.f * u + 1.f) - 1.f) * 0.5f) : -1;
    if (u >= 0) {
        while ((bi + 1) * (bi + 2) / 2 <= u) ++bi;
        while (bi * (bi + 1) / 2 > u) --bi;
    }
    const int bj = u - bi * (bi + 1) / 2;
    const int r0 = 2 * bi, c0 = 2 * bj;
    double v[2][2] = {{0.0, 0.0}, {0.0, 0.0}};
    if (u >= 0) {
#pragma unroll
        for (int a = 0; a < 2; ++a)
#pragma unroll
            for (int b = 0; b < 2; ++b) {
                const int i = r0 + a, j = c0 + b;
                if (i < w && j <= i) v[a][b] = C[(k0 + i) * r + k0 + j];
                else if (i == j) v[a][b] = sg[k0];           // padding: unit pivots of an accepted sign
            }
    }
    for (int k = 0; k < NB; ++k) {
        double* rw = raw[k & 1];
        const int a = k - r0, b = k - c0;
        if (u >= 0) {
            if (b == 0 || b == 1) {                          // column k, rows >= k
#pragma unroll
                for (int q = 0; q < 2; ++q)
                    if (r0 + q >= k) rw[r0 + q] = (b == 0) ? v[q][0] : v[q][1];
            }
            if (a == 0 || a == 1) {                          // row k of the inverse, columns < k
#pragma unroll
                for (int q = 0; q < 2; ++q)
                    if (c0 + q < k) rw[c0 + q] = (a == 0) ? v[0][q] : v[1][q];
            }
        }
        __syncthreads();
        const double J = k < w ? sg[k0 + k] : sg[k0];
        if (t < 32) {                                        // one warp: a second one would double the FP64 time
            double piv = J * rw[k];
            if (!(piv > 0.0) || !isfinite(piv)) {
                if (t == 0) *bad = 1;
                piv = 1.0;
            }
            const double il = rsqrt(piv);
#pragma unroll
            for (int c = t; c < NB; c += 32) {
                const double fc = c == k ? il : rw[c] * il;
                f[c] = fc;
                g[c] = J > 0.0 ? -fc : fc;
                // the finished column of L: l_kk = piv il, l_rk = J f[r]
                if (k < w && c >= k && c < w) C[(k0 + c) * r + k0 + k] = c == k ? piv * il : (J > 0.0 ? fc : -fc);
            }
        }
        __syncthreads();
        if (u >= 0) {
            const double fc0 = f[c0], fc1 = f[c0 + 1];
#pragma unroll
            for (int q = 0; q < 2; ++q) {
                const int i = r0 + q;
                if (i > k) {
                    const double l = g[i];
                    v[q][0] = fma(l, fc0, c0 == k ? 0.0 : v[q][0]);
                    v[q][1] = fma(l, fc1, c0 + 1 == k ? 0.0 : v[q][1]);
                } else if (i == k) {                         // the finished row of the inverse
                    if (c0 <= k) v[q][0] = fc0;
                    if (c0 + 1 <= k) v[q][1] = fc1;
                }
            }
        }
    }
    if (u >= 0) {
#pragma unroll
        for (int a = 0; a < 2; ++a)
#pragma unroll
            for (int b = 0; b < 2; ++b) {
                const int i = r0 + a, j = c0 + b;
                if (j <= i) D[i * NB + j] = v[a][b];
                if (j < i) D[j * NB + i] = 0.0;
            }
    }
}

// Panel below the diagonal tile: L_ic = J_c sum_{q <= c} A_iq D_cq for TR rows per CTA.
constexpr int TR = 16;
__global__ void __launch_bounds__(256) k_ldl_panel(double* __restrict__ C, int64_t r, int64_t k0,
                                                   const double* __restrict__ sg, const double* __restrict__ D) {
    __shared__ double Ds[NB][NB + 1];
    __shared__ double As[TR][NB];
    const int64_t i0 = k0 + NB + (int64_t)blockIdx.x * TR;
    for (int e = threadIdx.x; e < NB * NB; e += 256) Ds[e / NB][e % NB] = D[e];
    for (int e = threadIdx.x; e < TR * NB; e += 256) {
        const int64_t i = i0 + e / NB;
        As[e / NB][e % NB] = i < r ? C[i * r + k0 + e % NB] : 0.0;
    }
    __syncthreads();
    // thread: column c, rows rr, rr + 4, ...; a warp holds 32 columns of equal length to within 31
    const int c = threadIdx.x & 63, rr = threadIdx.x >> 6;
    double s[TR / 4] = {};
    for (int q = 0; q <= (c | 31); ++q) {
        const double d = Ds[c][q];                           // zero above the diagonal
#pragma unroll
        for (int e = 0; e < TR / 4; ++e) s[e] = fma(As[rr + 4 * e][q], d, s[e]);
    }
    const double J = sg[k0 + c];
#pragma unroll
    for (int e = 0; e < TR / 4; ++e) {
        const int64_t i = i0 + rr + 4 * e;
        if (i < r) C[i * r + k0 + c] = J * s[e];
    }
}

// Upper triangle: U = J L^T (U[k][i] = J_k L[i][k], k < i), in 32 x 32 tiles through shared memory.
__global__ void __launch_bounds__(256) k_ldl_mirror(double* __restrict__ C, int64_t r, const double* __restrict__ sg) {
    if (blockIdx.y < blockIdx.x) return;
    __shared__ double t[32][33];
    const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
    const int64_t i0 = blockIdx.y * 32ll, k0 = blockIdx.x * 32ll;
    for (int q = ty; q < 32; q += 8)
        if (i0 + q < r && k0 + tx < r) t[q][tx] = C[(i0 + q) * r + k0 + tx];
    __syncthreads();
    for (int q = ty; q < 32; q += 8) {
        const int64_t k = k0 + q, i = i0 + tx;
        if (k < i && i < r) C[k * r + i] = sg[k] * t[tx][q];
    }
}

// DU_b = (J L_bb^T)^-1 = D_b^T J.
__global__ void __launch_bounds__(256) k_ldl_dinvu(const double* __restrict__ D, const double* __restrict__ sg, int64_t r,
                                                   double* __restrict__ DU) {
    const int64_t b = blockIdx.x;
    for (int e = threadIdx.x; e < NB * NB; e += 256) {
        const int a = e / NB, c = e % NB;
        const int64_t k = min(b * NB + c, r - 1);
        DU[b * NB * NB + e] = D[b * NB * NB + c * NB + a] * sg[k];
    }
}

// Inverses of the diagonal tiles of a pivoted LU (unit lower, upper), identity beyond r: thread t
// < 64 forms column t of L^-1, thread 64 + t column t of U^-1.
__global__ void __launch_bounds__(128) k_lu_dinv(const double* __restrict__ LU, int64_t r, double* __restrict__ DL,
                                                 double* __restrict__ DU) {
    extern __shared__ double sh[];
    double* T = sh;                                          // NB x (NB + 1)
    double* X = sh + NB * (NB + 1);                          // two of them
    const int64_t b0 = (int64_t)blockIdx.x * NB;
    for (int e = threadIdx.x; e < NB * NB; e += 128) {
        const int i = e / NB, j = e % NB;
        T[i * (NB + 1) + j] = (b0 + i < r && b0 + j < r) ? LU[(b0 + i) * r + b0 + j] : (i == j ? 1.0 : 0.0);
    }
    __syncthreads();
    const int q = threadIdx.x & 63;
    double* Y = X + (threadIdx.x >> 6) * NB * (NB + 1);
    if (threadIdx.x < 64) {
        for (int i = 0; i < NB; ++i) {
            double s = i == q ? 1.0 : 0.0;
            for (int m = q; m < i; ++m) s -= T[i * (NB + 1) + m] * Y[m * (NB + 1) + q];
            Y[i * (NB + 1) + q] = i < q ? 0.0 : s;
        }
    } else {
        for (int i = NB - 1; i >= 0; --i) {
            double s = i == q ? 1.0 : 0.0;
            for (int m = i + 1; m <= q; ++m) s -= T[i * (NB + 1) + m] * Y[m * (NB + 1) + q];
            Y[i * (NB + 1) + q] = i > q ? 0.0 : s / T[i * (NB + 1) + i];
        }
    }
    __syncthreads();
    for (int e = threadIdx.x; e < NB * NB; e += 128) {
        DL[(int64_t)blockIdx.x * NB * NB + e] = X[(e / NB) * (NB + 1) + e % NB];
        DU[(int64_t)blockIdx.x * NB * NB + e] = X[NB * (NB + 1) + (e / NB) * (NB + 1) + e % NB];
    }
}

// ---------------------------------------------------------------------- substitutions
struct TriArgs {
    const double* M; int64_t r;          // L in the lower, U in the upper triangle (off-diagonal tiles)
    const double *DL, *DU;               // inverses of the diagonal tiles
    const int* rperm;                    // row a of the factors is row rperm[a] of the right-hand side
    const double* zi; double* y; double* zo;   // r x nc row-major: right-hand side, work, result
    int nc, nblk;                        // columns; 64-row blocks
    int group, nb;                       // columns of a group; CTAs of a group
    int* flags;                          // 2 nblk per group, zero at launch
    int* err;
};

__device__ __forceinline__ int ld_acquire(const int* p) {
    int v;
    asm volatile("ld.acquire.gpu.global.s32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ void st_release(int* p, int v) {
    asm volatile("st.release.gpu.global.s32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}

// GROUPS: P.nb CTAs per group of P.group columns (else all columns on all CTAs; kept apart because the
// strides at run time cost 2% at r = 6,693, 64 columns).
template <bool GROUPS>
__global__ void __launch_bounds__(256) k_tri_solve(TriArgs P) {
    extern __shared__ double sm[];
    const int nb = GROUPS ? P.nb : (int)gridDim.x;
    const int g = GROUPS ? (int)blockIdx.x / nb : 0, blk = (int)blockIdx.x - g * nb;
    const int c0 = GROUPS ? g * P.group : 0, ld = P.nc, nc = GROUPS ? min(P.group, ld - c0) : ld;     // its columns
    double* zs = sm;                     // the solved block being subtracted, NB x nc
    double* as = sm + NB * nc;           // this block's residual, NB x nc
    __shared__ int gave_up;
    const int t = threadIdx.x, row = t >> 2, qt = t & 3;
    int* flags = P.flags + (int64_t)g * 2 * P.nblk;
    if (t == 0) gave_up = 0;
    __syncthreads();
    // own blocks ascending (forward), then descending (backward): every wait is on a block that
    // comes earlier in this order, and the cooperative launch keeps all CTAs resident
    const int mine = (P.nblk - blk + nb - 1) / nb;
    for (int s = 0; s < 2 * mine; ++s) {
        const bool fwd = s < mine;
        const int rb = blk + (fwd ? s : 2 * mine - 1 - s) * nb;
        const int64_t i = (int64_t)rb * NB + row;
        for (int e = t; e < NB * nc; e += 256) {
            const int64_t a = (int64_t)rb * NB + e / nc;
            double v = 0.0;
            if (a < P.r) v = fwd ? P.zi[(int64_t)P.rperm[a] * ld + c0 + e % nc] : P.y[a * ld + c0 + e % nc];
            as[e] = v;
        }
        const int ndep = fwd ? rb : P.nblk - 1 - rb;
        auto tile = [&](int d, double* x) {                  // 16 entries of row `row` of the d-th tile
            const int b = fwd ? d : P.nblk - 1 - d;
            const int64_t j0 = (int64_t)b * NB + 16 * qt;
#pragma unroll
            for (int e = 0; e < 16; ++e) x[e] = (d < ndep && i < P.r && j0 + e < P.r) ? P.M[i * P.r + j0 + e] : 0.0;
        };
        double x[16], xn[16];
        tile(0, x);
        for (int d = 0; d < ndep; ++d) {
            const int b = fwd ? d : P.nblk - 1 - d;
            tile(d + 1, xn);                                 // in flight during the wait
            if (t == 0 && !gave_up) {
                const int* fl = flags + (fwd ? 0 : P.nblk) + b;
                if (!ld_acquire(fl)) {
                    const long long t0 = clock64();
                    while (!ld_acquire(fl))
                        if (clock64() - t0 > kWaitCycles) { gave_up = 1; atomicExch(P.err, 1); break; }
                }
            }
            __syncthreads();
            const double* src = (fwd ? P.y : P.zo) + (int64_t)b * NB * ld + c0;
            const int cnt = (int)min((int64_t)NB, P.r - (int64_t)b * NB) * nc;
            for (int e = t; e < NB * nc; e += 256)
                zs[e] = e < cnt ? __ldcg(src + (GROUPS ? (int64_t)(e / nc) * ld + e % nc : e)) : 0.0;
            __syncthreads();
            for (int j = 0; j < nc; ++j) {
                double a0 = 0.0, a1 = 0.0;
#pragma unroll
                for (int e = 0; e < 16; e += 2) {
                    a0 = fma(x[e], zs[(16 * qt + e) * nc + j], a0);
                    a1 = fma(x[e + 1], zs[(16 * qt + e + 1) * nc + j], a1);
                }
                a0 += a1;
                a0 += __shfl_xor_sync(0xffffffffu, a0, 1);
                a0 += __shfl_xor_sync(0xffffffffu, a0, 2);
                if (qt == 0) as[row * nc + j] -= a0;
            }
#pragma unroll
            for (int e = 0; e < 16; ++e) x[e] = xn[e];
        }
        // times the inverse of the diagonal tile
        const double* D = (fwd ? P.DL : P.DU) + (int64_t)rb * NB * NB + row * NB + 16 * qt;
#pragma unroll
        for (int e = 0; e < 16; ++e) x[e] = D[e];
        __syncthreads();
        double* dst = fwd ? P.y : P.zo;
        for (int j = 0; j < nc; ++j) {
            double a0 = 0.0, a1 = 0.0;
#pragma unroll
            for (int e = 0; e < 16; e += 2) {
                a0 = fma(x[e], as[(16 * qt + e) * nc + j], a0);
                a1 = fma(x[e + 1], as[(16 * qt + e + 1) * nc + j], a1);
            }
            a0 += a1;
            a0 += __shfl_xor_sync(0xffffffffu, a0, 1);
            a0 += __shfl_xor_sync(0xffffffffu, a0, 2);
            if (qt == 0 && i < P.r) dst[i * ld + c0 + j] = a0;
        }
        __threadfence();
        __syncthreads();
        if (t == 0) st_release(flags + (fwd ? 0 : P.nblk) + rb, 1);
    }
}

// out[perm a] = x_a (rows of nc values).
__global__ void k_scatter_rows(const double* __restrict__ x, double* __restrict__ out, int64_t r, int nc,
                               const int* __restrict__ perm) {
    const int64_t idx = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (idx >= r * nc) return;
    out[(int64_t)perm[idx / nc] * nc + idx % nc] = x[idx];
}

}  // namespace ldl

// Factors the core without pivoting: C (r x r) receives L in the lower and J L^T in the upper
// triangle, dperm the order (row a is column dperm[a] of U), dinv the inverses of the diagonal
// tiles (lower, then upper; 2 ceil(r / 64) 64 x 64).  HDF_ESINGULAR when lambda I + K~ is not
// positive definite to working precision (C is then undefined).  Synchronises.
hdf_status ldl_factor_device(int64_t r, const double* G, const std::vector<double>& Spad, const double* dS, double lambda,
                             double* C, DevBuf& dperm, DevBuf& dinv, int* err, cudaStream_t st) {
    using namespace ldl;
    std::vector<int> perm;
    std::vector<double> sg;
    perm.reserve(r);
    sg.reserve(r);
    for (int pass = 0; pass < 2; ++pass)
        for (int64_t a = 0; a < r; ++a)
            if ((Spad[a] < 0.0) == (pass == 1)) { perm.push_back((int)a); sg.push_back(pass ? -1.0 : 1.0); }
    const int64_t nblk = (r + NB - 1) / NB;
    DevBuf dsg, bad, work;
    HDF_CUDA(dperm.alloc(sizeof(int) * r));
    HDF_CUDA(dinv.alloc(sizeof(double) * 2 * (size_t)nblk * NB * NB));
    HDF_CUDA(dsg.alloc_on(sizeof(double) * r, st));
    HDF_CUDA(bad.alloc_on(sizeof(int), st));
    HDF_CUDA(work.alloc_on(tc_f64_update_bytes(r), st));
    HDF_CUDA(cudaMemcpyAsync(dperm.p, perm.data(), sizeof(int) * r, cudaMemcpyHostToDevice, st));
    HDF_CUDA(cudaMemcpyAsync(dsg.p, sg.data(), sizeof(double) * r, cudaMemcpyHostToDevice, st));
    HDF_CUDA(cudaMemsetAsync(bad.p, 0, sizeof(int), st));
    HDF_COUNT_LAUNCH();
    k_core_perm<<<(unsigned)((r * r + 255) / 256), 256, 0, st>>>(G, dS, dperm.as<int>(), lambda, r, C);
    HDF_CUDA(cudaGetLastError());
    double* DL = dinv.as<double>();
    double* DU = DL + nblk * NB * NB;
    int h = 0;
    for (int64_t b = 0; b < nblk; ++b) {
        const int64_t k0 = b * NB;
        const int w = (int)std::min<int64_t>(NB, r - k0);
        HDF_COUNT_LAUNCH();
        k_ldl_diag<<<1, PT, 0, st>>>(C, r, k0, w, dsg.as<double>(), DL + b * NB * NB, bad.as<int>());
        const int64_t m = r - k0 - w;
        if (m <= 0) break;
        HDF_COUNT_LAUNCH();
        k_ldl_panel<<<(unsigned)((m + TR - 1) / TR), 256, 0, st>>>(C, r, k0, dsg.as<double>(), DL + b * NB * NB);
        HDF_CUDA(cudaGetLastError());
        if (hdf_status e = tc_f64_update(C + (k0 + w) * r + k0, r, m, w, dsg.as<double>() + k0, nullptr, 0, m,
                                         C + (k0 + w) * r + k0 + w, r, work.p, err, st);
            e != HDF_OK)
            return e;
        if (b % kCheck == kCheck - 1) {                      // an indefinite system: stop early
            HDF_CUDA(cudaMemcpyAsync(&h, bad.p, sizeof(int), cudaMemcpyDeviceToHost, st));
            HDF_CUDA(cudaStreamSynchronize(st));
            if (h) return HDF_ESINGULAR;
        }
    }
    const unsigned nt = (unsigned)((r + 31) / 32);
    HDF_COUNT_LAUNCH();
    k_ldl_mirror<<<dim3(nt, nt), 256, 0, st>>>(C, r, dsg.as<double>());
    HDF_COUNT_LAUNCH();
    k_ldl_dinvu<<<(unsigned)nblk, 256, 0, st>>>(DL, dsg.as<double>(), r, DU);
    HDF_CUDA(cudaGetLastError());
    HDF_CUDA(cudaMemcpyAsync(&h, bad.p, sizeof(int), cudaMemcpyDeviceToHost, st));
    HDF_CUDA(cudaStreamSynchronize(st));
    return h ? HDF_ESINGULAR : HDF_OK;
}

// The inverses of the diagonal tiles of a pivoted LU, for tri_solve_device.
hdf_status lu_dinv_device(int64_t r, const double* LU, DevBuf& dinv, cudaStream_t st) {
    using namespace ldl;
    const int64_t nblk = (r + NB - 1) / NB;
    HDF_CUDA(dinv.alloc(sizeof(double) * 2 * (size_t)nblk * NB * NB));
    const size_t sm = sizeof(double) * 3 * NB * (NB + 1);
    HDF_CUDA(cudaFuncSetAttribute(k_lu_dinv, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm));
    HDF_COUNT_LAUNCH();
    k_lu_dinv<<<(unsigned)nblk, 128, sm, st>>>(LU, r, dinv.as<double>(), dinv.as<double>() + nblk * NB * NB);
    HDF_CUDA(cudaGetLastError());
    return HDF_OK;
}

// z (r x nc row-major, nc <= 64) = C^-1 zi with the factors of ldl_factor_device (symmetric: the
// order applies to rows and columns) or of lu_factor_device (to rows only); zi is left unchanged.
hdf_status tri_solve_device(int64_t r, const double* M, const DevBuf& dinv, const int* dperm, bool symmetric,
                            const double* zi, double* z, int nc, int* err, cudaStream_t st) {
    using namespace ldl;
    const int nblk = (int)((r + NB - 1) / NB);
    int dv = 0, nsm = 0;
    HDF_CUDA(cudaGetDevice(&dv));
    HDF_CUDA(cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dv));
    // CTAs that the blocks of rows leave over take groups of at least 8 columns of their own (64 columns in
    // one CTA, which a core of one block had, keep the FP64 pipe of its SM busy for 140 us)
    const int nb = std::min(nblk, nsm);
    const int most = std::min(nsm / nb, (nc + 7) / 8), group = (nc + most - 1) / most;
    const int groups = (nc + group - 1) / group;
    DevBuf work, flags;
    const size_t rows = (size_t)nblk * NB * nc;
    HDF_CUDA(work.alloc_on(sizeof(double) * 2 * rows, st));
    HDF_CUDA(flags.alloc_on(sizeof(int) * 2 * (size_t)nblk * groups, st));
    HDF_CUDA(cudaMemsetAsync(flags.p, 0, sizeof(int) * 2 * (size_t)nblk * groups, st));
    double* x = symmetric ? work.as<double>() + rows : z;
    TriArgs P{M, r, dinv.as<double>(), dinv.as<double>() + (int64_t)nblk * NB * NB, dperm, zi,
              work.as<double>(), x, nc, nblk, group, nb, flags.as<int>(), err};
    const size_t sm = sizeof(double) * 2 * NB * (size_t)group;
    void (*kern)(TriArgs) = groups > 1 ? k_tri_solve<true> : k_tri_solve<false>;
    HDF_CUDA(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm));
    void* args[] = {&P};
    HDF_COUNT_LAUNCH();
    HDF_CUDA(cudaLaunchCooperativeKernel(reinterpret_cast<void*>(kern), dim3((unsigned)(groups * nb)), dim3(256), args,
                                         sm, st));
    if (symmetric) {
        HDF_COUNT_LAUNCH();
        k_scatter_rows<<<(unsigned)((r * nc + 255) / 256), 256, 0, st>>>(x, z, r, nc, dperm);
        HDF_CUDA(cudaGetLastError());
    }
    return HDF_OK;
}

}  // namespace hdf
