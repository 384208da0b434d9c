// Adjoint of f = sum_j w_j^T K~ v_j with respect to the points and the lengthscale.
//
// The paper does not differentiate the factorization.  We use frozen-structure semantics:
// the scaling (c, R), the degree p, the radial-basis factor and the kept eigenvectors are
// those of the build, so that row i of U is an explicit smooth function of x_i,
//     U_i[(k,s,h)] = F_ks(|x'_i|) Y_k^h(x'_i / |x'_i|),  x' = (x - c)/(2R),
// and S depends on l only through the radial cores: S_k(l) = W_k^T R_f Gamma_k(l) R_f^T W_k.
// Then, with a = S U^T v and b = S U^T w,
//     grad_{x_i} f = (w_i a + v_i b) . dU_i/dx_i,     df/dl = (U^T w)^T (dS/dl) (U^T v).
// The kernel recomputes F, dF/drho, the harmonics and their gradients per point (nothing of
// U's Jacobian is stored): for a solid harmonic H of degree k (H(x_hat) = Y(x_hat)),
//     d/dx' [F(rho) Y(x'/rho)] = [F' - k F/rho] Y x_hat + (F/rho) grad H(x_hat).
// grad H comes from carrying d/dz and d/dq through the level recurrences
// P(n) = A z P(n-1) - B q P(n-2) (z = x_{D_j}, q = |x_{0..D_j}|^2) and from
// d(x0 + i x1)^mu = mu (x0 + i x1)^(mu-1) (dx0 + i dx1).
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <vector>

#include "hdf_kernels.cuh"
#include "internal.h"

#include <type_traits>
#include "planner.h"

namespace {

using hdf::dev::kMaxD;

template <typename T>
struct AdjParams {
    const double* x; int64_t n; int d; double c[kMaxD]; double inv2R;
    int L;                         // degrees of the harmonic tables (L_used)
    int Lr;                        // radial degree: basis sizes Lr+1 (even), Lr (odd)
    int tri;
    const double* Qm0; int nb0, m0;
    const double* Qm1; int nb1, m1;
    const float2* QC; int mtp;                     // FP32 factors: [Qm0 | Qm1] as float pairs, (Lr+1) x mtp
    const T* Wt; const uint8_t* colk; int nF;
    int nH, nk; const int* ktab;
    const int4* desc;                              // per harmonic (k_adj_desc)
    const int* desc2;                              // d >= 7: level offsets 4, 5
    const T* coefA; const T* coefB;
    const T* ab;                                   // (a, b) of every column
    const T* v; const T* w;                        // this column of V and W (length n)
    T* grad; int accumulate;
    int nb;                                        // points per batch of a warp (1, 2 or 4)
    int per_warp;                                  // bytes of shared memory per warp (a multiple of 16)
};
constexpr int kAdjBatch = 4;      // whole call at 500,000 points: 1 4.88, 2 4.55, 4 4.36, 8 4.79 ms

template <typename T> struct Pair;
template <> struct Pair<float> { typedef float2 type; };
template <> struct Pair<double> { typedef double2 type; };
template <typename T> struct Quad;
template <> struct Quad<float> { typedef float4 type; };
struct alignas(16) Double4 { double x, y, z, w; };
template <> struct Quad<double> { typedef Double4 type; };

// Shared memory of a warp: (value, d/dz, d/dq) of the level tables and (value, d/dx_0, d/dx_1) of the
// trigonometric factors, (F' - k F / rho, F / rho) per radial factor, T_l and T_l' of a batch of points (8
// bytes each), the radial basis and its derivative (8 bytes each).  The three values of a table entry
// lie together, in four elements that are read at once (packed), or in three arrays.
__host__ __device__ inline int adj_table_elems(int levels, int tri, int L, bool packed) {
    const int e = levels * tri + 2 * L + 1;
    return packed ? 4 * e : (3 * e + 1) / 2 * 2;
}
template <typename T>
size_t adj_per_warp(int levels, int tri, int L, int nF, int Lr, int m, int nb, bool packed) {
    return ((sizeof(T) * ((size_t)adj_table_elems(levels, tri, L, packed) + 2 * (size_t)nF) + 7) / 8 * 8 +
            8 * (2 * (size_t)nb * (Lr + 1) + 2 * (size_t)m) + 15) / 16 * 16;
}

// What the harmonic loop needs of harmonic gi, from five tables: first column, k | trigonometric index
// << 8, level offsets 0 | 1 << 16, 2 | 3 << 16 (, 4 | 5 << 16).
__global__ void k_adj_desc(const int16_t* __restrict__ chains, int nH, int cstride, int levels, int L,
                           const uint8_t* __restrict__ hk, const int* __restrict__ ktab, int4* __restrict__ desc,
                           int* __restrict__ desc2) {
    const int gi = blockIdx.x * blockDim.x + threadIdx.x;
    if (gi >= nH) return;
    const int k = hk[gi];
    const int* kt = ktab + hdf::kTabStride * k;
    const int16_t* ch = chains + (int64_t)gi * cstride;
    auto off = [&](int j) { return j < levels ? (int)(uint16_t)ch[j] << (16 * (j & 1)) : 0; };
    desc[gi] = make_int4(kt[2] + gi - kt[4], k | (L + ch[levels]) << 8, off(0) | off(1), off(2) | off(3));
    if (desc2) desc2[gi] = off(4) | off(5);
}

// Double-float helpers for the FP32 form (FP32 pairs, error-free products and sums).
__device__ __forceinline__ void df_two_sum(float a, float b, float& s, float& e) {
    s = a + b;
    const float bb = s - a;
    e = (a - (s - bb)) + (b - bb);
}
__device__ __forceinline__ float2 df_norm(float s, float e) {
    const float h = s + e;
    return make_float2(h, e - (h - s));
}
__device__ __forceinline__ float2 df_mul(float2 a, float2 b) {          // a * b
    const float p = a.x * b.x;
    float e = fmaf(a.x, b.x, -p);
    e = fmaf(a.x, b.y, fmaf(a.y, b.x, e));
    return df_norm(p, e);
}
__device__ __forceinline__ float2 df_add(float2 a, float2 b) {          // a + b
    float s, e;
    df_two_sum(a.x, b.x, s, e);
    e += a.y + b.y;
    return df_norm(s, e);
}
__device__ __forceinline__ void df_dot_step(float2 a, float2 b, float& sh, float& c) {   // Dot2 step
    const float ph = a.x * b.x;
    float pe = fmaf(a.x, b.x, -ph);
    pe = fmaf(a.x, b.y, fmaf(a.y, b.x, pe));
    float s2, es;
    df_two_sum(sh, ph, s2, es);
    sh = s2;
    c += es + pe;
}

// A warp takes batches of P.nb points: lane p forms the scaled coordinates of point p and runs its
// Chebyshev recurrences of T_l and T_l' (serial, in double-float arithmetic for FP32 factors some 70
// instructions a step, which one lane per point cost every lane), then the points follow one by one
// with the lanes over basis functions, radial factors and harmonics.  Bound by instruction issue and
// the latency of the table reads: 500,000 points, d = 4, 2,104 columns, 4.43 -> 3.19 ms with batches,
// one descriptor per harmonic and the tables' three values read together.  At high degrees a warp's
// tables leave few warps on an SM and their latency counts alone: there the three arrays, a quarter
// smaller, and CTAs of one or two warps are used (see run).  DD = the dimension d (a template parameter,
// so that the per-thread coordinate and gradient arrays stay in registers).
template <typename T, int DD, bool PACKED>
__global__ void __launch_bounds__(128) k_adjoint(AdjParams<T> P) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ int2 kts[HDF_MAX_L + 1];        // per k: F column | s_k << 16, columns per (k, s) block
    typedef typename Pair<T>::type T2;
    typedef typename Quad<T>::type T4;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
    constexpr int levels = DD - 2;
    for (int k = threadIdx.x; k < P.nk; k += blockDim.x) {
        const int* kt = P.ktab + hdf::kTabStride * k;
        kts[k] = make_int2(kt[0] | kt[1] << 16, kt[5]);
    }
    __syncthreads();
    // levels * tri entries of the level tables, then 2L+1 trigonometric ones
    T* tab = reinterpret_cast<T*>(smem_raw + (size_t)warp * P.per_warp);
    const int trig = levels * P.tri, entries = trig + 2 * P.L + 1;
    const int elems = adj_table_elems(levels, P.tri, P.L, PACKED);
    auto put = [&](int e, T v, T a, T b) {
        if constexpr (PACKED) {
            T4 w; w.x = v; w.y = a; w.z = b; w.w = (T)0;
            reinterpret_cast<T4*>(tab)[e] = w;
        } else {
            tab[e] = v; tab[entries + e] = a; tab[2 * entries + e] = b;
        }
    };
    auto get = [&](int e, T& v, T& a, T& b) {
        if constexpr (PACKED) {
            const T4 w = reinterpret_cast<const T4*>(tab)[e];
            v = w.x; a = w.y; b = w.z;
        } else {
            v = tab[e]; a = tab[entries + e]; b = tab[2 * entries + e];
        }
    };
    T2* RR = reinterpret_cast<T2*>(tab + elems);                               // nF
    double* Tl = reinterpret_cast<double*>(reinterpret_cast<unsigned char*>(tab) +
                                           (sizeof(T) * (elems + 2 * P.nF) + 7) / 8 * 8);
    const int nb = P.nb;
    double* dTl = Tl + nb * (P.Lr + 1);        // T_l(u), T_l'(u): [l][point]
    double* Q = dTl + nb * (P.Lr + 1);         // m0+m1
    double* dQ = Q + (P.m0 + P.m1);            // m0+m1
    const int64_t gw = (int64_t)blockIdx.x * nwarps + warp, nw = (int64_t)gridDim.x * nwarps;
    for (int64_t i0 = gw * nb; i0 < P.n; i0 += nw * nb) {
        // ---- this lane's point
        const int own = lane & (nb - 1);
        const int64_t io = min(i0 + own, P.n - 1);
        T xo[DD];
        double s2o = 0.0;
#pragma unroll
        for (int j = 0; j < DD; ++j) {
            const double xd = (P.x[io * DD + j] - P.c[j]) * P.inv2R;
            s2o += xd * xd;
            xo[j] = (T)xd;
        }
        const T wo = P.w[io], vo = P.v[io];
        T rhoo;
        if constexpr (sizeof(T) == 4) {
            rhoo = sqrtf((float)s2o);
            if (s2o > 0.0) { const float inv = 1.f / rhoo; for (int j = 0; j < DD; ++j) xo[j] *= inv; }
            else { for (int j = 0; j < DD; ++j) xo[j] = (j == 0) ? 1.f : 0.f; }
        } else {
            rhoo = sqrt(s2o);
            if (s2o > 0.0) { for (int j = 0; j < DD; ++j) xo[j] = xo[j] / rhoo; }
            else { for (int j = 0; j < DD; ++j) xo[j] = (j == 0) ? 1.0 : 0.0; }
        }
        if (lane < nb) {
            const double u = 8.0 * s2o - 1.0;
            if constexpr (sizeof(T) == 4) {
                // FP32 factors: the radial part in double-float / FP32 arithmetic (FP64 is slow here)
                float2* Tl2 = reinterpret_cast<float2*>(Tl) + lane;
                float2* dTl2 = reinterpret_cast<float2*>(dTl) + lane;
                const float uh = (float)u, ul = (float)(u - (double)uh);
                const float2 u2 = make_float2(2.f * uh, 2.f * ul);
                float2 t2 = make_float2(1.f, 0.f), t1 = make_float2(uh, ul);       // T_{l-2}, T_{l-1}
                float2 d2 = make_float2(0.f, 0.f), d1 = make_float2(1.f, 0.f);     // T'_{l-2}, T'_{l-1}
                Tl2[0] = t2; dTl2[0] = d2;
                if (P.Lr >= 1) { Tl2[nb] = t1; dTl2[nb] = d1; }
                for (int l = 2; l <= P.Lr; ++l) {
                    const float2 tn = df_add(df_mul(u2, t1), make_float2(-t2.x, -t2.y));
                    const float2 dn = df_add(df_add(make_float2(2.f * t1.x, 2.f * t1.y), df_mul(u2, d1)),
                                             make_float2(-d2.x, -d2.y));
                    Tl2[l * nb] = tn; dTl2[l * nb] = dn;
                    t2 = t1; t1 = tn;
                    d2 = d1; d1 = dn;
                }
            } else {
                double t2 = 1.0, t1 = u, d2 = 0.0, d1 = 1.0;
                Tl[lane] = t2; dTl[lane] = d2;
                if (P.Lr >= 1) { Tl[nb + lane] = t1; dTl[nb + lane] = d1; }
                for (int l = 2; l <= P.Lr; ++l) {
                    const double tn = 2.0 * u * t1 - t2, dn = 2.0 * t1 + 2.0 * u * d1 - d2;
                    Tl[l * nb + lane] = tn; dTl[l * nb + lane] = dn;
                    t2 = t1; t1 = tn;
                    d2 = d1; d1 = dn;
                }
            }
        }
        __syncwarp();
        for (int pt = 0; pt < nb && i0 + pt < P.n; ++pt) {
        const int64_t i = i0 + pt;
        T xh[kMaxD];
#pragma unroll
        for (int j = 0; j < DD; ++j) xh[j] = __shfl_sync(0xffffffffu, xo[j], pt);
        const T rhot = __shfl_sync(0xffffffffu, rhoo, pt);
        const T wi = __shfl_sync(0xffffffffu, wo, pt), vi = __shfl_sync(0xffffffffu, vo, pt);
        if constexpr (sizeof(T) == 4) {
            const float rhof = rhot, s2f = __shfl_sync(0xffffffffu, (float)s2o, pt);
            const float2* Tl2 = reinterpret_cast<const float2*>(Tl) + pt;
            const float2* dTl2 = reinterpret_cast<const float2*>(dTl) + pt;
            float* Qf = reinterpret_cast<float*>(Q);
            float* dQf = reinterpret_cast<float*>(dQ);
            // S_T[o] = sum_l T_l Qmat[l][o], S_dT[o] = sum_l T'_l Qmat[l][o] (Dot2); then
            // even: Q = S_T, dQ = 16 rho S_dT;  odd: Q = rho S_T, dQ = S_T + 16 rho^2 S_dT
            for (int o = lane; o < P.m0 + P.m1; o += 32) {
                const bool odd = o >= P.m0;
                const int nbas = odd ? P.nb1 : P.nb0;
                float th = 0.f, tc = 0.f, dh = 0.f, dc = 0.f;
                for (int l = 0; l < nbas; ++l) {
                    const float2 qm = P.QC[(size_t)l * P.mtp + o];
                    df_dot_step(Tl2[l * nb], qm, th, tc);
                    df_dot_step(dTl2[l * nb], qm, dh, dc);
                }
                const float st = th + tc, sd = dh + dc;
                if (!odd) { Qf[o] = st; dQf[o] = 16.f * rhof * sd; }
                else { Qf[o] = rhof * st; dQf[o] = st + 16.f * s2f * sd; }
            }
            __syncwarp();
            for (int col = lane; col < P.nF; col += 32) {
                const int k = P.colk[col];
                const int par = k & 1, ob = par ? P.m0 : 0, mp = par ? P.m1 : P.m0;
                float F = 0.f, dF = 0.f;
                for (int l = 0; l < mp; ++l) {
                    const float wv = (float)P.Wt[(int64_t)l * P.nF + col];
                    F += Qf[ob + l] * wv;
                    dF += dQf[ob + l] * wv;
                }
                T2 r;
                if (rhof > 1e-30f) { r.x = (T)(dF - k * F / rhof); r.y = (T)(F / rhof); }
                else { r.x = (T)dF; r.y = (T)0; }
                RR[col] = r;
            }
        } else {
        const double rho = rhot, s2 = __shfl_sync(0xffffffffu, s2o, pt);
        // Q = B Qmat and dQ/drho; B0 = T_l, B0' = 16 rho T_l'; B1 = rho T_l, B1' = T_l + 16 rho^2 T_l'
        for (int o = lane; o < P.m0 + P.m1; o += 32) {
            double q = 0.0, dq = 0.0;
            if (o < P.m0) {
                for (int l = 0; l < P.nb0; ++l) {
                    const double qm = P.Qm0[l * P.m0 + o];
                    q += Tl[l * nb + pt] * qm;
                    dq += 16.0 * rho * dTl[l * nb + pt] * qm;
                }
            } else {
                const int oo = o - P.m0;
                for (int l = 0; l < P.nb1; ++l) {
                    const double qm = P.Qm1[l * P.m1 + oo];
                    q += rho * Tl[l * nb + pt] * qm;
                    dq += (Tl[l * nb + pt] + 16.0 * s2 * dTl[l * nb + pt]) * qm;
                }
            }
            Q[o] = q;
            dQ[o] = dq;
        }
        __syncwarp();
        // radial factors: R1 = F' - k F / rho, R2 = F / rho (tangential term dropped at rho = 0)
        for (int col = lane; col < P.nF; col += 32) {
            const int k = P.colk[col];
            const int par = k & 1, ob = par ? P.m0 : 0, mp = par ? P.m1 : P.m0;
            double F = 0.0, dF = 0.0;
            for (int l = 0; l < mp; ++l) {
                const double wv = (double)P.Wt[(int64_t)l * P.nF + col];
                F += Q[ob + l] * wv;
                dF += dQ[ob + l] * wv;
            }
            T2 r;
            if (rho > 1e-30) { r.x = (T)(dF - k * F / rho); r.y = (T)(F / rho); }
            else { r.x = (T)dF; r.y = (T)0; }
            RR[col] = r;
        }
        }
        // level tables with d/dz and d/dq
        for (int j = 0; j < levels; ++j) {
            const int D = DD - 1 - j;
            T q = (T)0;
#pragma unroll
            for (int m = 0; m < DD; ++m)
                if (m <= D) q += xh[m] * xh[m];
            const T z = xh[D], qq = q;
            const T* A = P.coefA + j * P.tri;
            const T* B = P.coefB + j * P.tri;
            const int t0 = j * P.tri;
            for (int mu = lane; mu <= P.L; mu += 32) {
                const int o = mu * (P.L + 1) - mu * (mu - 1) / 2;
                const int nmax = P.L - mu;
                T v2 = A[o], z2 = (T)0, q2 = (T)0;
                put(t0 + o, v2, z2, q2);
                if (nmax >= 1) {
                    T v1 = A[o + 1] * z, z1 = A[o + 1], q1 = (T)0;
                    put(t0 + o + 1, v1, z1, q1);
                    for (int nn = 2; nn <= nmax; ++nn) {
                        const T an = A[o + nn], bn = B[o + nn];
                        const T v0 = an * z * v1 - bn * qq * v2;
                        const T z0 = an * (v1 + z * z1) - bn * qq * z2;
                        const T q0 = an * z * q1 - bn * (v2 + qq * q2);
                        put(t0 + o + nn, v0, z0, q0);
                        v2 = v1; z2 = z1; q2 = q1;
                        v1 = v0; z1 = z0; q1 = q0;
                    }
                }
            }
        }
        // (x0 + i x1)^mu and its derivatives, normalised as the harmonics
        typedef typename std::conditional<sizeof(T) == 4, float, double>::type TP;   // trig precision
        for (int mu = lane; mu <= P.L; mu += 32) {
            TP br = (TP)xh[0], bi = (TP)xh[1], rr = 1, ri = 0;     // z^mu
            TP pr = 1, pi = 0;                                      // z^(mu-1)
            int e = mu;
            while (e) {
                if (e & 1) { const TP t = rr * br - ri * bi; ri = rr * bi + ri * br; rr = t; }
                const TP t = br * br - bi * bi; bi = (TP)2 * br * bi; br = t;
                e >>= 1;
            }
            if (mu >= 1) {
                br = (TP)xh[0]; bi = (TP)xh[1]; e = mu - 1;
                while (e) {
                    if (e & 1) { const TP t = pr * br - pi * bi; pi = pr * bi + pi * br; pr = t; }
                    const TP t = br * br - bi * bi; bi = (TP)2 * br * bi; br = t;
                    e >>= 1;
                }
            }
            // value, d/dx_0, d/dx_1
            if (mu == 0) {
                put(trig + P.L, (T)0.3989422804014327, (T)0, (T)0);
            } else {
                const TP nm = (TP)0.5641895835477563;
                put(trig + P.L + mu, (T)(rr * nm), (T)(mu * pr * nm), (T)(-mu * pi * nm));      // Re z^mu
                put(trig + P.L - mu, (T)(ri * nm), (T)(mu * pi * nm), (T)(mu * pr * nm));       // Im z^mu
            }
        }
        __syncwarp();
        T g[kMaxD];
#pragma unroll
        for (int m = 0; m < kMaxD; ++m) g[m] = (T)0;
        T xt[kMaxD];
#pragma unroll
        for (int m = 0; m < DD; ++m) xt[m] = (T)xh[m];
        for (int gi = lane; gi < P.nH; gi += 32) {
            const int4 de = __ldg(P.desc + gi);
            const int2 kt = kts[de.y & 0xff];
            const T2* cp = reinterpret_cast<const T2*>(P.ab) + de.x;
            const T2* rp = RR + (kt.x & 0xffff);
            T al = (T)0, be = (T)0;
#pragma unroll 4
            for (int s = 0; s < kt.x >> 16; ++s) {
                const T2 c2 = __ldg(cp + (int64_t)s * kt.y), r2 = rp[s];
                const T cc = wi * c2.x + vi * c2.y;
                al += cc * r2.x;
                be += cc * r2.y;
            }
            T tr, tx, ty;
            get(trig + (de.y >> 8), tr, tx, ty);
            int of[kMaxD] = {de.z & 0xffff, (int)((unsigned)de.z >> 16), de.w & 0xffff, (int)((unsigned)de.w >> 16)};
            if constexpr (levels > 4) {
                const int e2 = __ldg(P.desc2 + gi);
                of[4] = e2 & 0xffff;
                of[5] = (int)((unsigned)e2 >> 16);
            }
            T pvv[kMaxD], pzz[kMaxD], pqq[kMaxD];
#pragma unroll
            for (int j = 0; j < levels; ++j) get(j * P.tri + of[j], pvv[j], pzz[j], pqq[j]);
            // suffix products suf[j] = prod_{j2 > j} P_j2, so that the product of all level
            // factors but one is (trig * prefix) * suffix: O(levels) per harmonic
            T suf[kMaxD];
            if (levels > 0) suf[levels - 1] = (T)1;
#pragma unroll
            for (int j = levels - 2; j >= 0; --j) suf[j] = suf[j + 1] * pvv[j + 1];
            const T pl = (levels > 0) ? pvv[0] * suf[0] : (T)1;      // all level factors
            const T prod = tr * pl;
            // Y x_hat term
#pragma unroll
            for (int m = 0; m < DD; ++m) g[m] += al * prod * xt[m];
            // grad H: level terms
            T pre = tr;                                  // trig * prod_{j2 < j} P_j2
#pragma unroll
            for (int j = 0; j < levels; ++j) {
                const T other = pre * suf[j];
                pre *= pvv[j];
                const int D = DD - 1 - j;
                const T cz = be * other * pzz[j], cq = be * other * pqq[j] * (T)2;
                g[D] += cz;
#pragma unroll
                for (int m = 0; m < DD; ++m)
                    if (m <= D) g[m] += cq * xt[m];
            }
            // grad H: trigonometric factor
            g[0] += be * pl * tx;
            g[1] += be * pl * ty;
        }
#pragma unroll
        for (int m = 0; m < DD; ++m) {
            T vsum = g[m];
            for (int o = 16; o > 0; o >>= 1) vsum += __shfl_xor_sync(0xffffffffu, vsum, o);
            g[m] = vsum;
        }
        if (lane < DD) {
            T vsum = (T)0;
#pragma unroll
    #pragma unroll
        for (int m = 0; m < DD; ++m) if (m == lane) vsum = g[m];
            const T out = vsum * (T)P.inv2R;
            T* dst = P.grad + i * DD + lane;
            *dst = P.accumulate ? *dst + out : out;
        }
        __syncwarp();
        }
    }
}

// dS_k/dl = W_k^T R_f (dGamma_k/dl) R_f^T W_k with dGamma from the Chebyshev coefficients of
// d kappa/d l truncated at the build's degree (frozen p, c, R).
void compute_dS(hdf_factor* f) {
    FactorPlan& P = f->plan;
    const int M = hdf::cheb_nodes(P.p_max);          // the build's node count
    std::vector<double> a(std::max(M, 2 * P.L + 2));
    hdf::cheb_coeffs(f->kernel, f->ell, 1.0 / P.inv2R, M, true, a.data());
    for (size_t i = 2 * P.L + 1; i < a.size(); ++i) a[i] = 0.0;
    std::vector<std::vector<double>> dG;
    hdf::radial_cores(a.data(), 2 * P.L, P.d, dG);
    P.dSk.assign(P.L + 1, std::vector<double>());
    for (int k = 0; k <= P.L; ++k) {
        const int sk = P.sk[k];
        if (sk == 0) continue;
        const int par = k & 1, nb = P.nb[par], mk = P.m[par];
        const std::vector<double>& Rf = P.Rf[par];
        const std::vector<double>& W = P.Wk[k];
        // T1 = R_f dG R_f^T (mk x mk)
        std::vector<double> A((size_t)mk * nb, 0.0), T1((size_t)mk * mk, 0.0), T2((size_t)sk * mk, 0.0);
        for (int o = 0; o < mk; ++o)
            for (int l = 0; l < nb; ++l) {
                double s = 0.0;
                for (int t = 0; t < nb; ++t) s += Rf[(size_t)o * nb + t] * dG[k][(size_t)t * nb + l];
                A[(size_t)o * nb + l] = s;
            }
        for (int o = 0; o < mk; ++o)
            for (int o2 = 0; o2 < mk; ++o2) {
                double s = 0.0;
                for (int l = 0; l < nb; ++l) s += A[(size_t)o * nb + l] * Rf[(size_t)o2 * nb + l];
                T1[(size_t)o * mk + o2] = s;
            }
        for (int s_ = 0; s_ < sk; ++s_)
            for (int o2 = 0; o2 < mk; ++o2) {
                double s = 0.0;
                for (int o = 0; o < mk; ++o) s += W[(size_t)o * sk + s_] * T1[(size_t)o * mk + o2];
                T2[(size_t)s_ * mk + o2] = s;
            }
        std::vector<double> dS((size_t)sk * sk, 0.0);
        for (int s_ = 0; s_ < sk; ++s_)
            for (int t_ = 0; t_ < sk; ++t_) {
                double s = 0.0;
                for (int o2 = 0; o2 < mk; ++o2) s += T2[(size_t)s_ * mk + o2] * W[(size_t)o2 * sk + t_];
                dS[(size_t)s_ * sk + t_] = s;
            }
        P.dSk[k].swap(dS);
    }
    P.have_dS = true;
}

template <typename T>
hdf_status run(hdf_factor* f, const double* x, const T* V, int64_t ldv, const T* Wv, int64_t ldw, int ncols,
               T* grad, double* grad_l, double* value, cudaStream_t st) {
    FactorPlan& P = f->plan;
    const int64_t n = f->info.n, r = (f->info.rank > 0) ? f->info.ldu : 0;   // padded width of U
    const int d = P.d;
    if (r == 0) {
        HDF_CUDA(cudaMemsetAsync(grad, 0, sizeof(T) * n * d, st));
        HDF_CUDA(cudaStreamSynchronize(st));
        if (grad_l) *grad_l = 0.0;
        if (value) *value = 0.0;
        return HDF_OK;
    }
    DevBuf ab, zd, vw;
    HDF_CUDA(ab.alloc_on(sizeof(T) * (size_t)r * ncols * 2, st));
    HDF_CUDA(zd.alloc_on(sizeof(double) * (size_t)r * ncols * 2, st));
    // U^T [V W] (FP64, r x 2 ncols row-major) in one pass over U when the 2 ncols columns fit
    // one group: [V W] is gathered into an n x 2 ncols column-major block first
    std::vector<double> hz((size_t)r * ncols * 2);
    const int c2 = 2 * ncols;
    if (c2 <= 64) {
        HDF_CUDA(vw.alloc_on(sizeof(T) * (size_t)n * c2, st));
        HDF_CUDA(cudaMemcpy2DAsync(vw.p, sizeof(T) * n, V, sizeof(T) * ldv, sizeof(T) * n, ncols,
                                   cudaMemcpyDeviceToDevice, st));
        HDF_CUDA(cudaMemcpy2DAsync(vw.as<T>() + (size_t)n * ncols, sizeof(T) * n, Wv, sizeof(T) * ldw, sizeof(T) * n,
                                   ncols, cudaMemcpyDeviceToDevice, st));
        hdf_status s = hdf::utv_reduce<T>(f, vw.as<T>(), n, c2, nullptr, nullptr, zd.as<double>(), st);
        if (s != HDF_OK) return s;
        HDF_CUDA(cudaMemcpyAsync(hz.data(), zd.p, sizeof(double) * hz.size(), cudaMemcpyDeviceToHost, st));
    } else {
        double* zv = zd.as<double>();
        double* zw = zv + (size_t)r * ncols;
        hdf_status s = hdf::utv_reduce<T>(f, V, ldv, ncols, nullptr, nullptr, zv, st);
        if (s != HDF_OK) return s;
        s = hdf::utv_reduce<T>(f, Wv, ldw, ncols, nullptr, nullptr, zw, st);
        if (s != HDF_OK) return s;
        std::vector<double> hv((size_t)r * ncols * 2);
        HDF_CUDA(cudaMemcpyAsync(hv.data(), zd.p, sizeof(double) * hv.size(), cudaMemcpyDeviceToHost, st));
        HDF_CUDA(cudaStreamSynchronize(st));
        for (int64_t col = 0; col < r; ++col)          // into the [V W] row layout
            for (int j = 0; j < ncols; ++j) {
                hz[(size_t)col * c2 + j] = hv[(size_t)col * ncols + j];
                hz[(size_t)col * c2 + ncols + j] = hv[(size_t)r * ncols + (size_t)col * ncols + j];
            }
    }
    HDF_CUDA(cudaStreamSynchronize(st));
    std::vector<T> hab((size_t)r * ncols * 2);     // per column of V: (S U^T v, S U^T w) of every column of U
    double fval = 0.0;
    for (int64_t col = 0; col < r; ++col)
        for (int j = 0; j < ncols; ++j) {
            const size_t q = 2 * ((size_t)j * r + col);
            const double sc = P.Spad[col];
            const double zv = hz[(size_t)col * c2 + j], zw = hz[(size_t)col * c2 + ncols + j];
            hab[q] = (T)(sc * zv);
            hab[q + 1] = (T)(sc * zw);
            fval += zw * sc * zv;
        }
    HDF_CUDA(cudaMemcpyAsync(ab.p, hab.data(), sizeof(T) * hab.size(), cudaMemcpyHostToDevice, st));

    AdjParams<T> A{};
    A.x = x;
    A.n = n; A.d = d;
    for (int j = 0; j < d; ++j) A.c[j] = P.c[j];
    A.inv2R = P.inv2R;
    A.L = P.L_used; A.Lr = P.L; A.tri = P.tri;
    A.Qm0 = P.dQ0.as<double>(); A.nb0 = P.nb[0]; A.m0 = P.m[0];
    A.Qm1 = P.dQ1.as<double>(); A.nb1 = P.nb[1]; A.m1 = P.m[1];
    A.QC = P.dQC.as<float2>(); A.mtp = ((P.m[0] + P.m[1] + 7) / 8) * 8;
    if (sizeof(T) == 4 && A.QC == nullptr)
        return hdf::fail(HDF_EINVAL, "hdf_matvec_adjoint: factor lacks its FP32 radial tables");
    A.Wt = P.dW.as<T>(); A.colk = P.dcolk.as<uint8_t>(); A.nF = P.nF;
    A.nH = P.nH; A.nk = P.L + 1; A.ktab = P.dktab.as<int>();
    DevBuf dd;
    HDF_CUDA(dd.alloc_on((sizeof(int4) + sizeof(int)) * (size_t)P.nH, st));
    A.desc = dd.as<int4>();
    A.desc2 = d >= 7 ? reinterpret_cast<const int*>(dd.as<int4>() + P.nH) : nullptr;
    HDF_COUNT_LAUNCH();
    k_adj_desc<<<(P.nH + 255) / 256, 256, 0, st>>>(P.dchains.as<int16_t>(), P.nH, hdf::chain_stride(d), d - 2, P.L_used,
                                                   P.dhk.as<uint8_t>(), A.ktab, dd.as<int4>(), const_cast<int*>(A.desc2));
    HDF_CUDA(cudaGetLastError());
    A.coefA = P.dA.as<T>(); A.coefB = P.dB.as<T>();
    A.grad = grad;
    const int levels = d - 2;
    int nsm = 0, dv = 0, occ = 0;
    HDF_CUDA(cudaGetDevice(&dv));
    HDF_CUDA(cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dv));
    // the limit of four warps' tables without batches and padding
    if (4 * (8 * (2 * ((size_t)P.L + 1) + 2 * (P.m[0] + P.m[1])) +
             sizeof(T) * ((2 * (size_t)P.nF + 3 * levels * P.tri + 3 * (2 * P.L_used + 1) + 3) & ~(size_t)3)) >
        200 * 1024)
        return hdf::fail(HDF_ETOOBIG, "hdf_matvec_adjoint: per-point tables exceed shared memory");
    using K = void (*)(AdjParams<T>);
    const K packed[] = {k_adjoint<T, 3, true>, k_adjoint<T, 4, true>, k_adjoint<T, 5, true>,
                        k_adjoint<T, 6, true>, k_adjoint<T, 7, true>, k_adjoint<T, 8, true>};
    const K narrow[] = {k_adjoint<T, 3, false>, k_adjoint<T, 4, false>, k_adjoint<T, 5, false>,
                        k_adjoint<T, 6, false>, k_adjoint<T, 7, false>, k_adjoint<T, 8, false>};
    // Batch, table layout and warps per CTA: the first in the order below that keeps kAdjFull warps on an
    // SM, else the one that keeps most (on a tie the smaller batch).  From about 28 warps on (FP64: 20, more
    // registers per thread) more of them gain nothing, while batches of four save up to 20% and packed
    // tables 4% (500,000 points, d = 4, 2,104 columns: 3.94 ms; three arrays 4.11; batches of one 4.43);
    // below, the time goes with the warps: d = 4, 30,000 points, 37,452 columns 7.14 ms on 8 warps (packed,
    // CTAs of four), 4.64 on 14; d = 5, 2,000 points, 523,787 columns 20.2 ms on 4, 8.5 on 8; d = 3,
    // 150,000 points, 8,997 columns 7.5 ms on 12, 5.9 on 18.
    constexpr int kAdjFull = sizeof(T) == 8 ? 20 : 28;
    K kern = nullptr;
    int warps = 0, best = 0;
    size_t sm = 0;
    int nb_max = kAdjBatch;
    while (nb_max > 1 && n < (int64_t)64 * nsm * nb_max) nb_max /= 2;
    for (int nb = nb_max; nb >= 1 && best < kAdjFull; nb /= 2)
        for (int pk = 1; pk >= 0 && best < kAdjFull; --pk) {
            const K k = (pk ? packed : narrow)[d - 3];
            const size_t pw = adj_per_warp<T>(levels, P.tri, P.L_used, P.nF, P.L, P.m[0] + P.m[1], nb, pk == 1);
            for (int w : {4, 2, 1}) {
                if (w * pw > 220 * 1024) continue;
                HDF_CUDA(cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)(w * pw)));
                int o = 0;
                HDF_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&o, k, w * 32, w * pw));
                if (o * w > best || (o * w == best && best < kAdjFull && nb < A.nb)) {
                    kern = k; warps = w; best = o * w; occ = o; sm = w * pw;
                    A.nb = nb;
                    A.per_warp = (int)pw;
                }
                if (best >= kAdjFull) break;
            }
        }
    HDF_CUDA(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm));
    const int grid = std::max(1, std::min<int>(nsm * std::max(occ, 1), (int)((n + warps * A.nb - 1) / (warps * A.nb))));
    for (int j = 0; j < ncols; ++j) {
        A.ab = ab.as<T>() + 2 * (size_t)j * r;
        A.v = V + j * ldv; A.w = Wv + j * ldw;
        A.accumulate = (j > 0);
        HDF_COUNT_LAUNCH();
        kern<<<grid, warps * 32, sm, st>>>(A);
        HDF_CUDA(cudaGetLastError());
    }
    // d f / d l on the host from U^T V, U^T W and the frozen dS_k/dl
    if (grad_l) {
        if (!P.have_dS) compute_dS(f);
        double gl = 0.0;
        std::vector<double> tmp;
        for (int k = 0; k <= P.L; ++k) {
            const int sk = P.sk[k];
            if (sk == 0) continue;
            const int dim = (int)hdf::harmonic_count(k, d);
            const int dimp = (k + 1 < (int)P.cbase.size() && sk > 0) ? (P.cbase[k + 1] - P.cbase[k]) / sk : dim;
            const std::vector<double>& dS = P.dSk[k];
            for (int j = 0; j < ncols; ++j)
                for (int h = 0; h < dim; ++h)
                    for (int s_ = 0; s_ < sk; ++s_) {
                        const int64_t cs = P.cbase[k] + (int64_t)s_ * dimp + h;
                        double acc = 0.0;
                        for (int t_ = 0; t_ < sk; ++t_) {
                            const int64_t ct = P.cbase[k] + (int64_t)t_ * dimp + h;
                            acc += dS[(size_t)s_ * sk + t_] * hz[(size_t)ct * c2 + j];
                        }
                        gl += hz[(size_t)cs * c2 + ncols + j] * acc;
                    }
        }
        *grad_l = gl;
    }
    if (value) *value = fval;
    HDF_CUDA(cudaStreamSynchronize(st));
    return hdf::take_device_error(f);
}

}  // namespace

extern "C" hdf_status hdf_matvec_adjoint(hdf_factor* f, const double* x_dev, const void* V_dev, int64_t ldv,
                                         const void* W_dev, int64_t ldw, int ncols, void* grad_x_dev,
                                         double* grad_l_host, double* value_host, hdf_stream stream) {
    if (!f || !x_dev || !V_dev || !W_dev || !grad_x_dev || ncols < 1 || ncols > 64 || ldv < f->info.n ||
        ldw < f->info.n)
        return hdf::fail(HDF_EINVAL, "hdf_matvec_adjoint: bad argument (1 <= ncols <= 64)");
    if (f->ypart) return hdf::fail(HDF_EINVAL, "hdf_matvec_adjoint: symmetric factors only");
    cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
    if (f->prec == HDF_FP64)
        return run<double>(f, x_dev, (const double*)V_dev, ldv, (const double*)W_dev, ldw, ncols, (double*)grad_x_dev,
                           grad_l_host, value_host, st);
    return run<float>(f, x_dev, (const float*)V_dev, ldv, (const float*)W_dev, ldw, ncols, (float*)grad_x_dev,
                      grad_l_host, value_host, st);
}
