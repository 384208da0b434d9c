// U rows of FP32 factors with few columns, straight from the points: lane = point.
//
// What bounds the two-kernel form (k_radial_F_df, then k_uwriter) at a loose tolerance: a point has
// about ten radial functions and a hundred harmonics, so the tiles of 32 points that 512 threads
// share have work for a few warps only, the F rows make a round trip through HBM padded to 128
// bytes, and a warp per point leaves most lanes without a recurrence of their own.  10,000,000
// points, d = 5, rank 125: 8.26 + 9.98 ms against 0.8 ms to write U.
//
// Here a lane owns one point from its coordinates to its row: the radial functions F = T (Qmat W_k)
// with T_l in double-float arithmetic and the dot products by Dot2 (see k_radial_F_df; the product
// Qmat W_k is formed on the host in FP64, since there are fewer radial functions than basis
// functions here), the level tables of the harmonics, and the row.  Nothing is shared between lanes
// but broadcast tables.  Two warps work on a tile of 32 points, since its rows and tables take the
// shared memory that more tiles would need: one forms the radial functions while the other forms
// the harmonics, then each writes half of every degree's columns.  A harmonic of the chain (mu_1, ..,
// mu_{d-2}) is a prefix (the levels but the last) times G[mu, m] = last level P(|m|, mu - |m|) times
// trigonometric factor m, mu = mu_{d-3} (the degree in d = 3); the 2 mu + 1 harmonics with one prefix
// are consecutive columns and consecutive entries of G, so an entry of U is one product and one
// store.  G is written as the last level's recurrence runs (no table of that level, no
// trigonometric table).  Rows are formed in shared memory, 4 floats longer than ldU (a stride of
// 4 x odd: four lanes per bank), and leave by one bulk copy per lane while the next tile's tables are
// formed.  Bound by the latency of shared memory at the tiles that an SM has room for: 2.9 ms for
// the 10,000,000 points above; 1,000,000 points, d = 5, rank 216: 0.62 ms (1.1 with one warp per tile
// and a table of every level).
//
// Used where a tile's tables and rows leave at least kMinPairs tiles per SM (rows_lane_plan); a
// point with more state keeps the warp-per-point writer, whose lanes then have work.  Radial factors and
// rows of 1,000,000 points, this kernel against the two: 8 tiles per SM 0.44 to 0.65 of their time, 5
// tiles 0.83 to 0.94 (d = 4, rank 200: 0.53 against 0.56 ms), 4 tiles 0.81 to 0.95 (d = 5, rank 252: 0.67
// and 0.71), 3 tiles 1.07 to 1.36 (d = 4, rank 310: 0.95 and 0.81), 2 tiles 1.40 to 1.72, 1 tile 2.6 to
// 3.2; at 30,000 points 4 tiles 0.74 to 0.84, 3 tiles 0.92 to 1.17.
#include <cuda_runtime.h>

#include <algorithm>
#include <cstring>
#include <vector>

#include "hdf_kernels.cuh"
#include "internal.h"
#include "planner.h"
#include "rows_lane.h"

namespace hdf {
namespace {

constexpr int kMinPairs = 4, kMaxPairs = 8;
constexpr size_t kBudget = 226 * 1024;

struct LaneParams {
    const double* x; int64_t n; dev::Center c; double inv2R;
    int L, nF, nF0, nFp;                 // radial degree; F columns, of them even; columns of RC
    int Lu, tri;                         // harmonics
    int ngrp, ndeg;                      // prefix groups, degrees with columns
    int ldU, rs;                         // row width and its stride in shared memory
    int lane_floats;                     // table entries per lane
    float* U;
    const float2* RC;                    // (L + 1) x nFp: Qmat W_k as (hi, lo) pairs
    const float* cA; const float* cB;
    const int* tab;                      // groups, degrees (see rows_lane_plan)
    int tab_ints;
};

__device__ __forceinline__ void bulk_store(void* g, const void* s, uint32_t bytes) {
    asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;" ::"l"(g),
                 "r"((uint32_t)__cvta_generic_to_shared(s)), "r"(bytes)
                 : "memory");
}

// F columns c0 .. c0 + NB - 1 (c0 a multiple of 16): sum_l T_l(u) RC[l][c] by Dot2 while the
// double-float recurrence of T runs in registers; odd columns times rho.
template <int NB>
__device__ __forceinline__ void radial_cols(const LaneParams& P, const float2* RC, double u, float rho, int c0, float* F) {
    float sh[NB], cc[NB];
#pragma unroll
    for (int j = 0; j < NB; ++j) sh[j] = cc[j] = 0.f;
    const float uh = (float)u, ul = (float)(u - (double)uh);
    const float u2h = 2.f * uh, u2l = 2.f * ul;
    float ah = uh, al = ul, bh = 1.f, bl = 0.f;              // T_{-1} = T_1 = u, T_0 = 1
    const float2* rc = RC + c0;
    for (int l = 0; l <= P.L; ++l, rc += P.nFp) {
        const float2 T = make_float2(bh, bl);
#pragma unroll
        for (int j = 0; j < NB; j += 2) {
            const float4 g = *reinterpret_cast<const float4*>(rc + j);
            dev::dot2_step(T, g.x, g.y, sh[j], cc[j]);
            if (j + 1 < NB) dev::dot2_step(T, g.z, g.w, sh[j + 1], cc[j + 1]);
        }
        // T_{l+1} = 2 u T_l - T_{l-1}
        const float ph = u2h * bh;
        float pl = fmaf(u2h, bh, -ph);
        pl = fmaf(u2h, bl, fmaf(u2l, bh, pl));
        float s, e;
        dev::two_sum(ph, -ah, s, e);
        e += pl - al;
        ah = bh; al = bl;
        dev::fast_two_sum(s, e, bh, bl);
    }
#pragma unroll
    for (int j = 0; j < NB; ++j) {
        float f = sh[j] + cc[j];
        if (c0 + j >= P.nF0) f *= rho;
        if (c0 + j < P.nF) F[32 * (c0 + j)] = f;
    }
}

// Columns of one prefix group for NS radial functions: row[s step + t] = f_s a G[t], t < LEN (LEN = 0:
// len, at run time).
template <int NS, int LEN>
__device__ __forceinline__ void group_run(const float* G, int len, const float* f, float* row, int step) {
    if constexpr (LEN > 0) {
#pragma unroll
        for (int t = 0; t < LEN; ++t) {
            const float y = G[32 * t];
#pragma unroll
            for (int s = 0; s < NS; ++s) row[s * step + t] = f[s] * y;
        }
    } else {
#pragma unroll 4
        for (int t = 0; t < len; ++t) {
            const float y = G[32 * t];
#pragma unroll
            for (int s = 0; s < NS; ++s) row[s * step + t] = f[s] * y;
        }
    }
}
// All groups [g0, g1) of one degree for NS of its radial functions.
template <int NS, int LV>
__device__ __forceinline__ void degree_cols(const int* grp, int g0, int g1, const float* tbl, const float* G,
                                            const float* F, float* row, int step) {
    float fs[NS];
#pragma unroll
    for (int s = 0; s < NS; ++s) fs[s] = F[32 * s];
    // G base | length << 16, column | prefix 4 << 16, prefixes 0 | 1 << 16, 2 | 3 << 16; the next
    // group's record and prefix are read while this group's columns are written
    auto prefix = [&](const int4& w) {
        float a = 1.f;
        if (LV >= 2) a = tbl[32 * (w.z & 0xffff)];
        if (LV >= 3) a *= tbl[32 * (w.z >> 16)];
        if (LV >= 4) a *= tbl[32 * (w.w & 0xffff)];
        if (LV >= 5) a *= tbl[32 * (w.w >> 16)];
        if (LV >= 6) a *= tbl[32 * (w.y >> 16)];
        return a;
    };
    int4 wn = *reinterpret_cast<const int4*>(grp + 4 * g0);
    float an = prefix(wn);
    for (int g = g0; g < g1; ++g) {
        const int4 w = wn;
        const float a = an;
        wn = *reinterpret_cast<const int4*>(grp + 4 * min(g + 1, g1 - 1));
        an = prefix(wn);
        const float* Gg = G + 32 * (w.x & 0xffff);
        const int len = w.x >> 16;
        float* out = row + (w.y & 0xffff);
        float f[NS];
#pragma unroll
        for (int s = 0; s < NS; ++s) f[s] = a * fs[s];
        switch (len) {
            case 1: group_run<NS, 1>(Gg, len, f, out, step); break;
            case 3: group_run<NS, 3>(Gg, len, f, out, step); break;
            case 5: group_run<NS, 5>(Gg, len, f, out, step); break;
            case 7: group_run<NS, 7>(Gg, len, f, out, step); break;
            case 9: group_run<NS, 9>(Gg, len, f, out, step); break;
            default: group_run<NS, 0>(Gg, len, f, out, step); break;
        }
    }
}

template <int DD>
__global__ void __launch_bounds__(64 * kMaxPairs, 1) k_rows_lane(const LaneParams P) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    constexpr int LV = DD - 2;
    const int lane = threadIdx.x & 31, pair = threadIdx.x >> 6, npairs = blockDim.x >> 6;
    const int role = (threadIdx.x >> 5) & 1;             // 0: radial functions and the copies, 1: harmonics
    // shared tables
    float2* RC = reinterpret_cast<float2*>(smem_raw);
    float* cA = reinterpret_cast<float*>(RC + (P.L + 1) * P.nFp);
    float* cB = cA + LV * P.tri;
    int* tab = reinterpret_cast<int*>(smem_raw +
                                      dev::align16(reinterpret_cast<unsigned char*>(cB + LV * P.tri) - smem_raw));
    for (int e = threadIdx.x; e < (P.L + 1) * P.nFp; e += blockDim.x) RC[e] = P.RC[e];
    for (int e = threadIdx.x; e < LV * P.tri; e += blockDim.x) { cA[e] = P.cA[e]; cB[e] = P.cB[e]; }
    for (int e = threadIdx.x; e < P.tab_ints; e += blockDim.x) tab[e] = P.tab[e];
    // this pair's rows and per-lane tables ([entry][lane])
    size_t off = (reinterpret_cast<unsigned char*>(tab + P.tab_ints) - smem_raw + 127) & ~(size_t)127;
    float* rows = reinterpret_cast<float*>(smem_raw + off) + (size_t)pair * 32 * (P.rs + P.lane_floats);
    float* base = rows + 32 * P.rs;
    for (int e = threadIdx.x & 63; e < 32 * P.rs; e += 64) rows[e] = 0.f;   // padding columns stay zero
    __syncthreads();
    float* row = rows + lane * P.rs;
    float* F = base + lane;                                              // nF
    float* tbl = base + 32 * P.nF + lane;                                // levels but the last
    float* G = tbl + 32 * (LV - 1) * P.tri;                              // (Lu + 1)^2
    const int* grp = tab;                                                // ngrp x 4
    const int* deg = tab + 4 * P.ngrp;                                   // ndeg x 8
    const int64_t ntiles = (P.n + 31) / 32, stride = (int64_t)gridDim.x * npairs;
    int64_t tile = (int64_t)blockIdx.x * npairs + pair;
    auto pair_sync = [&]() { asm volatile("bar.sync %0, 64;" ::"r"(pair + 1) : "memory"); };
    double xn[DD];
    auto load_x = [&](int64_t t) {
        const int64_t i = min(t * 32 + lane, P.n - 1);
#pragma unroll
        for (int j = 0; j < DD; ++j) xn[j] = P.x[i * DD + j];
    };
    if (tile < ntiles) load_x(tile);
    for (; tile < ntiles; tile += stride) {
        float xh[DD];
        double s64 = 0.0;
        float s = 0.f;
#pragma unroll
        for (int j = 0; j < DD; ++j) {
            const double y = (xn[j] - P.c.c[j]) * P.inv2R;
            s64 += y * y;
            xh[j] = (float)y;
            s += xh[j] * xh[j];
        }
        if (tile + stride < ntiles) load_x(tile + stride);               // in flight during this tile
        if (role == 0) {
        // ---- radial functions
        const double u = 8.0 * s64 - 1.0;
        const float rho = sqrtf((float)s64);
        int c0 = 0;
        for (; P.nF - c0 > 16; c0 += 16) radial_cols<16>(P, RC, u, rho, c0, F);
        const int left = P.nF - c0;
        if (left > 12) radial_cols<16>(P, RC, u, rho, c0, F);
        else if (left > 8) radial_cols<12>(P, RC, u, rho, c0, F);
        else if (left > 4) radial_cols<8>(P, RC, u, rho, c0, F);
        else if (left > 0) radial_cols<4>(P, RC, u, rho, c0, F);
        // the previous tile's copies have read the rows
        asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
        } else {
        // ---- direction, level tables, trigonometric powers
        if (s > 0.f) {
            const float inv = 1.f / sqrtf(s);
#pragma unroll
            for (int j = 0; j < DD; ++j) xh[j] *= inv;
        } else {
#pragma unroll
            for (int j = 0; j < DD; ++j) xh[j] = j == 0 ? 1.f : 0.f;
        }
        {
            // the levels' three-term recurrences side by side (LV independent chains), the last one (z =
            // x_2) times the trigonometric factors into G[mu^2 + mu +- m], mu = m + nn
            float z[LV], qq[LV];
#pragma unroll
            for (int j = 0; j < LV; ++j) {
                z[j] = xh[DD - 1 - j];
                qq[j] = 0.f;
#pragma unroll
                for (int m = 0; m < DD; ++m)
                    if (m <= DD - 1 - j) qq[j] += xh[m] * xh[m];
            }
            float rr = 0.3989422804014327f, ri = 0.f;                     // m = 0: 1 / sqrt(2 pi)
            int e = 0;                                                    // table index of (m, nn)
            for (int m = 0; m <= P.Lu; ++m) {
                float p1[LV], p2[LV];                                     // values at nn - 1 and nn - 2
                float* g = G + 32 * (m * m + m);
                const int nmax = P.Lu - m;
#pragma unroll 2
                for (int nn = 0; nn <= nmax; ++nn, ++e) {
#pragma unroll
                    for (int j = 0; j < LV; ++j) {
                        const float A = cA[j * P.tri + e], B = cB[j * P.tri + e];
                        const float v = nn == 0 ? A : nn == 1 ? A * z[j] : A * z[j] * p1[j] - B * qq[j] * p2[j];
                        p2[j] = nn == 0 ? 0.f : p1[j];
                        p1[j] = v;
                        if (j < LV - 1) tbl[32 * (j * P.tri + e)] = v;
                    }
                    g[32 * m] = p1[LV - 1] * rr;
                    if (m > 0) g[-32 * m] = p1[LV - 1] * ri;
                    g += 64 * (m + nn + 1);                               // mu^2 + mu to the next mu
                }
                const float cr = m == 0 ? 0.5641895835477563f : rr;       // 1 / sqrt(pi) from m = 1 on
                const float t = cr * xh[0] - ri * xh[1];
                ri = cr * xh[1] + ri * xh[0];
                rr = t;
            }
        }
        }
        pair_sync();
        // ---- the row: half of each degree's groups per warp
        for (int q = 0; q < P.ndeg; ++q) {
            // first group, the other warp's first group, end, F column | s_k << 16; step
            const int4 d4 = *reinterpret_cast<const int4*>(deg + 8 * q);
            const int step = deg[8 * q + 4];
            const int g0 = role ? d4.y : d4.x, g1 = role ? d4.z : d4.y;
            if (g0 >= g1) continue;
            const int sk = d4.w >> 16;
            for (int s0 = 0; s0 < sk; s0 += 4) {
                const float* Fk = F + 32 * ((d4.w & 0xffff) + s0);
                float* out = row + s0 * step;
                switch (sk - s0) {
                    case 1: degree_cols<1, LV>(grp, g0, g1, tbl, G, Fk, out, step); break;
                    case 2: degree_cols<2, LV>(grp, g0, g1, tbl, G, Fk, out, step); break;
                    case 3: degree_cols<3, LV>(grp, g0, g1, tbl, G, Fk, out, step); break;
                    default: degree_cols<4, LV>(grp, g0, g1, tbl, G, Fk, out, step); break;
                }
            }
        }
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        pair_sync();
        if (role == 0) {
            const int64_t i = tile * 32 + lane;
            if (i < P.n) bulk_store(P.U + i * P.ldU, row, 4u * (uint32_t)P.ldU);
            asm volatile("cp.async.bulk.commit_group;" ::: "memory");
        }
    }
    asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
}

}  // namespace

// Host tables and shared-memory plan.  Groups: runs of harmonics of one degree whose chains share
// every level but the last; each has to run through m = -mu .. mu of one mu in order.  False when
// it does not, or when the tables do not leave kMinPairs tiles per SM.
bool rows_lane_plan(int d, int L, const FactorChoice& fc, const DeviceTables& tb, RowsLanePlan& out) {
    const int levels = d - 2, cs = chain_stride(d), Lu = tb.L_used;
    const int lane_harm = (levels - 1) * tb.tri + (Lu + 1) * (Lu + 1);
    if (tb.nH == 0 || tb.nF >= (1 << 15) || lane_harm >= (1 << 15) || tb.ldU >= (1 << 15)) return false;
    out.lane_floats = (tb.nF + lane_harm + 3) / 4 * 4;
    out.rs = (int)tb.ldU + 4;
    const size_t pair = sizeof(float) * 32 * (size_t)(out.rs + out.lane_floats);
    if (kMinPairs * pair > kBudget) return false;
    std::vector<int> grp, deg;
    out.nF0 = 0;
    while (out.nF0 < tb.nF && tb.colpar[out.nF0] == 0) ++out.nF0;
    for (size_t k = 0; k + 1 < tb.hbase.size(); ++k) {
        const int* kt = &tb.ktab[kTabStride * k];
        if (kt[1] == 0 || kt[3] == 0) continue;
        const int first = (int)(grp.size() / 4);
        for (int h = 0; h < kt[3];) {
            const int16_t* c0 = &tb.chains[(size_t)(kt[4] + h) * cs];
            const int mu = -(int)c0[levels];
            if (mu < 0 || mu > Lu || h + 2 * mu + 1 > kt[3]) return false;
            for (int m = -mu; m <= mu; ++m) {
                const int16_t* c = &tb.chains[(size_t)(kt[4] + h + m + mu) * cs];
                const int am = std::abs(m);
                if (std::memcmp(c, c0, sizeof(int16_t) * (levels - 1)) != 0 || c[levels] != m ||
                    c[levels - 1] != am * (Lu + 1) - am * (am - 1) / 2 + (mu - am))
                    return false;
            }
            int pre[5] = {0, 0, 0, 0, 0};
            for (int j = 0; j < levels - 1; ++j) pre[j] = j * tb.tri + c0[j];
            grp.push_back((mu * mu) | ((2 * mu + 1) << 16));
            grp.push_back((kt[2] + h) | (pre[4] << 16));
            grp.push_back(pre[0] | (pre[1] << 16));
            grp.push_back(pre[2] | (pre[3] << 16));
            h += 2 * mu + 1;
        }
        // the second warp starts where half of the columns are passed (degrees of one group go to the
        // warps in turn)
        const int last = (int)(grp.size() / 4);
        int mid = first, cols = 0;
        while (mid < last && 2 * cols < kt[3]) cols += grp[4 * mid++] >> 16;
        if (last - first == 1) mid = (deg.size() / 8) % 2 ? first : last;
        const int dw[8] = {first, mid, last, kt[0] | (kt[1] << 16), kt[5], 0, 0, 0};
        deg.insert(deg.end(), dw, dw + 8);
    }
    out.ngrp = (int)(grp.size() / 4);
    out.ndeg = (int)(deg.size() / 8);
    out.tab = grp;
    out.tab.insert(out.tab.end(), deg.begin(), deg.end());
    out.nFp = (tb.nF + 15) / 16 * 16;
    const size_t shared = sizeof(float2) * (size_t)(L + 1) * out.nFp + sizeof(float) * 2 * (size_t)levels * tb.tri +
                          sizeof(int) * out.tab.size() + 256;
    if (shared + kMinPairs * pair > kBudget) return false;
    out.pairs = (int)std::min<size_t>(kMaxPairs, (kBudget - shared) / pair);
    out.smem = shared + out.pairs * pair;
    // Qmat W_k per parity, as (hi, lo) float pairs (odd columns: zero in row L)
    out.rc.assign((size_t)2 * (L + 1) * out.nFp, 0.f);
    for (size_t k = 0; k < fc.sk.size(); ++k) {
        const int par = (int)k % 2, nb = fc.nb[par], m = fc.m[par], sk = fc.sk[k];
        for (int l = 0; l < nb; ++l)
            for (int s = 0; s < sk; ++s) {
                double v = 0.0;
                for (int o = 0; o < m; ++o) v += fc.Qmat[par][(size_t)l * m + o] * fc.Wk[k][(size_t)o * sk + s];
                const float h = (float)v;
                float* p = &out.rc[2 * ((size_t)l * out.nFp + tb.fbase[k] + s)];
                p[0] = h;
                p[1] = (float)(v - (double)h);
            }
    }
    return true;
}

hdf_status rows_lane(const RowsLanePlan& pl, const double* x, int64_t n, int d, const dev::Center& c, double inv2R, int L,
                     const DeviceTables& tb, const float* cA, const float* cB, float* U, cudaStream_t st) {
    DevBuf dt;
    const size_t tb_bytes = sizeof(int) * pl.tab.size(), rc_bytes = sizeof(float) * pl.rc.size();
    HDF_CUDA(dt.alloc_on(rc_bytes + tb_bytes, st));
    unsigned char* p = dt.as<unsigned char>();
    HDF_CUDA(cudaMemcpyAsync(p, pl.rc.data(), rc_bytes, cudaMemcpyHostToDevice, st));
    HDF_CUDA(cudaMemcpyAsync(p + rc_bytes, pl.tab.data(), tb_bytes, cudaMemcpyHostToDevice, st));
    LaneParams P{x, n, c, inv2R, L, tb.nF, pl.nF0, pl.nFp, tb.L_used, tb.tri, pl.ngrp, pl.ndeg, (int)tb.ldU, pl.rs,
                 pl.lane_floats, U, reinterpret_cast<const float2*>(p), cA, cB, reinterpret_cast<const int*>(p + rc_bytes),
                 (int)pl.tab.size()};
    int dv = 0, nsm = 0;
    HDF_CUDA(cudaGetDevice(&dv));
    HDF_CUDA(cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dv));
    const int64_t tiles = (n + 31) / 32;
    const int grid = (int)std::max<int64_t>(1, std::min<int64_t>(nsm, (tiles + pl.pairs - 1) / pl.pairs));
    HDF_COUNT_LAUNCH();
#define HDF_RL(D)                                                                                                   \
    case D:                                                                                                         \
        HDF_CUDA(cudaFuncSetAttribute(k_rows_lane<D>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)pl.smem));  \
        k_rows_lane<D><<<grid, 64 * pl.pairs, pl.smem, st>>>(P);                                                    \
        break;
    switch (d) { HDF_RL(3) HDF_RL(4) HDF_RL(5) HDF_RL(6) HDF_RL(7) HDF_RL(8) }
#undef HDF_RL
    HDF_CUDA(cudaGetLastError());
    return HDF_OK;
}

}  // namespace hdf
