// FP64 products K~V on the tensor cores: U^T V and U W of FP64 factors by exact integer slices.
// Included by tc_gemm.cu (its PTX wrappers, tensor maps and bounded waits).
//
// Why.  GB300 retires 2 FP64 multiply-adds per clock and SM, 0.6e12 a second: at c columns an
// FP64 product needs 8 / c bytes of U per multiply-add and is bound by that pipe from c = 2 on
// (100,000 x 10,808, 64 columns: U^T V 114 ms, U W 130 ms, against 1.3 ms to read U).
//
// How (the error-free splitting of Ozaki, Ogita, Oishi and Rump, Numer. Algorithms 59, 2012, with
// integer digits).  Blocks of KB = 64 values along the contraction: of each MMA row of U and of
// each column of the small operand the block's largest exponent is taken and every value becomes
// the integer N = trunc(x 2^(55 - e)), |N| < 2^55 (x itself for every value within two binades of
// the largest, 55 bits below it for the others).  The small operand's N = sum_i d_i 256^(6 - i) has
// seven balanced digits -128 <= d_i <= 128, U's has the sign times the seven bytes of |N|; both
// are exact in FP16 (U's bytes as they are, i.e. as FP16 subnormals, 2^-24 per unit).  One
// kind::f16 MMA of slice i of U against the stacked slices 0 .. 7 - i of the other operand adds the
// products of levels l = i + j into the FP32 accumulators of the levels l = i .. 7; a level sums at
// most 7 x 64 products below 2^15, less than 2^24, so every FP32 sum is an exact integer.  The
// products of level > 7 are dropped (2^-63 of the block's largest product each; without level 7,
// dropping 2^-55, the error grew by half).  The promotion warps add the levels as one 64-bit integer
// in units of 2^-54 of the block's bound (levels 6 and 7 rounded into it), round it to FP64 with the
// two exponents, and add it to an FP64 register sum: two roundings per block where the multiply-add
// chain rounds 64 times.  Error against extended precision at 2,000 x 431, 1,500 x 10,064 and 3,001 x
// 1,960: 2.5 to 3.4e-16 relative (3.3 to 4.5e-16 while levels 6 and 7 were cut off instead of
// rounded), the streaming kernels of few_cols.cuh 1.9 to 3.5e-16, the register-tiled FP64 kernels 1.0
// to 4.8e-15.
//
// Why this split.  What bounds the kernel is the ALU pipe (64 lanes per clock and SM) of the
// converters and the promotion, then the read of U.  Splitting and packing a value takes about 14
// ALU operations (the FP64 pipe would take 16 clocks per warp and operation), hence sign and
// bytes instead of balanced digits on U's side, subnormals instead of an FP16 offset, shifts by
// the multiplier (hi + hi, 4 lo), and one promotion per 64 values: nine-bit digits need 21 slice
// products instead of 28 but leave K = 32 per promotion.  A first form with balanced digits on
// both sides, a bias, an FP16 subtraction and four promotion warps ran at 74% of the ALU pipe:
// U^T V 3.18 ms at 100,000 x 10,680 with 16 columns, 4.87 ms with 32; this one 2.15 and 3.39 ms
// (64 columns: two calls, 6.8 ms; the FP64 pipe took 114 ms), 4.0 TB/s of U at 16 columns, at 69%
// of the ALU pipe.  64 columns per launch would want two stages of 57 KB of slices beside the 128 KB of
// raw U, and twice the FP64 sums in the promotion threads' registers; not built.
//
// Data path of one block: TMA brings the raw 128 x 64 FP64 tile of U (64 KB, two stages) and the
// 64-deep stacked slices of the small operand (formed once per product by k_f64_prep_*); two
// converter sets of four warps take 32 of the 64 values each (registers, stage released at once),
// agree on the exponent through shared memory, and write 7 x 16 TMEM columns each; the MMA warp
// issues 7 MMAs per 16 values of K and group of 16 columns; two sets of four promotion warps (thread
// = MMA row) drain the levels of one group while the MMAs of the next run.
//
// TMEM: two accumulators (8 x 16 columns each) from column 0, A digits at 256 + 128 set.
#pragma once

namespace f64 {

constexpr int KB = 64;                   // values of K per block (one exponent, one promotion)
constexpr int NS = 7;                    // digits of 8 bits
constexpr int NL = 8;                    // levels kept
constexpr int NSETS = 2;                 // converter sets, KB / NSETS values each
constexpr int S_UD = 2;                  // raw U stages
constexpr int EX = 4;                    // ring of row exponents (converters -> promotion)
constexpr int NPROM = 2;                 // promotion sets of four warps
constexpr int THREADS = 32 * (3 + 4 * NSETS + 4 * NPROM);
constexpr uint32_t UBYTES_D = BM * KB * 8;
constexpr uint32_t kAcolD = 256;
// Exponents handed to level_sums: a zero block far below, one with infinities or NaN far above
// every sum of two finite ones.
constexpr int kZeroEab = -(1 << 20), kNanEab = 1 << 22;
__device__ __forceinline__ int special_exponent(int ex) {
    return ex == 0 ? kZeroEab : ex == 0x7ff ? kNanEab : ex;
}

constexpr int GC = 16;                   // columns per accumulator group
constexpr int NACC_ = 2;                 // accumulators, taken in turn by the (block, group) pairs
template <int CP> __host__ __device__ constexpr int sb() { return CP <= 16 ? 4 : 3; }
template <int CP> __host__ __device__ constexpr uint32_t bbytes() { return NS * CP * KB * 2; }

template <int CP>
struct Sm {
    unsigned char *U, *B;
    uint64_t *ufull, *uempty, *bfull, *bempty, *afull, *aempty, *done, *acce, *xfull, *efull, *drain;
    uint32_t *xch, *expo, *slot;
    __device__ explicit Sm(unsigned char* raw) {
        unsigned char* base = raw + ((1024u - (smem_u32(raw) & 1023u)) & 1023u);
        U = base;
        B = U + S_UD * UBYTES_D;
        xch = reinterpret_cast<uint32_t*>(B + sb<CP>() * bbytes<CP>());      // [2][NSETS][BM]
        expo = xch + 2 * NSETS * BM;                                        // [EX][BM]
        ufull = reinterpret_cast<uint64_t*>(expo + EX * BM);
        uempty = ufull + S_UD;
        bfull = uempty + S_UD;
        bempty = bfull + sb<CP>();
        afull = bempty + sb<CP>();
        aempty = afull + NSETS;
        done = aempty + NSETS;
        acce = done + NACC_;
        xfull = acce + NACC_;
        efull = xfull + 2;
        drain = efull + EX;
        slot = reinterpret_cast<uint32_t*>(drain + 1);
    }
    static constexpr size_t bytes() {
        return 1024 + (size_t)S_UD * UBYTES_D + (size_t)sb<CP>() * bbytes<CP>() + 4 * (2 * NSETS + EX) * BM +
               8 * (2 * S_UD + 2 * sb<CP>() + 2 * NSETS + 2 * NACC_ + 2 + EX + 1) + 16;
    }
};

struct Args {
    int64_t n, r;            // rows of U, columns of U (padded width)
    int nitems, nkb;         // work items; 64-value blocks along K of the whole contraction
    int kper;                // blocks per item (the last item of a row of items may have fewer)
    int mblocks;             // U^T V: 128-column blocks; U W: 128-row tiles
    int c;                   // columns of this call (<= ncg CP)
    const int* eb;           // exponents of the small operand (special_exponent): [block][ncg CP]
    double alpha, beta;
    const double* B; int64_t ldb;
    double* Y; int64_t ldy;  // U W: the result (null: write slices to part)
    double* part;            // slices: U^T V [(split ctot + j0 + j) r + a], U W [(split c + j) n + i]
    int ctot, j0;            // U^T V: columns of the whole group, first column of this call
    int ncg;                 // groups of CP columns of the small operand (items run over them too)
    double* C; int64_t ldc;  // U W of a trailing update: C[i ldc + col] -= the product
    int tri;                 // only for the tiles that meet the lower triangle (col <= i)
    int* err;
};

// Blocks of item `it`: [k0, k1) of the contraction (none for a tile above the diagonal of a
// trailing update), M block mb, column group cg with c columns, split index.
struct Item { int k0, k1, mb, cg, c, split; };
template <int CP>
__device__ __forceinline__ Item item_of(const Args& p, int it) {
    Item w;
    w.mb = it % p.mblocks;
    const int rest = it / p.mblocks;
    w.cg = rest % p.ncg;
    w.split = rest / p.ncg;
    w.c = min(CP, p.c - w.cg * CP);
    w.k0 = w.split * p.kper;
    w.k1 = min(p.nkb, w.k0 + p.kper);
    if (p.tri && w.mb * BM + BM <= w.cg * CP) w.k1 = w.k0;
    return w;
}

// Instruction descriptor: D FP32, A and B FP16, both K-major, M = 128.
__device__ __forceinline__ uint32_t idesc_f16(int n_) {
    return (1u << 4) | ((uint32_t)(n_ >> 3) << 17) | ((uint32_t)(BM >> 4) << 24);
}
__device__ __forceinline__ void mma_f16_ts(uint32_t d_tmem, uint32_t a_tmem, uint64_t b, uint32_t idesc, uint32_t acc) {
    asm volatile(
        "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n}\n" ::"r"(
            d_tmem),
        "r"(a_tmem), "l"(b), "r"(idesc), "r"(acc)
        : "memory");
}
// A bounded wait of a whole converged warp (false for every lane if one gave up).
__device__ __forceinline__ bool warp_wait(uint64_t* bar, uint32_t parity) {
    return __all_sync(0xffffffffu, mbar_wait(bar, parity));
}
__device__ __forceinline__ void tmem_st4(uint32_t taddr, uint32_t a, uint32_t b, uint32_t c, uint32_t d) {
    asm volatile("tcgen05.st.sync.aligned.32x32b.x4.b32 [%0], {%1, %2, %3, %4};" ::"r"(taddr), "r"(a), "r"(b), "r"(c),
                 "r"(d)
                 : "memory");
}
__device__ __forceinline__ void tmem_ld4(uint32_t taddr, uint32_t* r) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0, %1, %2, %3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(taddr));
}

// N + bias of x = (hi, lo) for the block exponent ex (biased, >= the value's own): the seven low
// bytes of the result minus 128 are the digits 6 .. 1, its bits 48 .. 56 minus 128 digit 0.
__device__ __forceinline__ uint64_t biased_int(uint32_t hi, uint32_t lo, uint32_t ex) {
    const uint32_t e = (hi >> 20) & 0x7ffu;
    const uint32_t t = min(ex - e, 63u);                 // zeros (e = 0, ex >= 64) shift out entirely
    const uint64_t m = ((uint64_t)((hi & 0xFFFFFu) | 0x100000u) << 32) | lo;
    const uint64_t v = (m << 2) >> t;
    const int64_t sg = (int64_t)(int32_t)hi >> 63;       // 0 or -1
    return (v ^ (uint64_t)sg) + (0x0080808080808080ull - (uint64_t)sg);
}
// Digit i (0 .. 6) of two values with neighbouring K as one FP16 pair.
template <int I>
__device__ __forceinline__ uint32_t digit_pair(uint64_t a, uint64_t b) {
    uint32_t w;
    if constexpr (I == 0) {
        w = (__byte_perm((uint32_t)(a >> 32), (uint32_t)(b >> 32), 0x7632) & 0x01ff01ffu) | 0x64006400u;
    } else {
        // byte 0 of the result from a, byte 2 from b
        constexpr uint32_t byte = (6 - I) & 3, sel = byte | ((4 + byte) << 8);
        w = (I <= 2) ? __byte_perm((uint32_t)(a >> 32), (uint32_t)(b >> 32), sel)
                     : __byte_perm((uint32_t)a, (uint32_t)b, sel);
        w = (w & 0x00ff00ffu) | 0x64006400u;
    }
    // 1024 + digit + 128 as FP16 integers; subtract 1152 (0x6480)
    const __half2 h = __hsub2(*reinterpret_cast<const __half2*>(&w), __half2half2(__ushort_as_half(0x6480)));
    return *reinterpret_cast<const uint32_t*>(&h);
}

// U's side: |N| of x = (hi, lo); exs = (block exponent << 21) | 0x1fffff, so that the shift
// ex - e is one subtraction and one shift (shr.u64 gives 0 from 64 on: zeros, e = 0, shift out).
__device__ __forceinline__ uint64_t magnitude_int(uint32_t hi, uint32_t lo, uint32_t exs) {
    const uint32_t t = (exs - (hi + hi)) >> 21;
    const uint32_t mh = (__funnelshift_l(lo, hi, 2) & 0x3FFFFFu) | 0x400000u;
    const uint64_t m = ((uint64_t)mh << 32) | (lo * 4u);
    uint64_t v;
    asm("shr.u64 %0, %1, %2;" : "=l"(v) : "l"(m), "r"(t));
    return v;
}
// Byte i of two magnitudes with neighbouring K as FP16 subnormals with the signs of sp.
template <int I>
__device__ __forceinline__ uint32_t byte_pair(uint64_t a, uint64_t b, uint32_t sp) {
    constexpr uint32_t byte = (6 - I) & 3, sel = byte | ((4 + byte) << 8);
    const uint32_t w = (I <= 2) ? __byte_perm((uint32_t)(a >> 32), (uint32_t)(b >> 32), sel)
                                : __byte_perm((uint32_t)a, (uint32_t)b, sel);
    return (w & 0x00ff00ffu) | sp;
}

// Exponent of a block from the largest |x| bit pattern's high word: below 2^-959 a block counts
// as zero (exponent 0): on U's side as it is (its other entries decide every sum there), while the small
// operand is scaled first.
__device__ __forceinline__ uint32_t block_exponent(uint32_t hmax) {
    const uint32_t e = hmax >> 20;
    return e < 64u ? 0u : e;
}

// Slices of the small operand: value(k, col) for K index k and column col < c, zero beyond kn and
// c, for cp columns (whole groups).  One warp per (64-deep block, column): lane l takes k = 2 l and
// 2 l + 1.  out[((col / 16 * 7 + slice) 16 + col mod 16) kpad + k], eb[block cp + col] (as level_sums
// takes it).  A block below 2^-959 is multiplied by 2^256 first, which is exact for subnormal numbers
// too, so that a column of any scale keeps its digits.
template <typename F>
__device__ __forceinline__ void prep_block(F value, int64_t kn, int c, int cp, int64_t kpad, __half* out, int* eb) {
    const int64_t wid = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    const int64_t blk = wid / cp;
    const int col = (int)(wid % cp);
    if (blk >= kpad / KB) return;
    const int64_t k = blk * KB + 2 * lane;
    double x0 = (col < c && k < kn) ? value(k, col) : 0.0;
    double x1 = (col < c && k + 1 < kn) ? value(k + 1, col) : 0.0;
    auto largest = [&]() {
        const uint32_t a = (uint32_t)__double2hiint(x0) & 0x7fffffffu, b = (uint32_t)__double2hiint(x1) & 0x7fffffffu;
        return __reduce_max_sync(0xffffffffu, max(a, b));
    };
    uint32_t ex = block_exponent(largest());
    int scale = 0;
    if (ex == 0u) {
        x0 *= 0x1p256;
        x1 *= 0x1p256;
        scale = 256;
        ex = block_exponent(largest());
    }
    if (lane == 0) eb[blk * cp + col] = special_exponent((int)ex) - scale;
    const uint32_t h0 = (uint32_t)__double2hiint(x0), h1 = (uint32_t)__double2hiint(x1);
    const uint64_t a = biased_int(h0, (uint32_t)__double2loint(x0), ex);
    const uint64_t b = biased_int(h1, (uint32_t)__double2loint(x1), ex);
    uint32_t* o = reinterpret_cast<uint32_t*>(out + (int64_t)(col / GC * NS * GC + col % GC) * kpad + k);
    const int64_t sl = (int64_t)GC * kpad / 2;
    const bool z = ex == 0u;
    o[0] = z ? 0u : digit_pair<0>(a, b);
    o[sl] = z ? 0u : digit_pair<1>(a, b);
    o[2 * sl] = z ? 0u : digit_pair<2>(a, b);
    o[3 * sl] = z ? 0u : digit_pair<3>(a, b);
    o[4 * sl] = z ? 0u : digit_pair<4>(a, b);
    o[5 * sl] = z ? 0u : digit_pair<5>(a, b);
    o[6 * sl] = z ? 0u : digit_pair<6>(a, b);
}
__global__ void __launch_bounds__(256) k_f64_prep_v(const double* __restrict__ V, int64_t ldv, int64_t n, int c, int cp,
                                                    int64_t kpad, __half* __restrict__ out, int* __restrict__ eb) {
    prep_block([&](int64_t k, int col) { return V[k + (int64_t)col * ldv]; }, n, c, cp, kpad, out, eb);
}
// W is r x ldw row-major.
__global__ void __launch_bounds__(256) k_f64_prep_w(const double* __restrict__ W, int64_t r, int64_t ldw, int c, int cp,
                                                    int64_t kpad, __half* __restrict__ out, int* __restrict__ eb) {
    prep_block([&](int64_t k, int col) { return W[k * ldw + col]; }, r, c, cp, kpad, out, eb);
}
// Column col is row col of the panel P (ldp), its entries times the signs sg.
__global__ void __launch_bounds__(256) k_f64_prep_panel(const double* __restrict__ P, int64_t ldp, int kn, int c, int cp,
                                                        const double* __restrict__ sg, __half* __restrict__ out,
                                                        int* __restrict__ eb) {
    prep_block([&](int64_t k, int col) { return sg[k] * P[(int64_t)col * ldp + k]; }, kn, c, cp, KB, out, eb);
}

// The rare results of level_sums: a 64-bit integer below 2^32 in magnitude, an exponent outside
// FP64's normal range (a subnormal number or infinity), a zero block, a block with infinities or NaN.
__device__ __noinline__ double level_sum_slow(uint64_t m, bool neg, int eab) {
    if (eab > kNanEab / 2) return __longlong_as_double(0x7ff8000000000000ll);
    if (m == 0) return 0.0;
    const int lz = __clzll((long long)m);
    const int e = eab - lz - 1012;
    if (e < -64) return 0.0;                                 // below half of 2^-1074
    const bool sub = e < 1;                                  // formed 2^128 above, then scaled down
    uint64_t bits = ((uint64_t)(uint32_t)(sub ? e + 127 : e - 1) << 52) + (((m << (lz - 1)) + 0x200u) >> 10);
    if (e > 2046) bits = 0x7ff0000000000000ull;
    const double v = __longlong_as_double((long long)(bits | (neg ? 0x8000000000000000ull : 0ull)));
    return sub ? v * 0x1p-128 : v;
}

// The values of the levels of four columns: sum_l L_l 256^(6 - l) 2^(eab - 2154 + 48), eab = ea + eb,
// in units of level 5 (2^-54 of the block's bound), each rounded to FP64 and added to acc.  The
// accumulators hold L_l 2^-24.  A unit of level l is 2^(-14 - 8 l) of the block's largest product.
// Levels 0 and 1 (below 2^22) are read off an FP32 sum with 1.5 2^23, levels 2-5 (below 2^24) are
// converted (16 conversions per clock and SM, so not all seven), and level 6, after taking in level 7,
// is read off a sum with 1.5 2^25 to a unit of 4; the sum starts at half a unit of level 5, so that the
// shift by which level 6 enters level 5 rounds.  (Without that half it cut off towards minus infinity,
// every block short by half a unit on average: an error of one sign that grew with the number of
// blocks.)  One branch for the special results of all four columns, so that their chains overlap.
__device__ __forceinline__ void level_sums(const uint32_t* L, const int* eab, double* acc) {
    constexpr float SC = 16777216.f, M1 = 12582912.f, M4 = 50331648.f + 128.f;
    constexpr uint32_t B1 = 0x4B400000u, B4 = 0x4C400000u;
    uint32_t hi[4], lo[4], sg[4];
    double out[4];
    bool special = false;
#pragma unroll
    for (int v = 0; v < 4; ++v) {
        const uint32_t l0 = __float_as_uint(fmaf(__uint_as_float(L[v]), SC, M1));
        const uint32_t l1 = __float_as_uint(fmaf(__uint_as_float(L[4 + v]), SC, M1));
        const int l2 = __float2int_rn(__uint_as_float(L[8 + v]) * SC);
        const int l3 = __float2int_rn(__uint_as_float(L[12 + v]) * SC);
        const int l4 = __float2int_rn(__uint_as_float(L[16 + v]) * SC);
        const int l5 = __float2int_rn(__uint_as_float(L[20 + v]) * SC);
        const float x6 = fmaf(__uint_as_float(L[28 + v]), 1.f / 256.f, __uint_as_float(L[24 + v]));
        const uint32_t l6 = __float_as_uint(fmaf(x6, SC, M4));
        // in units of 256 level-6 units: |T| < 2^62 (bits of l6: a quarter of level 6, plus 32)
        int64_t T = (int64_t)((int)((l6 >> 6) - (B4 >> 6)) + l5);
        T += (int64_t)l4 * 256;
        T += (int64_t)l3 * 65536;
        T += (int64_t)l2 * 16777216;
        const uint32_t th = (uint32_t)(T >> 32) + (l0 * 256u + l1 - (B1 * 256u + B1));
        sg[v] = (uint32_t)((int32_t)th >> 31);
        const uint64_t m = ((((uint64_t)th << 32) | (uint32_t)T) ^ (((uint64_t)sg[v] << 32) | sg[v])) + (sg[v] & 1u);
        hi[v] = (uint32_t)(m >> 32);
        lo[v] = (uint32_t)m;
        const int lz = __clz((int)hi[v]);
        const uint32_t e1 = (uint32_t)(eab[v] - lz - 1013);        // biased exponent of the result, minus 1
        // top bit to 62, then to 52 with rounding (a carry moves into the exponent field)
        const uint64_t q = ((m << ((lz - 1) & 63)) + 0x200u) >> 10;
        const uint32_t qh = (uint32_t)(q >> 32) + (e1 << 20);
        out[v] = __hiloint2double((int)((qh & 0x7fffffffu) | (sg[v] & 0x80000000u)), (int)(uint32_t)q);
        special |= hi[v] == 0u || e1 >= 2045u;
    }
    if (special) {
#pragma unroll
        for (int v = 0; v < 4; ++v) {
            const int lz = __clz((int)hi[v]);
            if (hi[v] == 0u || (uint32_t)(eab[v] - lz - 1013) >= 2045u)
                out[v] = level_sum_slow(((uint64_t)hi[v] << 32) | lo[v], sg[v] != 0u, eab[v]);
        }
    }
#pragma unroll
    for (int v = 0; v < 4; ++v) acc[v] += out[v];
}

// TRANS: U^T V (M = 128 columns of U, K = rows); otherwise U W (M = 128 rows, K = columns).
template <int CP, bool TRANS>
__global__ void __launch_bounds__(THREADS, 1)
    k_tc_f64(const __grid_constant__ CUtensorMap mU, const __grid_constant__ CUtensorMap mB, const Args p) {
    extern __shared__ unsigned char raw_f64[];
    Sm<CP> sm(raw_f64);
    constexpr int NG = CP / GC, SB_ = sb<CP>();
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (threadIdx.x == 0) {
        for (int s = 0; s < S_UD; ++s) { mbar_init(&sm.ufull[s], 1); mbar_init(&sm.uempty[s], 4 * NSETS); }
        for (int s = 0; s < SB_; ++s) { mbar_init(&sm.bfull[s], 1); mbar_init(&sm.bempty[s], 1); }
        for (int s = 0; s < NSETS; ++s) { mbar_init(&sm.afull[s], 4); mbar_init(&sm.aempty[s], 1); }
        for (int s = 0; s < NACC_; ++s) { mbar_init(&sm.done[s], 1); mbar_init(&sm.acce[s], 4 * NPROM / NG); }
        for (int s = 0; s < 2; ++s) mbar_init(&sm.xfull[s], 4 * NSETS);
        for (int s = 0; s < EX; ++s) mbar_init(&sm.efull[s], 4);
        mbar_init(sm.drain, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(sm.slot)),
                     "r"(kTmemCols));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *sm.slot;
    bool ok = true;

    if (warp == 0) {
        if (lane == 0) {                                 // raw U tiles
            uint32_t g = 0;
            for (int it = blockIdx.x; it < p.nitems && ok; it += gridDim.x) {
                const Item w = item_of<CP>(p, it);
                for (int kb = w.k0; kb < w.k1; ++kb, ++g) {
                    const uint32_t s = g % S_UD;
                    if (!mbar_wait(&sm.uempty[s], ((g / S_UD) & 1) ^ 1)) { ok = false; break; }
                    mbar_expect_tx(&sm.ufull[s], UBYTES_D);
                    unsigned char* dst = sm.U + s * UBYTES_D;
                    if constexpr (TRANS) {
                        tma_load_2d(dst, &mU, w.mb * BM, kb * KB, &sm.ufull[s]);
                    } else {
#pragma unroll
                        for (int q = 0; q < 4; ++q)
                            tma_load_2d(dst + q * (UBYTES_D / 4), &mU, kb * KB + 16 * q, w.mb * BM, &sm.ufull[s]);
                    }
                }
            }
            if (!producer_drain(sm.ufull, S_UD, g)) ok = false;
            if (!ok) atomicExch(p.err, 1);
        }
    } else if (warp == 2) {
        if (lane == 0) {                                 // stacked slices of the small operand
            uint32_t g = 0;
            for (int it = blockIdx.x; it < p.nitems && ok; it += gridDim.x) {
                const Item w = item_of<CP>(p, it);
                for (int kb = w.k0; kb < w.k1; ++kb, ++g) {
                    const uint32_t s = g % SB_;
                    if (!mbar_wait(&sm.bempty[s], ((g / SB_) & 1) ^ 1)) { ok = false; break; }
                    mbar_expect_tx(&sm.bfull[s], bbytes<CP>());
                    tma_load_2d(sm.B + s * bbytes<CP>(), &mB, kb * KB, w.cg * (NS * CP), &sm.bfull[s]);
                }
            }
            if (!producer_drain(sm.bfull, SB_, g)) ok = false;
            if (!ok) atomicExch(p.err, 1);
        }
    } else if (warp == 1) {                              // MMA issue (converged warp)
        uint32_t g = 0, u = 0;                           // blocks, (block, group) pairs
        for (int it = blockIdx.x; it < p.nitems && ok; it += gridDim.x) {
            const Item w = item_of<CP>(p, it);
            for (int kb = w.k0; kb < w.k1 && ok; ++kb, ++g) {
                const uint32_t s = g % SB_;
#pragma unroll
                for (int grp = 0; grp < NG; ++grp, ++u) {
                    const uint32_t acc = u % NACC_, d = tmem + acc * (NL * GC);
                    const uint64_t b0 = sw128_desc(sm.B + s * bbytes<CP>() + grp * bbytes<GC>());
                    const uint32_t wa = lane == 0 ? smem_u32(&sm.acce[acc]) : smem_u32(&sm.bfull[s]);
                    const uint32_t wp = lane == 0 ? ((u / NACC_) & 1) ^ 1 : (g / SB_) & 1;
                    if (!mbar_wait_lanes(wa, wp)) { ok = false; break; }
#pragma unroll
                    for (int h = 0; h < NSETS; ++h) {
                        if (grp == 0 && !warp_wait(&sm.afull[h], g & 1)) { ok = false; break; }
                        tc_fence_after();
                        if (elect_one()) {
#pragma unroll
                            for (int kk = 0; kk < 2; ++kk) {
                                const uint64_t db = b0 + (uint64_t)(((2 * h + kk) * 32) >> 4);
                                const uint32_t a = tmem + kAcolD + 128 * h + 8 * kk;
                                if (h + kk == 0) {
                                    // the first MMAs of a block clear level 0, then levels 1 .. 7
                                    mma_f16_ts(d, a, db, idesc_f16(GC), 0u);
                                    mma_f16_ts(d + GC, a + 16, db, idesc_f16(NS * GC), 0u);
                                    mma_f16_ts(d + GC, a, db + ((GC * KB * 2) >> 4), idesc_f16((NS - 1) * GC), 1u);
                                } else {
                                    mma_f16_ts(d, a, db, idesc_f16(NS * GC), 1u);
                                    mma_f16_ts(d + GC, a + 16, db, idesc_f16(NS * GC), 1u);
                                }
#pragma unroll
                                for (int i = 2; i < NS; ++i)
                                    mma_f16_ts(d + i * GC, a + 16 * i, db, idesc_f16((NL - i) * GC), 1u);
                            }
                            if (grp == NG - 1) mma_commit(&sm.aempty[h]);
                            if (h == NSETS - 1) {
                                if (grp == NG - 1) mma_commit(&sm.bempty[s]);
                                mma_commit(&sm.done[acc]);
                            }
                        }
                        __syncwarp();
                    }
                    if (!ok) break;
                }
            }
        }
        if (elect_one()) mma_commit(sm.drain);
        __syncwarp();
        if (!mbar_wait_for(sm.drain, 0, kDrainCycles)) ok = false;
        if (!ok && lane == 0) atomicExch(p.err, 1);
    } else if (warp < 3 + 4 * NSETS) {
        // converters: set h takes values 32 h .. 32 h + 31 of the block; a warp works on the TMEM
        // lanes 32 (warp mod 4), thread = MMA row m
        const int h = (warp - 3) >> 2, q = warp & 3, m = 32 * q + lane;
        const uint32_t ta = tmem + ((uint32_t)(32 * q) << 16) + kAcolD + 128 * h;
        uint32_t g = 0;
        for (int it = blockIdx.x; it < p.nitems && ok; it += gridDim.x) {
            const Item w = item_of<CP>(p, it);
            for (int kb = w.k0; kb < w.k1; ++kb, ++g) {
                const uint32_t s = g % S_UD;
                if (!warp_wait(&sm.ufull[s], (g / S_UD) & 1)) { ok = false; break; }
                const unsigned char* st = sm.U + s * UBYTES_D;
                uint32_t hi[32], lo[32];
                if constexpr (TRANS) {                   // [64 rows][128 columns]: lanes side by side
                    const double* R = reinterpret_cast<const double*>(st) + (32 * h) * BM + m;
#pragma unroll
                    for (int k = 0; k < 32; ++k) {
                        const uint2 v = *reinterpret_cast<const uint2*>(R + k * BM);
                        lo[k] = v.x;
                        hi[k] = v.y;
                    }
                } else {                                 // four [128 rows][16 values] boxes, SW128
                    const unsigned char* R = st + (2 * h) * (UBYTES_D / 4) + m * 128;
#pragma unroll
                    for (int j = 0; j < 16; ++j) {
                        const uint4 v = *reinterpret_cast<const uint4*>(R + (j >> 3) * (UBYTES_D / 4) +
                                                                        (((j & 7) ^ (m & 7)) << 4));
                        lo[2 * j] = v.x; hi[2 * j] = v.y;
                        lo[2 * j + 1] = v.z; hi[2 * j + 1] = v.w;
                    }
                }
                uint32_t hm = 0;                         // largest |x|, high word times 2
#pragma unroll
                for (int k = 0; k < 32; ++k) hm = max(hm, hi[k] + hi[k]);
                uint32_t* X = sm.xch + (g & 1) * (NSETS * BM);
                X[h * BM + m] = hm;
                __syncwarp();
                if (lane == 0) { mbar_arrive(&sm.uempty[s]); mbar_arrive(&sm.xfull[g & 1]); }
                if (!warp_wait(&sm.xfull[g & 1], (g >> 1) & 1)) { ok = false; break; }
                const uint32_t ex = block_exponent(max(hm, X[(h ^ 1) * BM + m]) >> 1);
                const uint32_t exs = (ex << 21) | 0x1fffffu;
                if (h == 0) {
                    sm.expo[(g % EX) * BM + m] = ex;
                    __syncwarp();
                    if (lane == 0) mbar_arrive(&sm.efull[g % EX]);
                }
                if (!warp_wait(&sm.aempty[h], (g & 1) ^ 1)) { ok = false; break; }
                tc_fence_after();
#pragma unroll
                for (int k = 0; k < 32; k += 8) {
                    uint64_t N[8];
                    uint32_t sp[4];
#pragma unroll
                    for (int u = 0; u < 8; ++u) N[u] = magnitude_int(hi[k + u], lo[k + u], exs);
#pragma unroll
                    for (int u = 0; u < 4; ++u)
                        sp[u] = __byte_perm(hi[k + 2 * u], hi[k + 2 * u + 1], 0x7030) & 0x80008000u;
                    const uint32_t t = ta + (k >> 1);
#define HDF_DIG(I)                                                                                      \
    tmem_st4(t + 16 * I, byte_pair<I>(N[0], N[1], sp[0]), byte_pair<I>(N[2], N[3], sp[1]),              \
             byte_pair<I>(N[4], N[5], sp[2]), byte_pair<I>(N[6], N[7], sp[3]));
                    HDF_DIG(0) HDF_DIG(1) HDF_DIG(2) HDF_DIG(3) HDF_DIG(4) HDF_DIG(5) HDF_DIG(6)
#undef HDF_DIG
                }
                tmem_st_wait();
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(&sm.afull[h]);
            }
        }
        if (!ok && lane == 0) atomicExch(p.err, 1);
    } else {
        // promotion: thread = MMA row, FP64 register sums.  With two groups each set of four warps
        // drains one (its accumulator is the group's); with one, each set takes half its columns
        constexpr int PC = CP / NPROM;                   // columns per thread
        const int set = (warp - 3 - 4 * NSETS) >> 2, q = warp & 3, m = 32 * q + lane;
        const int colg = NG == 1 ? PC * set : 0;         // first column within the group
        const int col0 = PC * set;                       // first column of the call
        const uint32_t tl = tmem + ((uint32_t)(32 * q) << 16) + colg;
        uint32_t g = 0;
        for (int it = blockIdx.x; it < p.nitems && ok; it += gridDim.x) {
            const Item w = item_of<CP>(p, it);
            double acc[PC];
#pragma unroll
            for (int j = 0; j < PC; ++j) acc[j] = 0.0;
            for (int kb = w.k0; kb < w.k1; ++kb, ++g) {
                const int eb = lane < PC ? p.eb[((int64_t)kb * p.ncg + w.cg) * CP + col0 + lane] : kZeroEab;
                if (!warp_wait(&sm.efull[g % EX], (g / EX) & 1)) { ok = false; break; }
                const int ea = special_exponent((int)sm.expo[(g % EX) * BM + m]);
                const uint32_t u = NG == 1 ? g : NG * g + set, b = u % NACC_;
                if (!warp_wait(&sm.done[b], (u / NACC_) & 1)) { ok = false; break; }
                tc_fence_after();
                const uint32_t td = tl + b * (NL * GC);
                auto four = [&](int c0) {
                    uint32_t L[NL * 4];
                    int eab[4];
#pragma unroll
                    for (int l = 0; l < NL; ++l) tmem_ld4(td + l * GC + c0, L + 4 * l);
#pragma unroll
                    for (int v = 0; v < 4; ++v) eab[v] = ea + __shfl_sync(0xffffffffu, eb, c0 + v);
                    tmem_ld_wait();
                    level_sums(L, eab, acc + c0);
                };
                if (col0 + PC <= w.c) {                  // straight-line: the four-column chains overlap
#pragma unroll
                    for (int c0 = 0; c0 < PC; c0 += 4) four(c0);
                } else {                                 // without the padding columns
#pragma unroll
                    for (int c0 = 0; c0 < PC; c0 += 4)
                        if (col0 + c0 < w.c) four(c0);
                }
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(&sm.acce[b]);
            }
            if (!ok) break;
            if constexpr (TRANS) {
                const int64_t a = (int64_t)w.mb * BM + m;
                if (a < p.r) {
#pragma unroll
                    for (int j = 0; j < PC; ++j)
                        if (col0 + j < w.c)
                            p.part[((int64_t)w.split * p.ctot + p.j0 + col0 + j) * p.r + a] = acc[j];
                }
            } else {
                const int64_t i = (int64_t)w.mb * BM + m;
                if (i < p.n && w.k0 < w.k1) {
#pragma unroll
                    for (int j = 0; j < PC; ++j) {
                        const int64_t col = col0 + j;
                        if (col < w.c) {
                            if (p.C) {
                                p.C[i * p.ldc + w.cg * CP + col] -= acc[j];
                            } else if (p.part) {
                                p.part[((int64_t)w.split * p.c + col) * p.n + i] = acc[j];
                            } else {
                                double out = p.alpha * acc[j];
                                if (p.B) out += p.beta * p.B[i + col * p.ldb];
                                p.Y[i + col * p.ldy] = out;
                            }
                        }
                    }
                }
            }
        }
        if (!ok && lane == 0) atomicExch(p.err, 1);
    }
    cta_teardown<16>(tmem, warp);
}

// Y = alpha (sum of the slices, in order) + beta B for a U W split along the columns of U.
__global__ void __launch_bounds__(256) k_f64_uw_finish(const double* __restrict__ part, int nsplit, int64_t n, int c,
                                                       double alpha, const double* __restrict__ B, int64_t ldb,
                                                       double beta, double* __restrict__ Y, int64_t ldy) {
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    const int j = blockIdx.y;
    if (i >= n) return;
    double s = 0.0;
    for (int k = 0; k < nsplit; ++k) s += part[((int64_t)k * c + j) * n + i];
    double out = alpha * s;
    if (B) out += beta * B[i + (int64_t)j * ldb];
    Y[i + (int64_t)j * ldy] = out;
}

// Split of nkb blocks of K over `mblocks` tiles: the blocks per item that minimise the longest
// CTA, rounds x (blocks per item + 6) with 6 blocks for filling the pipeline and writing the
// result, at most max_split splits.
inline void choose_split(int64_t mblocks, int64_t nkb, int64_t sms, int64_t max_split, int* kper, int* nsplit) {
    int64_t best = INT64_MAX;
    *kper = (int)nkb;
    *nsplit = 1;
    for (int64_t s = 1; s <= std::min<int64_t>(max_split, nkb); ++s) {
        const int64_t kp = (nkb + s - 1) / s, ns = (nkb + kp - 1) / kp;
        const int64_t cost = ((mblocks * ns + sms - 1) / sms) * (kp + 6);
        if (cost < best) { best = cost; *kper = (int)kp; *nsplit = (int)ns; }
    }
}

}  // namespace f64
