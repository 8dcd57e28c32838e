// k_attitude.cu -- the A block (Sect. 5.2): per-knot-interval partial normals from the
// time-ordered observations, assembly of the banded normals of each overlapping segment,
// and the segmented robust banded Cholesky (App. C restricted to the envelope).
#include <cuda_fp16.h>

#include "agis_internal.cuh"

namespace agis {

// linear index of the upper entry (i <= j) of a 16x16 symmetric matrix
__host__ __device__ constexpr int tri16(int i, int j) { return i * 16 - i * (i - 1) / 2 + (j - i); }
// 4x4 symmetric upper storage
__host__ __device__ constexpr int tri4(int i, int j) { return i * 4 - i * (i - 1) / 2 + (j - i); }

constexpr int kStage = 28;  // staged per observation: B[4], M[10], r[4], BB[10]
constexpr int kAccFP64 = 116;  // distinct products: BB[p] M[m] (10 x 10) and B[b] r[c] (4 x 4)

// One warp per knot interval l (left index), iv = l - 3.  For each observation
// dR/da = B (x) g and dD/da = -2 B (x) s (Eqs. dfadq, dDldan), so its contribution to the
// 16x16 block of the interval is W (B B') (x) (g g' + 4 lambda^2 s s') (Eq. normAmod) and
// to the right-hand side -W B (x) (R g [- 2 lambda^2 D s]).  The 136 upper entries of the
// block hold only 100 distinct products (the 10 upper entries of B B' times those of the
// symmetric 4x4 M), so the lanes accumulate those 100 and the 16 right-hand-side products
// (4 per lane) and expand them into the 152 outputs at the end.  W is the weight of the
// source update, or w_att[o] (Eqs. W, wl) when the excess attitude noise is estimated.
// accumulator of every block output
__device__ __forceinline__ void block_table(int16_t* src_tab) {
    for (int o = threadIdx.x; o < kBlkVals; o += blockDim.x) {
        int v;
        if (o < 136) {
            int i = 0;
            while (o >= tri16(i, 15) + 1) i++;
            const int jj = i + (o - tri16(i, i));
            const int bi = i >> 2, ci = i & 3, bj = jj >> 2, cj = jj & 3;
            v = tri4(bi, bj) * 10 + (ci <= cj ? tri4(ci, cj) : tri4(cj, ci));
        } else {
            v = 100 + (o - 136);
        }
        src_tab[o] = (int16_t)v;
    }
}

// one interval's products of every observation, by one warp, into red[kAccFP64]
__device__ __forceinline__ void interval_direct(const DevGeo& G, double lambda2, int rhs_norm,
                                                const uint32_t* __restrict__ perm_t, int64_t beg, int64_t end,
                                                const ObsRec* __restrict__ rec, const double* __restrict__ w_att,
                                                const double* __restrict__ att, int l, int lane, double* stg,
                                                double* red) {
    // this lane's accumulators s = lane + 32 k (k < 3: BB[p] M[m]; k = 3: lanes 0-3 BB M,
    // lanes 4-19 B[b] r[c] of the right-hand side, lanes 20-31 none): the staged factors
    int fa[4], fb[4];
#pragma unroll
    for (int k = 0; k < 4; k++) {
        const int sidx = lane + 32 * k;
        fa[k] = sidx < 100 ? 18 + sidx / 10 : (sidx < kAccFP64 ? (sidx - 100) >> 2 : 0);
        fb[k] = sidx < 100 ? 4 + sidx % 10 : 14 + ((sidx - 100) & 3);
    }
    const bool k3 = lane < 20;              // accumulator 3 in use
    const bool k3_rhs = lane >= 4 && k3;    // ... and it is a right-hand-side product
    double a[16];
#pragma unroll
    for (int k = 0; k < 16; k++) a[k] = att[4 * (int64_t)(l - 3) + k];
    double acc[4] = {0, 0, 0, 0};
    for (int64_t base = beg; base < end; base += kWarp) {
        const int64_t j = base + lane;
        double* st = stg + lane * kStage;
        if (j < end) {
            const uint32_t o = perm_t[j];
            const ObsRec r = rec[o];
            double B[4];
            bspline4(G, r.t_ns, l, B);
            double s[4];
#pragma unroll
            for (int c = 0; c < 4; c++) s[c] = B[0] * a[c] + B[1] * a[4 + c] + B[2] * a[8 + c] + B[3] * a[12 + c];
            const double W = w_att ? w_att[o] : r.W;
            const double l4 = 4.0 * lambda2;
#pragma unroll
            for (int c = 0; c < 4; c++) {
#pragma unroll
                for (int e = c; e < 4; e++) st[4 + tri4(c, e)] = W * (r.g[c] * r.g[e] + l4 * s[c] * s[e]);
            }
            double D = 1.0 - (s[0] * s[0] + s[1] * s[1] + s[2] * s[2] + s[3] * s[3]);
#pragma unroll
            for (int c = 0; c < 4; c++) {
                double v = r.R * r.g[c];
                if (rhs_norm) v -= 2.0 * lambda2 * D * s[c];
                st[14 + c] = W * v;
                st[c] = B[c];
            }
#pragma unroll
            for (int c = 0; c < 4; c++) {
#pragma unroll
                for (int e = c; e < 4; e++) st[18 + tri4(c, e)] = B[c] * B[e];
            }
        } else {
#pragma unroll
            for (int c = 0; c < kStage; c++) st[c] = 0.0;
        }
        __syncwarp();
        const int cnt = (int)((end - base) < kWarp ? (end - base) : kWarp);
        for (int q = 0; q < cnt; q++) {
            const double* sq = stg + q * kStage;
#pragma unroll
            for (int k = 0; k < 3; k++) acc[k] += sq[fa[k]] * sq[fb[k]];
            if (k3) acc[3] += sq[fa[3]] * sq[fb[3]];
        }
        __syncwarp();
    }
#pragma unroll
    for (int k = 0; k < 3; k++) red[lane + 32 * k] = acc[k];
    if (k3) red[lane + 96] = k3_rhs ? -acc[3] : acc[3];
    __syncwarp();
}

// One warp per interval, two FP64 factors from shared memory per product.
__global__ void __launch_bounds__(128) k_att_accum(DevGeo G, double lambda2, int rhs_norm,
                                                   const uint32_t* __restrict__ perm_t,
                                                   const int64_t* __restrict__ ivl_off, int n_iv,
                                                   const ObsRec* __restrict__ rec,
                                                   const double* __restrict__ w_att,
                                                   const double* __restrict__ att, double* __restrict__ blk) {
    __shared__ double stage_all[4][kWarp * kStage];
    __shared__ double red_all[4][kAccFP64];
    __shared__ int16_t src_tab[kBlkVals];
    const int lane = threadIdx.x & 31;
    const int wib = threadIdx.x >> 5;
    double* red = red_all[wib];
    block_table(src_tab);
    __syncthreads();
    const int nwarps = gridDim.x * (blockDim.x >> 5);
    for (int iv = blockIdx.x * (blockDim.x >> 5) + wib; iv < n_iv; iv += nwarps) {
        interval_direct(G, lambda2, rhs_norm, perm_t, ivl_off[iv], ivl_off[iv + 1], rec, w_att, att, iv + 3, lane,
                        stage_all[wib], red);
#pragma unroll
        for (int k = 0; k < 5; k++) {
            const int o = lane + 32 * k;
            if (o < kBlkVals) blk[(int64_t)iv * kBlkVals + o] = red[src_tab[o]];
        }
        __syncwarp();
    }
}

// ---------------------------------------------------------------------------------------
// Interval blocks by moments on the tensor cores.  In a regular knot interval the B-splines are
// cubic forms in u = (t - tau_l) / dt and v = 1 - u with coefficients c >= 0, so the block is
//   sum W BB[p] g g' = sum_k c[p][k] sum_o (W g g')_o (u^k v^(6-k))_o,   k = 0 .. 6,
// the right-hand side likewise with W R g (the cubics raised to degree 6), and the norm term, a
// form with the interval's coefficients alone, needs sum_o W u^k v^(12-k), k = 0 .. 12.  Rows
// W g g' (10), W R g (4), W v^6 and W u^6 by columns u^k v^(6-k): one 16 x 7 contraction over the
// interval's observations, and an expansion without cancellation.  Root mean square error of an entry
// relative to its place, against the products' sums: 0.54 of theirs with 24 observations in the interval, 0.36 with
// 54, 0.25 with 156 (the worst entry 0.81, 0.62, 0.44).
//
// It runs on mma.sync (a 128-row tcgen05 tile would hold one interval of 16 rows): every row value is
// a 62-bit and every column value a 61-bit fraction of its largest magnitude in the interval, cut into
// nine signed 7-bit digits kept as FP16 integers, and the products of the digit pairs i + j >= 7 are
// accumulated in FP32 by their weight 2^(7 (i + j)): 9 pairs x 448 observations x 2^12 are
// below 2^24, so every sum is exact, and the pairs left out are about 2^-69 of the largest term
// (FP64 rounds each product at 2^-53).  Products W g g', the forms and conversions are 64-bit
// integer arithmetic.
// Bound, by reading: integer and shared-memory issue (FP64 pipe 31% busy), and 68 FP64 instructions per
// interval for the expansion, where the FP64 form takes 116 FMAs and
// about 95 more FP64 instructions per observation (2 per clock and SM).
// Attitude update, the products' sums against this: 24.7M observations in 157,786 intervals 11.6 -> 5.3 ms, 7.1M in
// 131,490 4.62 -> 3.81 (a fifth of these intervals of 54 takes the products), 14M in 131,490 7.3 -> 4.4.
// Intervals next to the multiple end knots (two at each end), short ones, those that the
// observations do not cover and those with a sum far below its digits' scale sum the products one by one.
constexpr int kMomWarps = 4;
constexpr int kMomStride = 40;    // 64-bit values per row of the staged chunk (rows 64 B apart mod 128 B)
constexpr int kMomFlush = 448;    // observations per exact accumulation
constexpr int kMomMin = 24;       // shorter intervals: the sums of the products themselves
constexpr uint64_t kDigitBias = 0x4081020408102040ull;   // 64 in each of nine 7-bit digits

struct MomScale {                  // u with 63 fractional bits: 2^shift (t - tau) inv 2^-64, times 2
    uint64_t inv;
    int32_t shift;
    int32_t tshift;                // t - tau in 30 bits, and its unit in u
    float tinv;
};

// v 2^(62 - E) for |v| < 2^E, truncated
__device__ __forceinline__ long long to_fixed(double v, int E) {
    const uint32_t hi = (uint32_t)__double2hiint(v);
    const int sh = (int)((hi >> 20) & 0x7ffu) - 1023 + 10 - E;   // at most 9
    unsigned long long m = ((unsigned long long)((hi & 0xfffffu) | 0x100000u) << 32) | (uint32_t)__double2loint(v);
    m = sh >= 0 ? m << sh : (sh > -64 ? m >> -sh : 0ull);
    return (hi >> 31) ? -(long long)m : (long long)m;
}
// products of 62-bit fractions and of unsigned 63-bit ones, what is cut off at half its range
__device__ __forceinline__ long long mulq(long long a, long long b) { return (long long)((unsigned long long)__mul64hi(a, b) << 2) | 2; }
__device__ __forceinline__ uint64_t mulu(uint64_t a, uint64_t b) { return (__umul64hi(a, b) << 1) | 1; }
__device__ __forceinline__ long long shifted(uint64_t x, int n) { return (long long)(n >= 0 ? x << n : x >> -n); }
__device__ __forceinline__ double pow2(int n) { return __longlong_as_double((long long)(1023 + n) << 52); }

// fixed-point value -> its digits' bit fields; |q| <= 0.992 2^62
__device__ __forceinline__ uint2 digit_bits(long long q) {
    const uint64_t u = (uint64_t)q + kDigitBias;
    return make_uint2((uint32_t)u, (uint32_t)(u >> 32));
}
// the nine digits of a value of two observations (low and high words of each), as FP16 pairs
__device__ __forceinline__ uint32_t digit_half(uint32_t w) {   // digits in bits 0-6 and 16-22
    const uint32_t h = (w & 0x007f007fu) | 0x64006400u;        // 1024 + digit + 64
    const __half2 off = __halves2half2(__ushort_as_half(0xe440), __ushort_as_half(0xe440));   // -1088
    const __half2 r = __hadd2(*reinterpret_cast<const __half2*>(&h), off);
    return *reinterpret_cast<const uint32_t*>(&r);
}
__device__ __forceinline__ void digits4(uint32_t a, uint32_t b, uint32_t out[4]) {   // of bits 0 .. 27
    const uint32_t c0 = __byte_perm(a, b, 0x5410), c1 = __byte_perm(a >> 14, b >> 14, 0x5410);
    out[0] = digit_half(c0);
    out[1] = digit_half(c0 >> 7);
    out[2] = digit_half(c1);
    out[3] = digit_half(c1 >> 7);
}
__device__ __forceinline__ void digits9(const uint4 v, uint32_t out[9]) {
    digits4(v.x, v.z, out);
    digits4(__funnelshift_l(v.x, v.y, 4), __funnelshift_l(v.z, v.w, 4), out + 4);
    out[8] = digit_half(__byte_perm(v.y >> 24, v.w >> 24, 0x5410));
}
__device__ __forceinline__ void mma_f16(float c[4], const uint32_t a[4], uint32_t b0, uint32_t b1) {
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};\n"
        : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// the four B-splines' coefficients (over 6) of u^k v^(3-k), and the columns' scales 2^n at any u
__device__ constexpr int kSplineNum[4][4] = {{1, 0, 0, 0}, {4, 12, 6, 1}, {1, 6, 12, 4}, {0, 0, 0, 1}};
__device__ constexpr int kColShift[7] = {0, 3, 5, 5, 5, 3, 0};
// components c <= e of row tri4(c, e) of W g g'
__device__ __forceinline__ int row_first(int row) { return row < 4 ? 0 : row < 7 ? 1 : row < 9 ? 2 : 3; }
__device__ __forceinline__ int row_second(int row) { return row < 4 ? row : row < 7 ? row - 3 : row < 9 ? row - 5 : 3; }

// One interval's products from its moments, by one warp, into red[kAccFP64].  False (nothing written)
// if a sum on the diagonal is small beside the scale of its digits.
//
// Every row and column has a scale of its own (W, W R and each component of g by their largest
// values).  An observation's term is off by about 2^-63 of the row's largest value times the column's (two
// products cut at 2^-62), by 2^amp of that for a column that is shifted up by amp bits more than over a
// whole interval, and the sum by sqrt(n) of it.  The products' sums are off by 0.17 2^-52 sqrt(n) of a sum on the
// diagonal, and by about 0.28 2^-52 of its place in the matrix (the root of its two diagonal sums) where signs
// differ.  A diagonal sum of at least 2^(amp - 9) sqrt(n) of its two scales' product keeps the digits
// below 0.25 2^-52 of either; a smaller one (large weights that meet small components or lie at the other end
// of the interval) sends the interval to the products' sums.
__device__ __forceinline__ bool interval_moments(const DevGeo& G, MomScale ms, double lambda2,
                                                 const uint32_t* __restrict__ perm_t, int64_t beg, int64_t end, int iv,
                                                 const ObsRec* __restrict__ rec, const double* __restrict__ w_att,
                                                 const double* __restrict__ att, int EW, int ER, const int (&Eg)[4], float lu,
                                                 float lv, int lane, uint2* st, const double (*cbb)[8], const double (*cb)[8], double* wk,
                                                 double* red) {
    const int g = lane >> 2, q = lane & 3;
    const double l4 = 4.0 * lambda2;
    // every column to its largest value in the interval: u^k v^(6-k) 2^sh[k] < 1.  They are formed from
    // ua = u 2^a, vb = v 2^b and 4 u v, with cs[k] bits up to 61 fractional ones
    int sh[7], cs[7];
    const int a = (int)lu > 0, b = (int)lv > 0;
#pragma unroll
    for (int k = 0; k < 7; k++) {
        sh[k] = max(kColShift[k], (int)floorf((float)k * lu + (float)(6 - k) * lv - 1e-4f));
        const int m = k < 6 - k ? k : 6 - k;   // (4 u v)^m
        cs[k] = sh[k] - 2 - 2 * m - (k > 3 ? (2 * k - 6) * a : (6 - 2 * k) * b);
    }
    // moments of this lane: rows g and g + 8, columns 2 q and 2 q + 1
    double mom[4] = {0, 0, 0, 0};
    auto eg = [&](int c) { return c == 0 ? Eg[0] : c == 1 ? Eg[1] : c == 2 ? Eg[2] : Eg[3]; };
    auto unit = [&](int e) {   // power of two of mom[e]'s scale
        const int row = g + 8 * (e >> 1);
        const int ce = e & 1 ? (q == 0 ? sh[1] : q == 1 ? sh[3] : sh[5]) : (q == 0 ? sh[0] : q == 1 ? sh[2] : q == 2 ? sh[4] : sh[6]);
        return (row < 10 ? EW + eg(row_first(row)) + eg(row_second(row)) : (row < 14 ? ER + eg(row - 10) : EW)) - ce;
    };
    const int64_t tau = G.knot0_ns + (int64_t)iv * G.knot_dt_ns;
    for (int64_t f0 = beg; f0 < end; f0 += kMomFlush) {
        float acc[10][4];
#pragma unroll
        for (int s = 0; s < 10; s++)
#pragma unroll
            for (int e = 0; e < 4; e++) acc[s][e] = 0.0f;
        const int64_t f1 = end < f0 + kMomFlush ? end : f0 + kMomFlush;
        for (int64_t base = f0; base < f1; base += kWarp) {
            const int64_t j = base + lane;
            long long X[16], C[7];
            if (j < f1) {
                const uint32_t o = perm_t[j];
                const ObsRec& r = rec[o];
                const double W = w_att ? w_att[o] : r.W;
                const uint64_t u = __umul64hi((uint64_t)(r.t_ns - tau) << ms.shift, ms.inv) << 1, v = (1ull << 63) - u;
                const uint64_t ua = u << a, vb = v << b, p = mulu(ua, vb) << (2 - a - b), p2 = mulu(p, p);
                const uint64_t u2 = mulu(ua, ua), v2 = mulu(vb, vb), u4 = mulu(u2, u2), v4 = mulu(v2, v2);
                const uint64_t u6 = mulu(u4, u2), v6 = mulu(v4, v2);
                const long long Wq = to_fixed(W, EW), WR = to_fixed(W * r.R, ER);
                long long gq[4];
#pragma unroll
                for (int c = 0; c < 4; c++) gq[c] = to_fixed(r.g[c], Eg[c]);
#pragma unroll
                for (int c = 0; c < 4; c++) {
                    const long long Wg = mulq(Wq, gq[c]);
#pragma unroll
                    for (int e = c; e < 4; e++) X[tri4(c, e)] = mulq(Wg, gq[e]);
                    X[10 + c] = WR ? mulq(WR, gq[c]) : 0;   // zero residuals give zero sums
                }
                X[14] = mulq(Wq, (long long)(v6 >> (6 * b + 1)));
                X[15] = mulq(Wq, (long long)(u6 >> (6 * a + 1)));
                C[0] = shifted(v6, cs[0]);
                C[1] = shifted(mulu(p, v4), cs[1]);
                C[2] = shifted(mulu(p2, v2), cs[2]);
                C[3] = shifted(mulu(p2, p), cs[3]);
                C[4] = shifted(mulu(p2, u2), cs[4]);
                C[5] = shifted(mulu(p, u4), cs[5]);
                C[6] = shifted(u6, cs[6]);
            } else {
#pragma unroll
                for (int k = 0; k < 16; k++) X[k] = 0;
#pragma unroll
                for (int k = 0; k < 7; k++) C[k] = 0;
            }
            __syncwarp();
#pragma unroll
            for (int k = 0; k < 16; k++) st[k * kMomStride + lane] = digit_bits(X[k]);
#pragma unroll
            for (int k = 0; k < 7; k++) st[(16 + k) * kMomStride + lane] = digit_bits(C[k]);
            st[23 * kMomStride + lane] = digit_bits(0);
            __syncwarp();
#pragma unroll
            for (int h = 0; h < 2; h++) {
                const int k0 = 16 * h + 2 * q;
                uint32_t A[9][4], Bd[9][2];
#pragma unroll
                for (int e = 0; e < 4; e++) {   // rows g, g + 8 at k0; then at k0 + 8
                    uint32_t d[9];
                    digits9(*reinterpret_cast<const uint4*>(&st[(g + 8 * (e & 1)) * kMomStride + k0 + 8 * (e >> 1)]), d);
#pragma unroll
                    for (int t = 0; t < 9; t++) A[t][e] = d[t];
                }
#pragma unroll
                for (int e = 0; e < 2; e++) {
                    uint32_t d[9];
                    digits9(*reinterpret_cast<const uint4*>(&st[(16 + g) * kMomStride + k0 + 8 * e]), d);
#pragma unroll
                    for (int t = 0; t < 9; t++) Bd[t][e] = d[t];
                }
#pragma unroll
                for (int i = 0; i < 9; i++)
#pragma unroll
                    for (int jd = 0; jd < 9; jd++)
                        if (i + jd >= 7) mma_f16(acc[i + jd - 7], A[i], Bd[jd][0], Bd[jd][1]);
            }
        }
        // the exact sums by weight: H 2^84 + L 2^49, in units of 2^-123 of the scales
#pragma unroll
        for (int e = 0; e < 4; e++) {
            long long H = 0, L = 0;
#pragma unroll
            for (int s = 9; s >= 5; s--) H = (H << 7) + (long long)__float2int_rn(acc[s][e]);
#pragma unroll
            for (int s = 4; s >= 0; s--) L = (L << 7) + (long long)__float2int_rn(acc[s][e]);
            const int E = unit(e);
            mom[e] += fma((double)H, pow2(E - 39), (double)L * pow2(E - 74));
        }
    }
    bool good = true;
    const double root_n = (double)sqrtf((float)(end - beg));
#pragma unroll
    for (int e = 0; e < 4; e++) {   // rows 0, 4, 7 and 9, columns 0 .. 6
        const int row = g + 8 * (e >> 1);
        const int amp = e & 1 ? (q == 0 ? cs[1] + 1 : q == 1 ? cs[3] + 3 : cs[5] + 1) : (q == 0 ? cs[0] + 2 : q == 1 ? cs[2] + 1 : q == 2 ? cs[4] + 1 : cs[6] + 2);
        if ((row == 0 || row == 4 || row == 7 || row == 9) && 2 * q + (e & 1) < 7) good = good && mom[e] >= root_n * pow2(unit(e) + max(amp, 0) - 9);
    }
    if (!__all_sync(0xffffffffu, good)) return false;
    __syncwarp();
    // wk: moments [16][8] at 0, coefficients of s [4][4] at 128, of s s' [10][7] at 144, the moments
    // with the norm term [10][8] at 216
    wk[g * 8 + 2 * q] = mom[0];
    wk[g * 8 + 2 * q + 1] = mom[1];
    wk[(g + 8) * 8 + 2 * q] = mom[2];
    wk[(g + 8) * 8 + 2 * q + 1] = mom[3];
    if (lane < 16) {
        const int c = lane >> 2, k = lane & 3;
        double s = 0.0;
#pragma unroll
        for (int jj = 0; jj < 4; jj++) s = fma(att[4 * (int64_t)(iv + jj) + c], (double)kSplineNum[jj][k], s);
        wk[128 + lane] = s * (1.0 / 6.0);
    }
    __syncwarp();
#pragma unroll
    for (int t = 0; t < 3; t++) {
        const int idx = lane + 32 * t;
        if (idx < 70) {
            const int m = idx / 7, b = idx - 7 * m;
            int c = 0;
            while (m >= tri4(c, 3) + 1) c++;
            const int e = c + m - tri4(c, c);
            double s = 0.0;
#pragma unroll
            for (int a = 0; a < 4; a++)
                if (b - a >= 0 && b - a < 4) s = fma(wk[128 + 4 * c + a], wk[128 + 4 * e + b - a], s);
            wk[144 + idx] = s;
        }
    }
    __syncwarp();
#pragma unroll
    for (int t = 0; t < 3; t++) {
        const int idx = lane + 32 * t;
        if (idx < 70) {
            const int m = idx / 7, a = idx - 7 * m;
            double s = 0.0;
#pragma unroll
            for (int b = 0; b < 7; b++) {
                const int k = a + b;   // sum of W u^k v^(12-k): row 14, beyond k = 6 row 15
                s = fma(wk[144 + 7 * m + b], k < 7 ? wk[14 * 8 + k] : wk[15 * 8 + k - 6], s);
            }
            wk[216 + 8 * m + a] = fma(l4, s, wk[8 * m + a]);
        }
    }
    __syncwarp();
#pragma unroll
    for (int t = 0; t < 4; t++) {
        const int idx = lane + 32 * t;
        if (idx < 116) {
            double s = 0.0;
            if (idx < 100) {
                const int p = idx / 10, m = idx - 10 * p;
#pragma unroll
                for (int a = 0; a < 7; a++) s = fma(cbb[p][a], wk[216 + 8 * m + a], s);
                s *= 1.0 / 36.0;
            } else {
                const int b = (idx - 100) >> 2, c = idx & 3;
#pragma unroll
                for (int a = 0; a < 7; a++) s = fma(cb[b][a], wk[(10 + c) * 8 + a], s);
                s *= -1.0 / 6.0;
            }
            red[idx] = s;
        }
    }
    __syncwarp();
    return true;
}

__global__ void __launch_bounds__(32 * kMomWarps, 3) k_att_moments(DevGeo G, MomScale ms, double lambda2,
                                                                const uint32_t* __restrict__ perm_t,
                                                                const int64_t* __restrict__ ivl_off, int n_iv,
                                                                const ObsRec* __restrict__ rec,
                                                                const double* __restrict__ w_att,
                                                                const double* __restrict__ att, double* __restrict__ blk) {
    __shared__ __align__(16) double stage_all[kMomWarps][kWarp * kStage + kAccFP64];
    __shared__ double cbb[10][8], cb[4][8];   // coefficients of BB (over 36) and of B at degree 6 (over 6)
    __shared__ int16_t src_tab[kBlkVals];
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
    double* wk = stage_all[wib];   // after an interval's sums: moments and polynomials
    uint2* st = reinterpret_cast<uint2*>(wk);
    double* red = wk + kWarp * kStage;   // the products
    block_table(src_tab);
    for (int e = threadIdx.x; e < 80; e += blockDim.x) {
        const int p = e >> 3, k = e & 7;
        int i = 0;
        while (p >= tri4(i, 3) + 1) i++;
        const int j = i + p - tri4(i, i);
        int c = 0;
        for (int a = 0; a < 4; a++)
            if (k - a >= 0 && k - a < 4) c += kSplineNum[i][a] * kSplineNum[j][k - a];
        cbb[p][k] = (double)c;
    }
    if (threadIdx.x < 32) {
        const int i = threadIdx.x >> 3, k = threadIdx.x & 7;
        int c = 0;
        for (int a = 0; a < 4; a++)
            if (k - a >= 0 && k - a < 4) c += kSplineNum[i][a] * (k - a == 0 || k - a == 3 ? 1 : 3);
        cb[i][k] = (double)c;
    }
    __syncthreads();
    const int nwarps = gridDim.x * kMomWarps;
    for (int iv = blockIdx.x * kMomWarps + wib; iv < n_iv; iv += nwarps) {
        const int64_t beg = ivl_off[iv], end = ivl_off[iv + 1];
        bool done = false;
        if (iv >= 2 && iv < n_iv - 2 && end - beg >= kMomMin) {
            // the largest magnitudes of W, W R and g (bits of the high words)
            uint32_t mw = 0, mr = 0, mg[4] = {0, 0, 0, 0}, t_lo = 0xffffffffu, t_hi = 0;
            const int64_t tau = G.knot0_ns + (int64_t)iv * G.knot_dt_ns;
            for (int64_t j = beg + lane; j < end; j += kWarp) {
                const uint32_t o = perm_t[j];
                const ObsRec& r = rec[o];
                const double W = w_att ? w_att[o] : r.W;
                const double2 ga = *reinterpret_cast<const double2*>(r.g), gb = *reinterpret_cast<const double2*>(r.g + 2);
                const uint32_t tq = (uint32_t)((r.t_ns - tau) >> ms.tshift);
                t_lo = min(t_lo, tq);
                t_hi = max(t_hi, tq);
                mw = max(mw, (uint32_t)__double2hiint(W) & 0x7fffffffu);
                mr = max(mr, (uint32_t)__double2hiint(W * r.R) & 0x7fffffffu);
                mg[0] = max(mg[0], (uint32_t)__double2hiint(ga.x) & 0x7fffffffu);
                mg[1] = max(mg[1], (uint32_t)__double2hiint(ga.y) & 0x7fffffffu);
                mg[2] = max(mg[2], (uint32_t)__double2hiint(gb.x) & 0x7fffffffu);
                mg[3] = max(mg[3], (uint32_t)__double2hiint(gb.y) & 0x7fffffffu);
            }
            mw = __reduce_max_sync(0xffffffffu, mw);
            mr = __reduce_max_sync(0xffffffffu, mr);
            t_lo = __reduce_min_sync(0xffffffffu, t_lo);
            t_hi = __reduce_max_sync(0xffffffffu, t_hi);
            // -log2 of the largest u and v
            const float lu = -log2f((float)(t_hi + 1) * ms.tinv), lv = -log2f(fmaf(-(float)t_lo, ms.tinv, 1.0f) + 1e-6f);
            // 2^E above them; W and W R below 0.99 of it, for rows of 55 bits
            const int EW = (int)((mw + 0x5000) >> 20) - 1022, ER = (int)((mr + 0x5000) >> 20) - 1022;
            // scales in range: finite, and no power of two below under- or overflows (all residuals may be
            // zero); u and v each reach beyond 2^-1.5: columns near the outer B-splines' ends keep their bits
            bool ok = abs(EW) < 250 && ER < 250 && fmaxf(lu, lv) < 1.5f;
            int Eg[4];
#pragma unroll
            for (int c = 0; c < 4; c++) {
                Eg[c] = (int)(__reduce_max_sync(0xffffffffu, mg[c]) >> 20) - 1022;
                ok = ok && abs(Eg[c]) < 250;
            }
            if (ok)
                done = interval_moments(G, ms, lambda2, perm_t, beg, end, iv, rec, w_att, att, EW, max(ER, -250), Eg, lu, lv,
                                        lane, st, cbb, cb, wk, red);
        }
        if (!done) {
            __syncwarp();
            interval_direct(G, lambda2, 0, perm_t, beg, end, rec, w_att, att, iv + 3, lane, wk, red);
        }
#pragma unroll
        for (int k = 0; k < 5; k++) {
            const int o = lane + 32 * k;
            if (o < kBlkVals) blk[(int64_t)iv * kBlkVals + o] = red[src_tab[o]];
        }
        __syncwarp();
    }
}

// Band of every segment in column layout: bandc[(row0 + c)*16 + k] = N[c-k][c] (k = 0..15)
// and rhs[row0 + c], summed over the knot intervals of the segment only.  One warp per run of
// kAsmKnots consecutive knots of a segment: the interval blocks those knots touch (a
// contiguous range of blk) are copied into shared memory once, coalesced, and every band
// entry of the run is summed from there over its intervals in increasing order.
constexpr int kAsmKnots = 8;
constexpr int kAsmWarps = 4;
__global__ void __launch_bounds__(32 * kAsmWarps) k_att_assemble(int n_seg, int runs_per_seg,
                                                                 const int64_t* __restrict__ seg_row,
                                                                 const int32_t* __restrict__ seg_l,
                                                                 const int32_t* __restrict__ seg_n,
                                                                 const double* __restrict__ blk,
                                                                 double* __restrict__ bandc, double* __restrict__ rhs) {
    __shared__ double stage_all[kAsmWarps][(kAsmKnots + 3) * kBlkVals];
    const int lane = threadIdx.x & 31;
    const int wib = threadIdx.x >> 5;
    double* st = stage_all[wib];
    const int64_t n_units = (int64_t)n_seg * runs_per_seg;
    for (int64_t u = (int64_t)blockIdx.x * kAsmWarps + wib; u < n_units; u += (int64_t)gridDim.x * kAsmWarps) {
        const int sg = (int)(u / runs_per_seg);
        const int run = (int)(u % runs_per_seg);
        const int64_t row0 = seg_row[sg];
        const int n_knots = (int)((seg_row[sg + 1] - row0) / 4);
        const int k0 = run * kAsmKnots;
        if (k0 >= n_knots) continue;
        const int k1 = min(k0 + kAsmKnots, n_knots);
        const int l_lo = seg_l[2 * sg], l_hi = seg_l[2 * sg + 1];
        const int n_lo = seg_n[2 * sg];
        // intervals touched by the knots n_lo + k0 .. n_lo + k1 - 1 (l = n .. n + 3), within the segment
        const int lmin = max(n_lo + k0, l_lo), lmax = min(n_lo + k1 - 1 + 3, l_hi);
        const int nb = lmax - lmin + 1;
        __syncwarp();
        if (nb > 0) {
            const double* src = blk + (int64_t)(lmin - 3) * kBlkVals;
            for (int e = lane; e < nb * kBlkVals; e += kWarp) st[e] = src[e];
        }
        __syncwarp();
        const int n_ent = (k1 - k0) * 4 * 16;
        for (int e = lane; e < n_ent; e += kWarp) {
            const int c = 4 * k0 + (e >> 4);
            const int k = e & 15;
            const int v = c - k;
            double val = 0.0;
            if (v >= 0) {
                const int nc = n_lo + (c >> 2), cc = c & 3;
                const int nv = n_lo + (v >> 2), cv = v & 3;
                int lb = nc > nv ? nc : nv;
                int le = (nc < nv ? nc : nv) + 3;
                if (lb < l_lo) lb = l_lo;
                if (le > l_hi) le = l_hi;
                for (int l = lb; l <= le; l++) {
                    const int i = 4 * (nv - l + 3) + cv, j = 4 * (nc - l + 3) + cc;
                    val += st[(l - lmin) * kBlkVals + tri16(i, j)];
                }
            }
            bandc[(row0 + c) * 16 + k] = val;
        }
        for (int c = 4 * k0 + lane; c < 4 * k1; c += kWarp) {
            const int nc = n_lo + (c >> 2), cc = c & 3;
            double r = 0.0;
            int lb = nc < l_lo ? l_lo : nc;
            int le = nc + 3 > l_hi ? l_hi : nc + 3;
            for (int l = lb; l <= le; l++) r += st[(l - lmin) * kBlkVals + 136 + 4 * (nc - l + 3) + cc];
            rhs[row0 + c] = r;
        }
    }
}

// Robust factorisation of each segment's band (Algorithm C.1 on the envelope, in the
// square-root-free form N = V' D V with V unit upper triangular: U = sqrt(D) V, the same pivot
// test on D and the same zeroed rows for a failing pivot) with the forward substitution (C.2)
// fused, then the back substitution (C.3).  One segment per block of two warps.
//
// What bounds it: an FP64 instruction of a warp holds its SM sub-partition's FP64 unit for 64
// cycles, however many lanes it has active, and takes as long to its result, so a row costs 64
// cycles for every FP64 instruction that is issued or waited for.  Hence few instructions over
// full warps, and two warps that work at the same time:
//   pivot warp   V_{r,.} (one product over the 17 lanes of the pivot row), the next pivot row
//                ahead of the rest (one FMA), and its reciprocal in integer arithmetic
//   update warp  the rest of the window: the 136 entries of the 16x16 window of the partly
//                reduced matrix and its 16 right-hand sides are 152 unordered pairs of slots
//                (slot = row or column mod 16, 16 = right-hand side), five to a lane, in
//                registers: the window moves by one row without moving data, because a pair of
//                slots names one entry (row = early slot, column = late slot) at any time.  Five
//                FMAs update every pair; the pairs of the pivot's slot then take the column that
//                enters, from a ring filled by cp.async a knot (four rows) at a time.
// The pivot row, the row after it and V pass through shared memory, one barrier per row.
// Every entry receives the FMAs of the plain row-by-row elimination in its order.
// The back substitution (pivot warp) goes column by column: one FMA and one shuffle per row.
//
// Measured: 183 segments of 2988 rows 6.47 -> 1.29 ms (2.0 -> 0.43 us per row), 1827 segments of
// 11628 rows 26.5 -> 12.4 ms (before: one segment per 8 lanes, the window in shared memory, 15
// window instructions per row for four segments and an FP64 reciprocal from an FP32 seed).  With
// an FP64 reciprocal in this layout: 1.40 and 18.2 ms; with one warp for both parts: 2.1 and 13.5 ms.
constexpr int kColAhead = 16;      // ring slots of incoming columns
constexpr int kBackRows = 32;      // ring rows of the back substitution
constexpr int kPairs = 152;        // 136 of the matrix, 16 right-hand sides
constexpr int kPairSlots = 5;      // pairs per lane
struct __align__(16) SegWin {
    union {
        struct {
            double ring[kColAhead][16];  // incoming columns: 16 band values
            double rring[kColAhead];     // and their right-hand sides
            double A[2][18];             // pivot row by slot (16: right-hand side), alternating
            double B[2][18];             // the row after it, before this step's update
            double V[2][18];             // V_{r, .} by slot (16: w_r / D_r)
            double tdg[32];              // pivot tolerance times the original diagonal, row mod 32
        } f;
        struct {
            double U[kBackRows][16];     // rows of V (entry 0 unused), row mod kBackRows
            double y[kBackRows];
        } b;
    };
};
// order-preserving map of a double (not NaN) to a signed integer: comparing two of these takes a
// few integer cycles, an FP64 comparison 115
__device__ __forceinline__ long long ord_bits(double x) {
    const long long b = __double_as_longlong(x);
    return b ^ ((b >> 63) & 0x7fffffffffffffffll);
}
__device__ __forceinline__ bool is_nan_bits(double x) {
    return ((unsigned long long)__double_as_longlong(x) << 1) > 0xffe0000000000000ull;
}

__device__ __forceinline__ void cp_async16_att(void* smem, const void* gmem) {
    const unsigned sa = (unsigned)__cvta_generic_to_shared(smem);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(sa), "l"(gmem) : "memory");
}
__device__ __forceinline__ void cp_async8_att(void* smem, const void* gmem) {
    const unsigned sa = (unsigned)__cvta_generic_to_shared(smem);
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;\n" ::"r"(sa), "l"(gmem) : "memory");
}
__device__ __forceinline__ void cp_async_commit_att() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait_att() {
    asm volatile("cp.async.wait_group %0;\n" ::"n"(N) : "memory");
}

__device__ __forceinline__ void seg_barrier() { asm volatile("bar.sync 1, 64;" ::: "memory"); }
__global__ void __launch_bounds__(64) k_att_solve(int n_seg, const int64_t* __restrict__ seg_row,
                                                  const double* __restrict__ bandc, const double* __restrict__ rhs,
                                                  double* __restrict__ urow, double* __restrict__ yv,
                                                  double* __restrict__ x, double tol, int* __restrict__ seg_rd) {
    __shared__ SegWin sm;
    const int lane = threadIdx.x & 31;
    // the update warp issues five FP64 instructions per row, the pivot warp two: which warp of the
    // block is which alternates between waves of two blocks per SM, so that the SM's sub-partitions
    // carry both (1827 segments: 12.4 ms, 14.4 without)
    const bool pivot_warp = ((threadIdx.x >> 5) ^ ((blockIdx.x / (2 * 152)) & 1)) == 0;
    const int sg = blockIdx.x;
    const int64_t base = seg_row[sg];
    const int n = (int)(seg_row[sg + 1] - base);
    const double* bc = bandc + base * 16;
    const double* rh = rhs + base;
    double* ur = urow + base * 16;
    double* yr = yv + base;
    // pivot row 0 and row 1 by slot, right-hand side at 16, zero at 17
    if (threadIdx.x < 18) {
        sm.f.A[0][lane] = lane < 16 ? bc[(int64_t)lane * 16 + lane] : lane == 16 ? rh[0] : 0.0;
        sm.f.B[0][lane] = lane >= 1 && lane < 16 ? bc[(int64_t)lane * 16 + lane - 1] : lane == 16 ? rh[1] : 0.0;
        sm.f.A[1][lane] = sm.f.B[1][lane] = sm.f.V[0][lane] = sm.f.V[1][lane] = 0.0;
        if (lane < 16) sm.f.tdg[lane] = tol * bc[(int64_t)lane * 16];
    }
    __syncthreads();
    if (pivot_warp) {
        int rd = 0;
        // 1 / D_r for the pivot of row r; a failing pivot zeroes the row (rank defect)
        auto pivot_inverse = [&](double piv, double td) -> double {
            const bool pos = ord_bits(piv) > ord_bits(td) && !is_nan_bits(piv) && !is_nan_bits(td);
            rd += !pos;
            const double y = rcp_pos_int(piv);
            return pos && __double_as_longlong(piv) > 0 ? y : 0.0;
        };
        double invd = pivot_inverse(sm.f.A[0][0], sm.f.tdg[0]);
        const int l17 = lane < 17 ? lane : 17;
        double a0 = sm.f.A[0][l17];   // the pivot row (lane = slot; 16: right-hand side)
        double* up = ur;
        for (int r0 = 0; r0 < n; r0 += 4) {
#pragma unroll
            for (int h = 0; h < 4; h++) {
                const int r = r0 + h, s0 = r & 15, s1 = (r + 1) & 15;
                // V_{r, .} = W[0][.] / D_r and w_r / D_r
                const double v = invd * a0;
                if (lane < 17) sm.f.V[h & 1][lane] = v;
                const double v1 = __shfl_sync(0xffffffffu, v, s1);
                seg_barrier();   // V_r is out; row r + 1 (before this step's update) and column r + 16 are in
                const double* col = sm.f.ring[(r + 16) % kColAhead];
                const double b0 = sm.f.B[h & 1][l17];
                const double c15 = col[15], c0 = col[0], td = sm.f.tdg[(r + 1) & 31];
                // look ahead: the next pivot row, complete (lane s0: the entry of the column that enters)
                a0 = lane == s0 ? c15 : fma(-v1, a0, b0);
                const double piv = __shfl_sync(0xffffffffu, a0, s1);
                if (lane < 17) sm.f.A[(h + 1) & 1][lane] = a0;
                if (lane < 16) up[h * 16 + ((lane - s0) & 15)] = v;
                else if (lane == 16) yr[r] = v;
                else if (lane == 17) sm.f.tdg[(r + 16) & 31] = tol * c0;
                if (r + 1 < n) invd = pivot_inverse(piv, td);
            }
            up += 64;
        }
        if (lane == 0) seg_rd[sg] = rd;
        seg_barrier();
    } else {
        // this lane's pairs by early slot and late slot of the rows in the window, as byte offsets into
        // a row by slot, and their entries of the first window.  Pairs 0-135 are the matrix's (four for
        // every lane and a fifth in lanes 0-7), the right-hand sides of slots 0-15 are the fifth of
        // lanes 8-23 (late slot 16)
        int oe[kPairSlots], ol[kPairSlots];
        double e[kPairSlots];
#pragma unroll
        for (int t = 0; t < kPairSlots; t++) {
            int k = lane + kWarp * t, p = 0;
            oe[t] = ol[t] = 8 * 17;   // no pair: an entry that nothing uses
            e[t] = 0.0;
            if (k < 136) {
                while (k >= 16 - p) { k -= 16 - p; p++; }
                oe[t] = 8 * p;
                ol[t] = 8 * (p + k);
                e[t] = bc[(int64_t)(p + k) * 16 + k];   // n >= 16: a segment has 4 knots or more
            } else if (k < kPairs) {
                oe[t] = 8 * (k - 136);
                ol[t] = 8 * 16;
                e[t] = rh[k - 136];
            }
        }
        const bool z_lane = lane >= 8 && lane < 24;
        // the four columns of a knot (c a multiple of 4) into ring slots c mod kColAhead ..: a lane
        // copies 16 bytes of the 512, lanes 0 and 1 also 16 of the right-hand sides; zeros beyond the
        // segment (whose length is a multiple of 4)
        auto fetch = [&](int c) {
            double* slot = &sm.f.ring[c % kColAhead][0] + 2 * lane;
            double* rslot = &sm.f.rring[c % kColAhead] + 2 * lane;
            if (c < n) {
                cp_async16_att(slot, bc + (int64_t)c * 16 + 2 * lane);
                if (lane < 2) cp_async16_att(rslot, rh + c + 2 * lane);
            } else {
                slot[0] = slot[1] = 0.0;
                if (lane < 2) rslot[0] = rslot[1] = 0.0;
            }
            cp_async_commit_att();
        };
        constexpr int kKnotsAhead = kColAhead / 4 - 1;
#pragma unroll
        for (int q = 0; q < kKnotsAhead; q++) fetch(16 + 4 * q);
        for (int r0 = 0; r0 < n; r0 += 4) {
            cp_async_wait_att<kKnotsAhead - 1>();   // the columns r0 + 16 .. r0 + 19 have arrived
#pragma unroll
            for (int h = 0; h < 4; h++) {
                const int r = r0 + h, s0 = r & 15, s2 = (r + 2) & 15;
                seg_barrier();   // V_r and the pivot row are in; row r + 1 is out
                // the slots of the columns taken in the previous four steps are free
                if (h == 0) fetch(r0 + 12 + kColAhead);
                const char* A0 = (const char*)sm.f.A[h & 1];
                const char* V0 = (const char*)sm.f.V[h & 1];
                const char* col = (const char*)sm.f.ring[(r + 16) % kColAhead];
                // pairs of the other slots: W[a][b] -= V_a W[0][b]; pairs of slot s0 (their early one): the
                // entering column r + 16 (band entry N[c - k][c] or the right-hand side), the late slot of its pairs
#pragma unroll
                for (int t = 0; t < kPairSlots; t++) {
                    const double ve = *(const double*)(V0 + oe[t]);
                    const double wl = *(const double*)(A0 + ol[t]);
                    const bool mine = oe[t] == 8 * s0;
                    const char* src = col + ((8 * s0 - ol[t]) & 120);
                    if (t == 4) src = z_lane ? (const char*)&sm.f.rring[(r + 16) % kColAhead] : src;
                    const double in = *(const double*)src;
                    const double upd = fma(-ve, wl, e[t]);
                    e[t] = mine ? in : upd;
                    const bool turn = t == 4 ? mine && !z_lane : mine;
                    oe[t] = turn ? ol[t] : oe[t];
                    ol[t] = turn ? 8 * s0 : ol[t];
                }
                // publish row r + 2 for the next look-ahead: its slot is the early one of its pairs
                char* B1 = (char*)sm.f.B[(h + 1) & 1];
#pragma unroll
                for (int t = 0; t < kPairSlots; t++)
                    if (oe[t] == 8 * s2) *(double*)(B1 + ol[t]) = e[t];
            }
        }
        cp_async_wait_att<0>();
        seg_barrier();
        return;
    }
    cp_async_wait_att<0>();
    __syncwarp();
    // back substitution x_r = y_r - sum_k V_{r,r+k} x_{r+k}, column by column: lane j < 16 keeps the
    // partial sum of the row i = j mod 16 among the 16 rows at or below r; once x_r is known it is
    // broadcast and every pending row subtracts its product (one FMA per row and step).  Rows are
    // fetched a knot (four rows) at a time.
    auto fetch_rows = [&](int i) {   // i a multiple of 4
        if (i >= 0) {
            cp_async16_att(&sm.b.U[i % kBackRows][0] + 2 * lane, ur + (int64_t)i * 16 + 2 * lane);
            if (lane < 2) cp_async16_att(&sm.b.y[i % kBackRows] + 2 * lane, yr + i + 2 * lane);
        }
        cp_async_commit_att();
    };
    constexpr int kBackAhead = kBackRows / 4 - 5;   // knots fetched beyond the five that a step reads
#pragma unroll
    for (int q = 1; q <= 4 + kBackAhead; q++) fetch_rows(n - 4 * q);
    cp_async_wait_att<kBackAhead>();
    __syncwarp();
    const int j = lane & 15;
    double acc = sm.b.y[(n - 16 + ((j - (n - 16)) & 15)) % kBackRows];   // rows n-16 .. n-1 by slot
    double* xo = x + base;
    for (int r0 = n - 4; r0 >= 0; r0 -= 4) {
        cp_async_wait_att<kBackAhead - 1>();   // the rows r0 - 16 .. r0 - 13 have arrived
        __syncwarp();
        double u[4], yn[4];
#pragma unroll
        for (int h = 3; h >= 0; h--) {
            const int r = r0 + h, k = (r - j) & 15, i = r - k;
            u[h] = i >= 0 ? sm.b.U[i & (kBackRows - 1)][k] : 0.0;
            yn[h] = r >= 16 ? sm.b.y[(r - 16) & (kBackRows - 1)] : 0.0;
        }
#pragma unroll
        for (int h = 3; h >= 0; h--) {
            const int r = r0 + h;
            const double xr = __shfl_sync(0xffffffffu, acc, r & 15);
            const bool mine = j == (r & 15);
            if (lane == (r & 15)) xo[r] = xr;
            const double upd = fma(-u[h], xr, acc);
            acc = mine ? yn[h] : upd;
        }
        fetch_rows(r0 - 16 - 4 * kBackAhead);
    }
    cp_async_wait_att<0>();

}

// a_n += x for the coefficients each segment owns (n in [u_lo, u_hi]); one thread per
// coefficient.  The mixed form also accumulates the update in d_att (FP32); dx, if given,
// receives the update itself (FP64).
__global__ void k_att_apply(int n_coef, int n_seg, const int32_t* __restrict__ seg_u, const int32_t* __restrict__ seg_n,
                            const int64_t* __restrict__ seg_row, const double* __restrict__ x,
                            double* __restrict__ att, float* __restrict__ d_att, double* __restrict__ dx) {
    for (int n = blockIdx.x * blockDim.x + threadIdx.x; n < n_coef; n += gridDim.x * blockDim.x) {
        int lo = 0, hi = n_seg - 1;
        while (lo < hi) {
            int mid = (lo + hi + 1) >> 1;
            if (seg_u[2 * mid] <= n) lo = mid; else hi = mid - 1;
        }
        const int sg = lo;
        const int64_t r0 = seg_row[sg] + 4 * (int64_t)(n - seg_n[2 * sg]);
#pragma unroll
        for (int c = 0; c < 4; c++) {
            att[4 * (int64_t)n + c] += x[r0 + c];
            if (d_att) d_att[4 * (int64_t)n + c] += (float)x[r0 + c];
            if (dx) dx[4 * (int64_t)n + c] = x[r0 + c];
        }
    }
}

void launch_att_accum(const DevGeo& G, double lambda2, int rhs_norm, const uint32_t* perm_t, const int64_t* ivl_off,
                      int n_iv, const ObsRec* rec, const double* w_att, const double* att, double* blk, bool moments,
                      const Shapes& sh, cudaStream_t s) {
    const int bps = sh.att_bps > 0 ? sh.att_bps : 32;
    int blocks = (n_iv + 3) / 4;
    if (blocks > 152 * bps) blocks = 152 * bps;
    if (blocks < 1) blocks = 1;
    // the norm term of degree 12 has no columns of its own and loses 4 bits in its middle: it must be small
    // beside g g' (|g| about 2; the usual lambda^2 is 1e-6)
    if (moments && !rhs_norm && lambda2 <= 1.0 / 64.0) {
        int nb = 0;   // significant bits of dt
        while (nb < 62 && (G.knot_dt_ns >> nb) > 0) nb++;
        MomScale ms;
        ms.shift = 64 - nb;
        ms.tshift = nb > 30 ? nb - 30 : 0;
        ms.tinv = (float)((double)((int64_t)1 << ms.tshift) / (double)G.knot_dt_ns);
        ms.inv = (uint64_t)(((unsigned __int128)1 << (62 + nb)) / (unsigned __int128)G.knot_dt_ns);
        k_att_moments<<<blocks, 32 * kMomWarps, 0, s>>>(G, ms, lambda2, perm_t, ivl_off, n_iv, rec, w_att, att, blk);
        return;
    }
    k_att_accum<<<blocks, 128, 0, s>>>(G, lambda2, rhs_norm, perm_t, ivl_off, n_iv, rec, w_att, att, blk);
}

// d_att (mixed form only, else null) accumulates the applied update in FP32
void launch_att_solve(int n_seg, int max_seg_knots, int n_coef, int64_t n_rows, const int64_t* seg_row, const int32_t* seg_l,
                      const int32_t* seg_n, const int32_t* seg_u, const double* blk, double* bandc, double* rhs,
                      double* urow, double* yv, double* x, double tol, int* seg_rd, double* att, float* d_att,
                      double* dx, cudaStream_t s) {
    // knot runs per segment, enough for the largest segment
    const int runs_per_seg = (max_seg_knots + kAsmKnots - 1) / kAsmKnots;
    int64_t units = (int64_t)n_seg * runs_per_seg;
    int blocks = (int)((units + kAsmWarps - 1) / kAsmWarps);
    if (blocks > 152 * 16) blocks = 152 * 16;
    if (blocks < 1) blocks = 1;
    k_att_assemble<<<blocks, 32 * kAsmWarps, 0, s>>>(n_seg, runs_per_seg, seg_row, seg_l, seg_n, blk, bandc, rhs);
    k_att_solve<<<n_seg, 64, 0, s>>>(n_seg, seg_row, bandc, rhs, urow, yv, x, tol, seg_rd);
    k_att_apply<<<(n_coef + 255) / 256, 256, 0, s>>>(n_coef, n_seg, seg_u, seg_n, seg_row, x, att, d_att, dx);
}

// Block Gauss-Seidel (Sect. 4.6, Eq. precond): before the C block the hand-over residuals
// take the attitude update to first order, R += sum_j B_j g . dx[l-3+j] (dR/da_n = g B_n,
// Eq. dfadq); one thread per observation, FP64.
__global__ void k_rec_att_correct(DevGeo G, int64_t n_obs, ObsRec* __restrict__ rec, const double* __restrict__ dx) {
    for (int64_t o = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; o < n_obs; o += (int64_t)gridDim.x * blockDim.x) {
        ObsRec& r = rec[o];
        const int l = left_index(G, r.t_ns);
        double B[4];
        bspline4(G, r.t_ns, l, B);
        const double* d = dx + 4 * (int64_t)(l - 3);
        double corr = 0.0;
#pragma unroll
        for (int j = 0; j < 4; j++)
            corr += B[j] * (r.g[0] * d[4 * j] + r.g[1] * d[4 * j + 1] + r.g[2] * d[4 * j + 2] + r.g[3] * d[4 * j + 3]);
        r.R += corr;
    }
}
void launch_rec_att_correct(const DevGeo& G, int64_t n_obs, ObsRec* rec, const double* dx, cudaStream_t s) {
    int64_t b = (n_obs + 255) / 256;
    if (b > 152 * 32) b = 152 * 32;
    if (b < 1) b = 1;
    k_rec_att_correct<<<(int)b, 256, 0, s>>>(G, n_obs, rec, dx);
}

}  // namespace agis
