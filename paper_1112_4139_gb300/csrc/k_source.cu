// k_source.cu -- the observation pass in source order and the S block (Sect. 5.1).
//
// The observation pass (one thread per observation) leaves residual h, design row A and sigma^2
// in a 64-byte scratch row.  The inner iteration of Sect. 5.1.2 then runs as passes over the
// rows (one warp per source, largest first) and 5x5 solves (one thread per source) in turn:
//   k_src_first   sigma per class, robust scale and round 0's class sums
//   k_src_solve5  the 5x5 algebra of the excess-noise steps
//   k_src_round   the next round's class sums, and the weights of the last round
//   k_src_sums    class sums of every row, a block per source, in place of the above where the set is small
//   k_src_final   the hand-over records (t, R = h - A d, W, g, meta) that the time-ordered
//                 attitude pass and the calibration pass gather
//   k_src_general sources whose sigma differs within a class: all rounds in one warp
//
// What bounds it: the FP64 pipe (2 FMA per clock and SM; 86 to 92% busy in the passes over the rows, 63% in
// k_src_round, which waits for rows at 12 warps an SM).  A 5x5 solve of one lane costs a warp as
// many FP64 cycles as 32 of them, hence a thread per source there.  Downweighting leaves w = 1
// wherever |z| <= 2 (Eqs. dw, dwH), about 95% of the observations, so for long sources the 21
// products of a row within two robust scales are summed once, with unit weights; a round evaluates z in
// FP32 (with a bound on its error), and only the rows that may exceed 2 or that those sums do not hold are
// gathered, 32 to a warp, for the FP64 weight and 27 products: a round then costs about a fifth of
// the FP64 work of the direct sums.
// Measured, source solves of the S block: 6.6M observations of 8000 sources 4.75 -> 2.9 ms with direct
// sums (first pass 0.12 ms, sums 5 x 0.47), 1.5 with corrections (first sums 0.37, rounds 4 x 0.175); 0.5M of
// 3000 sources 1.68 -> 0.57 with direct sums.  Before, one persistent kernel ran all rounds of a batch of sources in a
// warp, with the 5x5 solves in one lane each.
#include <type_traits>

#include "agis_internal.cuh"

namespace agis {



// k-th smallest (0-based) of the keys[0..n) (order-preserving maps of h / sigma, one 8-byte key
// per observation, contiguous) by a radix select of 8-bit digits with a 256-bin shared-memory
// histogram per warp.  A pass whose chosen digit holds a single key ends the select: one more
// pass finds that key (on continuous data about 4 passes instead of 8).
__device__ uint64_t warp_select(const uint64_t* __restrict__ keys, int n, int k, int* hist, int lane) {
    uint64_t prefix = 0, pmask = 0;
    int kk = k;
    for (int d = 7; d >= 0; d--) {
        int shift = 8 * d;
#pragma unroll
        for (int i = 0; i < 8; i++) hist[lane * 8 + i] = 0;
        __syncwarp();
        for (int j = lane; j < n; j += kWarp) {
            const uint64_t key = keys[j];
            if ((key & pmask) == prefix) atomicAdd(&hist[(key >> shift) & 255u], 1);
        }
        __syncwarp();
        int c[8];
        int tot = 0;
#pragma unroll
        for (int i = 0; i < 8; i++) { c[i] = hist[lane * 8 + i]; tot += c[i]; }
        // inclusive scan across lanes
        int incl = tot;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            int v = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += v;
        }
        int excl = incl - tot;
        unsigned ball = __ballot_sync(0xffffffffu, incl > kk);
        int src_lane = __ffs(ball) - 1;
        int bin = 0, below = 0, cnt = 0;
        if (lane == src_lane) {
            int acc = excl;
            int bsel = 7;
#pragma unroll
            for (int i = 0; i < 8; i++) {
                if (acc + c[i] > kk) { bsel = i; break; }
                acc += c[i];
            }
            bin = lane * 8 + bsel;
            below = acc;
            cnt = hist[bin];
        }
        bin = __shfl_sync(0xffffffffu, bin, src_lane);
        below = __shfl_sync(0xffffffffu, below, src_lane);
        cnt = __shfl_sync(0xffffffffu, cnt, src_lane);
        kk -= below;
        prefix |= (uint64_t)bin << shift;
        pmask |= (uint64_t)0xffu << shift;
        __syncwarp();
        if (cnt == 1 && d > 0) {
            // the only key with this prefix is the k-th smallest
            uint64_t found = 0;
            for (int j = lane; j < n; j += kWarp) {
                const uint64_t key = keys[j];
                if ((key & pmask) == prefix) found = key;
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                const uint64_t v = __shfl_xor_sync(0xffffffffu, found, o);
                found = v > found ? v : found;
            }
            return found;
        }
    }
    return prefix;
}

// the (k)-th and (k+1)-th smallest values (k+1 capped at n-1)
__device__ void warp_select_pair(const uint64_t* __restrict__ keys, int n, int k, int* hist, int lane, double& v0,
                                 double& v1) {
    uint64_t K = warp_select(keys, n, k, hist, lane);
    v0 = dkey_inv(K);
    if (k + 1 >= n) { v1 = v0; return; }
    int less = 0, eq = 0;
    uint64_t nxt = ~0ull;
    for (int j = lane; j < n; j += kWarp) {
        const uint64_t key = keys[j];
        less += key < K;
        eq += key == K;
        if (key > K && key < nxt) nxt = key;
    }
    less = warp_sum_int(less);
    eq = warp_sum_int(eq);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        uint64_t v = __shfl_xor_sync(0xffffffffu, nxt, o);
        nxt = v < nxt ? v : nxt;
    }
    v1 = (k + 1 < less + eq) ? v0 : dkey_inv(nxt);
}

// Per-source geometry for the observation pass: p, q, r (Eq. normal-triad), parameters, cos(delta).
__global__ void k_src_geo(int32_t n_src, const double* __restrict__ src, double* __restrict__ geo) {
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n_src; i += gridDim.x * blockDim.x) {
        SrcGeo S;
        source_geo(src + 5 * (size_t)i, S);
        double* g = geo + 16 * (size_t)i;
        for (int k = 0; k < 3; k++) { g[k] = S.p[k]; g[3 + k] = S.q[k]; g[6 + k] = S.r[k]; }
        g[9] = S.par; g[10] = S.pma; g[11] = S.pmd; g[12] = S.cosd;
        // slots 13-15: p and q rounded to FP32 (six floats)
        float* gf = reinterpret_cast<float*>(g + 13);
        for (int k = 0; k < 3; k++) { gf[k] = (float)S.p[k]; gf[3 + k] = (float)S.q[k]; }
    }
}

// Observation pass, one thread per observation (source order): residual h, design row A and
// attitude partial g at the current parameters.  Scratch row: h, A[5], weight 1, sigma^2;
// with the excess attitude noise on, sigma~^2 = sigma^2 + eps_a^2(t) in place of sigma^2 (Eq. W).
__global__ void __launch_bounds__(256) k_obs_forward(DevGeo G, AttNoise an, int64_t n_obs, const int64_t* __restrict__ t_ns,
                                                     const uint32_t* __restrict__ meta,
                                                     const float* __restrict__ sigma, const double* __restrict__ mu,
                                                     const int32_t* __restrict__ obs_src,
                                                     const double* __restrict__ geo, const double* __restrict__ att,
                                                     const double* __restrict__ cal, double* __restrict__ scr,
                                                     uint64_t* __restrict__ skey, ObsRec* __restrict__ rec) {
    for (int64_t o = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; o < n_obs; o += (int64_t)gridDim.x * blockDim.x) {
        const double* g = geo + 16 * (size_t)obs_src[o];
        SrcGeo S;
        for (int k = 0; k < 3; k++) { S.p[k] = g[k]; S.q[k] = g[3 + k]; S.r[k] = g[6 + k]; }
        S.par = g[9]; S.pma = g[10]; S.pmd = g[11]; S.cosd = g[12];
        const int64_t t = t_ns[o];
        const uint32_t m = meta[o];
        const double muv = (G.cg.on || meta_kind(m)) ? mu[o] : 0.0;
        ObsOut ob;
        observe<1>(G, S, t, m, muv, att, cal, ob);
        const double sg = (double)sigma[o];
        double s2 = sg * sg, x = ob.R * rcp_pos(sg);
        if (an.eps2) {
            s2 = s2 + an.eps2[an_index(an, t, m)];
            x = ob.R * rsqrt(s2);
        }
        double* e = scr + (size_t)o * kScr;
        e[0] = ob.R;
        e[1] = ob.A[0]; e[2] = ob.A[1]; e[3] = ob.A[2]; e[4] = ob.A[3]; e[5] = ob.A[4];
        skey[o] = dkey(x);
        e[6] = 1.0;
        e[7] = s2;
        ObsRec* r = rec + o;
        r->t_ns = t;
        r->meta = m;
        r->pad = 0;
        r->g[0] = ob.g[0]; r->g[1] = ob.g[1]; r->g[2] = ob.g[2]; r->g[3] = ob.g[3];
    }
}

// ---------------------------------------------------------------------------------------
// class-sum path (one sigma per class and source)
// ---------------------------------------------------------------------------------------
constexpr int kPassWarps = 4;      // warps per block of the passes over the rows

// Sums of kSumVals lane values over the warp by recursive halving: in each step a lane gives one
// half of its values to its partner and adds the partner's other half, 23 additions instead of
// the 105 of butterflies.  out[i] (i < kSumVals) is written by the lane that ends up with it.
__device__ __forceinline__ void reduce_vals(double* v, int lane, double* out) {
    int off = 0, cnt = kSumVals;   // this lane's values are off .. off + cnt - 1
    auto step = [&](auto nc, int bit) {
        constexpr int n = decltype(nc)::value, h = (n + 1) / 2;
        const bool up = lane & bit;
#pragma unroll
        for (int k = 0; k < h; k++) {
            const double lo = v[k], hi = k + h < n ? v[k + h] : 0.0;
            const double got = __shfl_xor_sync(0xffffffffu, up ? lo : hi, bit);
            v[k] = (up ? hi : lo) + got;
        }
        off += up ? h : 0;
        cnt = up ? cnt - h : (cnt < h ? cnt : h);
    };
    step(std::integral_constant<int, 21>{}, 16);
    step(std::integral_constant<int, 11>{}, 8);
    step(std::integral_constant<int, 6>{}, 4);
    step(std::integral_constant<int, 3>{}, 2);
    step(std::integral_constant<int, 2>{}, 1);
    if (cnt > 0) out[off] = v[0];
}

// Adds u times the products of the rows listed in shared memory (m <= 32 of them) to corr, lane by
// lane.  first: w = wfun(h rx), the initial downweighting by the robust scale; else w = wfun((h - A d)
// isd).  kAll: u = w.  Otherwise a row that the unit-weight sums hold (weight slot 1) takes u = w - 1
// and counts into what is taken off (sub_n rows, sub_hh of h^2), one that they do not hold (weight
// slot 0) takes u = w.  last: w goes to the scratch row for the hand-over records.
template <bool kAll>
__device__ __forceinline__ void weigh_rows(double* scr, const uint32_t* list, int m, int lane, bool first,
                                           const double* d, double scale, int wfn, bool last, double* corr, int& nout,
                                           int& sub_n, double& sub_hh) {
    if (lane >= m) return;
    double* e = scr + (size_t)list[lane] * kScr;
    double h, A[5];
    row_load(e, h, A);
    const double w = wfun((first ? h : h - row_dot(A, d)) * scale, wfn);
    const bool held = !kAll && e[6] != 0.0;
    if (last) e[6] = w;
    nout += w < 0.2;
    const double u = held ? w - 1.0 : w;
#pragma unroll
    for (int a = 0; a < 5; a++) {
        const double ua = u * A[a];
#pragma unroll
        for (int b = a; b < 5; b++) corr[up5(a, b)] = fma(ua, A[b], corr[up5(a, b)]);
        corr[15 + a] = fma(ua, h, corr[15 + a]);
    }
    const double uh = u * h;
    corr[20] = fma(uh, h, corr[20]);
    if (held) {
        sub_n++;
        sub_hh = fma(-uh, h, sub_hh);
    }
}

// Sums of w times the products over all rows of a class, for rounds that would take off too much of
// the unit-weight sums.
__device__ __noinline__ void direct_rows(double* scr, int lo, int hi, uint32_t* list, int lane, const double* d, double scale,
                                         int wfn, bool last, double* sums, int& nout) {
    int sub_n = 0;
    double sub_hh = 0.0;
#pragma unroll
    for (int k = 0; k < kSumVals; k++) sums[k] = 0.0;
    for (int j0 = lo; j0 < hi; j0 += kWarp) {
        list[lane] = (uint32_t)(j0 + lane);
        __syncwarp();
        weigh_rows<true>(scr, list, min(hi - j0, kWarp), lane, false, d, scale, wfn, last, sums, nout, sub_n, sub_hh);
        __syncwarp();
    }
}

// Appends the row j of every lane with cand set to the list (n entries so far); a full list of 32
// is worked off by `flush`.
template <class F>
__device__ __forceinline__ void append_rows(bool cand, int j, uint32_t* list, int& n, int lane, F flush) {
    const unsigned ball = __ballot_sync(0xffffffffu, cand);
    if (!ball) return;
    const int pos = n + __popc(ball & ((1u << lane) - 1u));
    if (cand && pos < 32) list[pos] = (uint32_t)j;
    n += __popc(ball);
    if (n < 32) return;
    __syncwarp();
    flush(32);
    __syncwarp();
    if (cand && pos >= 32) list[pos - 32] = (uint32_t)j;
    n -= 32;
}

// Per source: sigma per class, robust scale of x = h / sigma (Sect. 5.1.2: half the intersextile
// range), unit-weight class sums, and round 0's downweighting.  The unit-weight sums hold the rows with
// |x| below twice the robust scale and no others: a row further out (5 to 8% of them, however far) has
// 0 in its weight slot and is added with its weight in every round, so that nothing large is ever
// summed only to be taken off again.  A robust scale of 0 leaves all rows to be added.
template <bool kDirect>
__global__ void __launch_bounds__(32 * kPassWarps) k_src_first(Settings st, const int64_t* __restrict__ src_off,
                                                               const int32_t* __restrict__ src_nal,
                                                               const int32_t* __restrict__ src_order, int32_t n_src,
                                                               int batch, double* __restrict__ scratch,
                                                               const uint64_t* __restrict__ skey,
                                                               SrcWork* __restrict__ work) {
    extern __shared__ __align__(16) unsigned char first_smem[];
    SelWork& sw = reinterpret_cast<SelWork*>(first_smem)[threadIdx.x >> 5];
    __shared__ uint32_t list_all[kPassWarps][32];
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
    uint32_t* list = list_all[wib];
    const int step = gridDim.x * kPassWarps * batch;
    for (int base = (blockIdx.x * kPassWarps + wib) * batch; base < n_src; base += step)
        for (int q = base; q < min(base + batch, n_src); q++) {
            const int i = src_order[q];
            const int64_t o0 = src_off[i];
            const int n = (int)(src_off[i + 1] - o0), nal = src_nal[i];
            SrcWork& w = work[i];
            if (n == 0) {
                if (lane == 0) w.flags = 2;
                continue;
            }
            double* scr = scratch + (size_t)o0 * kScr;
            double vs = 0.0;
            const bool in_smem = n <= kKeyCap64;
            const uint64_t* keys = in_smem ? sw.keys : skey + o0;
            if (st.robust) {
                float lo = INFINITY, hi = -INFINITY;
                bool nan = false;
                for (int j = lane; j < n; j += kWarp) {
                    const uint64_t key = skey[o0 + j];
                    if (in_smem) sw.keys[j] = key;
                    const float x = trunc_f32(dkey_inv(key));
                    nan = nan || !isfinite(x);
                    lo = fminf(lo, x);
                    hi = fmaxf(hi, x);
                }
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) {
                    lo = fminf(lo, __shfl_xor_sync(0xffffffffu, lo, o));
                    hi = fmaxf(hi, __shfl_xor_sync(0xffffffffu, hi, o));
                }
                nan = __any_sync(0xffffffffu, nan);
                __syncwarp();
                const double h1 = __dmul_rn(1.0 / 6.0, (double)(n - 1)), h5 = __dmul_rn(5.0 / 6.0, (double)(n - 1));
                const int lo1 = (int)floor(h1), lo5 = (int)floor(h5);
                double x[4];
                if (nan || !select_quantiles(keys, n, lo1, lo5, lo, hi, sw, lane, x)) {
                    warp_select_pair(keys, n, lo1, sw.hist, lane, x[0], x[1]);
                    warp_select_pair(keys, n, lo5, sw.hist, lane, x[2], x[3]);
                }
                // products and differences rounded one by one (h - floor(h) is exact)
                const double g1 = __dadd_rn(h1, -(double)lo1), g5 = __dadd_rn(h5, -(double)lo5);
                vs = 0.5 * ((x[2] + g5 * (x[3] - x[2])) - (x[0] + g1 * (x[1] - x[0])));
                __syncwarp();
            }
            // x of the key, to 2^-22 relative: at or above 2 robust scales within that, or not finite
            const float ivs = (float)(1.0 / vs);
            auto beyond = [&](int j) {
                return st.robust && !(fabsf(trunc_f32(dkey_inv(keys[j])) * ivs) < 1.99999f);
            };
            // unit-weight sums and sigma of each class; sums only while its sigma is one value
            // (bit patterns: variances are not negative, and comparisons hold the FP64 unit)
            double s2c[2] = {1.0, 1.0};
            uint64_t s2m = __double_as_longlong(1e300);
            bool uni = true;
            for (int c = 0; c < 2; c++) {
                const int lo = c ? nal : 0, hi = c ? n : nal;
                double v[kSumVals];
#pragma unroll
                for (int k = 0; k < kSumVals; k++) v[k] = 0.0;
                if (lo < hi) {
                    const double s2 = scr[(size_t)lo * kScr + 7];
                    const uint64_t s2b = __double_as_longlong(s2);
                    bool same = s2 == s2;
                    for (int j0 = lo; j0 < hi; j0 += kWarp) {
                        const int j = j0 + lane;
                        if (j < hi) {
                            double* e = scr + (size_t)j * kScr;
                            const uint64_t sj = __double_as_longlong(e[7]);
                            s2m = sj < s2m ? sj : s2m;
                            same = same && sj == s2b;
                            if (!kDirect && uni) {
                                double h, A[5];
                                row_load(e, h, A);
                                if (beyond(j)) {
                                    e[6] = 0.0;
                                } else {
#pragma unroll
                                    for (int a = 0; a < 5; a++) {
#pragma unroll
                                        for (int b = a; b < 5; b++) v[up5(a, b)] = fma(A[a], A[b], v[up5(a, b)]);
                                        v[15 + a] = fma(A[a], h, v[15 + a]);
                                    }
                                    v[20] = fma(h, h, v[20]);
                                }
                            }
                        }
                        uni = __all_sync(0xffffffffu, uni && same);
                    }
                    s2c[c] = s2;
                }
                if (!kDirect && uni) reduce_vals(v, lane, w.T[c]);
            }
            const double s2min = warp_min(__longlong_as_double(s2m));
            if (lane == 0) {
                w.s2c[0] = s2c[0];
                w.s2c[1] = s2c[1];
                w.s2min = s2min;
                w.vs = vs;
                w.flags = uni ? 1 : 0;
            }
            if (!uni) continue;
            const bool last = st.robust ? st.n_rounds == 0 : true;
            int nout = 0;
            if constexpr (kDirect) {
                // round 0's weights are wfun(h rx); all 1 for a robust scale of 0
                if (lane < 2) w.isd[lane] = vs > 0.0 ? 1.0 / (sqrt(lane ? s2c[1] : s2c[0]) * vs) : 0.0;
                if (lane < 2) w.all[lane] = 0;
                for (int k = lane; k < kRedVals; k += kWarp) (&w.C[0][0])[k] = 0.0;
                continue;
            } else
            for (int c = 0; c < 2; c++) {
                const int lo = c ? nal : 0, hi = c ? n : nal;
                double corr[kSumVals];
#pragma unroll
                for (int k = 0; k < kSumVals; k++) corr[k] = 0.0;
                int m = 0, listed = 0, sub_n = 0;
                double sub_hh = 0.0;
                const double rx = vs > 0.0 ? 1.0 / (sqrt(s2c[c]) * vs) : 0.0;
                auto flush = [&](int k) {
                    weigh_rows<true>(scr, list, k, lane, true, nullptr, rx, st.weight_fn, last, corr, nout, sub_n, sub_hh);
                    listed += k;
                };
                if (st.robust)
                    for (int j0 = lo; j0 < hi; j0 += kWarp) {
                        const int j = j0 + lane;
                        append_rows(j < hi && beyond(j), j, list, m, lane, flush);
                    }
                __syncwarp();
                if (m > 0) flush(m);
                __syncwarp();
                if (lane == 0) w.all[c] = 0;
                if (listed) reduce_vals(corr, lane, w.C[c]);
                else if (lane < kSumVals) w.C[c][lane] = 0.0;
            }
            nout = warp_sum_int(nout);
            if (lane == 0) w.nout = nout;
            __syncwarp();
        }
}

// Class sums of a later round: w = wfun((h - A d) / sqrt(sigma_c^2 + y)) with the previous round's
// (d, y).  z = (h - A d) isd in FP32 from truncated values: its error is below
// 2^-19 isd (|h| + sum |A_k d_k|) (truncation 2^-23 of each factor, ten roundings of 2^-24).  Rows that
// the unit-weight sums do not hold are added with their weights, the others that may exceed 2 have
// (1 - w) taken off.  Their |h| is below two robust scales, but the rounds may still reject many of
// them: where more than a third of a class's rows or a quarter of its sum of h^2 is taken off, the class is
// summed over all its rows instead, so that the difference loses less than a bit.
__global__ void __launch_bounds__(32 * kPassWarps) k_src_round(Settings st, int last, const int64_t* __restrict__ src_off,
                                                               const int32_t* __restrict__ src_nal,
                                                               const int32_t* __restrict__ src_order, int32_t n_src,
                                                               int batch, double* __restrict__ scratch,
                                                               SrcWork* __restrict__ work) {
    __shared__ uint32_t list_all[kPassWarps][32];
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
    uint32_t* list = list_all[wib];
    const int step = gridDim.x * kPassWarps * batch;
    for (int base = (blockIdx.x * kPassWarps + wib) * batch; base < n_src; base += step)
        for (int q = base; q < min(base + batch, n_src); q++) {
            const int i = src_order[q];
            SrcWork& w = work[i];
            if (w.flags != 1) continue;
            const int64_t o0 = src_off[i];
            const int n = (int)(src_off[i + 1] - o0), nal = src_nal[i];
            double* scr = scratch + (size_t)o0 * kScr;
            double d[5];
            float df[5];
#pragma unroll
            for (int k = 0; k < 5; k++) { d[k] = w.d[k]; df[k] = (float)d[k]; }
            int nout = 0;
            for (int c = 0; c < 2; c++) {
                const int lo = c ? nal : 0, hi = c ? n : nal;
                const double isd = w.isd[c];
                const float isf = (float)isd;
                double corr[kSumVals];
#pragma unroll
                for (int k = 0; k < kSumVals; k++) corr[k] = 0.0;
                int m = 0, listed = 0, sub_n = 0;
                double sub_hh = 0.0;
                const int nout0 = nout;
                auto flush = [&](int k) {
                    weigh_rows<false>(scr, list, k, lane, false, d, isd, st.weight_fn, last, corr, nout, sub_n, sub_hh);
                    listed += k;
                };
                auto screen = [&](double h, const double A[5]) {
                    const float hf = trunc_f32(h);
                    float Rf = hf, S = fabsf(hf);
#pragma unroll
                    for (int k = 0; k < 5; k++) {
                        const float t = trunc_f32(A[k]) * df[k];
                        Rf -= t;
                        S += fabsf(t);
                    }
                    return !((fabsf(Rf) + S * 1.9073486e-6f) * isf < 2.0f);
                };
                for (int j0 = lo; j0 < hi; j0 += 2 * kWarp) {   // two rows in flight per lane
                    const int ja = j0 + lane, jb = ja + kWarp;
                    double ha = 0.0, hb = 0.0, Aa[5], Ab[5];
                    long long wa = 0, wb = 0;   // weight slots: 1, or 0 for a row beyond
                    if (ja < hi) {
                        row_load(scr + (size_t)ja * kScr, ha, Aa);
                        wa = __double_as_longlong(scr[(size_t)ja * kScr + 6]);
                    }
                    if (jb < hi) {
                        row_load(scr + (size_t)jb * kScr, hb, Ab);
                        wb = __double_as_longlong(scr[(size_t)jb * kScr + 6]);
                    }
                    const bool ca = ja < hi && (wa == 0 || screen(ha, Aa));
                    const bool cb = jb < hi && (wb == 0 || screen(hb, Ab));
                    append_rows(ca, ja, list, m, lane, flush);
                    append_rows(cb, jb, list, m, lane, flush);
                }
                __syncwarp();
                if (m > 0) flush(m);
                __syncwarp();
                const bool all = 3 * warp_sum_int(sub_n) > hi - lo || 4.0 * warp_sum(sub_hh) > w.T[c][20];
                if (all) {
                    double sums[kSumVals];   // (in memory: corr stays in registers)
                    int cnt = 0;
                    direct_rows(scr, lo, hi, list, lane, d, isd, st.weight_fn, last, sums, cnt);
                    nout = nout0 + cnt;
#pragma unroll
                    for (int k = 0; k < kSumVals; k++) corr[k] = sums[k];
                }
                if (lane == 0) w.all[c] = all;
                if (listed) reduce_vals(corr, lane, w.C[c]);
                else if (lane < kSumVals) w.C[c][lane] = 0.0;
            }
            nout = warp_sum_int(nout);
            if (lane == 0) w.nout = nout;
        }
}

// Direct class sums of one round, a block per source.  Every row is weighted: w = wfun(h rx) in
// round 0 (kSumFirst, rx in SrcWork::isd), wfun((h - A d) isd) later (kSumLater), 1 for plain
// weights (kSumOne).  Lane partials over the rows lane, lane + 32, ... of each class, then the 32
// partials of a value are added in lane order.  last: w goes to the scratch row.
//
// Bound by FP64 instructions (64 cycles each on a sub-partition, whatever the active lanes), so
// the four warps split them without doing any twice: the arguments z by chunks of 32 rows, the
// products by the row of A that they share.  Only rows with |z| >= 2 are listed for the weight
// function, for full warps of its polynomial, exponential and division.  With a warp per
// source and the weight function in every row: 800 sources of 165 45 us a round (the largest one's
// chain), 3000 81, 8000 of 840 512; so 28, 61, 470
// (10,000 of 165: 181).
enum SumMode { kSumFirst, kSumLater, kSumOne };
constexpr int kSumChunks = 16;     // chunks of 32 rows between two flushes of the list
struct SumShared {
    double red[kRedVals * kRedStride];
    double w[kSumChunks * kWarp];      // weights of the group's rows
    double z[kSumChunks * kWarp];      // listed arguments and their rows
    uint16_t slot[kSumChunks * kWarp];
    int m[2], nout;
};

// the products of one row of A (kRole = 0, 1, 2 with sum w h^2, or 3 with row 4) over a group's chunks
template <int kRole>
__device__ __forceinline__ void sum_role(double* scr, SumShared& sh, int q0, int q1, int n_al, int nal, int n, int lane,
                                         bool last, double (&v)[7]) {
    for (int q = q0; q < q1; q++) {
        const bool ac = q >= n_al;
        if (q == n_al) {
            // the AL class is complete
            int k = 0;
#pragma unroll
            for (int b = kRole; b < 5; b++) sh.red[up5(kRole, b) * kRedStride + lane] = v[k++];
            sh.red[(15 + kRole) * kRedStride + lane] = v[k++];
            if (kRole == 2) sh.red[20 * kRedStride + lane] = v[k++];
            if (kRole == 3) {
                sh.red[up5(4, 4) * kRedStride + lane] = v[k++];
                sh.red[19 * kRedStride + lane] = v[k++];
            }
#pragma unroll
            for (int e = 0; e < 7; e++) v[e] = 0.0;
        }
        const int j = (ac ? nal + (q - n_al) * kWarp : q * kWarp) + lane;
        if (j < (ac ? n : nal)) {
            double* e = scr + (size_t)j * kScr;
            const double w = sh.w[(q - q0) * kWarp + lane], h = e[0];
            if (kRole == 0 && last) e[6] = w;
            const double wa = w * e[1 + kRole];
            int k = 0;
#pragma unroll
            for (int b = kRole; b < 5; b++, k++) v[k] += wa * e[1 + b];
            v[k++] += wa * h;
            if (kRole == 2) v[k++] += w * h * h;
            if (kRole == 3) {
                const double w4 = w * e[5];
                v[k++] += w4 * e[5];
                v[k++] += w4 * h;
            }
        }
    }
}

__global__ void __launch_bounds__(128) k_src_sums(Settings st, int mode, int last, const int64_t* __restrict__ src_off,
                                                  const int32_t* __restrict__ src_nal,
                                                  const int32_t* __restrict__ src_order, int32_t n_src,
                                                  double* __restrict__ scratch, SrcWork* __restrict__ work) {
    __shared__ SumShared sh;
    const int tid = threadIdx.x, lane = tid & 31, wib = tid >> 5;
    if (tid < 2) sh.m[tid] = 0;
    if (tid == 2) sh.nout = 0;
    __syncthreads();
    int par = 0;
    for (int q_ = blockIdx.x; q_ < n_src; q_ += gridDim.x) {
        const int i = src_order[q_];
        SrcWork& w = work[i];
        if (w.flags != 1) continue;
        const int64_t o0 = src_off[i];
        const int n = (int)(src_off[i + 1] - o0), nal = src_nal[i];
        double* scr = scratch + (size_t)o0 * kScr;
        const int n_al = (nal + kWarp - 1) / kWarp, n_chunk = n_al + (n - nal + kWarp - 1) / kWarp;
        const double isd0 = w.isd[0], isd1 = w.isd[1];
        double d[5], v[7];
#pragma unroll
        for (int k = 0; k < 5; k++) d[k] = w.d[k];
#pragma unroll
        for (int k = 0; k < 7; k++) v[k] = 0.0;
        int cnt = 0;
        for (int q0 = 0; q0 < n_chunk; q0 += kSumChunks, par ^= 1) {
            const int q1 = min(q0 + kSumChunks, n_chunk);
            for (int e = tid; e < (q1 - q0) * kWarp; e += 128) sh.w[e] = 1.0;
            if (mode != kSumOne)
                for (int q = q0 + wib; q < q1; q += 4) {
                    const bool ac = q >= n_al;
                    const int j = (ac ? nal + (q - n_al) * kWarp : q * kWarp) + lane;
                    double z = 0.0;
                    if (j < (ac ? n : nal)) {
                        double h, A[5];
                        row_load(scr + (size_t)j * kScr, h, A);
                        const double f = ac ? isd1 : isd0;
                        if (mode == kSumFirst) z = h * f;
                        else z = (h - row_dot(A, d)) * f;
                    }
                    const bool cand = (__double2hiint(z) & 0x7fffffff) >= 0x40000000;   // |z| >= 2, or not a number
                    const unsigned ball = __ballot_sync(0xffffffffu, cand);
                    if (ball) {
                        int pos = 0;
                        if (lane == 0) pos = atomicAdd(&sh.m[par], __popc(ball));
                        pos = __shfl_sync(0xffffffffu, pos, 0) + __popc(ball & ((1u << lane) - 1u));
                        if (cand) {
                            sh.z[pos] = z;
                            sh.slot[pos] = (uint16_t)((q - q0) * kWarp + lane);
                        }
                    }
                }
            __syncthreads();
            const int m = sh.m[par];
            for (int e = tid; e < m; e += 128) {
                const double wt = wfun(sh.z[e], st.weight_fn);
                sh.w[sh.slot[e]] = wt;
                cnt += wt < 0.2;
            }
            if (tid == 0) sh.m[par ^ 1] = 0;
            __syncthreads();
            if (wib == 0) sum_role<0>(scr, sh, q0, q1, n_al, nal, n, lane, last, v);
            else if (wib == 1) sum_role<1>(scr, sh, q0, q1, n_al, nal, n, lane, last, v);
            else if (wib == 2) sum_role<2>(scr, sh, q0, q1, n_al, nal, n, lane, last, v);
            else sum_role<3>(scr, sh, q0, q1, n_al, nal, n, lane, last, v);
            __syncthreads();
        }
        // the last class (AL, with AC zero, if no AC rows follow)
        const int base = n_chunk > n_al ? kSumVals : 0;
        auto put = [&](int val, double x) {
            sh.red[(base + val) * kRedStride + lane] = x;
            if (base == 0) sh.red[(kSumVals + val) * kRedStride + lane] = 0.0;
            else if (n_al == 0) sh.red[val * kRedStride + lane] = 0.0;
        };
        int k = 0;
        for (int b = wib; b < 5; b++) put(up5(wib, b), v[k++]);
        put(15 + wib, v[k++]);
        if (wib == 2) put(20, v[k++]);
        if (wib == 3) {
            put(up5(4, 4), v[k++]);
            put(19, v[k++]);
        }
        cnt = warp_sum_int(cnt);
        if (lane == 0 && cnt) atomicAdd(&sh.nout, cnt);
        __syncthreads();
        // the partials of lanes without rows are zeros: one addition stands for them
        if (tid < 64 && lane < kSumVals) {
            const int cls = tid >> 5, val = cls * kSumVals + lane, rows = cls ? n - nal : nal, cols = min(rows, kWarp);
            const double* col = sh.red + val * kRedStride;
            double t = col[0];
            for (int e = 1; e < cols; e++) t += col[e];
            (&w.T[0][0])[val] = t + 0.0;
        } else if (tid == 64) {
            w.nout = sh.nout;
        }
        __syncthreads();
        if (tid == 64) sh.nout = 0;
    }
}

// the 5x5 algebra of one round, one thread (kPair: two neighbouring lanes) per source: y = 0 first,
// then the rational steps of the excess variance.  Leaves (d, 1 / sqrt(sigma_c^2 + y)) for the next
// round; after the last round the update, 1 / (sigma_c^2 + y) and the per-source results.
template <bool kPair>
__global__ void __launch_bounds__(128) k_src_solve5(Settings st, int last, const int64_t* __restrict__ src_off,
                                                    int32_t n_src, SrcOutPtrs out, SrcWork* __restrict__ work) {
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    const int h = kPair ? t & 1 : 0;
    const int it_ = kPair ? t >> 1 : t;
    const int i = it_ < n_src ? it_ : n_src - 1;   // lanes beyond the sources repeat the last one for the shuffles
    const bool mine = it_ < n_src && h == 0;
    if (!kPair && !mine) return;
    SrcWork& w = work[i];
    const int flags = w.flags;
    if (mine && (flags & 2) && last) {
        for (int k = 0; k < 5; k++) out.d[5 * (size_t)i + k] = 0.0;
        for (int k = 0; k < 25; k++) out.cov[25 * (size_t)i + k] = 0.0;
        out.eps2[i] = out.q[i] = out.dsig[i] = out.chi2[i] = 0.0;
        out.nu[i] = out.nout[i] = out.rankdef[i] = 0;
    }
    if (!kPair && flags != 1) return;
    const int n = (int)(src_off[i + 1] - src_off[i]);
    ClassSums S;
    HalfSums H;
    const int all[2] = {w.all[0], w.all[1]};
    auto sum_of = [&](int c, int k) { return (c ? all[1] : all[0]) ? w.C[c][k] : w.T[c][k] + w.C[c][k]; };
    if (kPair) {
        for (int c = 0; c < 2; c++)
            for (int k = 0; k < 10; k++) H.E[c][k] = sum_of(c, 10 * h + k);
        for (int k = 0; k < 15; k++) H.AA[k] = sum_of(h, k);
        for (int k = 0; k < 5; k++) H.Ah[k] = sum_of(h, 15 + k);
        H.hh = sum_of(h, 20);
    } else {
#pragma unroll
        for (int c = 0; c < 2; c++) {
#pragma unroll
            for (int k = 0; k < 15; k++) S.AA[c][k] = sum_of(c, k);
#pragma unroll
            for (int k = 0; k < 5; k++) S.Ah[c][k] = sum_of(c, 15 + k);
            S.hh[c] = sum_of(c, 20);
        }
    }
    const double s2c[2] = {w.s2c[0], w.s2c[1]};
    const int nout = w.nout, nu = n - nout - 5;
    double U[kU5], d[5], y = 0.0, Q, S2;
    int rd;
    auto solve = [&](double yy) {
        if (kPair) class_solve_pair(H, h, s2c, yy, st.pivot_tol, U, d, rd, Q, S2);
        else class_solve(S, s2c, yy, st.pivot_tol, U, d, rd, Q, S2);
    };
    solve(0.0);
    const double Q0 = Q;
    // the two lanes of a pair hold the same values; the pairs of a warp leave the loop together
    bool go = st.robust && flags == 1 && nu > 0 && Q0 > (double)nu;
    const double tol = 1e-12 * w.s2min;
    for (int it = 0; it < st.n_eps; it++) {
        if (kPair ? !__any_sync(0xffffffffu, go) : !go) break;
        const double dy = (1.0 - Q / (double)nu) * Q / (-S2);
        if (kPair) {
            // a pair that is done keeps its solution: solve again at its y (the same values)
            y = go ? fmax(0.0, y + dy) : y;
            solve(y);
            go = go && !(fabs(dy) <= tol);
        } else {
            y = fmax(0.0, y + dy);
            solve(y);
            if (fabs(dy) <= tol) break;
        }
    }
    if (!mine || flags != 1) return;
#pragma unroll
    for (int k = 0; k < 5; k++) w.d[k] = d[k];
    if (!last) {
        for (int c = 0; c < 2; c++) w.isd[c] = 1.0 / sqrt(s2c[c] + y);
        return;
    }
    for (int c = 0; c < 2; c++) w.isd[c] = 1.0 / (s2c[c] + y);
    double* sp = out.src + 5 * (size_t)i;
    const double cosd = cos(sp[1]);
    sp[0] += d[0] / cosd;
    for (int k = 1; k < 5; k++) sp[k] += d[k];
    for (int k = 0; k < 5; k++) out.d[5 * (size_t)i + k] = d[k];
    for (int c = 0; c < 5; c++) {
        double e[5] = {0, 0, 0, 0, 0};
        e[c] = 1.0;
        double x[5];
        chol5_solve(U, e, x);
        for (int k = 0; k < 5; k++) out.cov[25 * (size_t)i + 5 * k + c] = x[k];
    }
    out.eps2[i] = y;
    out.q[i] = Q;
    out.nu[i] = nu;
    out.nout[i] = nout;
    out.dsig[i] = nu > 0 ? (Q0 - (double)nu) / sqrt(2.0 * (double)nu) : 0.0;
    out.rankdef[i] = rd;
}

// hand-over records R = h - A d, W = w / (sigma_c^2 + y) and chi^2 of the class-sum sources
__global__ void __launch_bounds__(32 * kPassWarps) k_src_final(Settings st, const int64_t* __restrict__ src_off,
                                                               const int32_t* __restrict__ src_nal,
                                                               const int32_t* __restrict__ src_order, int32_t n_src,
                                                               int batch, const double* __restrict__ scratch,
                                                               const SrcWork* __restrict__ work, SrcOutPtrs out,
                                                               ObsRec* __restrict__ rec) {
    const int lane = threadIdx.x & 31;
    const int step = gridDim.x * kPassWarps * batch;
    for (int base = (blockIdx.x * kPassWarps + (threadIdx.x >> 5)) * batch; base < n_src; base += step)
        for (int q = base; q < min(base + batch, n_src); q++) {
            const int i = src_order[q];
            const SrcWork& w = work[i];
            if (w.flags != 1) continue;
            const int64_t o0 = src_off[i];
            const int n = (int)(src_off[i + 1] - o0), nal = src_nal[i];
            const double* scr = scratch + (size_t)o0 * kScr;
            const double d[5] = {w.d[0], w.d[1], w.d[2], w.d[3], w.d[4]};
            const double iw[2] = {w.isd[0], w.isd[1]};
            double chi = 0.0;
            for (int j = lane; j < n; j += kWarp) {
                const double* e = scr + (size_t)j * kScr;
                double h, A[5];
                row_load(e, h, A);
                const double R = h - (A[0] * d[0] + A[1] * d[1] + A[2] * d[2] + A[3] * d[3] + A[4] * d[4]);
                const double W = e[6] * (j < nal ? iw[0] : iw[1]);
                ObsRec* r = rec + (o0 + j);
                r->R = st.handover_h ? h : R;
                r->W = W;
                chi += W * R * R;
            }
            chi = warp_sum(chi);
            if (lane == 0) out.chi2[i] = chi;
        }
}

// ---------------------------------------------------------------------------------------
// General path (any sigma per observation): per-observation passes for every excess-noise step.
// Bound by FP64 instructions (64 cycles each on a sub-partition): 33 per observation of a round's
// normals and 15 of its Q, where divisions and square roots in every row made it about 135.  The
// weight is 1 up to |z| = 2, decided by z^2 = R^2 / (sigma^2 + y) without a root; the other rows
// (5 to 8%) are listed and worked off 32 at a time, so that their roots and exponentials run with
// full warps.  4.1M observations of 5000 sources, converged noise: 5.1 -> 3.5 ms, the first
// update with three noise steps in every round 13 -> 9.2 ms.
// ---------------------------------------------------------------------------------------
struct GenWork {
    double sums[kSumVals + 1];
    uint32_t list[32];
};

enum GenMode { kGenOne, kGenFirst, kGenRefresh, kGenKeep };

// Normal equations with W = w / (sigma^2 + y).  Weights: all 1 (kGenOne), w(h / (sigma vs))
// (kGenFirst, iz2 = 1 / vs^2), w(R / sqrt(sigma^2 + yp)) of R = h - A dp (kGenRefresh), or those
// of the row (kGenKeep); new weights go to the row.  nout: weights below 0.2 (left alone by kGenKeep).
template <GenMode kMode>
__device__ __forceinline__ void pass_normals(double* scr, int n, int lane, double y, const double* dp, double yp,
                                             double iz2, int wfn, GenWork& g, double* N, double* b, int& nout) {
    double v[kSumVals];
#pragma unroll
    for (int i = 0; i < kSumVals; i++) v[i] = 0.0;
    auto add = [&](double W, double h, const double A[5]) {
#pragma unroll
        for (int a = 0; a < 5; a++) {
            const double wa = W * A[a];
#pragma unroll
            for (int c = a; c < 5; c++) v[up5(a, c)] = fma(wa, A[c], v[up5(a, c)]);
            v[15 + a] = fma(wa, h, v[15 + a]);
        }
    };
    // z^2 of a row and 1 / (sigma^2 + y)
    auto z2_of = [&](double h, const double A[5], double s2, double& iv) {
        iv = rcp_pos(s2 + y);
        if (kMode == kGenFirst) return h * h * (iv * iz2);   // y = 0
        const double R = h - row_dot(A, dp);
        return R * R * (yp == y ? iv : rcp_pos(s2 + yp));
    };
    int cnt = 0, m = 0;
    auto flush = [&](int k) {
        if (lane >= k) return;
        double* e = scr + (size_t)g.list[lane] * kScr;
        double h, A[5], iv;
        row_load(e, h, A);
        const double w = wfun(sqrt(z2_of(h, A, e[7], iv)), wfn);
        e[6] = w;
        cnt += w < 0.2;
        add(w * iv, h, A);
    };
    for (int j0 = 0; j0 < n; j0 += kWarp) {
        const int j = j0 + lane;
        bool cand = false;
        if (j < n) {
            double* e = scr + (size_t)j * kScr;
            double h, A[5];
            row_load(e, h, A);
            const double2 ws = *reinterpret_cast<const double2*>(e + 6);
            if (kMode == kGenKeep) {
                add(ws.x * rcp_pos(ws.y + y), h, A);
            } else {
                double iv;
                if (kMode == kGenOne)
                    iv = rcp_pos(ws.y + y);
                else
                    cand = (__double2hiint(z2_of(h, A, ws.y, iv)) & 0x7fffffff) >= 0x40100000;   // 4 and above, or not a number
                if (!cand) {
                    e[6] = 1.0;
                    add(iv, h, A);
                }
            }
        }
        if (kMode == kGenFirst || kMode == kGenRefresh) append_rows(cand, j, g.list, m, lane, flush);
    }
    __syncwarp();
    if (m > 0) flush(m);
    reduce_vals(v, lane, g.sums);
    __syncwarp();
#pragma unroll
    for (int i = 0; i < 15; i++) N[i] = g.sums[i];
#pragma unroll
    for (int i = 0; i < 5; i++) b[i] = g.sums[15 + i];
    __syncwarp();
    if (kMode != kGenKeep) nout = warp_sum_int(cnt);
}

// Q(y) = sum w R^2 / (s2 + y) and S2 = sum w R^2 / (s2 + y)^2 for R = h - A d
__device__ __forceinline__ void pass_q(const double* scr, int n, int lane, const double* d, double y, double& Q,
                                       double& S2) {
    double q = 0.0, s = 0.0;
    for (int j = lane; j < n; j += kWarp) {
        const double* e = scr + (size_t)j * kScr;
        double h, A[5];
        row_load(e, h, A);
        const double2 ws = *reinterpret_cast<const double2*>(e + 6);
        const double R = h - row_dot(A, d);
        const double iv = rcp_pos(ws.y + y);
        const double t = ws.x * R * R * iv;
        q += t;
        s = fma(t, iv, s);
    }
    Q = warp_sum(q);
    S2 = warp_sum(s);
}

// One source, whole warp; the robust sigma vs is given.
__device__ __noinline__ void solve_general(const Settings& st, int i, int64_t o0, int n, const double* s5, double cosd,
                                           double* scr, double s2min, double vs, const SrcOutPtrs& out,
                                           ObsRec* __restrict__ rec, int lane, GenWork& g) {
    double d[5] = {0, 0, 0, 0, 0};
    double U[kU5];
    double y = 0.0, Q = 0.0, Q0 = 0.0;
    int nu = 0, nout = 0, rd = 0;
    const int rounds = st.robust ? st.n_rounds + 1 : 1;
    for (int rnd = 0; rnd < rounds; rnd++) {
        double N[15], b[5];
        double dprev[5] = {d[0], d[1], d[2], d[3], d[4]};
        const double yprev = y;
        y = 0.0;
        if (rnd > 0)
            pass_normals<kGenRefresh>(scr, n, lane, 0.0, dprev, yprev, 0.0, st.weight_fn, g, N, b, nout);
        else if (st.robust && vs > 0.0)
            pass_normals<kGenFirst>(scr, n, lane, 0.0, dprev, 0.0, 1.0 / (vs * vs), st.weight_fn, g, N, b, nout);
        else
            pass_normals<kGenOne>(scr, n, lane, 0.0, dprev, 0.0, 0.0, st.weight_fn, g, N, b, nout);
        nu = n - nout - 5;
        rd = chol5(N, U, st.pivot_tol);
        chol5_solve(U, b, d);
        double S2;
        pass_q(scr, n, lane, d, 0.0, Q, S2);
        Q0 = Q;
        if (st.robust && nu > 0 && Q0 > (double)nu) {
            const double tol = 1e-12 * s2min;
            for (int it = 0; it < st.n_eps; it++) {
                double dy = (1.0 - Q / (double)nu) * Q / (-S2);
                y = fmax(0.0, y + dy);
                pass_normals<kGenKeep>(scr, n, lane, y, dprev, 0.0, 0.0, st.weight_fn, g, N, b, nout);
                rd = chol5(N, U, st.pivot_tol);
                chol5_solve(U, b, d);
                pass_q(scr, n, lane, d, y, Q, S2);
                if (fabs(dy) <= tol) break;
            }
        }
        __syncwarp();
    }
    double chi = 0.0;
    for (int j = lane; j < n; j += kWarp) {
        const double* e = scr + (size_t)j * kScr;
        double h, A[5];
        row_load(e, h, A);
        const double R = h - row_dot(A, d);
        const double W = e[6] * rcp_pos(e[7] + y);
        ObsRec* r = rec + (o0 + j);
        r->R = st.handover_h ? h : R;
        r->W = W;
        chi += W * R * R;
    }
    chi = warp_sum(chi);
    if (lane == 0) {
        double* sp = out.src + 5 * (size_t)i;
        sp[0] = s5[0] + d[0] / cosd;
        sp[1] = s5[1] + d[1];
        sp[2] = s5[2] + d[2];
        sp[3] = s5[3] + d[3];
        sp[4] = s5[4] + d[4];
        for (int k = 0; k < 5; k++) out.d[5 * (size_t)i + k] = d[k];
        for (int c = 0; c < 5; c++) {
            double e[5] = {0, 0, 0, 0, 0};
            e[c] = 1.0;
            double x[5];
            chol5_solve(U, e, x);
            for (int k = 0; k < 5; k++) out.cov[25 * (size_t)i + 5 * k + c] = x[k];
        }
        out.eps2[i] = y;
        out.q[i] = Q;
        out.nu[i] = nu;
        out.nout[i] = nout;
        out.dsig[i] = nu > 0 ? (Q0 - (double)nu) / sqrt(2.0 * (double)nu) : 0.0;
        out.chi2[i] = chi;
        out.rankdef[i] = rd;
    }
    __syncwarp();
}

// sources whose sigma differs within a class: all rounds by per-observation passes
__global__ void __launch_bounds__(32 * kPassWarps) k_src_general(Settings st, const int64_t* __restrict__ src_off,
                                                                 const int32_t* __restrict__ src_order, int32_t n_src,
                                                                 SrcOutPtrs out, ObsRec* __restrict__ rec,
                                                                 double* __restrict__ scratch,
                                                                 const SrcWork* __restrict__ work) {
    __shared__ __align__(16) GenWork gen[kPassWarps];
    const int lane = threadIdx.x & 31;
    const int nw = gridDim.x * kPassWarps;
    for (int q = blockIdx.x * kPassWarps + (threadIdx.x >> 5); q < n_src; q += nw) {
        const int i = src_order[q];
        const SrcWork& w = work[i];
        if (w.flags != 0) continue;
        const int64_t o0 = src_off[i];
        const int n = (int)(src_off[i + 1] - o0);
        double s5[5];
        for (int k = 0; k < 5; k++) s5[k] = out.src[5 * (size_t)i + k];
        solve_general(st, i, o0, n, s5, cos(s5[1]), scratch + (size_t)o0 * kScr, w.s2min, w.vs, out, rec, lane, gen[threadIdx.x >> 5]);
    }
}

// Residuals at the current parameters, one thread per observation (no update).
__global__ void k_evaluate(DevGeo G, const int64_t* __restrict__ t_ns, const uint32_t* __restrict__ meta,
                           const double* __restrict__ mu, const int32_t* __restrict__ obs_src, int64_t n_obs,
                           const double* __restrict__ src, const double* __restrict__ att,
                           const double* __restrict__ cal, double* __restrict__ R) {
    for (int64_t o = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; o < n_obs; o += (int64_t)gridDim.x * blockDim.x) {
        SrcGeo S;
        source_geo(src + 5 * (size_t)obs_src[o], S);
        uint32_t m = meta[o];
        ObsOut ob;
        observe<0>(G, S, t_ns[o], m, (G.cg.on || meta_kind(m)) ? mu[o] : 0.0, att, cal, ob);
        R[o] = ob.R;
    }
}

// the observation pass of the S block: source geometry, then the model at every observation
void launch_obs_pass(const DevGeo& G, const AttNoise& an, const int64_t* t_ns, const uint32_t* meta, const float* sigma,
                     const double* mu, const int32_t* obs_src, int64_t n_obs, int32_t n_src, const double* src,
                     const double* att, const double* cal, ObsRec* rec, double* geo, double* scratch,
                     uint64_t* skey, const Shapes& sh, cudaStream_t stream) {
    k_src_geo<<<n_src > 0 ? (n_src + 31) / 32 : 1, 32, 0, stream>>>(n_src, src, geo);
    const int th = sh.obs_threads;
    int64_t fb = (n_obs + th - 1) / th;
    if (fb > 152 * (int64_t)sh.obs_bps) fb = 152 * (int64_t)sh.obs_bps;
    if (fb < 1) fb = 1;
    k_obs_forward<<<(int)fb, th, 0, stream>>>(G, an, n_obs, t_ns, meta, sigma, mu, obs_src, geo, att, cal, scratch, skey,
                                              rec);
}

// The inner iteration of the S block on the scratch rows of the observation pass.  corrections:
// rounds correct unit-weight sums by the rows beyond |z| = 2; else each round sums every row.
void launch_source_solve(const Settings& st, bool corrections, const int64_t* src_off, const int32_t* src_nal,
                         const int32_t* src_order, int32_t n_src, const SrcOutPtrs& out, ObsRec* rec, double* scratch,
                         const uint64_t* skey, SrcWork* work, const Shapes& sh, cudaStream_t stream) {
    if (n_src == 0) return;
    // consecutive sources of the largest-first order per warp and step: one, unless the autotuner
    // chose more (grids of at most 16 blocks per SM, a warp per source up to 9728 sources)
    const int batch = sh.src_batch > 0 ? sh.src_batch : 1;
    const int64_t warps = ((int64_t)n_src + batch - 1) / batch;
    int64_t blocks = (warps + kPassWarps - 1) / kPassWarps;
    if (blocks > 152 * 16) blocks = 152 * 16;
    const int nb = (int)blocks, th = 32 * kPassWarps;
    const int rounds = st.robust ? st.n_rounds + 1 : 1;
    // a warp of 5x5 algebra is a chain of FP64 instructions (64 cycles each): two lanes per source and
    // one warp per block while that leaves sub-partitions idle (800 sources: 38 us a round, one
    // lane 48), one lane beyond (30,000 sources: 100 us)
    const bool pair = n_src <= 152 * 4 * 16;
    constexpr size_t first_smem = kPassWarps * sizeof(SelWork);
    for (int r = 0; r < rounds; r++) {
        const int last = r == rounds - 1;
        if (r == 0 && corrections)
            k_src_first<false><<<nb, th, first_smem, stream>>>(st, src_off, src_nal, src_order, n_src, batch, scratch, skey,
                                                               work);
        else if (corrections)
            k_src_round<<<nb, th, 0, stream>>>(st, last, src_off, src_nal, src_order, n_src, batch, scratch, work);
        else {
            if (r == 0)
                k_src_first<true><<<nb, th, first_smem, stream>>>(st, src_off, src_nal, src_order, n_src, batch, scratch,
                                                                  skey, work);
            const int mode = !st.robust ? kSumOne : (r == 0 ? kSumFirst : kSumLater);
            k_src_sums<<<n_src < 152 * 64 ? n_src : 152 * 64, 128, 0, stream>>>(st, mode, last, src_off, src_nal,
                                                                                src_order, n_src, scratch, work);
        }
        if (pair) k_src_solve5<true><<<(2 * n_src + 31) / 32, 32, 0, stream>>>(st, last, src_off, n_src, out, work);
        else k_src_solve5<false><<<(n_src + 127) / 128, 128, 0, stream>>>(st, last, src_off, n_src, out, work);
    }
    k_src_final<<<nb, th, 0, stream>>>(st, src_off, src_nal, src_order, n_src, batch, scratch, work, out, rec);
    k_src_general<<<nb, th, 0, stream>>>(st, src_off, src_order, n_src, out, rec, scratch, work);
}

// kernels of one call: sums (a first pass and one pass per further round, or one per round) and 5x5 algebra of
// every round, the hand-over records and the per-observation path
int source_solve_kernels(const Settings& st, bool corrections) {
    const int rounds = st.robust ? st.n_rounds + 1 : 1;
    return 1 + (corrections ? rounds - 1 : rounds) + rounds + 2;
}

void launch_src_geo(int32_t n_src, const double* src, double* geo, cudaStream_t s) {
    k_src_geo<<<n_src > 0 ? (n_src + 31) / 32 : 1, 32, 0, s>>>(n_src, src, geo);
}

void launch_evaluate(const DevGeo& G, const int64_t* t_ns, const uint32_t* meta, const double* mu,
                     const int32_t* obs_src, int64_t n_obs, const double* src, const double* att, const double* cal,
                     double* R, cudaStream_t stream) {
    int blocks = (int)((n_obs + 255) / 256);
    if (blocks > 152 * 32) blocks = 152 * 32;
    if (blocks < 1) blocks = 1;
    k_evaluate<<<blocks, 256, 0, stream>>>(G, t_ns, meta, mu, obs_src, n_obs, src, att, cal, R);
}

}  // namespace agis
