// Test harness for the interval blocks of the FP64 attitude accumulation: both kernels on the same
// records (host arrays in and out).
#include "k_attitude.cu"

extern "C" int att_blocks_eval(int64_t knot0, int64_t dt, int n_coef, double lambda2, int64_t n, const int64_t* t,
                               const double* R, const double* W, const double* g4, const int64_t* ivl_off,
                               const double* att, double* out_direct, double* out_moments) {
    const int n_iv = n_coef - 3;
    agis::DevGeo G;
    memset(&G, 0, sizeof(G));
    G.knot0_ns = knot0;
    G.knot_dt_ns = dt;
    G.inv_knot_dt = 1.0 / (double)dt;
    G.n_coef = n_coef;
    agis::ObsRec* rec = nullptr;
    uint32_t* perm = nullptr;
    int64_t* off = nullptr;
    double *da = nullptr, *blk = nullptr;
    const size_t nb = (size_t)n_iv * agis::kBlkVals * sizeof(double);
    int rc = cudaMallocManaged(&rec, (n + 1) * sizeof(agis::ObsRec)) != cudaSuccess ||
             cudaMallocManaged(&perm, (n + 1) * 4) != cudaSuccess || cudaMallocManaged(&off, (n_iv + 1) * 8) != cudaSuccess ||
             cudaMallocManaged(&da, 4 * (size_t)n_coef * 8) != cudaSuccess || cudaMallocManaged(&blk, 2 * nb) != cudaSuccess;
    if (!rc) {
        memset(blk, 0xff, 2 * nb);
        for (int64_t i = 0; i < n; i++) {
            const int64_t o = n - 1 - i;   // records in another order than time
            memset(&rec[o], 0, sizeof(agis::ObsRec));
            rec[o].t_ns = t[i];
            rec[o].R = R[i];
            rec[o].W = W[i];
            for (int c = 0; c < 4; c++) rec[o].g[c] = g4[4 * i + c];
            perm[i] = (uint32_t)o;
        }
        memcpy(off, ivl_off, (n_iv + 1) * 8);
        memcpy(da, att, 4 * (size_t)n_coef * 8);
        for (int m = 0; m < 2; m++)
            agis::launch_att_accum(G, lambda2, 0, perm, off, n_iv, rec, nullptr, da, blk + m * (nb / 8), m == 1,
                                   agis::Shapes{}, 0);
        rc = cudaDeviceSynchronize() != cudaSuccess || cudaGetLastError() != cudaSuccess;
    }
    if (!rc) {
        memcpy(out_direct, blk, nb);
        memcpy(out_moments, blk + nb / 8, nb);
    }
    cudaFree(rec);
    cudaFree(perm);
    cudaFree(off);
    cudaFree(da);
    cudaFree(blk);
    return rc;
}
