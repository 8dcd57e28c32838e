// Test harness for the quantile select of the source updates: a warp per set of values (host arrays
// in and out).  A set that is refused has its histogram cleared at once, as the radix select does.
#include "agis_internal.cuh"

__global__ void __launch_bounds__(32) k_select(const int64_t* off, const double* x, int* ok, double* out) {
    __shared__ __align__(16) agis::SelWork sw;
    const int lane = threadIdx.x, n = (int)(off[blockIdx.x + 1] - off[blockIdx.x]);
    const double* v = x + off[blockIdx.x];
    float lo = INFINITY, hi = -INFINITY;
    for (int j = lane; j < n; j += 32) {
        sw.keys[j] = agis::dkey(v[j]);
        lo = fminf(lo, agis::trunc_f32(v[j]));
        hi = fmaxf(hi, agis::trunc_f32(v[j]));
    }
    for (int o = 16; o > 0; o >>= 1) {
        lo = fminf(lo, __shfl_xor_sync(0xffffffffu, lo, o));
        hi = fmaxf(hi, __shfl_xor_sync(0xffffffffu, hi, o));
    }
    __syncwarp();
    double q[4] = {0, 0, 0, 0};
    const bool done = agis::select_quantiles(sw.keys, n, (int)floor(1.0 / 6.0 * (n - 1)), (int)floor(5.0 / 6.0 * (n - 1)), lo,
                                             hi, sw, lane, q);
    if (!done)
        for (int i = 0; i < 8; i++) sw.hist[lane * 8 + i] = 0;
    ok[blockIdx.x * 32 + lane] = done;
    if (lane == 0)
        for (int k = 0; k < 4; k++) out[4 * blockIdx.x + k] = q[k];
}

extern "C" int select_eval(int n_set, int64_t n, const int64_t* off, const double* x, int* ok, double* out) {
    int64_t* d_off = nullptr;
    double *d_x = nullptr, *d_out = nullptr;
    int* d_ok = nullptr;
    int rc = cudaMalloc(&d_off, (n_set + 1) * 8) != cudaSuccess || cudaMalloc(&d_x, n * 8) != cudaSuccess ||
             cudaMalloc(&d_ok, n_set * 32 * 4) != cudaSuccess || cudaMalloc(&d_out, n_set * 4 * 8) != cudaSuccess;
    if (!rc) {
        cudaMemcpy(d_off, off, (n_set + 1) * 8, cudaMemcpyHostToDevice);
        cudaMemcpy(d_x, x, n * 8, cudaMemcpyHostToDevice);
        k_select<<<n_set, 32>>>(d_off, d_x, d_ok, d_out);
        rc = cudaMemcpy(ok, d_ok, n_set * 32 * 4, cudaMemcpyDeviceToHost) != cudaSuccess ||
             cudaMemcpy(out, d_out, n_set * 4 * 8, cudaMemcpyDeviceToHost) != cudaSuccess;
    }
    cudaFree(d_off);
    cudaFree(d_x);
    cudaFree(d_ok);
    cudaFree(d_out);
    return rc;
}
