// Test harness for the integer reciprocal rcp_pos_int of the banded attitude solve: evaluates it
// and the correctly rounded division 1.0 / d on the same inputs (host arrays in and out).
#include "agis_internal.cuh"

__global__ void k_rcp_int(const double* __restrict__ d, double* __restrict__ y, double* __restrict__ q, int64_t n) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        y[i] = agis::rcp_pos_int(d[i]);
        q[i] = 1.0 / d[i];
    }
}

extern "C" int rcp_int_eval(const double* d_host, double* y_host, double* q_host, int64_t n) {
    double* buf = nullptr;
    const size_t b = (size_t)n * sizeof(double);
    if (cudaMalloc(&buf, 3 * b) != cudaSuccess) return 1;
    int rc = cudaMemcpy(buf, d_host, b, cudaMemcpyHostToDevice) != cudaSuccess;
    if (!rc) {
        k_rcp_int<<<152 * 4, 256>>>(buf, buf + n, buf + 2 * n, n);
        rc = cudaDeviceSynchronize() != cudaSuccess || cudaMemcpy(y_host, buf + n, b, cudaMemcpyDeviceToHost) != cudaSuccess ||
             cudaMemcpy(q_host, buf + 2 * n, b, cudaMemcpyDeviceToHost) != cudaSuccess;
    }
    cudaFree(buf);
    return rc;
}
