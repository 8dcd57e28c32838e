// Test harness for the inner iteration of the FP64 source update (host arrays in and out): given rows
// (h, A, sigma^2) of every source, AL rows first, either form of the weight rounds.
#include <cstring>

#include "k_source.cu"

extern "C" int src_solve_eval(int robust, int n_rounds, int n_eps, int weight_fn, int corrections, int n_src, int64_t n,
                              const int64_t* off, const int32_t* nal, const double* rows, double* src, double* eps2,
                              double* q, int* nu, int* nout, double* R, double* W) {
    using namespace agis;
    Settings st;
    memset(&st, 0, sizeof(st));
    st.robust = robust;
    st.n_rounds = n_rounds;
    st.n_eps = n_eps;
    st.weight_fn = weight_fn;
    st.pivot_tol = 1e-12;
    SrcOutPtrs o;
    memset(&o, 0, sizeof(o));
    int64_t* d_off = nullptr;
    int32_t *d_nal = nullptr, *order = nullptr;
    double* scr = nullptr;
    uint64_t* key = nullptr;
    ObsRec* rec = nullptr;
    SrcWork* work = nullptr;
    auto make = [](auto** p, size_t count) { return cudaMallocManaged(p, (count + 1) * sizeof(**p)) == cudaSuccess; };
    int rc = !(make(&d_off, n_src + 1) && make(&d_nal, n_src) && make(&order, n_src) && make(&scr, n * kScr) &&
               make(&key, n) && make(&rec, n) && make(&work, n_src) && make(&o.src, 5 * n_src) && make(&o.d, 5 * n_src) &&
               make(&o.eps2, n_src) && make(&o.q, n_src) && make(&o.dsig, n_src) && make(&o.chi2, n_src) &&
               make(&o.cov, 25 * n_src) && make(&o.nu, n_src) && make(&o.nout, n_src) && make(&o.rankdef, n_src));
    if (!rc) {
        memcpy(d_off, off, (n_src + 1) * sizeof(int64_t));
        memcpy(d_nal, nal, n_src * sizeof(int32_t));
        for (int i = 0; i < n_src; i++) order[i] = i;
        for (int64_t j = 0; j < n; j++) {
            double* e = scr + j * kScr;
            for (int k = 0; k < 6; k++) e[k] = rows[7 * j + k];
            e[6] = 1.0;
            e[7] = rows[7 * j + 6];
            const double x = e[0] / sqrt(e[7]);
            uint64_t b;
            memcpy(&b, &x, 8);
            key[j] = b >> 63 ? ~b : b | 0x8000000000000000ull;
        }
        memcpy(o.src, src, 5 * (size_t)n_src * sizeof(double));
        launch_source_solve(st, corrections != 0, d_off, d_nal, order, n_src, o, rec, scr, key, work, Shapes{}, 0);
        rc = cudaDeviceSynchronize() != cudaSuccess || cudaGetLastError() != cudaSuccess;
    }
    if (!rc) {
        memcpy(src, o.src, 5 * (size_t)n_src * sizeof(double));
        memcpy(eps2, o.eps2, n_src * sizeof(double));
        memcpy(q, o.q, n_src * sizeof(double));
        memcpy(nu, o.nu, n_src * sizeof(int));
        memcpy(nout, o.nout, n_src * sizeof(int));
        for (int64_t j = 0; j < n; j++) {
            R[j] = rec[j].R;
            W[j] = rec[j].W;
        }
    }
    for (void* p : {(void*)d_off, (void*)d_nal, (void*)order, (void*)scr, (void*)key, (void*)rec, (void*)work, (void*)o.src,
                    (void*)o.d, (void*)o.eps2, (void*)o.q, (void*)o.dsig, (void*)o.chi2, (void*)o.cov, (void*)o.nu,
                    (void*)o.nout, (void*)o.rankdef})
        cudaFree(p);
    return rc;
}
