// ts_probe.cu -- the eigensolvers' FP64 products (tallskinny.cu) as calls of their own.
#include "spmm_probe.h"
#include "tallskinny.h"

using namespace spmm;

static bool bad_sizes(const void* a, const void* b, const void* c, int64_t lda, int32_t p, int64_t ldb, int32_t q,
                      int64_t n) {
    if (a && b && c && n >= 1 && p >= 1 && p <= 64 && q >= 1 && q <= 64 && lda >= p && ldb >= q) return false;
    set_error("spmm_probe_ts: need non-NULL arrays, n >= 1, 1 <= p, q <= 64 and leading dimensions that hold a row");
    return true;
}

extern "C" int spmm_probe_ts_tn(const double* A, int64_t lda, int32_t p, const double* B, int64_t ldb, int32_t q,
                                int64_t n, double* C, void* stream) {
    if (bad_sizes(A, B, C, lda, p, ldb, q, n)) return SPMM_ERR_ARG;
    cudaStream_t s = (cudaStream_t)stream;
    double* partial = nullptr;
    cudaError_t e = cudaMalloc((void**)&partial, ts_partial_doubles(n, 64) * sizeof(double));
    if (e == cudaSuccess) e = ts_tn(A, lda, p, B, ldb, q, n, partial, C, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    cudaFree(partial);
    return e == cudaSuccess ? SPMM_OK : cuda_fail(e, "spmm_probe_ts_tn");
}

extern "C" int spmm_probe_ts_nn(const double* A, int64_t lda, int32_t p, const double* C, int32_t q, double* Out,
                                int64_t ldo, int64_t n, double alpha, double beta, void* stream) {
    if (bad_sizes(A, C, Out, lda, p, ldo, q, n)) return SPMM_ERR_ARG;
    cudaStream_t s = (cudaStream_t)stream;
    cudaError_t e = ts_nn(A, lda, p, C, q, Out, ldo, n, alpha, beta, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    return e == cudaSuccess ? SPMM_OK : cuda_fail(e, "spmm_probe_ts_nn");
}

extern "C" int spmm_probe_chol_inv(const double* G, int32_t b, double* Rinv, int32_t* flag, void* stream) {
    if (!G || !Rinv || !flag || b < 1 || b > 32) {
        set_error("spmm_probe_chol_inv: need non-NULL arrays and 1 <= b <= 32");
        return SPMM_ERR_ARG;
    }
    cudaStream_t s = (cudaStream_t)stream;
    cudaError_t e = chol_inverse(G, b, Rinv, flag, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    return e == cudaSuccess ? SPMM_OK : cuda_fail(e, "spmm_probe_chol_inv");
}
