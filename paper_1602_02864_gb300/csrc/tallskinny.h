// tallskinny.h -- FP64 products of tall, narrow matrices (tallskinny.cu) and the Cholesky factor of a Gram matrix.
#pragma once

#include "internal.h"

namespace spmm {

// doubles of scratch that ts_tn needs for matrices of n rows and at most m <= 64 columns
size_t ts_partial_doubles(int64_t n, int m);
// out (p x q, row-major) = A^T B; A n x p, B n x q with leading dimensions
// lda, ldb; 1 <= p, q <= 64.  The sums have a fixed order.
cudaError_t ts_tn(const double* A, int64_t lda, int p, const double* B, int64_t ldb, int q, int64_t n,
                  double* partial, double* out, cudaStream_t s);
// Out (n x q) = beta Out + alpha A C; A n x p, C p x q row-major; 1 <= p, q <= 64; Out does not overlap A or C.
cudaError_t ts_nn(const double* A, int64_t lda, int p, const double* C, int q, double* Out, int64_t ldo, int64_t n,
                  double alpha, double beta, cudaStream_t s);
// the column norms squared of R = AU - U diag(theta) (n x q, contiguous): out[j] = sum_i R[i][j]^2
cudaError_t ts_residuals(const double* AU, const double* U, const double* theta, int q, int64_t n, double* partial,
                         double* out, cudaStream_t s);

// Rinv (b x b, upper) = R^-1 of the Cholesky factor G = R^T R, b <= 32 (eigs.cu); *flag = 1 and the identity
// where a pivot is not safely positive
cudaError_t chol_inverse(const double* G, int b, double* Rinv, int32_t* flag, cudaStream_t s);

}  // namespace spmm
