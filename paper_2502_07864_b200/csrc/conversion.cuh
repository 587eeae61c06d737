// GQA -> MLA conversion on calibration activations (Sec. 4.2, 4.3; App. B, C, D): launchers.
// Everything here is fp32 on the device (the orthonormalisation inside the subspace iteration runs in fp64):
// the conversion is a one-off whose results are eigenvectors, which bf16 would not resolve.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include "common.cuh"
#include "transmla.h"

namespace transmla {
namespace conv {

// C[M,N] = alpha * op(A) op(B); op(A) is A [M,K] (ta = 0, row stride lda) or the transpose of A [K,M] (ta = 1), likewise
// op(B) from B [K,N] or B [N,K].  `batch` problems, strides in elements.  A barrier wait that gives up
// sets TRANSMLA_DEV_TIMEOUT in *dev_status (if there is one) and leaves NaN in the tiles of C that it concerns.
cudaError_t gemm_f32(int ta, int tb, int M, int N, int K, float alpha, const float* A, int lda, long long strideA,
                     const float* B, int ldb, long long strideB, float* C, int ldc, long long strideC, int batch,
                     int32_t* dev_status, cudaStream_t stream);
// The same of dense matrices by the kernel for single CTAs or pairs, with waits that give up at once (for a test).
cudaError_t gemm_f32_gives_up(int pairs, int M, int N, int K, const float* A, const float* B, float* C, int32_t* dev_status,
                              cudaStream_t stream);
// seg[G][2n][g*fold]: rows 0..n-1 the real parts, n..2n-1 the imaginary parts of group G's dimensions (App. B, C)
cudaError_t gather_segments(const float* K, int n, int g, int d, int fold, float* seg, cudaStream_t stream);
// Symmetric eigendecomposition of `batch` matrices of order m <= 128 (parallel cyclic Jacobi, one block each).
cudaError_t sym_eig(float* a, int batch, int m, float* eigvals, float* eigvecs, int32_t* dev_status, cudaStream_t stream);
cudaError_t rorope_apply(const float* X, int C, const float* U, int g, int d, int fold, float* Y, cudaStream_t stream);
cudaError_t row_norm_ratio(const float* k_nope, int n, int mk, const float* v, int mv, float* scratch, float* alpha_out,
                           cudaStream_t stream);
cudaError_t balance_concat(const float* k_nope, int n, int mk, const float* v, int mv, const float* alpha, float* Z,
                           cudaStream_t stream);
// Cholesky QR: Q [m,r] = Y L^-T with Y^T Y = L L^T, r <= 1024.  Scratch: partial [gram_slices(r)][r,r], G [r,r] and X [r,r]
// in fp64, X32 [r,r] (L^-T in fp32).  Q must not alias Y.  Sets TRANSMLA_DEV_NUMERIC if the Gram matrix is not positive definite.
// most_ctas: the factor's cluster is no larger (a power of two).
constexpr int kOrthCluster = 16;
int gram_slices(int r);
cudaError_t cholesky_qr(const float* Y, int m, int r, double* partial, double* G, double* X, float* X32, float* Q,
                        int32_t* dev_status, cudaStream_t stream, int most_ctas = kOrthCluster);
// The pass that leaves the result, in place: Q <- Q L^-T, rounded once.  P [m,r] is scratch; the rest as above.
cudaError_t cholesky_qr_last(float* Q, int m, int r, double* partial, double* G, double* X, float* X32, float* P,
                             int32_t* dev_status, cudaStream_t stream, int most_ctas = kOrthCluster);

// For a test: out [n][3] = the factor's 1 / sqrt(d), CUDA's rsqrt(d), the approximation that the first begins with.
cudaError_t inverse_roots(const double* d, int n, double* out, int32_t* dev_status, cudaStream_t stream);

}  // namespace conv
}  // namespace transmla
