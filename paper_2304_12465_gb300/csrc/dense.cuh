// Dense building blocks (dense.cu, digits.cu): products by digits, the Gram
// product, the blocked float64 Cholesky factorisation and the inverse of a
// lower-triangular factor.
#pragma once

#include "common.cuh"

namespace krr {

// C (N x nc, ldc) -= A (N x K, lda) B^T in float64, on the tensor cores by digits
// (digits.cuh): row c of B starts at B + rows[c] (rows NULL: B + c) with a step of
// ldb between its K entries and updates column cmap[c] of C (cmap NULL: c).  an2,
// bn2: the squared norms of the rows of A and of B (bn2 indexed like the rows), to
// rounding; they scale the rows, and an entry is off by about 2^-57 of the two
// norms' product.  img: dig_image_bytes(nc, K) bytes of scratch.  A bounded wait
// that gives up sets the flag that tc5_check_fault reads.
size_t dig_image_bytes(int nc, int K);
krr_status dig_gemm_sub(const double *A, int64_t lda, int64_t N, int K, const double *an2,
                        const double *B, int64_t ldb, const int64_t *rows, const double *bn2,
                        int nc, double *C, int64_t ldc, const int *cmap, uint4 *img,
                        cudaStream_t s);

// Lower triangle of C (r x r, column-major) = F^T F for F N x r column-major.
// float F: float32 products summed in float32 over 16-term chunks, the chunk
// sums in float-float (slices added in float64); double F: float64.  The
// strict upper triangle of C is untouched.
template <typename T>
krr_status gram_lower(const T *F, int64_t N, int r, double *C, cudaStream_t s);

// In-place lower Cholesky of the n x n column-major matrix A (lda): on return
// the lower triangle holds L with A = L L^T (the upper triangle is scratch).
// Returns KRR_ECHOL if a pivot is not positive (NaN included).
krr_status potrf_lower(double *A, int n, int64_t lda, cudaStream_t s);

// W (n x n, column-major) = L^{-1} for the lower-triangular L (lda); the upper
// triangle of W is zero.
krr_status trinv_lower(const double *L, int n, int64_t lda, double *W, cudaStream_t s);

// A(i, i) += v for i < n.
krr_status add_diagonal(double *A, int n, int64_t lda, double v, cudaStream_t s);

// B = A^T for n x n column-major matrices (no aliasing).
krr_status transpose_square(const double *A, int n, double *B, cudaStream_t s);

}  // namespace krr
