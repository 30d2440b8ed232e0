// Internal interface of the digit-split products (split_gemm.cu).
#pragma once

#include "common.cuh"

namespace rbfsl {

constexpr int kSplitChunk = 128;  // inner entries per exact digit sum; rows of a solve's block

// Radial functions of the global method (Gaussian, inverse multiquadric) from r^2.
__device__ __forceinline__ double global_radial(int kind, double eps2, double d2) {
    return kind == RBFSL_GAUSS ? exp(-eps2 * d2) : rsqrt(1.0 + eps2 * d2);
}

// Triangular solves with an LU factor: factor holds what split_solve_prepare makes of LU once
// (inverted 64 x 64 diagonal blocks), scratch the digits of one block of right-hand sides.
size_t split_solve_factor_bytes(int64_t N);
size_t split_solve_scratch_bytes(int64_t N, int T);
int split_solve_prepare(const double *LU, int64_t N, void *factor, cudaStream_t s);
int split_solve(const double *LU, const int32_t *perm, int64_t N, const double *Q, int T, double *C, const void *factor,
                void *scratch, cudaStream_t s);

// out = A x for an M x K matrix A and T columns: split_apply with a stored A (RBFSL_F64 or
// RBFSL_F32X2, as x and out), split_eval with A_ik = phi(|P_i - X_k|), c FP64, out RBFSL_F64 or
// RBFSL_F32X2. ws: at least split_product_bytes(M, K, T, out's type), 256-byte aligned. The splits
// of the inner dimension are added in a fixed order.
size_t split_product_bytes(int64_t M, int64_t K, int T, int out_dtype);
int split_apply(const void *E, int64_t M, int64_t K, const void *x, int T, int dtype, void *out, void *ws,
                cudaStream_t s);
int split_eval(const double *P, int64_t M, const double *X, int64_t K, int kind, double eps, const double *c, int T,
               int out_dtype, void *out, void *ws, cudaStream_t s);

}  // namespace rbfsl
