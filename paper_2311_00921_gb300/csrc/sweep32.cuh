// FP32 products with few columns and inverses of triangular blocks, for the sweeps
// of the mixed factors (sweep32.cu).
#pragma once
#include <cuda_runtime.h>

// C (m x n) = alpha op(A) B (+ Cin, may be null) for `batch` problems, n <= 16:
// op(A) = A (m x k) or Aᵀ (ta: A is k x m), B k x n, column-major.  Cin may be C.
cudaError_t narrow32(int m, int n, int k, const float* A, int lda, long long sA, bool ta,
                     const float* B, int ldb, long long sB, float alpha, const float* Cin,
                     int ldcin, long long sCin, float* C, int ldc, long long sC, int batch,
                     cudaStream_t st);

// Inverses of the diagonal blocks (128 columns each, the last one fewer) of the c x c
// lower triangle at the head of every matrix M (ld ldm, stride sM): block q at
// X + node sX + q lb², ld lb = min(c, 128), zeros above the diagonal.
cudaError_t launch_inv32(const float* M, int ldm, long long sM, int c, float* X, long long sX,
                         int nodes, cudaStream_t st);
