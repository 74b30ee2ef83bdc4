// FP64 products on the tensor cores by exact slicing (fxgemm.cu).
#pragma once
#include <cuda_runtime.h>

// One operand, rows x K, batched: element (row, k) is p1[k + row ld1] (kc) or
// p1[row + k ld1].  With p2 (in both operands of a call) K is twice the inner
// indices of each array: k >= K / 2 is the same in p2 at k - K / 2.
struct FxOperand {
  const double* p1;
  int ld1;
  long long s1;   // batch stride
  bool kc;        // K is the contiguous index
  const double* p2 = nullptr;
  int ld2 = 0;
  long long s2 = 0;
};

// C (m x n) = alpha a bᵀ + beta Cin for `batch` problems, a m x K and b n x K.
// lower: only elements on and below the diagonal (m = n).  PA (may be null):
// node z's result also goes, both triangles, to the diagonal block at offset
// (z & 1) m of parent block z / 2.  Cin may be C.  components: every element
// within about the bound of a DFMA chain, K 2^-53 Σ|a||b|; else (Householder
// transformations) within K 2^-58.5 of the largest |a| times the largest |b| of its row
// and column in each 128 inner indices.  skip (may be null): problem z is left out where
// skip[z skip_stride] is not zero, its C as it was.
cudaError_t fx_gemm(int m, int n, int K, const FxOperand& a, const FxOperand& b, double alpha,
                    double beta, const double* Cin, int ldcin, long long sCin, double* C, int ldc,
                    long long sC, int batch, bool lower, double* PA, int ldpa, long long sPA,
                    cudaStream_t st, bool components = true, const int* skip = nullptr,
                    int skip_stride = 0);

// opts a kernel into `bytes` of dynamic shared memory, once per device and kernel
cudaError_t fx_allow_smem(const void* kernel, int bytes);

// The FP64 products of the library, column-major with batch strides in elements
// (semantics of gemm_batched, syr2k_lower_batched, syrk_lower_batched and
// syrk_lower_merge_batched in common.cuh): sliced products except where the rule
// in fxgemm.cu leaves them on the FP64 pipe.
void dgemm_batched(bool transA, bool transB, int m, int n, int k, double alpha, const double* A,
                   int lda, long long sA, const double* B, int ldb, long long sB, double beta,
                   double* C, int ldc, long long sC, int batch, cudaStream_t st,
                   bool components = true);
void dsyr2k_lower_batched(int m, int k, const double* A, int lda, long long sA, const double* P,
                          int ldp, long long sP, const double* Q, int ldq, long long sQ, double* M,
                          int ldm, long long sM, int batch, cudaStream_t st);
// PA = null: no merge
void dsyrk_lower_batched(int m, int k, const double* A, int lda, long long sA, const double* P,
                         int ldp, long long sP, double* M, int ldm, long long sM, double* PA,
                         int ldpa, long long sPA, int batch, cudaStream_t st);
