// Shared device helpers for the HSS-ULV kernels (sm_103a).
//
// Storage convention everywhere: column-major blocks, element (i, j) of a
// block with leading dimension ld at [i + j * ld]; blocks of one tree level
// are contiguous in node order with a fixed batch stride.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#define HSS_DEVINL __device__ __forceinline__

// Chained launches.  A level of the tree is a row of short kernels that each need the
// one before: launch_chained lets the next one's blocks be placed while this one still
// runs (programmatic dependent launch), which takes the placement, the kernel's
// parameters and its index arithmetic out of the chain.  chain_wait, before the first
// access to global memory, waits until the kernel before has ended and its writes are
// visible (so also every one before that); chain_release, called by every block right
// after it, lets the next kernel's blocks in where there is room, one kernel ahead.  A
// kernel started with launch_chained must call chain_wait in every block.
// Used by the narrow products and the row copies, the kernels of the sweeps: solve of
// N = 4096 294 -> 164 us, product with an operator of N = 1024 78 -> 52 us.  The factor's
// kernels are left out: their waiting blocks keep registers and shared memory from the
// other streams' kernels (with them chained a batch of ten took 14.5 ms, now 11.3).
HSS_DEVINL void chain_release() { asm volatile("griddepcontrol.launch_dependents;"); }
HSS_DEVINL void chain_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

template <typename... P, typename... A>
cudaError_t launch_chained(void (*kernel)(P...), dim3 grid, int threads, int smem, cudaStream_t st,
                           const A&... args) {
  cudaLaunchAttribute at{};
  at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at.val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = grid;
  cfg.blockDim = dim3(threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cfg.attrs = &at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kernel, P(args)...);
}

// status word layout (device int32[8]): [0] error code (0 = ok),
// [1] level, [2] node, [3] column, [4] timeout site
enum { ST_CODE = 0, ST_LEVEL = 1, ST_NODE = 2, ST_COL = 3, ST_SITE = 4 };

// record the first failure only
HSS_DEVINL void report_failure(int* status, int code, int level, int node, int col) {
  if (atomicCAS(status + ST_CODE, 0, code) == 0) {
    status[ST_LEVEL] = level;
    status[ST_NODE] = node;
    status[ST_COL] = col;
  }
}

// 1 / sqrt(d), d > 0: y0 from FP32 on d scaled to [1, 4) by a power of four, then
// y = y0 + y0 e (1/2 + 3/8 e), e = 1 - d y0² (Householder's iteration of third order,
// the binomial series of (1 - e)^(-1/2) up to e²): the estimate's 2^-22 becomes 2^-63
// before rounding.  Denormals, infinities and NaN take CUDA's square root and division.
HSS_DEVINL double inv_sqrt(double d) {
  const int hi = __double2hiint(d), ex = (hi >> 20) & 0x7ff;
  if (ex == 0 || ex == 0x7ff) return 1.0 / sqrt(d);
  const int e = ex - 1023, p = e >> 1;
  const double m =
      __hiloint2double((hi & 0xfffff) | ((1023 + e - 2 * p) << 20), __double2loint(d));
  const double y0 = (double)rsqrtf((float)m);
  const double r = fma(-m, y0 * y0, 1.0);
  const double y = fma(y0 * r, fma(0.375, r, 0.5), y0);
  return __hiloint2double(__double2hiint(y) - (p << 20), __double2loint(y));
}

// sqrt(d), d > 0, from inv = inv_sqrt(d): d inv and one step of Heron's (Newton's)
// iteration with the reciprocal at hand; infinity for infinity
HSS_DEVINL double sqrt_from(double d, double inv) {
  const double s = d * inv;
  return inv == 0.0 ? d : fma(fma(-s, s, d), 0.5 * inv, s);
}

// 1 / d, d > 0: y = y0 (1 + e + e²), e = 1 - d y0, y0 the FP32 reciprocal of d scaled to
// [1, 2) (Householder's iteration of third order, the geometric series up to e²).
// Results near the ends of the range take CUDA's division.
HSS_DEVINL double inv_pos(double d) {
  const int hi = __double2hiint(d), ex = (hi >> 20) & 0x7ff;
  if (ex < 32 || ex > 0x7ff - 32) return 1.0 / d;
  const double m = __hiloint2double((hi & 0xfffff) | (1023 << 20), __double2loint(d));
  const double y0 = (double)(1.f / (float)m);
  const double e = fma(-m, y0, 1.0);
  const double y = fma(y0, fma(e, e, e), y0);
  return __hiloint2double(__double2hiint(y) - ((ex - 1023) << 20), __double2loint(y));
}

template <typename T>
HSS_DEVINL T warp_sum(T v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// Sum over the 32 lanes of acc[k] lands in lane k (k < NV; NV = 16 or 32):
// a transposing butterfly, NV - 1 (+ NV for NV = 16) shuffles instead of NV * 5.
template <typename T, int NV>
HSS_DEVINL T warp_transpose_reduce(T (&acc)[NV], int lane) {
  if (NV == 16) {
#pragma unroll
    for (int i = 0; i < NV; ++i) acc[i] += __shfl_xor_sync(0xffffffffu, acc[i], 16);
  }
#pragma unroll
  for (int s = NV / 2; s >= 1; s >>= 1) {
    const bool upper = (lane & s) != 0;
#pragma unroll
    for (int i = 0; i < s; ++i) {
      const T send = upper ? acc[i] : acc[i + s];
      const T keep = upper ? acc[i + s] : acc[i];
      acc[i] = keep + __shfl_xor_sync(0xffffffffu, send, s);
    }
  }
  return acc[0];
}

// block-wide sum over blockDim.x threads (multiple of 32); `red` holds >= 32
// elements of shared scratch.  Every thread gets the total.
template <typename T>
HSS_DEVINL T block_sum(T v, T* red) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const int nw = blockDim.x >> 5;
  v = warp_sum(v);
  __syncthreads();
  if (lane == 0) red[wid] = v;
  __syncthreads();
  T t = (threadIdx.x < nw) ? red[threadIdx.x] : T(0);
  if (wid == 0) {
    t = warp_sum(t);
    if (lane == 0) red[0] = t;
  }
  __syncthreads();
  T r = red[0];
  return r;
}

// ---------------------------------------------------------------- batched GEMM
// C = alpha * op(A) * op(B) + beta * C for `batch` independent problems.
// op(X) = X or Xᵀ.  Column-major; batch strides in elements.
template <typename T>
void gemm_batched(bool transA, bool transB, int m, int n, int k, T alpha,
                  const T* A, int lda, long long sA, const T* B, int ldb, long long sB,
                  T beta, T* C, int ldc, long long sC, int batch, cudaStream_t st);

// M(i, j) = A(i, j) - sum_k [P(i,k) Q(j,k) + Q(i,k) P(j,k)] on the lower
// triangle (i >= j); P, Q are m x k.  A may alias M.
template <typename T>
void syr2k_lower_batched(int m, int k, const T* A, int lda, long long sA,
                         const T* P, int ldp, long long sP, const T* Q, int ldq, long long sQ,
                         T* M, int ldm, long long sM, int batch, cudaStream_t st);

// As syrk_lower_batched, and the result of node z (both triangles) also goes to
// the diagonal block at offset (z & 1) m of parent block z / 2 of PA (ld ldpa,
// stride sPA): the merge step of Alg. 2 fused into the last Schur update.
template <typename T>
void syrk_lower_merge_batched(int m, int k, const T* A, int lda, long long sA, const T* P,
                              int ldp, long long sP, T* M, int ldm, long long sM, T* PA, int ldpa,
                              long long sPA, int batch, cudaStream_t st);

// M(i, j) = A(i, j) - sum_k P(i,k) P(j,k) on the lower triangle; A may alias M.
template <typename T>
void syrk_lower_batched(int m, int k, const T* A, int lda, long long sA, const T* P, int ldp,
                        long long sP, T* M, int ldm, long long sM, int batch, cudaStream_t st);
