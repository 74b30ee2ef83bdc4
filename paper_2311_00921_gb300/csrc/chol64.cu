// Cholesky factor and inverse of 64 x 64 FP64 blocks, one CTA per tree node.
//
// The FP64 pipe retires half a lane per clock in each quarter of an SM, so a
// warp-wide DFMA costs 64 clocks whatever its neighbours do: a block factored by
// one warp (one lane a row) leaves three quarters of the pipe idle and pays a
// square root and a division, tens of such instructions each, per column.  Here
// four warps share a 32 x 32 diagonal block, each owning every fourth column of
// L and every fourth row of L⁻¹ in registers; a column costs one inverse square
// root (a FP32 estimate and one third-order Newton step: five FP64 instructions),
// one barrier, and at most 24 DFMA a warp.  The 64 x 64 block is two such blocks, the
// rows below the first eliminated with it (by substitution: a product with the
// inverse instead, as fast, loses accuracy with the block's condition number), and
// three 32 x 32 products.
#include "chol64.cuh"
#include "common.cuh"

namespace {

constexpr int kT = 128;   // threads
constexpr int kN = 64;    // order of the block
constexpr int kP = 65;    // pitch of its columns in shared memory

// factor and inverse of the 32 x 32 diagonal block at offset o: S (L, lower) and X;
// BELOW: the next 32 rows of S too, L21 = A21 L⁻ᵀ.  Columns from `cols` on are those of
// the identity and left out (root of order 8: FP32 factor of five levels 392 -> 373 us).
template <bool BELOW>
HSS_DEVINL void factor32(double* S, double* X, int o, int cols, double (*col)[64],
                         double (*xrow)[32], int level, int node, int col0, int* status) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  double a[8], x[8];   // a: column w + 4 u of the block (lane = row); x: row w + 4 u of L⁻¹
  double a2[8];        // the column's rows 32 + lane
#pragma unroll
  for (int u = 0; u < 8; ++u) {
    const int t = w + 4 * u;
    a[u] = lane >= t ? S[(o + t) * kP + o + lane] : 0.0;
    x[u] = lane == t ? 1.0 : 0.0;
    if (BELOW) a2[u] = S[(o + t) * kP + o + 32 + lane];
  }
#pragma unroll
  for (int j = 0; j < 32; ++j) {
    if (j >= cols) break;
    const int buf = j & 1, u = j >> 2;
    if (w == (j & 3)) {
      const double d = __shfl_sync(0xffffffffu, a[u], j);
      double inv = 0.0, s = 0.0;
      if (d > 0.0) {
        inv = inv_sqrt(d);
        s = sqrt_from(d, inv);
      } else if (lane == 0) {
        report_failure(status, -3 /*NOT_SPD*/, level, node, col0 + o + j);
      }
      const double v = a[u] * inv;
      a[u] = lane == j ? s : v;
      x[u] *= inv;
      col[buf][lane] = lane > j ? v : 0.0;
      if (BELOW) col[buf][32 + lane] = a2[u] *= inv;
      xrow[buf][lane] = x[u];
    }
    __syncthreads();
    if (j < 31) {
      const double c = col[buf][lane], xr = xrow[buf][lane];
      const double c2 = BELOW ? col[buf][32 + lane] : 0.0;
#pragma unroll
      for (int q = (j + 1) >> 2; q < 8; ++q) {
        const int t = w + 4 * q;
        if (t > j) {
          const double l = col[buf][t];
          a[q] = fma(-c, l, a[q]);
          if (BELOW) a2[q] = fma(-c2, l, a2[q]);
          x[q] = fma(-l, xr, x[q]);
        }
      }
    }
  }
#pragma unroll
  for (int u = 0; u < 8; ++u) {
    const int t = w + 4 * u;
    if (lane >= t) S[(o + t) * kP + o + lane] = a[u];
    if (BELOW) S[(o + t) * kP + o + 32 + lane] = a2[u];
    X[(o + lane) * kP + o + t] = x[u];
  }
  __syncthreads();
}

// 32 x 32 product of blocks in shared memory, out(i, j) = Σ_k A(i, k) B(k, j),
// i = lane, j = w + 4 u: A(i, k) = A[k as + i], B(k, j) = B[k bk + j bj]; terms
// with k outside [lo, hi] of their column are zero and left out
template <typename Keep>
HSS_DEVINL void product32(const double* A, int as, const double* B, int bk, int bj,
                          double (&out)[8], Keep keep) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
#pragma unroll
  for (int u = 0; u < 8; ++u) out[u] = 0.0;
#pragma unroll 4
  for (int k = 0; k < 32; ++k) {
    const double a = A[k * as + lane];
#pragma unroll
    for (int u = 0; u < 8; ++u)
      if (keep(k, w + 4 * u)) out[u] = fma(a, B[k * bk + (w + 4 * u) * bj], out[u]);
  }
}

// high word without the sign
HSS_DEVINL int high(double v) { return __double2hiint(v) & 0x7fffffff; }

// *flag = 1 where the block needs no correction (see chol64.cuh): max|L| max|L⁻¹| < 16 at
// most, from the threads' largest high words; h: shared scratch
HSS_DEVINL void block_flag(int hl, int hx, int* h, int* flag) {
  if (threadIdx.x < 2) h[threadIdx.x] = 0;
  __syncthreads();
  hl = __reduce_max_sync(0xffffffffu, hl);
  hx = __reduce_max_sync(0xffffffffu, hx);
  if ((threadIdx.x & 31) == 0) {
    atomicMax(h, hl);
    atomicMax(h + 1, hx);
  }
  __syncthreads();
  if (threadIdx.x == 0) *flag = (h[0] >> 20) + (h[1] >> 20) - 2 * 1023 <= 2;
}

// the same for the kb x kb blocks, kb <= 128, one CTA of 128 threads per node
__global__ void __launch_bounds__(2 * kN)
inv_flag_kernel(const double* __restrict__ Lb, int ldl, long long sL, const double* __restrict__ Xb,
                int ldx, long long sX, int kb, int* flag, int flag_stride) {
  __shared__ int hmax[2];
  const long long node = blockIdx.x;
  const double *L = Lb + node * sL, *X = Xb + node * sX;
  const int i = threadIdx.x;
  int hl = 0, hx = 0;
  if (i < kb) {
#pragma unroll 16
    for (int j = 0; j < kb; ++j) {   // zeros above the diagonals
      hl = max(hl, high(L[i + (long long)j * ldl]));
      hx = max(hx, high(X[i + (long long)j * ldx]));
    }
  }
  block_flag(hl, hx, hmax, flag + node * flag_stride);
}

__global__ void __launch_bounds__(kT)
chol64_kernel(double* Mb, int ldm, long long sM, int kb, double* Xb, int ldx, long long sX,
              int above, double* Pb, int rows, double* part, int level, int node0, int col0,
              int* status, int accumulate, int* flag, int flag_stride) {
  const long long node = blockIdx.x;
  double* M = Mb + node * sM;
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  if (blockIdx.y > 0) {   // the rows below the block, for the product that solves them
    double* P = Pb + node * 64 * rows;
    const int step = (gridDim.y - 1) * kT;
    for (int e = (blockIdx.y - 1) * kT + tid; e < rows * kb; e += step)
      P[e] = M[kb + e % rows + (long long)(e / rows) * ldm];
    return;
  }
  extern __shared__ __align__(16) double sm[];
  double* S = sm;
  double* X = sm + kN * kP;
  __shared__ double col[2][64], xrow[2][32];
  __shared__ int hmax[2];
  for (int e = tid; e < kN * kN; e += kT) {
    const int i = e % kN, j = e / kN;
    S[j * kP + i] = (i < kb && j <= i) ? M[i + (long long)j * ldm] : (i == j ? 1.0 : 0.0);
    X[j * kP + i] = 0.0;
  }
  __syncthreads();
  factor32<true>(S, X, 0, kb, col, xrow, level, node0 + (int)node, col0, status);
  if (kb > 32) {
    double o[8];
    product32(S + 32, kP, S + 32, kP, 1, o, [](int, int) { return true; });
#pragma unroll
    for (int u = 0; u < 8; ++u)
      if (lane >= w + 4 * u) S[(32 + w + 4 * u) * kP + 32 + lane] -= o[u];
    __syncthreads();
    factor32<false>(S, X, 32, kb - 32, col, xrow, level, node0 + (int)node, col0, status);
    // X21 = -X22 (L21 X11); the product in brackets waits in X's upper block
    product32(S + 32, kP, X, 1, kP, o, [](int k, int j) { return k >= j; });
#pragma unroll
    for (int u = 0; u < 8; ++u) X[(32 + w + 4 * u) * kP + lane] = o[u];
    __syncthreads();
    product32(X + 32 * kP + 32, kP, X + 32 * kP, 1, kP, o, [](int, int) { return true; });
    __syncthreads();
#pragma unroll
    for (int u = 0; u < 8; ++u) X[(w + 4 * u) * kP + 32 + lane] = -o[u];
    __syncthreads();
  }
  double* Xo = Xb + node * sX;
  int hl = 0, hx = 0;
  for (int e = tid; e < kN * kb; e += kT) {
    const int i = e % kN, j = e / kN;
    if (i >= kb) continue;
    const double l = i >= j ? S[j * kP + i] : 0.0, x = i >= j ? X[j * kP + i] : 0.0;
    M[i + (long long)j * ldm] = l;
    Xo[i + (long long)j * ldx] = x;
    hl = max(hl, high(l));
    hx = max(hx, high(x));
  }
  block_flag(hl, hx, hmax, flag + node * flag_stride);
  for (int e = tid; e < above * kb; e += kT) {
    Xo[e % above - above + (long long)(e / above) * ldx] = 0.0;
    M[e % above - above + (long long)(e / above) * ldm] = 0.0;
  }
  if (w == 0 && part) {
    double s = lane < kb ? log(S[lane * kP + lane]) : 0.0;
    if (lane + 32 < kb) s += log(S[(lane + 32) * kP + lane + 32]);
    s = 2.0 * warp_sum(s);
    if (lane == 0) part[node] = accumulate ? part[node] + s : s;
  }
}

template <typename T>
__global__ void copy_rows_kernel(const T* __restrict__ src, int lds, long long ss,
                                 T* __restrict__ dst, int ldd, long long sd, int r, int nc) {
  const long long node = blockIdx.x;
  chain_wait();
  chain_release();
  for (int e = blockIdx.y * blockDim.x + threadIdx.x; e < r * nc; e += gridDim.y * blockDim.x) {
    const int i = e % r, j = e / r;
    dst[node * sd + i + (long long)j * ldd] = src[node * ss + i + (long long)j * lds];
  }
}

}  // namespace

cudaError_t launch_chol64(double* M, int ldm, long long sM, int kb, double* X, int ldx,
                          long long sX, int above, double* P, int rows, double* part, int level,
                          int node0, int col0, int* status, int nodes, bool accumulate,
                          int* flag, int flag_stride, cudaStream_t st) {
  if (kb < 1 || kb > kN || nodes < 1) return cudaErrorInvalidValue;
  const int smem = 2 * kN * kP * (int)sizeof(double);
  const cudaError_t e = fx_allow_smem((const void*)chol64_kernel, smem);
  if (e != cudaSuccess) return e;
  // copies: 8 elements a thread
  const int copies = rows > 0 ? (rows * kb + 8 * kT - 1) / (8 * kT) : 0;
  chol64_kernel<<<dim3(nodes, 1 + copies), kT, smem, st>>>(M, ldm, sM, kb, X, ldx, sX, above, P,
                                                           rows, part, level, node0, col0, status,
                                                           accumulate ? 1 : 0, flag, flag_stride);
  return cudaGetLastError();
}

cudaError_t launch_inv_flag(const double* L, int ldl, long long sL, const double* X, int ldx,
                            long long sX, int kb, int* flag, int flag_stride, int nodes,
                            cudaStream_t st) {
  if (kb < 1 || kb > 2 * kN || nodes < 1) return cudaErrorInvalidValue;
  inv_flag_kernel<<<nodes, 2 * kN, 0, st>>>(L, ldl, sL, X, ldx, sX, kb, flag, flag_stride);
  return cudaGetLastError();
}

template <typename T>
cudaError_t launch_copy_rows(const T* src, int lds, long long ss, T* dst, int ldd, long long sd,
                             int r, int nc, int nodes, cudaStream_t st) {
  if (r <= 0 || nc <= 0 || nodes <= 0) return cudaSuccess;
  return launch_chained(copy_rows_kernel<T>, dim3(nodes, (r * nc + 255) / 256), 256, 0, st, src, lds,
                        ss, dst, ldd, sd, r, nc);
}

template cudaError_t launch_copy_rows<double>(const double*, int, long long, double*, int, long long,
                                              int, int, int, cudaStream_t);
template cudaError_t launch_copy_rows<float>(const float*, int, long long, float*, int, long long, int,
                                             int, int, cudaStream_t);
