// Cholesky factor and inverse of 64 x 64 FP64 blocks, one CTA per tree node.
//
// The FP64 pipe retires half a lane per clock in each quarter of an SM, so a
// warp-wide DFMA costs 64 clocks whatever its neighbours do: a block factored by
// one warp (one lane a row) leaves three quarters of the pipe idle and pays a
// square root and a division, tens of such instructions each, per column.  Here
// four warps share a 32 x 32 diagonal block, each owning every fourth column of
// L and every fourth row of L⁻¹ in registers; a column costs one inverse square
// root (a FP32 estimate and one third-order Newton step: five FP64 instructions),
// one barrier, and at most 16 DFMA a warp.  The 64 x 64 block is two such blocks
// and four 32 x 32 products.
#include "chol64.cuh"
#include "common.cuh"

namespace {

constexpr int kT = 128;   // threads
constexpr int kN = 64;    // order of the block
constexpr int kP = 65;    // pitch of its columns in shared memory

// factor and inverse of the 32 x 32 diagonal block at offset o: S (L, lower) and X
HSS_DEVINL void factor32(double* S, double* X, int o, double (*col)[32], double (*xrow)[32],
                         int level, int node, int col0, int* status) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  double a[8], x[8];   // a: column w + 4 u of the block (lane = row); x: row w + 4 u of L⁻¹
#pragma unroll
  for (int u = 0; u < 8; ++u) {
    const int t = w + 4 * u;
    a[u] = lane >= t ? S[(o + t) * kP + o + lane] : 0.0;
    x[u] = lane == t ? 1.0 : 0.0;
  }
#pragma unroll
  for (int j = 0; j < 32; ++j) {
    const int buf = j & 1, u = j >> 2;
    if (w == (j & 3)) {
      const double d = __shfl_sync(0xffffffffu, a[u], j);
      double inv = 0.0, s = 0.0;
      if (d > 0.0) {
        inv = inv_sqrt(d);
        s = d * inv;
        s = fma(fma(-s, s, d), 0.5 * inv, s);
      } else if (lane == 0) {
        report_failure(status, -3 /*NOT_SPD*/, level, node, col0 + o + j);
      }
      const double v = a[u] * inv;
      a[u] = lane == j ? s : v;
      x[u] *= inv;
      col[buf][lane] = lane > j ? v : 0.0;
      xrow[buf][lane] = x[u];
    }
    __syncthreads();
    if (j < 31) {
      const double c = col[buf][lane], xr = xrow[buf][lane];
#pragma unroll
      for (int q = (j + 1) >> 2; q < 8; ++q) {
        const int t = w + 4 * q;
        if (t > j) {
          const double l = col[buf][t];
          a[q] = fma(-c, l, a[q]);
          x[q] = fma(-l, xr, x[q]);
        }
      }
    }
  }
#pragma unroll
  for (int u = 0; u < 8; ++u) {
    const int t = w + 4 * u;
    if (lane >= t) S[(o + t) * kP + o + lane] = a[u];
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

__global__ void __launch_bounds__(kT)
chol64_kernel(double* Mb, int ldm, long long sM, int kb, double* Xb, int ldx, long long sX,
              int above, double* Pb, int rows, double* part, int level, int node0, int col0,
              int* status, int accumulate) {
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
  __shared__ double col[2][32], xrow[2][32];
  for (int e = tid; e < kN * kN; e += kT) {
    const int i = e % kN, j = e / kN;
    S[j * kP + i] = (i < kb && j <= i) ? M[i + (long long)j * ldm] : (i == j ? 1.0 : 0.0);
    X[j * kP + i] = 0.0;
  }
  __syncthreads();
  factor32(S, X, 0, col, xrow, level, node0 + (int)node, col0, status);
  if (kb > 32) {
    double o[8];
    // L21 = A21 X11ᵀ: X11(j, k), k <= j
    product32(S + 32, kP, X, kP, 1, o, [](int k, int j) { return k <= j; });
    __syncthreads();
#pragma unroll
    for (int u = 0; u < 8; ++u) S[(w + 4 * u) * kP + 32 + lane] = o[u];
    __syncthreads();
    product32(S + 32, kP, S + 32, kP, 1, o, [](int, int) { return true; });
#pragma unroll
    for (int u = 0; u < 8; ++u)
      if (lane >= w + 4 * u) S[(32 + w + 4 * u) * kP + 32 + lane] -= o[u];
    __syncthreads();
    factor32(S, X, 32, col, xrow, level, node0 + (int)node, col0, status);
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
  for (int e = tid; e < kN * kb; e += kT) {
    const int i = e % kN, j = e / kN;
    if (i >= kb) continue;
    if (i >= j) M[i + (long long)j * ldm] = S[j * kP + i];
    Xo[i + (long long)j * ldx] = i >= j ? X[j * kP + i] : 0.0;
  }
  for (int e = tid; e < above * kb; e += kT)
    Xo[e % above - above + (long long)(e / above) * ldx] = 0.0;
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
                          cudaStream_t st) {
  if (kb < 1 || kb > kN || nodes < 1) return cudaErrorInvalidValue;
  const int smem = 2 * kN * kP * (int)sizeof(double);
  const cudaError_t e = fx_allow_smem((const void*)chol64_kernel, smem);
  if (e != cudaSuccess) return e;
  // copies: 8 elements a thread
  const int copies = rows > 0 ? (rows * kb + 8 * kT - 1) / (8 * kT) : 0;
  chol64_kernel<<<dim3(nodes, 1 + copies), kT, smem, st>>>(M, ldm, sM, kb, X, ldx, sX, above, P,
                                                           rows, part, level, node0, col0, status,
                                                           accumulate ? 1 : 0);
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
