// Kernels of the mixed factors' sweeps (sweep32.cuh).
//
// A node's triangular sweep in one CTA is a chain of 32-column steps on 8 warps,
// 84 us a level of the tree at rank 128 with 16 columns whatever the node count.  With
// the 128 x 128 diagonal blocks inverted once, a level is two products per 128 eliminated
// columns and three for Q, each a launch over the whole level: a sweep of N = 262144
// 2.7 -> 1.3 ms (its factor read once: 0.12 ms).
#include "sweep32.cuh"

#include "common.cuh"
#include "fxgemm.cuh"

namespace {

// ------------------------------------------------------------------ products
// CTA: 64 rows and every column of one problem, 8 warps.  Warp w takes the chunks
// w, w + 8, .. of 16 inner indices on its own (no barrier), lane = rows lane and
// lane + 32: per index one coalesced load of A a row (Aᵀ: through the warp's own
// shared tile, read along its contiguous index), the row of B broadcast.  The
// warps' sums are added at the end.  Upper levels are bound by this chain, one chunk
// a warp at k <= 128; the leaves by reading A, for which two rows a lane halve the
// broadcasts per product.
constexpr int kRows = 64, kChunk = 16, kWarps = 8, kThreads = 32 * kWarps;

struct Narrow {
  int m, n, k, lda, ldb, ldcin, ldc, tiles;
  long long sA, sB, sCin, sC;
  float alpha;
  const float *A, *B, *Cin;
  float* C;
};

template <int NC, bool TA>
__global__ void __launch_bounds__(kThreads)
narrow32_kernel(const __grid_constant__ Narrow s) {
  constexpr int PB = NC + 4;   // pitch of B's rows: 16-byte aligned, few conflicts
  __shared__ float buf[kWarps][kRows * 17];
  __shared__ __align__(16) float bs[kWarps][kChunk * PB];
  const long long z = blockIdx.x / s.tiles;
  const int i0 = (int)(blockIdx.x % s.tiles) * kRows;
  const float* A = s.A + z * s.sA;
  const float* B = s.B + z * s.sB;
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  const int kk0 = lane & 15, half = lane >> 4;
  float acc[2][NC];
#pragma unroll
  for (int h = 0; h < 2; ++h)
#pragma unroll
    for (int j = 0; j < NC; ++j) acc[h][j] = 0.f;
  chain_wait();
  chain_release();
  for (int kc = kChunk * w; kc < s.k; kc += kChunk * kWarps) {
    float a[2][kChunk];
    if (TA) {
#pragma unroll
      for (int q = 0; q < kChunk; ++q)
#pragma unroll
        for (int h = 0; h < 2; ++h) {   // row half + 2 (q + 16 h), index kk0
          const int i = i0 + half + 2 * q + 32 * h;
          a[h][q] = i < s.m && kc + kk0 < s.k ? A[kc + kk0 + (long long)i * s.lda] : 0.f;
        }
    } else {
#pragma unroll
      for (int q = 0; q < kChunk; ++q)
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const int i = i0 + lane + 32 * h;
          a[h][q] = i < s.m && kc + q < s.k ? A[i + (long long)(kc + q) * s.lda] : 0.f;
        }
    }
#pragma unroll
    for (int q = 0; q < NC / 2; ++q) {
      const int j = half + 2 * q;
      bs[w][kk0 * PB + j] =
          j < s.n && kc + kk0 < s.k ? B[kc + kk0 + (long long)j * s.ldb] : 0.f;
    }
    if (TA) {
#pragma unroll
      for (int q = 0; q < kChunk; ++q)
#pragma unroll
        for (int h = 0; h < 2; ++h) buf[w][(half + 2 * q + 32 * h) * 17 + kk0] = a[h][q];
    }
    __syncwarp();
#pragma unroll
    for (int q = 0; q < kChunk; ++q) {
      const float a0 = TA ? buf[w][lane * 17 + q] : a[0][q];
      const float a1 = TA ? buf[w][(lane + 32) * 17 + q] : a[1][q];
#pragma unroll
      for (int j = 0; j < NC; j += 4) {
        const float4 b = *reinterpret_cast<const float4*>(&bs[w][q * PB + j]);
        const float bj[4] = {b.x, b.y, b.z, b.w};
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          acc[0][j + e] = fmaf(a0, bj[e], acc[0][j + e]);
          acc[1][j + e] = fmaf(a1, bj[e], acc[1][j + e]);
        }
      }
    }
    __syncwarp();
  }
#pragma unroll
  for (int h = 0; h < 2; ++h)
#pragma unroll
    for (int j = 0; j < NC; ++j) buf[w][(lane + 32 * h) * 17 + j] = acc[h][j];
  __syncthreads();
  for (int e = tid; e < kRows * s.n; e += kThreads) {
    const int r = e % kRows, j = e / kRows, i = i0 + r;
    if (i >= s.m) continue;
    float v = 0.f;
#pragma unroll
    for (int u = 0; u < kWarps; ++u) v += buf[u][r * 17 + j];
    v *= s.alpha;
    if (s.Cin) v += s.Cin[z * s.sCin + i + (long long)j * s.ldcin];
    s.C[z * s.sC + i + (long long)j * s.ldc] = v;
  }
}

// ------------------------------------------------------------------ inverses
// A CTA per block, a thread per column x of the inverse: 32 rows at a time in
// registers, first minus L's rows times the x known so far (L broadcast four rows a
// load, x from the thread's own column in shared memory), then the 32 x 32 triangle
// unrolled.  Rows above a warp's columns are zero and left out.
constexpr int kOrder = 128;
constexpr int kPL = kOrder + 4, kPX = kOrder + 1;
constexpr int kInvSmem = kOrder * (kPL + kPX + 1) * (int)sizeof(float);

__global__ void __launch_bounds__(kOrder)
inv32_kernel(const float* __restrict__ Mb, int ldm, long long sM, int c, float* __restrict__ Xb,
             long long sX, int lb) {
  extern __shared__ __align__(16) float smem[];
  float* Ls = smem;                    // L(i, k) at k kPL + i
  float* Xs = Ls + kOrder * kPL;       // X(i, j) at i kPX + j
  float* dinv = Xs + kOrder * kPX;
  const int k0 = kOrder * blockIdx.y, kb = min(kOrder, c - k0), kr = (kb + 31) & ~31;
  const float* M = Mb + blockIdx.x * sM + k0 + (long long)k0 * ldm;
  float* X = Xb + blockIdx.x * sX + (long long)blockIdx.y * lb * lb;
  const int tid = threadIdx.x, w = tid >> 5;
  for (int k = 0; k < kr; ++k) {
    const int i = tid;
    Ls[k * kPL + i] = (i >= k && i < kb) ? M[i + (long long)k * ldm] : (i == k ? 1.f : 0.f);
  }
  __syncthreads();
  dinv[tid] = tid < kr ? 1.f / Ls[tid * kPL + tid] : 1.f;
  __syncthreads();
  for (int I = 0; 32 * I < kr; ++I) {
    if (I < w) {
      for (int i = 0; i < 32; ++i) Xs[(32 * I + i) * kPX + tid] = 0.f;
      continue;
    }
    float acc[32];
#pragma unroll
    for (int i = 0; i < 32; ++i) acc[i] = 32 * I + i == tid ? 1.f : 0.f;
    for (int k = 32 * w; k < 32 * I; ++k) {
      const float x = Xs[k * kPX + tid];
#pragma unroll
      for (int i = 0; i < 32; i += 4) {
        const float4 l = *reinterpret_cast<const float4*>(Ls + k * kPL + 32 * I + i);
        acc[i] = fmaf(-l.x, x, acc[i]);
        acc[i + 1] = fmaf(-l.y, x, acc[i + 1]);
        acc[i + 2] = fmaf(-l.z, x, acc[i + 2]);
        acc[i + 3] = fmaf(-l.w, x, acc[i + 3]);
      }
    }
#pragma unroll
    for (int i = 0; i < 32; ++i) {
      const float x = acc[i] * dinv[32 * I + i];
      Xs[(32 * I + i) * kPX + tid] = x;
#pragma unroll
      for (int u = i + 1; u < 32; ++u)
        acc[u] = fmaf(-Ls[(32 * I + i) * kPL + 32 * I + u], x, acc[u]);
    }
  }
  __syncthreads();
  for (int j = 0; j < kb; ++j)
    if (tid < kb) X[tid + (long long)j * lb] = tid >= j ? Xs[tid * kPX + j] : 0.f;
}

template <int NC>
cudaError_t run_narrow(const Narrow& s, bool ta, int batch, cudaStream_t st) {
  return launch_chained(ta ? narrow32_kernel<NC, true> : narrow32_kernel<NC, false>,
                        dim3((unsigned)((long long)s.tiles * batch)), kThreads, 0, st, s);
}

}  // namespace

cudaError_t narrow32(int m, int n, int k, const float* A, int lda, long long sA, bool ta,
                     const float* B, int ldb, long long sB, float alpha, const float* Cin,
                     int ldcin, long long sCin, float* C, int ldc, long long sC, int batch,
                     cudaStream_t st) {
  if (m <= 0 || n <= 0 || batch <= 0) return cudaSuccess;
  if (n > 16 || k <= 0) return cudaErrorInvalidValue;
  const Narrow s{m,  n,  k,    lda, ldb,   ldcin, ldc, (m + kRows - 1) / kRows, sA, sB, sCin,
                 sC, alpha, A, B,   Cin, C};
  if (n <= 4) return run_narrow<4>(s, ta, batch, st);
  if (n <= 8) return run_narrow<8>(s, ta, batch, st);
  return run_narrow<16>(s, ta, batch, st);
}

cudaError_t launch_inv32(const float* M, int ldm, long long sM, int c, float* X, long long sX,
                         int nodes, cudaStream_t st) {
  if (c <= 0 || nodes <= 0) return cudaSuccess;
  const cudaError_t e = fx_allow_smem((const void*)inv32_kernel, kInvSmem);
  if (e != cudaSuccess) return e;
  inv32_kernel<<<dim3(nodes, (c + kOrder - 1) / kOrder), kOrder, kInvSmem, st>>>(
      M, ldm, sM, c, X, sX, c < kOrder ? c : kOrder);
  return cudaGetLastError();
}
