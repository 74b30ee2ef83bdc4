// Panel and T-block kernels of the blocked Householder QL (qlpanel.cuh).
//
// A node's whole QL in one CTA (ql_basis_kernel) runs its block reflectors, 9/10 of
// the flops, on that SM's pipe: in FP64 18.9 ms for 512 leaves of 512 x 128 and
// 2.7 ms for any level with fewer nodes than SMs.  Here only the panels, whose
// columns depend on one another, stay in a CTA.
//
// Panel: the thread's rows of all columns in registers; per column one reduction of
// the Gram row g_k = Σ_{i>j} x_ij x_ik (k >= j) -- its first entry is the squared
// norm below the pivot, and with the pivot row it gives every v_jᵀ x_k -- and one
// barrier.  In FP64 a warp instruction takes 64 clocks of its SM quarter, so the
// reduction (31 additions a warp) costs as much as the products: 4 warps with up
// to 4 rows a thread reduce half as many partial sums as 8 warps, and the scalars
// come from FP32 estimates with one Newton step (inv_sqrt, inv_pos).
#include "qlpanel.cuh"

namespace {

// reflector of (alpha, x), |x|² = sigma (LAPACK's dlarfg signs): beta, tau and the
// factor that turns x into v below its unit entry
HSS_DEVINL void reflector(double alpha, double sigma, double* beta, double* tau, double* scale) {
  if (sigma == 0.0) {
    *tau = 0.0;
    *beta = alpha;
    *scale = 1.0;
    return;
  }
  const double s = fma(alpha, alpha, sigma), inv = inv_sqrt(s), aa = fabs(alpha);
  const double nrm = sqrt_from(s, inv), sc = inv_pos(aa + nrm);
  *beta = alpha >= 0.0 ? -nrm : nrm;
  *tau = fma(aa, inv, 1.0);
  *scale = alpha >= 0.0 ? sc : -sc;
}
HSS_DEVINL void reflector(float alpha, float sigma, float* beta, float* tau, float* scale) {
  if (sigma == 0.f) {
    *tau = 0.f;
    *beta = alpha;
    *scale = 1.f;
    return;
  }
  const float nrm = sqrtf(alpha * alpha + sigma);
  *beta = alpha >= 0.f ? -nrm : nrm;
  *tau = (*beta - alpha) / *beta;
  *scale = 1.f / (alpha - *beta);
}

template <typename T, int NB, int NT, int RPT>
__global__ void __launch_bounds__(NT)
ql_panel_kernel(const T* __restrict__ Bb, T* __restrict__ Wb, T* __restrict__ Vb,
                T* __restrict__ Tb, T* __restrict__ Lb, int b, int r, int j0, int nb) {
  constexpr int NW = NT / 32;
  __shared__ T red[2][NW][NB];
  __shared__ T prow[2][NB];
  __shared__ T tau_s[NB];
  __shared__ T Gs[NW][NB][NB + 1];
  const long long node = blockIdx.x;
  const T* B = Bb + node * b * r;
  T* W = Wb + node * b * r;
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  if (blockIdx.y > 0) {   // first panel: the later columns, reversed, to W
    const int step = (gridDim.y - 1) * NT;
    for (int e = (blockIdx.y - 1) * NT + tid; e < b * (r - nb); e += step) {
      const int i = e % b, j = nb + e / b;
      W[i + (long long)j * b] = B[i + (long long)(r - 1 - j) * b];
    }
    return;
  }
  T* V = Vb + node * b * r;
  T* Tn = Tb + node * r * r;
  T* Ln = Lb + node * r * r;
  // column j0 + k at src + k dir b (row i of the elimination order at b - 1 - i)
  const T* src = j0 == 0 ? B + (long long)(r - 1) * b : W + (long long)j0 * b;
  const long long dir = j0 == 0 ? -b : b;
  T x[RPT][NB];
#pragma unroll
  for (int s = 0; s < RPT; ++s) {
    const int i = j0 + tid + NT * s;
#pragma unroll
    for (int k = 0; k < NB; ++k) x[s][k] = (i < b && k < nb) ? src[(b - 1 - i) + k * dir] : T(0);
  }
#pragma unroll
  for (int jj = 0; jj < NB; ++jj) {
    if (jj >= nb) break;
    const int j = j0 + jj, buf = jj & 1;
    if (tid == jj) {   // the pivot row (row j is thread jj's first row)
#pragma unroll
      for (int k = 0; k < NB; ++k) prow[buf][k] = x[0][k];
    }
    T g[NB];
#pragma unroll
    for (int k = 0; k < NB; ++k) g[k] = T(0);
#pragma unroll
    for (int s = 0; s < RPT; ++s) {
      const int i = j0 + tid + NT * s;
      const T a = i > j ? x[s][jj] : T(0);   // rows past b are zero
#pragma unroll
      for (int k = jj; k < NB; ++k) g[k] = fma(a, x[s][k], g[k]);
    }
    const T gw = warp_transpose_reduce<T, NB>(g, lane);
    if (lane < NB) red[buf][wid][lane] = gw;
    __syncthreads();
    T gk = T(0);   // Σ_{i>j} x_ij x_ik for k = lane
    if (lane < NB) {
#pragma unroll
      for (int w = 0; w < NW; ++w) gk += red[buf][w][lane];
    }
    const T sigma = __shfl_sync(0xffffffffu, gk, jj);
    T tau, beta, scale;
    reflector(prow[buf][jj], sigma, &beta, &tau, &scale);
    if (tid == 0) tau_s[jj] = tau;
    // v_jᵀ x_k = x_jk + scale g_k, held by lane k; then x_k -= tau (v_jᵀ x_k) v_j
    const T tw = lane < NB ? tau * fma(scale, gk, prow[buf][lane]) : T(0);
    T v[RPT];
#pragma unroll
    for (int s = 0; s < RPT; ++s) {
      const int i = j0 + tid + NT * s;
      v[s] = i > j ? x[s][jj] * scale : (i == j ? T(1) : T(0));
    }
#pragma unroll
    for (int k = jj + 1; k < NB; ++k) {
      const T twk = __shfl_sync(0xffffffffu, tw, k);
#pragma unroll
      for (int s = 0; s < RPT; ++s) x[s][k] = fma(-twk, v[s], x[s][k]);
    }
#pragma unroll
    for (int s = 0; s < RPT; ++s) {
      const int i = j0 + tid + NT * s;
      if (i > j) x[s][jj] = v[s];
      if (i == j) x[s][jj] = beta;   // R(j, j)
    }
  }
  // L_B's columns (R above and on the diagonal; rows before the panel are final in
  // src) and the reflectors
#pragma unroll
  for (int s = 0; s < RPT; ++s) {
    const int i = j0 + tid + NT * s;
    if (i < b) {
#pragma unroll
      for (int k = 0; k < NB; ++k) {
        if (k >= nb) break;
        const int d = j0 + k;
        if (i < r) Ln[(r - 1 - i) + (long long)(r - 1 - d) * r] = i <= d ? x[s][k] : T(0);
        x[s][k] = i > d ? x[s][k] : (i == d ? T(1) : T(0));
        V[(b - 1 - i) + (long long)d * b] = x[s][k];
      }
    }
  }
  for (int e = tid; e < j0 * nb; e += NT) {
    const int i = e % j0, k = e / j0;
    Ln[(r - 1 - i) + (long long)(r - 1 - j0 - k) * r] = src[(b - 1 - i) + k * dir];
    V[(b - 1 - i) + (long long)(j0 + k) * b] = T(0);
  }
  if (j0 + nb >= r) {   // no later column needs the panel's T: only tau
    __syncthreads();
    if (tid < nb) Tn[(j0 + tid) * (long long)(r + 1)] = tau_s[tid];
    return;
  }
  // panel Gram G(a, c) = v_aᵀ v_c (a < c): the columns c and NB - c share one
  // transposing reduction (c + (NB - c) = NB products)
#pragma unroll
  for (int c = 1; c <= NB / 2; ++c) {
    const int c2 = NB - c;
    T g[NB];
#pragma unroll
    for (int q = 0; q < NB; ++q) g[q] = T(0);
#pragma unroll
    for (int s = 0; s < RPT; ++s) {
#pragma unroll
      for (int q = 0; q < NB; ++q) {
        if (q < c) g[q] = fma(x[s][q], x[s][c], g[q]);
        else if (c2 != c) g[q] = fma(x[s][q - c], x[s][c2], g[q]);
      }
    }
    const T gw = warp_transpose_reduce<T, NB>(g, lane);
    if (lane < c) Gs[wid][c][lane] = gw;
    else if (lane < NB && c2 != c) Gs[wid][c2][lane - c] = gw;
  }
  __syncthreads();
  for (int e = tid; e < NB * NB; e += NT) {
    const int c = e / NB, a = e % NB;
    if (a < c) {
      T gm = Gs[0][c][a];
#pragma unroll
      for (int w = 1; w < NW; ++w) gm += Gs[w][c][a];
      Gs[0][c][a] = gm;
    }
  }
  __syncthreads();
  // panel T (forward dlarft): T(0:c, c) = -tau_c T(0:c, 0:c) G(0:c, c), lane a keeps
  // row a
  if (wid == 0) {
    T tp[NB];
#pragma unroll
    for (int c = 0; c < NB; ++c) {
      if (c < nb) {
        T v = T(0);
#pragma unroll
        for (int m = 0; m < c; ++m) v = fma(tp[m], Gs[0][c][m], v);
        const T tc = tau_s[c];
        tp[c] = lane < c ? -tc * v : (lane == c ? tc : T(0));
      } else {
        tp[c] = T(0);
      }
    }
#pragma unroll
    for (int m = 0; m < NB; ++m)
      if (lane < nb && m < nb) Tn[(j0 + lane) + (long long)(j0 + m) * r] = tp[m];
  }
}

// ------------------------------------------------------------------ T blocks
constexpr int kT = 128, kN = 64, kP = 65;

// inverse X of the 32 x 32 lower triangular block of S at offset o, its diagonal
// given by its reciprocals tau; a zero there leaves a zero row and column
template <typename T>
HSS_DEVINL void inverse32(const T* S, const T* tau, T* X, int o, T (*xrow)[32]) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  T x[8];   // row w + 4 u of X, lane = column
#pragma unroll
  for (int u = 0; u < 8; ++u) x[u] = lane == w + 4 * u ? T(1) : T(0);
#pragma unroll
  for (int j = 0; j < 32; ++j) {
    const int buf = j & 1;
    if (w == (j & 3)) {
      x[j >> 2] *= tau[o + j];
      xrow[buf][lane] = x[j >> 2];
    }
    __syncthreads();
    if (j < 31) {
      const T xr = xrow[buf][lane];
#pragma unroll
      for (int q = (j + 1) >> 2; q < 8; ++q) {
        const int t = w + 4 * q;
        if (t > j) x[q] = fma(-S[(o + j) * kP + o + t], xr, x[q]);
      }
    }
  }
#pragma unroll
  for (int u = 0; u < 8; ++u) X[(o + lane) * kP + o + w + 4 * u] = x[u];
  __syncthreads();
}

template <typename T>
__global__ void __launch_bounds__(kT)
ql_tblock_kernel(const T* __restrict__ Gb, T* Tb, int r) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  T* S = reinterpret_cast<T*>(smem_raw);
  T* X = S + kN * kP;
  __shared__ T xrow[2][32], tau[kN];
  const long long node = blockIdx.x;
  const int c0 = kN * blockIdx.y, kb = min(kN, r - c0);
  const T* G = Gb + node * r * r + c0 + (long long)c0 * r;
  T* Tn = Tb + node * r * r + (long long)c0 * r;
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  for (int e = tid; e < kN * kN; e += kT) {
    const int i = e % kN, j = e / kN;
    S[j * kP + i] = (i < kb && j < i) ? G[i + (long long)j * r] : T(0);
    X[j * kP + i] = T(0);
  }
  if (tid < kN) tau[tid] = tid < kb ? Tn[c0 + tid + (long long)tid * r] : T(1);
  __syncthreads();
  inverse32(S, tau, X, 0, xrow);
  if (kb > 32) {
    inverse32(S, tau, X, 32, xrow);
    // X21 = -X22 (L21 X11)
    T o[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) o[u] = T(0);
#pragma unroll 4
    for (int k = 0; k < 32; ++k) {
      const T a = S[k * kP + 32 + lane];
#pragma unroll
      for (int u = 0; u < 8; ++u)
        if (k >= w + 4 * u) o[u] = fma(a, X[(w + 4 * u) * kP + k], o[u]);
    }
#pragma unroll
    for (int u = 0; u < 8; ++u) S[(w + 4 * u) * kP + lane] = o[u];   // S's first block is done with
    __syncthreads();
#pragma unroll
    for (int u = 0; u < 8; ++u) o[u] = T(0);
#pragma unroll 4
    for (int k = 0; k < 32; ++k) {
      const T a = X[(32 + k) * kP + 32 + lane];
#pragma unroll
      for (int u = 0; u < 8; ++u) o[u] = fma(a, S[(w + 4 * u) * kP + k], o[u]);
    }
#pragma unroll
    for (int u = 0; u < 8; ++u) X[(w + 4 * u) * kP + 32 + lane] = -o[u];
    __syncthreads();
  }
  // T = Xᵀ, and zeros below the diagonal block
  for (int e = tid; e < (r - c0) * kb; e += kT) {
    const int i = e % (r - c0), j = e / (r - c0);
    Tn[c0 + i + (long long)j * r] = i <= j ? X[i * kP + j] : T(0);
  }
}

template <typename T, int NB, int NT, int RPT>
cudaError_t run_panel(const T* B, T* W, T* V, T* Tm, T* LB, int b, int r, int j0, int nb,
                      int nodes, cudaStream_t st) {
  const long long rest = j0 == 0 ? (long long)b * (r - nb) : 0;   // 16 copies a thread
  const int copies = (int)((rest + 16 * NT - 1) / (16 * NT));
  ql_panel_kernel<T, NB, NT, RPT>
      <<<dim3(nodes, 1 + copies), NT, 0, st>>>(B, W, V, Tm, LB, b, r, j0, nb);
  return cudaGetLastError();
}

}  // namespace

template <typename T>
cudaError_t launch_ql_panel(const T* B, T* W, T* V, T* Tm, T* LB, int b, int r, int j0, int nb,
                            int panel, int nodes, cudaStream_t st) {
  const int rows = b - j0;
  if (rows > 1024 || nb < 1 || nb > ql_panel_width(sizeof(T), b, panel))
    return cudaErrorInvalidValue;
#define QL_PANEL(NB, NT, RPT) \
  return run_panel<T, NB, NT, RPT>(B, W, V, Tm, LB, b, r, j0, nb, nodes, st)
  if constexpr (sizeof(T) == 8) {
    if (rows <= 128) QL_PANEL(16, 128, 1);
    if (rows <= 256) QL_PANEL(16, 128, 2);
    if (rows <= 384) QL_PANEL(16, 128, 3);
    if (rows <= 512) QL_PANEL(16, 128, 4);
    if (rows <= 768) QL_PANEL(16, 256, 3);
    QL_PANEL(16, 256, 4);
  } else {
    if (ql_panel_width(sizeof(T), b, panel) == 32) {
      if (rows <= 256) QL_PANEL(32, 256, 1);
      if (rows <= 512) QL_PANEL(32, 256, 2);
      QL_PANEL(32, 256, 3);
    }
    if (rows <= 256) QL_PANEL(16, 256, 1);
    if (rows <= 512) QL_PANEL(16, 256, 2);
    if (rows <= 768) QL_PANEL(16, 256, 3);
    QL_PANEL(16, 256, 4);
  }
#undef QL_PANEL
}

template <typename T>
cudaError_t launch_ql_tblocks(const T* G, T* Tm, int r, int nodes, cudaStream_t st) {
  const int smem = 2 * kN * kP * (int)sizeof(T);
  const cudaError_t e = fx_allow_smem((const void*)ql_tblock_kernel<T>, smem);
  if (e != cudaSuccess) return e;
  ql_tblock_kernel<T><<<dim3(nodes, (r + kN - 1) / kN), kT, smem, st>>>(G, Tm, r);
  return cudaGetLastError();
}

#define INST(T)                                                                                  \
  template cudaError_t launch_ql_panel<T>(const T*, T*, T*, T*, T*, int, int, int, int, int, int, \
                                          cudaStream_t);                                         \
  template cudaError_t launch_ql_tblocks<T>(const T*, T*, int, int, cudaStream_t);
INST(double)
INST(float)
