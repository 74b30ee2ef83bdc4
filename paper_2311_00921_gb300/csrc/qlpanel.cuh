// Basis completion of a whole tree level by blocked Householder QL: one panel
// kernel per 16 or 32 columns (qlpanel.cu), everything else as products over the
// level.
#pragma once
#include <cuda_runtime.h>

#include <algorithm>
#include <type_traits>

#include "../../include/hss.h"
#include "common.cuh"
#include "fxgemm.cuh"

// One panel (columns j0 .. j0 + nb - 1, nb <= NB) of the QL factorization of every
// node's basis, in the order of elimination (column j is the basis' column
// r - 1 - j, pivot row b - 1 - j).  W (b x r) holds the columns not yet factored;
// the first panel reads them from B and copies the later ones to W.  Writes the
// reflectors (unit diagonal and zeros written out) to V, their compact-WY factor
// to the diagonal block of Tm (ld r), and the panel's columns of L_B.
template <typename T>
cudaError_t launch_ql_panel(const T* B, T* W, T* V, T* Tm, T* LB, int b, int r, int j0, int nb,
                            int panel, int nodes, cudaStream_t st);

// The 64 x 64 diagonal blocks of T = (diag(1 / tau) + striu(VᵀV))⁻¹ from the Gram
// matrix G (r x r, its lower triangle) and tau = diag(T); zeros below them.
template <typename T>
cudaError_t launch_ql_tblocks(const T* G, T* Tm, int r, int nodes, cudaStream_t st);

// Whether the Householder basis completion runs as panels and level-wide products.
// In FP64 from the second 16-column panel on (level of 256 x 128 bases, any node
// count up to the SMs: 2.7 -> 1.45 ms; 512 leaves of 512 x 128: 18.9 -> 8.4 ms; 16 of
// 256 x 32: 0.29 -> 0.24 ms).  In FP32 the one-CTA kernel's products are fast and the
// launches count: rank 96 loses 2 % of a step, rank 256 gains (leaf 1024: 8.9 ->
// 3.1 ms, the levels above 2.2 -> 1.3 ms).  At lower ranks it gains on a level with more
// nodes than SMs and more rows than a CTA has threads, where the one-CTA kernel runs in
// several waves of two rows a thread (512 leaves of 512 x 128, 3.0 ms of the critical path:
// the step 22.1 -> 21.0 ms; FP32 factor by one CTA a node and by panels, leaf x rank,
// leaves: 300 x 64, 256: 3.18 and 3.02 ms; 512 x 64, 256: 5.02 and 4.75; 512 x 96, 256:
// 6.72 and 6.40; 260 x 96, 512: 6.94 and 6.50; 300 x 127, 256: 7.26 and 6.73).
template <typename T>
bool ql_blocked(int b, int r, int nodes) {
  if (sizeof(T) == 8) return r > 16;
  return r > 128 || (r >= 64 && b > 256 && nodes >= 152);
}

template <typename T>
void level_gemm(bool ta, bool tb, int m, int n, int k, T alpha, const T* A, int lda, long long sA,
                const T* B, int ldb, long long sB, T beta, T* C, int ldc, long long sC, int batch,
                cudaStream_t st) {
  if constexpr (std::is_same<T, double>::value)
    dgemm_batched(ta, tb, m, n, k, alpha, A, lda, sA, B, ldb, sB, beta, C, ldc, sC, batch, st,
                  /*components=*/false);
  else
    gemm_batched<T>(ta, tb, m, n, k, alpha, A, lda, sA, B, ldb, sB, beta, C, ldc, sC, batch, st);
}

#define QL_TRY(kind, flops, call)           \
  do {                                      \
    cudaError_t e_ = cudaSuccess;           \
    log(kind, flops, [&] { e_ = (call); }); \
    if (e_ != cudaSuccess) return e_;       \
  } while (0)

// Columns per panel.
inline int ql_panel_width(size_t elem, int b, int panel) {
  return elem == 8 || panel == 16 || b > 768 ? 16 : 32;
}

// V, L_B and the panels' blocks of T for n nodes of a level (scratch per node: W
// b r, W1 and W2 r r elements).  Right-looking: after
// a panel, the later columns get A -= V_p (T_pᵀ V_pᵀ A) as three products.
template <typename T, typename Log>
cudaError_t ql_level(const T* B, T* V, T* Tm, T* LB, int b, int r, int n, T* W, T* W1, T* W2,
                     int panel, cudaStream_t st, const Log& log) {
  const int NB = ql_panel_width(sizeof(T), b, panel);
  const long long br = (long long)b * r, rr = (long long)r * r;
  for (int j0 = 0; j0 < r; j0 += NB) {
    const int nb = std::min(NB, r - j0), k0 = j0 + nb, nk = r - k0, rows = b - j0;
    QL_TRY(HSS_K_QL, 3.0 * rows * nb * nb * n,
           launch_ql_panel<T>(B, W, V, Tm, LB, b, r, j0, nb, panel, n, st));
    if (nk <= 0) break;
    const T* Vp = V + (long long)j0 * b;
    T* A = W + (long long)k0 * b;
    auto gemm = [&](bool ta, bool tb, int m, int nn, int k, T alpha, const T* X, int ldx,
                    long long sX, const T* Y, int ldy, long long sY, T beta, T* C, int ldc,
                    long long sC) {
      log(nn <= 32 ? HSS_K_GEMM_SKINNY : HSS_K_GEMM, 2.0 * m * nn * k * n, [&] {
        level_gemm<T>(ta, tb, m, nn, k, alpha, X, ldx, sX, Y, ldy, sY, beta, C, ldc, sC, n, st);
      });
    };
    gemm(true, false, nk, nb, rows, T(1), A, b, br, Vp, b, br, T(0), W1, nk, rr);
    gemm(false, false, nk, nb, nb, T(1), W1, nk, rr, Tm + j0 + (long long)j0 * r, r, rr, T(0), W2,
         nk, rr);
    gemm(false, true, rows, nk, nb, T(-1), Vp, b, br, W2, nk, rr, T(1), A, b, br);
  }
  return cudaGetLastError();
}

// The whole of T, from V and tau = diag(T): T = (diag(1 / tau) + striu(VᵀV))⁻¹
// (Puglisi 1992; Joffrain, Low, Quintana-Orti, van de Geijn, Van Zee 2006), its 64 x 64
// diagonal blocks by a kernel, the rest by products, T12 = -T11 G12 T22, blocks of
// 64, 128.  G and P: scratch of r r elements a node.
template <typename T, typename Log>
cudaError_t ql_tfactor(const T* V, T* Tm, int b, int r, int n, T* G, T* P, cudaStream_t st,
                       const Log& log) {
  const long long br = (long long)b * r, rr = (long long)r * r;
  log(HSS_K_GEMM, 1.0 * r * r * b * n, [&] {
    if constexpr (std::is_same<T, double>::value) {
      const FxOperand v{V, b, br, true};
      fx_gemm(r, r, b, v, v, 1.0, 0.0, nullptr, 0, 0, G, r, rr, n, /*lower=*/true, nullptr, 0, 0,
              st, /*components=*/false);
    } else {
      level_gemm<T>(true, false, r, r, b, T(1), V, b, br, V, b, br, T(0), G, r, rr, n, st);
    }
  });
  QL_TRY(HSS_K_BASIS_NODE, 64.0 * 64 * r / 3 * n, launch_ql_tblocks<T>(G, Tm, r, n, st));
  for (int s = 64; s < r; s *= 2)
    for (int i = 0; i + s < r; i += 2 * s) {
      const int m2 = std::min(s, r - i - s);
      const T* T11 = Tm + i + (long long)i * r;
      const T* T22 = Tm + (i + s) + (long long)(i + s) * r;
      const T* G21 = G + (i + s) + (long long)i * r;
      log(HSS_K_GEMM, 2.0 * s * m2 * s * n, [&] {   // T11 G21ᵀ
        level_gemm<T>(false, true, s, m2, s, T(1), T11, r, rr, G21, r, rr, T(0), P, s, rr, n, st);
      });
      log(HSS_K_GEMM, 2.0 * s * m2 * m2 * n, [&] {
        level_gemm<T>(false, false, s, m2, m2, T(-1), P, s, rr, T22, r, rr, T(0),
                      Tm + i + (long long)(i + s) * r, r, rr, n, st);
      });
    }
  return cudaGetLastError();
}
