// Blocked FP64 Cholesky, and triangular solves (FP64 and FP32), of a whole tree level
// as products (chol64.cu and sweep32.cu hold the kernels; the level routines are below).
#pragma once
#include <cuda_runtime.h>

#include <algorithm>
#include <type_traits>

#include "../../include/hss.h"
#include "fxgemm.cuh"
#include "sweep32.cuh"

// Cholesky factor of the kb x kb block (kb <= 64) at the head of every matrix of a
// batch, and its inverse: L to M (ld ldm, stride sM), L⁻¹ to X (ld ldx, stride sX),
// both with zeros above the diagonal and in the `above` rows above the block.  The `rows` rows of M below the block go to P (ld rows,
// stride rows 64).  Writes (or, with accumulate, adds) 2 Σ log diag to part[node];
// a pivot that is not positive is reported at (level, node0 + node, col0 + column).
// flag[node flag_stride]: 1 where the inverse can be used without a correction.
cudaError_t launch_chol64(double* M, int ldm, long long sM, int kb, double* X, int ldx,
                          long long sX, int above, double* P, int rows, double* part, int level,
                          int node0, int col0, int* status, int nodes, bool accumulate,
                          int* flag, int flag_stride, cudaStream_t st);

// the flags of kb x kb blocks L and their inverses X, kb <= 128, zeros above the diagonals
cudaError_t launch_inv_flag(const double* L, int ldl, long long sL, const double* X, int ldx,
                            long long sX, int kb, int* flag, int flag_stride, int nodes,
                            cudaStream_t st);

// dst (r rows per node, ld ldd, stride sd) = src (ld lds, stride ss), nc columns
template <typename T>
cudaError_t launch_copy_rows(const T* src, int lds, long long ss, T* dst, int ldd, long long sd,
                             int r, int nc, int nodes, cudaStream_t st);

// Order of the inverted diagonal blocks, and the elements they take per node, for
// c eliminated columns.  128: a triangular solve of c columns is then c / 128
// pairs of products, two for every level above the leaves at rank <= 128.
constexpr int kInvOrder = 128;
inline int inv_order(int c) { return std::min(c, kInvOrder); }
inline long long inv_size(int c) {
  const long long lb = inv_order(c);
  return c > 0 ? (c + lb - 1) / lb * lb * lb : 0;
}

// Flags of a node: one per 64-column block, then one per 128-column block.
inline int flag_size(int c) { return (c + 63) / 64 + (c + kInvOrder - 1) / kInvOrder; }

// One tree level of the factor: n nodes of order b, c columns eliminated.
template <typename T>
struct LevelOf {
  int n, b, c;
  T* M;    // n x b x b, the factored blocks
  T* Li;   // n x inv_size(c), the inverted diagonal blocks
  int* Fl = nullptr;   // n x flag_size(c) (FP64)

  LevelOf part(int first, int count) const {
    return {count, b, c, M + (long long)first * b * b, Li + (long long)first * inv_size(c),
            Fl + (long long)first * flag_size(c)};
  }
};

using Level64 = LevelOf<double>;

// Where the merge puts a level's Schur complements: the diagonal blocks of the
// parents PA (ld, stride) for the first `split` nodes, and those of PA2 for the
// others (a forest's trees whose roots come next).  split is even.
struct Merge64 {
  double* PA = nullptr;
  int ld = 0;
  long long stride = 0;
  int split = 0;
  double* PA2 = nullptr;
};

// C (m x n) = alpha op(A) B + beta Cin, nc columns
inline cudaError_t skinny(int m, int nc, int k, const double* A, int lda, long long sA, bool ta,
                          const double* B, int ldb, long long sB, double alpha, const double* Cin,
                          int ldcin, long long sCin, double* C, int ldc, long long sC, int batch,
                          cudaStream_t st, bool components = true, const int* skip = nullptr,
                          int skip_stride = 0) {
  const FxOperand a{A, lda, sA, ta}, b{B, ldb, sB, true};
  return fx_gemm(m, nc, k, a, b, alpha, Cin ? 1.0 : 0.0, Cin, ldcin, sCin, C, ldc, sC, batch, false,
                 nullptr, 0, 0, st, components, skip, skip_stride);
}

inline cudaError_t skinny(int m, int nc, int k, const float* A, int lda, long long sA, bool ta,
                          const float* B, int ldb, long long sB, float alpha, const float* Cin,
                          int ldcin, long long sCin, float* C, int ldc, long long sC, int batch,
                          cudaStream_t st, bool = true) {
  return narrow32(m, nc, k, A, lda, sA, ta, B, ldb, sB, alpha, Cin, ldcin, sCin, C, ldc, sC, batch,
                  st);
}

#define LV_TRY(kind, flops, call)                                       \
  do {                                                                  \
    cudaError_t e_ = cudaSuccess;                                       \
    log(kind, flops, [&] { e_ = (call); });                             \
    if (e_ != cudaSuccess) return e_;                                   \
  } while (0)

// Partial Cholesky of every node of a level (Eq. partial-Cholesky): in 128-column
// panels, each factored as two 64-column blocks (launch_chol64, the rows below a
// block by a product with its inverse and one correction, the second block's columns
// updated first), then one update of the trailing triangle with 128 inner indices -- a whole
// scaling group of the sliced product, which at 32 inner indices spends most of
// its time putting the digits' sums together (512 nodes, order 480: 1.45 ms for 32,
// 1.4 ms for 128).  The last update merges into the parents where given.
// The correction: L21 = A21 X is as inaccurate as the block is ill-conditioned (a
// Gaussian covariance of condition 1e10 solved to a residual of 1.6e-5 where
// substitution leaves 1.2e-6), L21 + (A21 - L21 L11ᵀ) Xᵀ as accurate as substitution.
// So it needs the components of the residual only, not those of the products with X.
// Nodes whose block has max|L| max|X| < 16 leave it out (their flag is set): there the
// inverse amplifies rounding less than the 128 steps of a substitution may.  Without
// any correction the residuals of the Gaussian covariance were those of substitution
// or below up to a condition of 3e5.  Factor + solve N = 262144: 57.0 ms without
// corrections, 61.8 with all of them, 56.3 so; solve 3.56, 4.94 and 3.73 ms; solve of
// N = 4096 171, 259 and 194 us (launches that return at once).
// P: scratch of n b 64 doubles.  log(kind, flops, fn) runs fn, one launch.
template <typename Log>
cudaError_t chol_level64(const Level64& lv, double* P, double* part, int level, int node0,
                         int* status, const Merge64& up, cudaStream_t st, const Log& log) {
  const int b = lv.b, c = lv.c, n = lv.n, lb = inv_order(c);
  const long long bb = (long long)b * b, sX = inv_size(c);
  const int nf = flag_size(c);
  for (int k0 = 0; k0 < c; k0 += kInvOrder) {
    const int kb = std::min(kInvOrder, c - k0);
    double* X = lv.Li + (long long)(k0 / lb) * lb * lb;
    int* flag = lv.Fl + (c + 63) / 64 + k0 / kInvOrder;   // the panel's
    for (int h0 = 0; h0 < kb; h0 += 64) {
      const int kh = std::min(64, kb - h0), col = k0 + h0, rows = b - col - kh;
      double* Mk = lv.M + col + (long long)col * b;
      double* Xh = X + h0 + (long long)h0 * lb;
      int* ok = kb > 64 ? lv.Fl + col / 64 : flag;
      LV_TRY(HSS_K_PCHOL, (double)kh * kh * kh / 3.0 * n,
             launch_chol64(Mk, b, bb, kh, Xh, lb, sX, h0, P, rows, part, level, node0, col, status,
                           n, col > 0, ok, nf, st));
      if (rows <= 0) continue;
      const FxOperand pa{P, rows, 64LL * rows, false}, xb{Xh, lb, sX, false};
      const FxOperand l21{Mk + kh, b, bb, false}, l11{Mk, b, bb, false};
      LV_TRY(HSS_K_GEMM, (double)rows * kh * kh * n,
             fx_gemm(rows, kh, kh, pa, xb, 1.0, 0.0, nullptr, 0, 0, Mk + kh, b, bb, n, false,
                     nullptr, 0, 0, st, /*components=*/false));
      LV_TRY(HSS_K_GEMM, 0.0,
             fx_gemm(rows, kh, kh, l21, l11, -1.0, 1.0, P, rows, 64LL * rows, P, rows, 64LL * rows,
                     n, false, nullptr, 0, 0, st, true, ok, nf));
      LV_TRY(HSS_K_GEMM, 0.0,
             fx_gemm(rows, kh, kh, pa, xb, 1.0, 1.0, Mk + kh, b, bb, Mk + kh, b, bb, n, false,
                     nullptr, 0, 0, st, /*components=*/false, ok, nf));
      if (h0 == 0 && kb > 64) {
        double* C = Mk + 64 + 64LL * b;
        const FxOperand l{Mk + 64, b, bb, false};
        LV_TRY(HSS_K_SYR2K, 2.0 * rows * (kb - 64) * 64 * n,
               fx_gemm(rows, kb - 64, 64, l, l, -1.0, 1.0, C, b, bb, C, b, bb, n, false, nullptr,
                       0, 0, st));
      }
    }
    double* Mk = lv.M + k0 + (long long)k0 * b;
    const int rows = b - k0 - kb;
    if (rows > 0) {
      auto update = [&](int first, int count, double* PA) {
        double* L = Mk + kb + first * bb;
        double* C = L + (long long)kb * b;
        LV_TRY(HSS_K_SYR2K, (double)rows * (rows + 1.0) * kb * count,
               (dsyrk_lower_batched(rows, kb, C, b, bb, L, b, bb, C, b, bb, PA, up.ld, up.stride,
                                    count, st),
                cudaGetLastError()));
        return cudaSuccess;
      };
      cudaError_t e = cudaSuccess;
      if (k0 + kb < c || !(up.PA || up.PA2)) {
        e = update(0, n, nullptr);
      } else {
        if (up.split > 0) e = update(0, up.split, up.PA);
        if (e == cudaSuccess && n > up.split) e = update(up.split, n - up.split, up.PA2);
      }
      if (e != cudaSuccess) return e;
    }
    if (kb > 64) {   // off-diagonal block of the inverse: -X22 (L21 X11)
      const int k2 = kb - 64;
      LV_TRY(HSS_K_GEMM, 2.0 * k2 * 64 * 64 * n,
             skinny(k2, 64, 64, Mk + 64, b, bb, false, X, lb, sX, 1.0, nullptr, 0, 0, P, k2,
                    64LL * k2, n, st, /*components=*/false));
      LV_TRY(HSS_K_GEMM, 2.0 * k2 * 64 * k2 * n,
             skinny(k2, 64, k2, X + 64 + 64LL * lb, lb, sX, false, P, k2, 64LL * k2, -1.0, nullptr,
                    0, 0, X + 64, lb, sX, n, st, /*components=*/false));
      LV_TRY(HSS_K_OTHER, 0.0, launch_inv_flag(Mk, b, bb, X, lb, sX, kb, flag, nf, n, st));
    }
  }
  return cudaSuccess;
}

// Forward triangular sweep of a level on nc columns: z = L^RR⁻¹ y^R, and
// y^S - L^SR z to the parent's vector par (r = b - c rows per node; null at the
// root).  y and z: ld ldy and ldz, b rows per node.  y is overwritten.  In FP64 with
// one correction per diagonal block, z = X y and z += X (y - L z), for the reason and
// with the exception given at chol_level64.  An FP32 factor is a preconditioner: none
// there (the iteration counts of refinement are those of substitution).
template <typename T, typename Log>
cudaError_t fwd_level(const LevelOf<T>& lv, T* y, int ldy, T* z, int ldz, T* par, int ldpar,
                      int nc, cudaStream_t st, const Log& log) {
  const int b = lv.b, c = lv.c, n = lv.n, lb = inv_order(c), r = b - c;
  const long long bb = (long long)b * b, sX = inv_size(c);
  if (c == 0 && par)
    LV_TRY(HSS_K_OTHER, 0.0, launch_copy_rows<T>(y, ldy, b, par, ldpar, r, r, nc, n, st));
  for (int k0 = 0; k0 < c; k0 += kInvOrder) {
    const int kb = std::min(kInvOrder, c - k0), rows = b - k0 - kb;
    const T* X = lv.Li + (long long)(k0 / lb) * lb * lb;
    LV_TRY(HSS_K_TRSV_FWD, (double)kb * kb * nc * n,
           skinny(kb, nc, kb, X, lb, sX, false, y + k0, ldy, b, T(1), static_cast<const T*>(nullptr),
                  0, 0, z + k0, ldz, b, n, st, /*components=*/false));
    if constexpr (std::is_same<T, double>::value) {
      const int* ok = lv.Fl + (c + 63) / 64 + k0 / kInvOrder;
      LV_TRY(HSS_K_TRSV_FWD, 0.0,
             skinny(kb, nc, kb, lv.M + k0 + (long long)k0 * b, b, bb, false, z + k0, ldz, b, -1.0,
                    y + k0, ldy, b, y + k0, ldy, b, n, st, true, ok, flag_size(c)));
      LV_TRY(HSS_K_TRSV_FWD, 0.0,
             skinny(kb, nc, kb, X, lb, sX, false, y + k0, ldy, b, 1.0, z + k0, ldz, b, z + k0, ldz,
                    b, n, st, /*components=*/false, ok, flag_size(c)));
    }
    if (rows <= 0) continue;
    const bool last = k0 + kb == c;   // only the S rows are left: the parent's
    T* yb = y + k0 + kb;
    LV_TRY(HSS_K_TRSV_FWD, 2.0 * rows * kb * nc * n,
           skinny(rows, nc, kb, lv.M + (k0 + kb) + (long long)k0 * b, b, bb, false, z + k0, ldz, b,
                  T(-1), yb, ldy, b, last && par ? par : yb, last && par ? ldpar : ldy,
                  last && par ? r : b, n, st));
  }
  return cudaSuccess;
}

// Backward sweep: x^S from the parent's vector, x^R = L^RR⁻ᵀ (z - L^SRᵀ x^S),
// into y; z is overwritten.
template <typename T, typename Log>
cudaError_t bwd_level(const LevelOf<T>& lv, T* y, int ldy, T* z, int ldz, const T* par, int ldpar,
                      int nc, cudaStream_t st, const Log& log) {
  const int b = lv.b, c = lv.c, n = lv.n, lb = inv_order(c), r = b - c;
  const long long bb = (long long)b * b, sX = inv_size(c);
  if (par && r > 0)
    LV_TRY(HSS_K_OTHER, 0.0, launch_copy_rows<T>(par, ldpar, r, y + c, ldy, b, r, nc, n, st));
  for (int k0 = c > 0 ? (c - 1) / kInvOrder * kInvOrder : -1; k0 >= 0; k0 -= kInvOrder) {
    const int kb = std::min(kInvOrder, c - k0), rows = b - k0 - kb;
    const T* X = lv.Li + (long long)(k0 / lb) * lb * lb;
    if (rows > 0)
      LV_TRY(HSS_K_TRSV_BWD, 2.0 * rows * kb * nc * n,
             skinny(kb, nc, rows, lv.M + (k0 + kb) + (long long)k0 * b, b, bb, true, y + k0 + kb,
                    ldy, b, T(-1), z + k0, ldz, b, z + k0, ldz, b, n, st));
    LV_TRY(HSS_K_TRSV_BWD, (double)kb * kb * nc * n,
           skinny(kb, nc, kb, X, lb, sX, true, z + k0, ldz, b, T(1), static_cast<const T*>(nullptr),
                  0, 0, y + k0, ldy, b, n, st, /*components=*/false));
    if constexpr (std::is_same<T, double>::value) {
      const int* ok = lv.Fl + (c + 63) / 64 + k0 / kInvOrder;
      LV_TRY(HSS_K_TRSV_BWD, 0.0,
             skinny(kb, nc, kb, lv.M + k0 + (long long)k0 * b, b, bb, true, y + k0, ldy, b, -1.0,
                    z + k0, ldz, b, z + k0, ldz, b, n, st, true, ok, flag_size(c)));
      LV_TRY(HSS_K_TRSV_BWD, 0.0,
             skinny(kb, nc, kb, X, lb, sX, true, z + k0, ldz, b, 1.0, y + k0, ldy, b, y + k0, ldy, b,
                    n, st, /*components=*/false, ok, flag_size(c)));
    }
  }
  return cudaSuccess;
}
