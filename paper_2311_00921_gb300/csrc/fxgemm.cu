// FP64 products on the tensor cores by exact slicing (the Ozaki scheme: Ozaki,
// Ogita, Oishi, Rump 2012; on tensor cores Mukunoki, Ozaki, Ogita, Imamura 2020).
//
// The chip's FP64 pipe gives 1.05 TFLOP/s (2 DFMA per clock per SM); its FP16
// MMA 600 TFLOP/s with FP32 accumulation, which is exact as long as every
// partial sum is an integer of at most 24 bits.  Within a group of kGroup = 128
// inner indices, each row of an operand is scaled by the power of two e of its
// largest element and cut to a 64-bit integer q, |q| < 2^63; q is written as
// eight digits of base 256 in [-128, 127] (exact in FP16), and of the 64 digit
// products the 36 with weight i + j <= 7 are accumulated, those of equal weight
// in one FP32 accumulator: at most 8 x 128 products of magnitude <= 2^14, a sum
// of at most 2^24, so every MMA is exact.  At the end of a group the eight
// accumulators are put together as two integers and added to the FP64 result.
//
// Error of one group: cutting each operand at 2^-63 of its row's scale (at most twice
// its largest element), and the dropped digit products, together at most 2^-60.5 of
// the scales' product per inner index (2^-64 √K in the mean over random digits).  That
// is relative to the rows' largest elements; a DFMA chain is within K 2^-53 of Σ|a||b|,
// far less where the large elements of one row meet zeros or small elements of the
// other.  So each element's S = Σ|a||b| is accumulated beside its digits' products, by a
// 37th MMA on the two leading digits' absolute values (FP16 accumulators: S above
// 65504 is as good as infinite).  Where S is below 2^-8 of the scales' product, the
// group's part of that element is summed by DFMA; elsewhere the error is at most
// K 2^-52.5 of Σ|a||b|, 2^-56 √K in the mean.  The products of the Householder
// transformations, whose error in any arithmetic is relative to the norms of rows and
// columns (a chain's bound K 2^-53 of them is 2^5 of the above), do without S
// (components = false): the reflectors' unit entries and zeros would send up to 22 % of
// their elements to the DFMA pipe.  Batch of ten: 11.4 ms without S, 13.9 ms with S
// in all products, 12.2 ms so; D x of 512 leaves and 16 columns is 5 % slower with S.
// The merges' products, L_B (nearly diagonal) times couplings of a wide range, send 5 to
// 30 % of their elements there: factor of the sphere workload's matrix, N = 262144, 52
// ms without S and 57.7 with it, of random generators 52 and 53.
// (Seven digits, whose error is 2^-56 of max|a| max|b|, are not enough: the solves of
// kernel matrices lost a factor of three to five against the DFMA chain.)
//
// Rows with an element that is not finite or whose largest magnitude is outside
// [2^-470, 2^470] take a DFMA loop as a whole, so that infinities, NaN, overflow and
// denormals behave as in the plain product.
//
// Layout: a CTA has 4 warps and a 64 x BN tile of C (BN = 32, 16 or 8 columns;
// a warp 16 rows and every column).  Per group the operands' strips are read
// once for the row maxima and, from L1 or L2, again in chunks of 32 inner indices
// for the conversion to digits in shared memory (80-byte rows: ldmatrix and
// 16-byte stores without bank conflicts); 8 weights x BN / 2 FP32 accumulators
// live in registers.  Several CTAs share an SM, one converting while another
// issues MMAs.
#include <stdint.h>

#include <mutex>
#include <set>
#include <utility>

#include "common.cuh"
#include "fxgemm.cuh"

namespace {

constexpr int kThreads = 128;
constexpr int kRows = 64;       // rows of a CTA's tile
constexpr int kChunk = 32;      // inner indices converted at a time
constexpr int kGroup = 128;     // inner indices with one scale
constexpr int kDigits = 8;
constexpr int kPitch = 2 * kChunk + 16;   // bytes of a row of digits in shared memory
constexpr int kHiBig = (1023 + 470) << 20, kHiSmall = (1023 - 470) << 20;
constexpr int kZeroRow = 1 << 16;   // exponent of a row of zeros: shifts every digit out
constexpr float kLeast = 64.f;      // 2^-8 of the scales' product, in the unit of S (128 a scale)

struct FxShape {
  int m, n, K, K1;   // K1: inner indices of each part, K in all
  FxOperand a, b;
  double alpha, beta;
  const double* Cin;
  int ldcin;
  long long sCin;
  double* C;
  int ldc;
  long long sC;
  int lower;
  double* PA;
  int ldpa;
  long long sPA;
  int tiles_m, tiles_n, tiles;
  int components;
  const int* skip;
  int skip_stride;
};

HSS_DEVINL uint32_t smem_of(const void* p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

HSS_DEVINL uint32_t prmt(uint32_t a, uint32_t b, uint32_t sel) { return __byte_perm(a, b, sel); }

// fp16x2 of two digits held as 1024 + (digit + 128): minus 1152
HSS_DEVINL uint32_t unbias(uint32_t v) {
  uint32_t r;
  asm("sub.f16x2 %0, %1, %2;" : "=r"(r) : "r"(v), "r"(0x64806480u));
  return r;
}

HSS_DEVINL uint32_t shr(uint32_t v, uint32_t n) {   // 0 for n >= 32
  uint32_t r;
  asm("shr.u32 %0, %1, %2;" : "=r"(r) : "r"(v), "r"(n));
  return r;
}

// v 2^(63 - e), cut to an integer, + 0x8080808080808080: its bytes are the digits
// plus 128, least significant first; E1 = e + 1023, e + 1022 the row's biased
// exponent.  The mantissa, its leading one at bit 63, is shifted right and
// negated with the sign; zeros and denormals (exponent field 0) are shifted out.
HSS_DEVINL uint64_t fixed_point(double v, int E1) {
  const uint32_t hi = (uint32_t)__double2hiint(v), lo = (uint32_t)__double2loint(v);
  const uint32_t n = (uint32_t)(E1 - (int)((hi >> 20) & 0x7ffu));
  const uint32_t top = __funnelshift_l(lo, hi, 11) | 0x80000000u;
  const uint32_t tl = shr(__funnelshift_rc(lo << 11, top, n), (uint32_t)max((int)n - 32, 0));
  const uint32_t th = shr(top, n);
  const uint32_t s = (uint32_t)((int)hi >> 31);
  return (((uint64_t)(th ^ s) << 32) | (tl ^ s)) +
         ((0x80808080ull << 32) | (uint64_t)(0x80808080u - s));
}

// digit pairs of the elements u0 (lower half) and u1, most significant first
HSS_DEVINL void digits(uint64_t u0, uint64_t u1, uint32_t (&d)[kDigits]) {
  const uint32_t w0[2] = {(uint32_t)(u0 >> 32), (uint32_t)u0},
                 w1[2] = {(uint32_t)(u1 >> 32), (uint32_t)u1};
  const uint32_t c = 0x64646464u;
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    const uint32_t up = prmt(w0[h], w1[h], 0x7362), dn = prmt(w0[h], w1[h], 0x5140);
    d[4 * h + 0] = unbias(prmt(up, c, 0x4342));
    d[4 * h + 1] = unbias(prmt(up, c, 0x4140));
    d[4 * h + 2] = unbias(prmt(dn, c, 0x4342));
    d[4 * h + 3] = unbias(prmt(dn, c, 0x4140));
  }
}

HSS_DEVINL void ldmatrix4(uint32_t (&r)[4], uint32_t addr) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(addr));
}

HSS_DEVINL void mma_f16(float (&c)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, "
      "{%8, %9}, {%0, %1, %2, %3};"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// S += |a| |b| in FP16, of the operands' absolute leading parts
HSS_DEVINL void mma_abs(uint32_t (&c)[2], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f16.f16.f16.f16 {%0, %1}, {%2, %3, %4, %5}, {%6, %7}, "
      "{%0, %1};"
      : "+r"(c[0]), "+r"(c[1])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// |d0 + d1 / 256|, two digits of a pair of elements (digit units of the first)
HSS_DEVINL uint32_t leading(uint32_t d0, uint32_t d1) {
  uint32_t r;
  asm("fma.rn.f16x2 %0, %1, %2, %3;" : "=r"(r) : "r"(d1), "r"(0x1c001c00u), "r"(d0));
  return r & 0x7fff7fffu;
}

// half h of an fp16x2
HSS_DEVINL float half_of(uint32_t v, int h) {
  float f;
  asm("{.reg .b16 t; cvt.u16.u32 t, %1; cvt.f32.f16 %0, t;}" : "=f"(f) : "r"(h ? v >> 16 : v));
  return f;
}

// magnitude of v for the row maxima: its high word, not zero if v is not
HSS_DEVINL int magnitude(double v) {
  return (__double2hiint(v) & 0x7fffffff) | (__double2loint(v) != 0);
}

// biased exponent (+ 1) of a row's scale from its largest magnitude: |v| < 0.996 2^(E - 1022),
// a mantissa near 2 goes up to the next power, so that the digits' range holds it;
// odd: the row is outside the sliced range
HSS_DEVINL int row_exponent(int h, int& odd) {
  odd |= h >= kHiBig || (h > 0 && h < kHiSmall);
  return h ? ((h + 0x2100) >> 20) + 1 : kZeroRow;
}

// R rows (from row0 on) of one operand's part (contiguous inner indices 0 .. K-1
// of one array).  Rows past the last are read as copies of it: their results are
// not stored.
template <int R, bool KC>
struct Strip {
  const double* p;   // KC: element (0, 0) of the operand; else the same
  int ld, row0, last;

  HSS_DEVINL const double* row(int r) const {
    const int i = min(row0 + r, last);
    return KC ? p + (long long)i * ld : p + i;
  }
  HSS_DEVINL double at(int r, int k) const { return row(r)[KC ? (long long)k : (long long)k * ld]; }

  // mx[r] = largest magnitude() of row r over [k0, k1); mx is cleared
  HSS_DEVINL void maxima(int k0, int k1, int* mx) const {
    const int tid = threadIdx.x;
    if (KC) {
      const int lane = tid & 31, w = tid >> 5;
      constexpr int U = R / 4 < 4 ? R / 4 : 4;
      for (int r = w; r < R; r += 4 * U) {
        int v[U][kGroup / 32];
#pragma unroll
        for (int u = 0; u < U; ++u) {
          const double* q = row(r + 4 * u) + k0 + lane;
#pragma unroll
          for (int j = 0; j < kGroup / 32; ++j)
            v[u][j] = k0 + lane + 32 * j < k1 ? magnitude(q[32 * j]) : 0;
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
          int h = 0;
#pragma unroll
          for (int j = 0; j < kGroup / 32; ++j) h = max(h, v[u][j]);
          h = __reduce_max_sync(0xffffffffu, h);
          if (lane == 0) mx[r + 4 * u] = h;
        }
      }
    } else {
      constexpr int S = kThreads / R;   // threads per row
      const int r = tid % R, n = k1 - k0;
      int k = tid / R, h = 0;
      const double* q = row(r) + (long long)(k0 + k) * ld;
      const long long step = (long long)S * ld;
      for (; k + 15 * S < n; k += 16 * S) {
        int v[16];
#pragma unroll
        for (int j = 0; j < 16; ++j, q += step) v[j] = magnitude(*q);
#pragma unroll
        for (int j = 0; j < 16; ++j) h = max(h, v[j]);
      }
#pragma unroll 4
      for (; k < n; k += S, q += step) h = max(h, magnitude(*q));
      atomicMax(mx + r, h);
    }
  }

  // digits of [k0, k0 + kChunk) (zero from k1 on) to shared memory, digit s of
  // row r, index k at sm + s R kPitch + r kPitch + 2 (k - k0)
  template <bool WHOLE>
  HSS_DEVINL void convert(int k0, int k1, const int* E1, unsigned char* sm) const {
    const int tid = threadIdx.x;
    if (KC) {
      constexpr int UNITS = R * kChunk / 2 / kThreads;   // (row, pair of k) per thread
      double v[UNITS][2];
      const int kp = 2 * (tid & 15);
      // pairs past the end read the last pair's place
      const bool ok0 = WHOLE || k0 + kp < k1, ok1 = WHOLE || k0 + kp + 1 < k1;
#pragma unroll
      for (int u = 0; u < UNITS; ++u) {
        const double* q = row((tid >> 4) + 8 * u) + k0 + kp;
        v[u][0] = ok0 ? q[0] : 0.0;
        v[u][1] = ok1 ? q[1] : 0.0;
      }
#pragma unroll
      for (int u = 0; u < UNITS; ++u) {
        const int r = (tid >> 4) + 8 * u;
        uint32_t d[kDigits];
        digits(fixed_point(v[u][0], E1[r]), fixed_point(v[u][1], E1[r]), d);
#pragma unroll
        for (int s = 0; s < kDigits; ++s)
          *reinterpret_cast<uint32_t*>(sm + (s * R + r) * kPitch + 2 * kp) = d[s];
      }
    } else {
      for (int u = tid; u < 4 * R; u += kThreads) {   // (row, 8 consecutive k)
        const int r = u % R, o = u / R;
        double v[8];
        const double* q = row(r) + (long long)(k0 + 8 * o) * ld;
#pragma unroll
        for (int j = 0; j < 8; ++j, q += ld) v[j] = (WHOLE || k0 + 8 * o + j < k1) ? *q : 0.0;
        const int e = E1[r];
        uint32_t d[4][kDigits];
#pragma unroll
        for (int j = 0; j < 4; ++j)
          digits(fixed_point(v[2 * j], e), fixed_point(v[2 * j + 1], e), d[j]);
#pragma unroll
        for (int s = 0; s < kDigits; ++s)
          *reinterpret_cast<uint4*>(sm + (s * R + r) * kPitch + 16 * o) =
              make_uint4(d[0][s], d[1][s], d[2][s], d[3][s]);
      }
    }
  }
};

// res += Σ_k A B over [k0, k1) by a DFMA chain, for the elements set in `which`
// (bit 4 b + e: fragment register e of column block b)
template <int NB, typename SA, typename SB>
HSS_DEVINL void plain_group(const SA& A, const SB& B, int k0, int k1, uint32_t which,
                            double (&res)[NB][4]) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  for (int k = k0; k < k1; ++k)
#pragma unroll
    for (int b = 0; b < NB; ++b)
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const int r = w * 16 + (lane >> 2) + 8 * (e >> 1);
        const int c = 8 * b + 2 * (lane & 3) + (e & 1);
        if (which >> (4 * b + e) & 1) res[b][e] = fma(A.at(r, k), B.at(c, k), res[b][e]);
      }
}

// Σ_k a(l, k) b(l, k) over [k0, k1) for the lanes l set in `bad`, by the warp together; the
// lane's own sum is returned.  A warp-wide FP64 instruction takes 64 clocks of its SM
// quarter: four sums at a time on eight lanes each cost 300 clocks a sum, one on 32
// lanes 600, a lane's own chain 8192.
template <typename At, typename Bt>
HSS_DEVINL double warp_dots(uint32_t bad, int k0, int k1, At a, Bt b) {
  const int lane = threadIdx.x & 31;
  double mine = 0.0;
  while (bad) {
    const bool four = __popc(bad) > 2;
    const int width = four ? 8 : 32;
    int src[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      src[q] = __ffs(bad) - 1;   // -1: none left
      if (q == 0 || four) bad &= bad - 1;
    }
    int l = src[0];
#pragma unroll
    for (int q = 1; q < 4; ++q)
      if (four && lane >> 3 == q && src[q] >= 0) l = src[q];
    double v = 0.0;
#pragma unroll 4
    for (int k = k0 + (lane & (width - 1)); k < k1; k += width) v = fma(a(l, k), b(l, k), v);
    if (!four) {
      v += __shfl_xor_sync(0xffffffffu, v, 16);
      v += __shfl_xor_sync(0xffffffffu, v, 8);
    }
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const double x = __shfl_sync(0xffffffffu, v, 8 * q);
      if (lane == src[q] && (q == 0 || four)) mine = x;
    }
  }
  return mine;
}

// plain_group's sums by the warp together where they are few.  Called by whole warps.
template <int NB, typename SA, typename SB>
__device__ __noinline__ void small_sums(const SA& A, const SB& B, int k0, int k1, uint32_t which,
                                        double (&res)[NB][4]) {
  const int w = threadIdx.x >> 5;
  // of 128 NB: there 300 clocks a sum meet the chains' 8192 a fragment register (merges of
  // real couplings: factor of the grid covariance, N = 65536, 21.3 ms with the line at
  // half, 19.8 here)
  if (__reduce_add_sync(0xffffffffu, __popc(which)) > 104 * NB) {
    plain_group<NB>(A, B, k0, k1, which, res);
    return;
  }
#pragma unroll
  for (int b = 0; b < NB; ++b)
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      const uint32_t bad = __ballot_sync(0xffffffffu, which >> (4 * b + e) & 1);
      if (!bad) continue;
      res[b][e] += warp_dots(
          bad, k0, k1, [&](int l, int k) { return A.at(w * 16 + (l >> 2) + 8 * (e >> 1), k); },
          [&](int l, int k) { return B.at(8 * b + 2 * (l & 3) + (e & 1), k); });
    }
}

template <int BN>
constexpr int fx_smem() {
  return kDigits * (kRows + BN) * kPitch;
}

template <int BN, bool AKC, bool BKC>
__global__ void __launch_bounds__(kThreads, BN == 32 ? 2 : 3)
fx_gemm_kernel(const __grid_constant__ FxShape s) {
  constexpr int NB = BN / 8;
  extern __shared__ __align__(16) unsigned char sm[];
  __shared__ int ex[kRows + BN];   // row maxima, then the rows' exponents
  unsigned char* smA = sm;
  unsigned char* smB = sm + kDigits * kRows * kPitch;
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  const long long z = blockIdx.x / s.tiles;
  if (s.skip && s.skip[z * s.skip_stride]) return;
  int t = (int)(blockIdx.x % s.tiles), tm, tn;
  if (s.lower) {   // row block tm has the column blocks that start at or left of its last row
    tm = 0;
    for (;; ++tm) {
      const int have = min(s.tiles_n, (kRows * tm + kRows - 1) / BN + 1);
      if (t < have) break;
      t -= have;
    }
    tn = t;
  } else {
    tm = t % s.tiles_m;
    tn = t / s.tiles_m;
  }
  const int i0 = tm * kRows, j0 = tn * BN;

  float acc[kDigits][NB][4];
  double res[NB][4];
#pragma unroll
  for (int b = 0; b < NB; ++b)
#pragma unroll
    for (int e = 0; e < 4; ++e) res[b][e] = 0.0;

  // parts of the inner index (two arrays per operand in the rank-2k update)
  for (int part = 0; part * s.K1 < s.K; ++part) {
  const Strip<kRows, AKC> A{(part ? s.a.p2 : s.a.p1) + z * (part ? s.a.s2 : s.a.s1),
                            part ? s.a.ld2 : s.a.ld1, i0, s.m - 1};
  const Strip<BN, BKC> B{(part ? s.b.p2 : s.b.p1) + z * (part ? s.b.s2 : s.b.s1),
                         part ? s.b.ld2 : s.b.ld1, j0, s.n - 1};
  for (int kg = 0; kg < s.K1; kg += kGroup) {
    const int ke = min(s.K1, kg + kGroup);
    for (int r = tid; r < kRows + BN; r += kThreads) ex[r] = 0;
    __syncthreads();
    A.maxima(kg, ke, ex);
    B.maxima(kg, ke, ex + kRows);
    __syncthreads();
    int odd = 0;
    for (int r = tid; r < kRows + BN; r += kThreads) ex[r] = row_exponent(ex[r], odd);
    if (__syncthreads_or(odd)) {   // plain FP64 for this group
      plain_group<NB>(A, B, kg, ke, 0xffffffffu, res);
      __syncthreads();
      continue;
    }
    uint32_t abs_sum[NB][2];
#pragma unroll
    for (int b = 0; b < NB; ++b) abs_sum[b][0] = abs_sum[b][1] = 0;
#pragma unroll
    for (int q = 0; q < kDigits; ++q)
#pragma unroll
      for (int b = 0; b < NB; ++b)
#pragma unroll
        for (int e = 0; e < 4; ++e) acc[q][b][e] = 0.f;
    for (int kc = kg; kc < ke; kc += kChunk) {
      if (kc + kChunk <= ke) {
        A.template convert<true>(kc, ke, ex, smA);
        B.template convert<true>(kc, ke, ex + kRows, smB);
      } else {
        A.template convert<false>(kc, ke, ex, smA);
        B.template convert<false>(kc, ke, ex + kRows, smB);
      }
      __syncthreads();
#pragma unroll 1
      for (int ks = 0; ks < kChunk / 16; ++ks) {
        if (kc + 16 * ks >= ke) break;
        uint32_t a[kDigits][4];
        const uint32_t aa =
            smem_of(smA) + (w * 16 + (lane & 15)) * kPitch + ks * 32 + (lane >> 4) * 16;
#pragma unroll
        for (int q = 0; q < kDigits; ++q) ldmatrix4(a[q], aa + q * kRows * kPitch);
        uint32_t la[4];
        if (s.components) {
#pragma unroll
          for (int p = 0; p < 4; ++p) la[p] = leading(a[0][p], a[1][p]);
        }
        // two blocks of 8 columns per load (BN = 8: both halves of the 16 indices of one)
        const uint32_t ba = smem_of(smB) + ks * 32 + ((lane >> 3) & 1) * 16 +
                            ((lane & 7) + (NB > 1 ? (lane >> 4) << 3 : 0)) * kPitch;
#pragma unroll
        for (int b = 0; b < NB; b += 2) {
          uint32_t v0[4];
#pragma unroll
          for (int j = 0; j < kDigits; ++j) {
            uint32_t v[4];
            ldmatrix4(v, ba + (j * BN + 8 * b) * kPitch);
            if (j == 0) {
#pragma unroll
              for (int p = 0; p < 4; ++p) v0[p] = v[p];
            }
            if (j == 1 && s.components) {
              mma_abs(abs_sum[b], la, leading(v0[0], v[0]), leading(v0[1], v[1]));
              if (NB > 1)
                mma_abs(abs_sum[b + (NB > 1)], la, leading(v0[2], v[2]), leading(v0[3], v[3]));
            }
#pragma unroll
            for (int i = 0; i + j < kDigits; ++i) {
              mma_f16(acc[i + j][b], a[i], v[0], v[1]);
              if (NB > 1) mma_f16(acc[i + j][b + (NB > 1)], a[i], v[2], v[3]);
            }
          }
        }
      }
      __syncthreads();
    }
    // the group's sum: 2^(ea + eb - 70) (H 2^32 + L); by DFMA where S is small
    uint32_t small = 0;
#pragma unroll
    for (int b = 0; b < NB; ++b)
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        long long H = 0, L = 0;
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          H += (long long)__float2int_rn(acc[q][b][e]) * (1 << (24 - 8 * q));
          L += (long long)__float2int_rn(acc[q + 4][b][e]) * (1 << (24 - 8 * q));
        }
        const int r = w * 16 + (lane >> 2) + 8 * (e >> 1);
        const int c = 8 * b + 2 * (lane & 3) + (e & 1);
        const int E = ex[r] + ex[kRows + c];
        if (E >= kZeroRow) continue;
        if (s.components && half_of(abs_sum[b][e >> 1], e & 1) < kLeast) {
          // not for results that are not stored
          if (i0 + r < s.m && j0 + c < s.n) small |= 1u << (4 * b + e);
          continue;
        }
        const double scale = __hiloint2double((E - 1093) << 20, 0);
        res[b][e] = fma(fma((double)H, 4294967296.0, (double)L), scale, res[b][e]);
      }
    if (__any_sync(0xffffffffu, small)) small_sums<NB>(A, B, kg, ke, small, res);
    __syncthreads();
  }
  }

  double* C = s.C + z * s.sC;
  const double* Ci = s.Cin + z * s.sCin;
#pragma unroll
  for (int b = 0; b < NB; ++b)
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      const int i = i0 + w * 16 + (lane >> 2) + 8 * (e >> 1);
      const int j = j0 + 8 * b + 2 * (lane & 3) + (e & 1);
      if (i >= s.m || j >= s.n || (s.lower && i < j)) continue;
      double v = s.alpha * res[b][e];
      if (s.beta != 0.0) v = fma(s.beta, Ci[i + (long long)j * s.ldcin], v);
      C[i + (long long)j * s.ldc] = v;
      if (s.PA) {
        double* pa = s.PA + (z >> 1) * s.sPA;
        const int off = (int)(z & 1) * s.m;
        pa[(off + i) + (long long)(off + j) * s.ldpa] = v;
        if (i != j) pa[(off + j) + (long long)(off + i) * s.ldpa] = v;
      }
    }
}

// ------------------------------------------------------------------ narrow products
// n <= 16 columns (right-hand sides; B's inner index contiguous), a CTA 16 rows and
// every column.  The four warps of a team take 32 inner indices each of a group of
// 128, hold them as the MMA's fragments (inner index kw + 16 q + t + 4 j for lane t of
// a quad, in both operands) and convert them in registers: every operand element is
// read once, and the row maxima are the only thing the warps exchange before the
// MMAs.  The team's accumulators, exact integers up to 2^24, are then added through
// shared memory, each warp putting a quarter of the sums together.  TEAMS = 2: two
// groups at a time.  At the sizes of the upper levels a launch is one such chain, bound
// by its latency: a 128 x 256 node and 16 columns 8.4 us where fx_gemm_kernel, which
// reads the strips twice and passes them through shared memory, takes 24.7 us.
template <int NB, int TEAMS>
constexpr int skinny_smem() {
  return TEAMS * 4 * NB * (4 * 2 * 32 * (int)sizeof(float4) + 2 * 32 * (int)sizeof(uint32_t));
}

template <int NB, int TEAMS, bool AKC>
__global__ void __launch_bounds__(128 * TEAMS, (NB == 1 ? 4 : 2) / TEAMS)
fx_skinny_kernel(const __grid_constant__ FxShape s) {
  constexpr int R = 16, BN = 8 * NB, E = 4 * NB;   // E: fragment registers
  extern __shared__ __align__(16) float4 xch[];    // [team][warp][E][2][lane], then the
  uint32_t* xsum = reinterpret_cast<uint32_t*>(xch + TEAMS * 4 * E * 64);   // S's [..][NB][2][lane]
  __shared__ int mx[TEAMS][4][R + BN];
  const int tid = threadIdx.x, lane = tid & 31, w = (tid >> 5) & 3, team = tid >> 7;
  const int g = lane >> 2, t = lane & 3;
  const long long z = blockIdx.x / s.tiles;
  const int i0 = (int)(blockIdx.x % s.tiles) * R;
  const double* A = s.a.p1 + z * s.a.s1;
  const double* B = s.b.p1 + z * s.b.s1;
  const long long lda = s.a.ld1, ldb = s.b.ld1;
  // rows and columns past the last are read as copies of it: not stored
  const double *pa[2], *pb[NB];
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    const int i = min(i0 + 8 * h + g, s.m - 1);
    pa[h] = A + (AKC ? i * lda : i);
  }
#pragma unroll
  for (int b = 0; b < NB; ++b) pb[b] = B + min(8 * b + g, s.n - 1) * ldb;

  double res[NB];
#pragma unroll
  for (int b = 0; b < NB; ++b) res[b] = 0.0;
  chain_wait();
  chain_release();
  if (s.skip && s.skip[z * s.skip_stride]) return;

  for (int kt = 0; kt < s.K; kt += kGroup * TEAMS) {
    const int kg = kt + kGroup * team, ke = min(s.K, kg + kGroup), kw = kg + 32 * w;
    double av[2][2][4], bv[NB][2][4];   // [half of the rows or block, half of 32 indices, j]
#pragma unroll
    for (int q = 0; q < 2; ++q)
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const int k = kw + 16 * q + t + 4 * j;
        const bool in = k < ke;
#pragma unroll
        for (int h = 0; h < 2; ++h) av[h][q][j] = in ? pa[h][AKC ? (long long)k : k * lda] : 0.0;
#pragma unroll
        for (int b = 0; b < NB; ++b) bv[b][q][j] = in ? pb[b][k] : 0.0;
      }
    auto quad_max = [&](const double (&v)[2][4]) {   // over the quad's 32 indices
      int x = 0;
#pragma unroll
      for (int q = 0; q < 2; ++q)
#pragma unroll
        for (int j = 0; j < 4; ++j) x = max(x, magnitude(v[q][j]));
      x = max(x, __shfl_xor_sync(0xffffffffu, x, 1));
      return max(x, __shfl_xor_sync(0xffffffffu, x, 2));
    };
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int x = quad_max(av[h]);
      if (t == 0) mx[team][w][8 * h + g] = x;
    }
#pragma unroll
    for (int b = 0; b < NB; ++b) {
      const int x = quad_max(bv[b]);
      if (t == 0) mx[team][w][R + 8 * b + g] = x;
    }
    __syncthreads();
    int odd = 0;
    auto exponent = [&](int r) {
      return row_exponent(
          max(max(mx[team][0][r], mx[team][1][r]), max(mx[team][2][r], mx[team][3][r])), odd);
    };
    int ea[2], eb[NB];
#pragma unroll
    for (int h = 0; h < 2; ++h) ea[h] = exponent(8 * h + g);
#pragma unroll
    for (int b = 0; b < NB; ++b) eb[b] = exponent(R + 8 * b + g);
    const bool plain = __any_sync(0xffffffffu, odd);   // the same in the team's warps
    float acc[kDigits][NB][4];
#pragma unroll
    for (int d = 0; d < kDigits; ++d)
#pragma unroll
      for (int b = 0; b < NB; ++b)
#pragma unroll
        for (int e = 0; e < 4; ++e) acc[d][b][e] = 0.f;
    uint32_t abs_sum[NB][2];
#pragma unroll
    for (int b = 0; b < NB; ++b) abs_sum[b][0] = abs_sum[b][1] = 0;
    if (!plain) {
#pragma unroll
      for (int q = 0; q < 2; ++q) {
        if (kw + 16 * q < ke) {
          uint32_t bd[NB][2][kDigits], ad[4][kDigits];
#pragma unroll
          for (int b = 0; b < NB; ++b)
#pragma unroll
            for (int p = 0; p < 2; ++p)
              digits(fixed_point(bv[b][q][2 * p], eb[b]), fixed_point(bv[b][q][2 * p + 1], eb[b]),
                     bd[b][p]);
#pragma unroll
          for (int p = 0; p < 4; ++p)   // fragment register p: row half p & 1, indices p >> 1
            digits(fixed_point(av[p & 1][q][2 * (p >> 1)], ea[p & 1]),
                   fixed_point(av[p & 1][q][2 * (p >> 1) + 1], ea[p & 1]), ad[p]);
          if (s.components) {
            uint32_t la[4];
#pragma unroll
            for (int p = 0; p < 4; ++p) la[p] = leading(ad[p][0], ad[p][1]);
#pragma unroll
            for (int b = 0; b < NB; ++b)
              mma_abs(abs_sum[b], la, leading(bd[b][0][0], bd[b][0][1]),
                      leading(bd[b][1][0], bd[b][1][1]));
          }
#pragma unroll
          for (int i = 0; i < kDigits; ++i) {
            const uint32_t a[4] = {ad[0][i], ad[1][i], ad[2][i], ad[3][i]};
#pragma unroll
            for (int j = 0; i + j < kDigits; ++j)
#pragma unroll
              for (int b = 0; b < NB; ++b) mma_f16(acc[i + j][b], a, bd[b][0][j], bd[b][1][j]);
          }
        }
      }
    }
    float4* mine = xch + (team * 4 + w) * (E * 64) + lane;
#pragma unroll
    for (int b = 0; b < NB; ++b)
#pragma unroll
      for (int e = 0; e < 4; ++e)
#pragma unroll
        for (int h = 0; h < 2; ++h)
          mine[((b * 4 + e) * 2 + h) * 32] = make_float4(acc[4 * h][b][e], acc[4 * h + 1][b][e],
                                                         acc[4 * h + 2][b][e], acc[4 * h + 3][b][e]);
#pragma unroll
    for (int b = 0; b < NB; ++b)
#pragma unroll
      for (int h = 0; h < 2; ++h)
        xsum[((team * 4 + w) * NB + b) * 64 + h * 32 + lane] = abs_sum[b][h];
    __syncthreads();
    // warp w: fragment register w of every block, row g + 8 (w >> 1), column 2 t + (w & 1)
#pragma unroll
    for (int b = 0; b < NB; ++b) {
      const int ex =
          __shfl_sync(0xffffffffu, eb[b], (2 * t + (w & 1)) * 4) + (w & 2 ? ea[1] : ea[0]);
      const int row = 8 * (w >> 1) + g, col = 8 * b + 2 * t + (w & 1);
      if (!plain) {
        float sum = 0.f;
#pragma unroll
        for (int u = 0; u < 4; ++u)
          sum += half_of(xsum[((team * 4 + u) * NB + b) * 64 + (w >> 1) * 32 + lane], w & 1);
        const bool zero = ex >= kZeroRow, small = s.components && !zero && sum < kLeast;
        // by DFMA; not for results that are not stored
        const uint32_t bad = __ballot_sync(0xffffffffu, small && i0 + row < s.m && col < s.n);
        if (bad)
          res[b] += warp_dots(
              bad, kg, ke,
              [&](int l, int k) {
                const long long i = i0 + 8 * (w >> 1) + (l >> 2);
                return A[AKC ? i * lda + k : i + k * lda];
              },
              [&](int l, int k) { return B[(8 * b + 2 * (l & 3) + (w & 1)) * ldb + k]; });
        if (zero || small) continue;
        long long v[2];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          float4 x = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
          for (int u = 0; u < 4; ++u) {
            const float4 y = xch[(team * 4 + u) * (E * 64) + ((b * 4 + w) * 2 + h) * 32 + lane];
            x.x += y.x, x.y += y.y, x.z += y.z, x.w += y.w;
          }
          v[h] = (long long)__float2int_rn(x.x) * (1 << 24) +
                 (long long)__float2int_rn(x.y) * (1 << 16) +
                 (long long)__float2int_rn(x.z) * (1 << 8) + __float2int_rn(x.w);
        }
        const double scale = __hiloint2double((ex - 1093) << 20, 0);
        res[b] = fma(fma((double)v[0], 4294967296.0, (double)v[1]), scale, res[b]);
      } else {   // plain FP64 for this group
        const int i = min(i0 + row, s.m - 1), j = min(col, s.n - 1);
        for (int k = kg; k < ke; ++k)
          res[b] = fma(A[AKC ? i * lda + k : i + k * lda], B[j * ldb + k], res[b]);
      }
    }
  }

  if (TEAMS > 1) {
    double* sum = reinterpret_cast<double*>(xch);
    __syncthreads();
    if (team == 1) {
#pragma unroll
      for (int b = 0; b < NB; ++b) sum[b * 128 + (tid & 127)] = res[b];
    }
    __syncthreads();
    if (team == 1) return;
#pragma unroll
    for (int b = 0; b < NB; ++b) res[b] += sum[b * 128 + tid];
  }
  double* C = s.C + z * s.sC;
  const double* Ci = s.Cin + z * s.sCin;
#pragma unroll
  for (int b = 0; b < NB; ++b) {
    const int i = i0 + 8 * (w >> 1) + g, j = 8 * b + 2 * t + (w & 1);
    if (i >= s.m || j >= s.n) continue;
    double v = s.alpha * res[b];
    if (s.beta != 0.0) v = fma(s.beta, Ci[i + (long long)j * s.ldcin], v);
    C[i + (long long)j * s.ldc] = v;
  }
}

template <int NB, int TEAMS>
cudaError_t launch_skinny(FxShape& s, int batch, cudaStream_t st) {
  s.tiles = (s.m + 15) / 16;
  const auto kernel = s.a.kc ? fx_skinny_kernel<NB, TEAMS, true> : fx_skinny_kernel<NB, TEAMS, false>;
  const int bytes = skinny_smem<NB, TEAMS>();
  const cudaError_t e = fx_allow_smem(reinterpret_cast<const void*>(kernel), bytes);
  if (e != cudaSuccess) return e;
  return launch_chained(kernel, dim3((unsigned)((long long)s.tiles * batch)), 128 * TEAMS, bytes,
                        st, s);
}

template <int BN, bool AKC, bool BKC>
cudaError_t launch(FxShape& s, int batch, cudaStream_t st) {
  s.tiles_m = (s.m + kRows - 1) / kRows;
  s.tiles_n = (s.n + BN - 1) / BN;
  s.tiles = s.tiles_m * s.tiles_n;
  if (s.lower) {
    s.tiles = 0;
    for (int tm = 0; tm < s.tiles_m; ++tm) {
      const int have = (kRows * tm + kRows - 1) / BN + 1;
      s.tiles += have < s.tiles_n ? have : s.tiles_n;
    }
  }
  const cudaError_t e = fx_allow_smem(
      reinterpret_cast<const void*>(fx_gemm_kernel<BN, AKC, BKC>), fx_smem<BN>());
  if (e != cudaSuccess) return e;
  fx_gemm_kernel<BN, AKC, BKC>
      <<<(unsigned)((long long)s.tiles * batch), kThreads, fx_smem<BN>(), st>>>(s);
  return cudaGetLastError();
}

template <int BN>
cudaError_t launch_modes(FxShape& s, int batch, cudaStream_t st) {
  if (s.a.kc) return s.b.kc ? launch<BN, true, true>(s, batch, st) : launch<BN, true, false>(s, batch, st);
  return s.b.kc ? launch<BN, false, true>(s, batch, st) : launch<BN, false, false>(s, batch, st);
}

}  // namespace

cudaError_t fx_allow_smem(const void* kernel, int bytes) {
  static std::mutex mu;
  static std::set<std::pair<int, const void*>> memo;
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  std::lock_guard<std::mutex> g(mu);
  const auto key = std::make_pair(dev, kernel);
  if (memo.count(key)) return cudaSuccess;
  e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
  if (e == cudaSuccess) memo.insert(key);   // a failure is tried, and reported, again
  return e;
}

cudaError_t fx_gemm(int m, int n, int K, const FxOperand& a, const FxOperand& b, double alpha,
                    double beta, const double* Cin, int ldcin, long long sCin, double* C, int ldc,
                    long long sC, int batch, bool lower, double* PA, int ldpa, long long sPA,
                    cudaStream_t st, bool components, const int* skip, int skip_stride) {
  FxShape s{m, n, K, a.p2 ? K / 2 : K, a, b, alpha, beta, Cin ? Cin : C, ldcin, sCin, C, ldc, sC, lower ? 1 : 0,
            PA, ldpa, sPA, 0, 0, 0, components ? 1 : 0, skip, skip_stride};
  // Narrow products (B's inner index contiguous).  Up to 8 columns fx_skinny_kernel is
  // the faster one at every size (512 x 512, 512 nodes: 481 against 506 us; 128 nodes:
  // 128 against 150; 128 x 128, 8 nodes: 6.2 against 10.5).  With 9 to 16 it wins while
  // the 64-row tiles of the other kernel leave SMs idle (128 x 256, 16 nodes: 8.4
  // against 24.7 us; 33 nodes 12.5 against 22.7), and loses where they fill the chip (256
  // nodes: 62 against 57; 512 x 512, 512 nodes: 950 against 660): there the 64 rows
  // share one conversion of B.  Two groups at a time while a wave of CTAs takes them
  // all (8 nodes of 128 x 256, 8 columns: 6.3 against 8.2 us; 264 tiles: 14.5
  // against 12.5).
  if (n <= 16 && b.kc && !a.p2 && !lower) {
    const bool two = K > kGroup && (long long)((m + 15) / 16) * batch <= 152;
    if (n <= 8) return two ? launch_skinny<1, 2>(s, batch, st) : launch_skinny<1, 1>(s, batch, st);
    if ((long long)((m + kRows - 1) / kRows) * batch <= 304)
      return two ? launch_skinny<2, 2>(s, batch, st) : launch_skinny<2, 1>(s, batch, st);
  }
  if (n <= 8) return launch_modes<8>(s, batch, st);
  if (n <= 16) return launch_modes<16>(s, batch, st);
  return launch_modes<32>(s, batch, st);
}

void dgemm_batched(bool transA, bool transB, int m, int n, int k, double alpha, const double* A,
                   int lda, long long sA, const double* B, int ldb, long long sB, double beta,
                   double* C, int ldc, long long sC, int batch, cudaStream_t st, bool components) {
  if (m <= 0 || n <= 0 || k <= 0 || batch <= 0) return;
  // A few inner indices and columns on few rows (the tree of a rank <= 8 matrix):
  // the FP64 pipe's kernels take 4.2 us against 6.2 us, whose digits are padded to
  // 32 indices.  From 16 indices, or 32 columns, on the sliced product is the
  // faster one at every size (16 indices: 6.2 us both; 128 rows, 128 indices, 1
  // column: 10.3 against 22.6 us; 512 x 128 x 512, 512 nodes: 4.6 against 27.5 ms).
  if (k <= 8 && n <= 16 && (long long)m * batch <= 16384) {
    gemm_batched<double>(transA, transB, m, n, k, alpha, A, lda, sA, B, ldb, sB, beta, C, ldc, sC,
                         batch, st);
    return;
  }
  const FxOperand a{A, lda, sA, transA}, b{B, ldb, sB, !transB};
  fx_gemm(m, n, k, a, b, alpha, beta, C, ldc, sC, C, ldc, sC, batch, false, nullptr, 0, 0, st,
          components);
}

void dsyr2k_lower_batched(int m, int k, const double* A, int lda, long long sA, const double* P,
                          int ldp, long long sP, const double* Q, int ldq, long long sQ, double* M,
                          int ldm, long long sM, int batch, cudaStream_t st) {
  if (m <= 0 || k <= 0 || batch <= 0) return;
  // A - [P Q] [Q P]ᵀ, a Householder transformation
  const FxOperand a{P, ldp, sP, false, Q, ldq, sQ}, b{Q, ldq, sQ, false, P, ldp, sP};
  fx_gemm(m, m, 2 * k, a, b, -1.0, 1.0, A, lda, sA, M, ldm, sM, batch, true, nullptr, 0, 0, st,
          /*components=*/false);
}

void dsyrk_lower_batched(int m, int k, const double* A, int lda, long long sA, const double* P,
                         int ldp, long long sP, double* M, int ldm, long long sM, double* PA,
                         int ldpa, long long sPA, int batch, cudaStream_t st) {
  if (m <= 0 || k <= 0 || batch <= 0) return;
  const FxOperand a{P, ldp, sP, false};
  fx_gemm(m, m, k, a, a, -1.0, 1.0, A, lda, sA, M, ldm, sM, batch, true, PA, ldpa, sPA, st);
}
