// Offline rotation calibration on the GPU (Sec. 4.2-4.5; Appendix, "OptR
// Algorithm"): per KV head, Adam on the skew generators A_K and A_V of
//   R_K = R_K^0 exp(A_K - A_K^T),  R_V = R_V^0 exp(A_V - A_V^T)
// against the output-aware objectives
//   L_K = mean_{t,j} KL(p_t || p_t^K) + lambda ||e_K(t,j)||^2 / d_model,
//   L_V = mean_{t,j} ||e_V(t,j)||^2 / d_model,
// with the cache's INT2 quantizer Q2 inside the effective keys and values and
// its straight-through gradient, and held-out selection of the rotations.
//
// Everything is float64: the calibration is a one-time offline pass, and float64
// keeps its trajectory reproducible.  The matrix products, its bulk, run on the
// fp16 tensor cores as exact products of digits (gemm_digits_kernel), the rest on
// the CUDA cores.
// The gradient is written out (no autograd):
//   keys    Z = (K - mu) R, Zh = Q2(Z), Kt = Zh R^T, l = scale q Kt^T
//           dl = c [(pk - p) + pk (gv - sum_s pk gv)],  gv = U V^T,
//           U = (2 lambda / d_model) e W_O,  c = 1 / (nt g)
//           dKt = dl^T q,  dR = dKt^T Zh + (K - mu)^T (1{inside} (dKt R))
//   values  Vt = Q2(V R) R^T, e = phat_nw (Vt - V) W_O^T
//           dVt = phat_nw^T U,  U = 2 c / d_model e W_O
//           dR = dVt^T Zh + V^T (1{inside} (dVt R))
//   both    dE = R0^T dR, dS = L_exp(S^T, dE), dA = dS - dS^T
// where L_exp(X, H) is the Frechet derivative of the matrix exponential
// (the adjoint of L_exp(S, .) is L_exp(S^T, .)); it is taken as
// dS^T = L_exp(S, dR^T R0).  exp comes from a Taylor polynomial with scaling
// and squaring, L_exp from the same chain of products differentiated
// (mat_product_kernel, expm and generator_grad below).
#include <math.h>
#include <string.h>

#include <algorithm>
#include <vector>

#include "optr_internal.cuh"

namespace optr {
namespace {

constexpr int kCD = 128;  // head dimension d

// ------------------------------------------------------------------ GEMM
// C[b] = alpha op(A[b]) op(B[b]), float64, row-major with leading dimensions;
// op = transpose when tA / tB (gemm_digits_kernel below).
struct Gemm {
  int M, N, K;
  const double* A;
  long long lda, sA;
  int tA;
  const double* B;
  long long ldb, sB;
  int tB;
  double* C;
  long long ldc, sC;
  double alpha;
  // depth continued with a second pair of the same shape and layout (null: no)
  const double *A2, *B2;
  const double* mul;  // C = mul .* (..) when given, row-major with ldc
  const double* sub;  // C = .. - sub when given, likewise
};

// The product runs on the fp16 tensor cores after a split of both factors into
// small integers, whose products are exact (the scheme of Ozaki, Ogita, Oishi and
// Rump, "Error-free transformations of matrix multiplication", 2012): this GPU does
// 2 float64 FMAs per clock and SM, three orders of magnitude below its tensor
// cores.  Per k chunk of 128, a row of A (a column of B) is rounded to
// fixed-point numbers under its own largest exponent, 62 bits and sign, in
// eight balanced base-256 digits d_0 .. d_7 (|d_0| <= 64, else |d| <= 128),
// which are exact fp16 values.  All digit products of one weight d = i + j are
// summed in one float32 accumulator: at most 128 x 7 x 2^14 < 2^24, so every
// sum is exact.  The weights 0 .. 8 (43 of the 64 products; what is left out of
// one product is below 2^-67 of the largest one) are put together in 64-bit
// integers and added to the float64 result, one rounding per 128 products.
//
// What the split loses is bounded by the largest elements of the row and of the
// column, about 2^-62 of max|a| max|b| per chunk, not by the sum: far better than
// a float64 FMA chain while large elements meet large ones, unbounded where they
// do not (an outlier channel against a zero of the rotation).  So one more mma
// per step multiplies the magnitudes, two digits each, and outputs with
// sum |a b| below 1/1024 of the largest product possible take their chunk's sum
// from float64 FMAs (float64_sums; as good as none in a calibration on synthetic
// traces), rows and columns with a NaN or an infinity too.  Largest error against
// sum |a b| at depth 128, float64 FMA chain / digits alone / both as here: normal
// 6e-16 / 5e-17 / 5e-17; softmax of logits of deviation 3 and 10 x t(4) 2e-15 /
// 1e-14 / 3e-16; exponents spread over 80 bits 1.4e-15 / 9e-9 / 3e-16; an outlier
// channel of 1e8 2.7e-15 / 6e-15 / 6e-16, times an identity 0 / 4e-6 / 0.  (Seven
// digits, 54 bits, need that line at 1/8 for the errors of an FMA chain: 6% of the
// probabilities x values of a calibration, 20 + 20 steps 33.7 ms instead of 26.2.)
// What bounds it: per CTA and chunk 352 mma a warp (5.7 us at one m16n8k16 per 8
// cycles and SM quarter), the split of both tiles (24 values a thread, ~50
// integer instructions each, 2.5 us) and the load's latency, one after the
// other, as 197 KB of digits leave room for one CTA per SM.  64 x 32 tiles make
// the calibration's products (2048 or 4 x 64 rows, 128 columns or the reverse)
// one wave of 128 CTAs: 2048 x 128 x 128 takes 20.6 us from cold caches (with
// seven digits 17.8, 25 with 32 x 32 tiles in two waves, 21 with 64-deep chunks
// and two CTAs per SM).
// Products with fewer than half as many tiles and chunks as SMs take 32 x 16
// tiles (8 steps on 256 tokens: 4.4 ms, 5.0 with 64 x 32 throughout).
//
// With kc > 1 CTA z of a product covers the z-th part of k and writes its sum
// to P[z][b]; the last of the tile's kc CTAs to finish (a per-tile arrival
// counter, left at 0 again) adds the parts in a fixed order, z = 0 .. kc-1,
// so the result does not depend on which CTA that is.
constexpr int kGK = 128;     // k chunk
constexpr int kDigits = 8;
constexpr int kWeights = 9;
constexpr int kBadExp = 1 << 20;  // exponent of a row with a non-finite value

// MT x NT outputs, one warp per 16 x 8 of them
template <int MT, int NT>
struct GemmTile {
  static constexpr int kThreads = MT / 16 * (NT / 8) * 32;
  // digit planes [digit][row][k]; 16-byte piece p of row r at p ^ (r % 8)
  __half a[kDigits][MT][kGK];
  __half b[kDigits][NT][kGK];
  int emax[MT + NT][17];  // largest exponents of a row's sixteen 8-element pieces
  int e[MT + NT];
};

__device__ __forceinline__ void digits_mma(float (&d)[4], const uint32_t (&a)[4], uint32_t b0,
                                           uint32_t b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 "
      "{%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};\n"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
__device__ __forceinline__ void digits_ldsm(uint32_t (&r)[4], const void* p) {
  const unsigned s = static_cast<unsigned>(__cvta_generic_to_shared(p));
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];\n"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(s));
}

// |x| = m 2^(e - 1075), m < 2^53, e = max(biased exponent, 1).  The largest
// exponent of a row: the maximum over its values of field(x), then row_exponent.
__device__ __forceinline__ int field(double x) { return __double2hiint(x) & 0x7ff00000; }
__device__ __forceinline__ int row_exponent(int f) {
  return f == 0x7ff00000 ? kBadExp : max(f >> 20, 1);
}

// x as a fixed-point integer with unit 2^(e_row - 1084), rounded, |result| <=
// 2^62, plus the bias that makes its bytes digit + 128.
constexpr unsigned long long kBias = 0x8080808080808080ull;
__device__ __noinline__ unsigned long long fixed_point_small(double x, int e_row) {
  const unsigned long long bits = __double_as_longlong(x);
  if (bits << 1 == 0) return kBias;
  const int e = (int)(bits >> 52) & 2047;
  unsigned long long m = (bits & 0xfffffffffffffull) | (e ? 1ull << 52 : 0ull);
  const int sh = e_row - max(e, 1);
  m <<= 9;
  if (sh > 0) m = sh < 64 ? (m + (1ull << (sh - 1))) >> sh : 0ull;
  const long long f = (long long)bits < 0 ? -(long long)m : (long long)m;
  return (unsigned long long)f + kBias;
}
// The same for e_row >= kFastExp, in 15 integer instructions: zeros and
// subnormals (no implicit bit) are shifted out with the rest of what is below
// the unit.
constexpr int kFastExp = 66;
__device__ __forceinline__ unsigned long long fixed_point(double x, int e_row) {
  const int hi = __double2hiint(x);
  const unsigned lo = (unsigned)__double2loint(x);
  const unsigned mh = ((unsigned)hi & 0xfffffu) | 0x100000u;
  // one fractional bit more, then one addition rounds (half away from zero)
  const unsigned long long m = ((unsigned long long)__funnelshift_l(lo, mh, 10) << 32) | (lo << 10);
  const int sh = min(e_row - ((hi >> 20) & 2047), 63);
  const unsigned long long t = ((m >> sh) + 1) >> 1;
  const unsigned long long sg = (long long)(hi >> 31);
  return (t ^ sg) - sg + kBias;
}

// The digits of eight k of row r (piece kg) into the planes.
template <int ROWS, int KS>
__device__ __forceinline__ void store_digits(__half (*planes)[ROWS][KS], int r, int kg,
                                             const double (&x)[8], int e_row) {
  uint32_t h[kDigits][4];
  const __half2 off = __float2half2_rn(1152.f);  // 1024 + byte - 1152 = digit
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    unsigned long long f0, f1;
    if (e_row >= kFastExp) {
      f0 = fixed_point(x[2 * q], e_row);
      f1 = fixed_point(x[2 * q + 1], e_row);
    } else {
      f0 = fixed_point_small(x[2 * q], e_row);
      f1 = fixed_point_small(x[2 * q + 1], e_row);
    }
    const uint32_t l0 = (uint32_t)f0, l1 = (uint32_t)f1, u0 = (uint32_t)(f0 >> 32), u1 = (uint32_t)(f1 >> 32);
    const uint32_t b01 = __byte_perm(l0, l1, 0x5140), b23 = __byte_perm(l0, l1, 0x7362),
                   b45 = __byte_perm(u0, u1, 0x5140), b67 = __byte_perm(u0, u1, 0x7362);
    const uint32_t w[kDigits] = {
        __byte_perm(b67, 0x64646464u, 0x4342), __byte_perm(b67, 0x64646464u, 0x4140),
        __byte_perm(b45, 0x64646464u, 0x4342), __byte_perm(b45, 0x64646464u, 0x4140),
        __byte_perm(b23, 0x64646464u, 0x4342), __byte_perm(b23, 0x64646464u, 0x4140),
        __byte_perm(b01, 0x64646464u, 0x4342), __byte_perm(b01, 0x64646464u, 0x4140)};
#pragma unroll
    for (int d = 0; d < kDigits; ++d) {
      const __half2 v = __hsub2(*reinterpret_cast<const __half2*>(&w[d]), off);
      h[d][q] = *reinterpret_cast<const uint32_t*>(&v);
    }
  }
#pragma unroll
  for (int d = 0; d < kDigits; ++d)
    *reinterpret_cast<uint4*>(&planes[d][r][(kg ^ (r & 7)) * 8]) =
        make_uint4(h[d][0], h[d][1], h[d][2], h[d][3]);
}

// |256 d_0 + d_1| of two values as fp16 (at most 16512)
__device__ __forceinline__ uint32_t digits_abs(uint32_t d0, uint32_t d1) {
  const __half2 m = __hfma2(*reinterpret_cast<const __half2*>(&d0), __float2half2_rn(256.f),
                            *reinterpret_cast<const __half2*>(&d1));
  return *reinterpret_cast<const uint32_t*>(&m) & 0x7fff7fffu;
}

// One 16-deep step of the 43 digit products on the 16 x 8 outputs at (r0, c0),
// and of the magnitudes in mag; p0: first of the step's two 16-byte pieces.
template <int MT, int NT, int KS>
__device__ __forceinline__ void digits_step(float (&acc)[kWeights][4], float (&mag)[4],
                                            const __half (*a)[MT][KS], const __half (*b)[NT][KS],
                                            int r0, int c0, int p0, int lane) {
  uint32_t fb[kDigits][2];
  {
    // lanes 0-15 address digit j, 16-31 digit j + 1
    const int r = c0 + (lane & 7), p = p0 + ((lane >> 3) & 1);
#pragma unroll
    for (int j = 0; j < kDigits; j += 2) {
      uint32_t x[4];
      digits_ldsm(x, &b[j + (lane >> 4)][r][(p ^ (r & 7)) * 8]);
      fb[j][0] = x[0];
      fb[j][1] = x[1];
      fb[j + 1][0] = x[2];
      fb[j + 1][1] = x[3];
    }
  }
  const int r = r0 + (lane & 15), p = p0 + (lane >> 4);
  uint32_t ma[4];
#pragma unroll
  for (int i = 0; i < kDigits; ++i) {
    uint32_t fa[4];
    digits_ldsm(fa, &a[i][r][(p ^ (r & 7)) * 8]);
#pragma unroll
    for (int j = 0; j < kDigits; ++j)
      if (i + j < kWeights) digits_mma(acc[i + j], fa, fb[j][0], fb[j][1]);
    if (i < 2) {
#pragma unroll
      for (int x = 0; x < 4; ++x) ma[x] = i == 0 ? fa[x] : digits_abs(ma[x], fa[x]);
      if (i == 1)
        digits_mma(mag, ma, digits_abs(fb[0][0], fb[1][0]), digits_abs(fb[0][1], fb[1][1]));
    }
  }
}

// Whether a chunk's sum of digit products is too small against its row's and
// column's largest elements (exponents e0, e1; all zero or below 2^-1021: e = 1)
// to be as accurate as float64 operations, or has a factor that is not finite:
// see gemm_digits_kernel.
constexpr float kMagMin = 262144.f;  // 2^28 / 1024
__device__ __forceinline__ bool digits_lost(float mag, int e0, int e1) {
  return max(e0, e1) >= kBadExp || (mag < kMagMin && min(e0, e1) > 1);
}

// For the lanes with `lost`: v = sum_{k < n} a[k sa] b[k sb] in float64.  Four of
// them at a time, eight lanes each; the whole warp calls it.
__device__ __forceinline__ void float64_sums(bool lost, const double* a, long long sa,
                                             const double* b, long long sb, int n, double& v) {
  const int lane = threadIdx.x & 31;
  unsigned todo = __ballot_sync(0xffffffffu, lost);
  while (todo != 0) {
    int who[4];  // -1: none left
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      who[i] = __ffs(todo) - 1;
      todo &= todo - 1;
    }
    const int lo = lane & 8 ? who[1] : who[0], hi = lane & 8 ? who[3] : who[2];
    const int src = lane & 16 ? hi : lo;
    const double* x = reinterpret_cast<const double*>(
        __shfl_sync(0xffffffffu, reinterpret_cast<unsigned long long>(a), src & 31));
    const double* y = reinterpret_cast<const double*>(
        __shfl_sync(0xffffffffu, reinterpret_cast<unsigned long long>(b), src & 31));
    double s = 0.0;
    if (src >= 0) {
#pragma unroll 4
      for (int k = lane & 7; k < n; k += 8) s = fma(__ldcg(x + k * sa), __ldcg(y + k * sb), s);
    }
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const double r = __shfl_sync(0xffffffffu, s, 8 * i);
      if (lane == who[i]) v = r;
    }
  }
}

// sum_d acc_d 256^-d of output i as hi 2^-24 + lo 2^-64 (|sum| < 2^20 over a depth
// of 128).  A weight alone is below 2^24, a pair of them past 32 bits: |w_7|
// reaches 128 x 7 x 2^14 where digits repeat (constant rows).
struct DigitSum {
  long long hi, lo;
};
__device__ __forceinline__ DigitSum digits_sum(const float (&acc)[kWeights][4], int i) {
  int w[kWeights];
#pragma unroll
  for (int d = 0; d < kWeights; ++d) w[d] = __float2int_rn(acc[d][i]);
  auto pair = [&](int d) { return (long long)w[d] * 256 + w[d + 1]; };
  return {(pair(0) << 16) + pair(2), (pair(4) << 24) + (pair(6) << 8) + w[8]};
}

// v + t 2^(E0 + E1 - 12 - f), |x| < 2^E in a row, E = e - 1022; of t at least the
// first 61 bits are kept
__device__ __forceinline__ double digits_add(double v, DigitSum t, int e0, int e1, int f) {
  const int drop = max(43 - __clzll(t.hi ^ (t.hi >> 63)), 0);  // of the 40 bits below hi
  const long long n = (t.hi << (40 - drop)) + ((t.lo + ((1ll << drop) >> 1)) >> drop);
  const int sc = e0 + e1 - 2 * 1022 - 76 + drop - f;
  if (sc >= -1022 && sc <= 1023)
    return fma((double)n, __hiloint2double((sc + 1023) << 20, 0), v);
  return v + scalbn((double)n, sc);
}

// The pieces of a tile of R rows that a thread loads and splits: piece p of a
// row holds k = p, p + 16, .. p + 112 (both operands alike); lanes run along the
// contiguous dimension (`rows`: k), so that a warp reads whole sectors.
template <int R, int THR>
struct Pieces {
  static constexpr int kN = R * 16 / THR;
  double x[kN][8];
  __device__ __forceinline__ static int row(bool rows, int u) {
    const int t = threadIdx.x + u * THR;
    return rows ? t >> 4 : t % R;
  }
  __device__ __forceinline__ static int piece(bool rows, int u) {
    const int t = threadIdx.x + u * THR;
    return rows ? t & 15 : t / R;
  }
  // rows r0 .. of nr, depth k0 .. ke; zeros outside
  __device__ __forceinline__ void load(const double* A, long long ld, bool rows, int r0, int nr,
                                       int k0, int ke) {
#pragma unroll
    for (int u = 0; u < kN; ++u) {
      const int r = r0 + row(rows, u), k = k0 + piece(rows, u);
      const double* a = rows ? A + r * ld + k : A + k * ld + r;
      const long long step = rows ? 16 : 16 * ld;
      if (r < nr && k + 112 < ke) {
#pragma unroll
        for (int i = 0; i < 8; ++i) x[u][i] = __ldcg(a + i * step);
      } else {
#pragma unroll
        for (int i = 0; i < 8; ++i) x[u][i] = r < nr && k + 16 * i < ke ? __ldcg(a + i * step) : 0.0;
      }
    }
  }
  __device__ __forceinline__ void exponents(int (*emax)[17], bool rows) const {
#pragma unroll
    for (int u = 0; u < kN; ++u) {
      int e = 0;
#pragma unroll
      for (int i = 0; i < 8; ++i) e = max(e, field(x[u][i]));
      emax[row(rows, u)][piece(rows, u)] = e;
    }
  }
  __device__ __forceinline__ void split(__half (*planes)[R][kGK], const int (*emax)[17], int* er,
                                        bool rows) const {
#pragma unroll
    for (int u = 0; u < kN; ++u) {
      const int r = row(rows, u), p = piece(rows, u);
      int e = emax[r][0];
#pragma unroll
      for (int i = 1; i < 16; ++i) e = max(e, emax[r][i]);
      e = row_exponent(e);
      store_digits(planes, r, p, x[u], e);
      if (p == 0) er[r] = e;
    }
  }
};

template <int MT, int NT>
__global__ void __launch_bounds__(GemmTile<MT, NT>::kThreads)
    gemm_digits_kernel(Gemm g, int kc, double* P, int* tcnt) {
  using Tile = GemmTile<MT, NT>;
  constexpr int THR = Tile::kThreads;
  extern __shared__ __align__(16) unsigned char gsm_[];
  Tile& S = *reinterpret_cast<Tile*>(gsm_);
  __shared__ int s_last;
  const int b = blockIdx.z / kc, z = blockIdx.z % kc;
  const int tn = (g.N + NT - 1) / NT;  // row tiles may exceed a grid's y limit
  const int m0 = blockIdx.x / tn * MT, n0 = blockIdx.x % tn * NT;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  double* C = g.C + (long long)b * g.sC;
  pdl_wait();
  pdl_trigger();
  // this CTA's chunks: part z of kc
  const int n1 = (g.K + kGK - 1) / kGK, nsl = g.A2 != nullptr ? 2 * n1 : n1;
  const int cb = (int)((long long)z * nsl / kc), ce = (int)((long long)(z + 1) * nsl / kc);
  const bool a_rows = !g.tA, b_rows = g.tB;  // k contiguous
  const int wm = 16 * (warp % (MT / 16)), wn = 8 * (warp / (MT / 16));
  double out[4] = {0.0, 0.0, 0.0, 0.0};
  for (int ch = cb; ch < ce; ++ch) {
    const bool second = ch >= n1;
    const double* A = (second ? g.A2 : g.A) + (long long)b * g.sA;
    const double* B = (second ? g.B2 : g.B) + (long long)b * g.sB;
    const int k0 = (second ? ch - n1 : ch) * kGK;
    {
      Pieces<MT, THR> pa;
      Pieces<NT, THR> pb;
      pa.load(A, g.lda, a_rows, m0, g.M, k0, g.K);
      pb.load(B, g.ldb, b_rows, n0, g.N, k0, g.K);
      pa.exponents(S.emax, a_rows);
      pb.exponents(S.emax + MT, b_rows);
      __syncthreads();  // (and the previous chunk's digits and exponents have been read)
      pa.split(S.a, S.emax, S.e, a_rows);
      pb.split(S.b, S.emax + MT, S.e + MT, b_rows);
      __syncthreads();
    }
    float acc[kWeights][4], mag[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
    for (int d = 0; d < kWeights; ++d)
#pragma unroll
      for (int i = 0; i < 4; ++i) acc[d][i] = 0.f;
#pragma unroll 1
    for (int ks = 0; ks < kGK / 16; ++ks) digits_step(acc, mag, S.a, S.b, wm, wn, 2 * ks, lane);
    unsigned lost = 0;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int r = wm + (lane >> 2) + 8 * (i >> 1), c = wn + 2 * (lane & 3) + (i & 1);
      const int e0 = S.e[r], e1 = S.e[MT + c];
      if (!digits_lost(mag[i], e0, e1)) out[i] = digits_add(out[i], digits_sum(acc, i), e0, e1, 0);
      else if (m0 + r < g.M && n0 + c < g.N) lost |= 1u << i;
    }
    if (__any_sync(0xffffffffu, lost != 0)) {
#pragma unroll 1
      for (int i = 0; i < 4; ++i) {
        const int r = m0 + wm + (lane >> 2) + 8 * (i >> 1), c = n0 + wn + 2 * (lane & 3) + (i & 1);
        double x = 0.0;
        float64_sums(lost >> i & 1, a_rows ? A + r * g.lda + k0 : A + k0 * g.lda + r,
                     a_rows ? 1 : g.lda, b_rows ? B + c * g.ldb + k0 : B + k0 * g.ldb + c,
                     b_rows ? 1 : g.ldb, min(kGK, g.K - k0), x);
#pragma unroll
        for (int j = 0; j < 4; ++j)
          if (j == i) out[j] += x;
      }
    }
    if (ch + 1 < ce) __syncthreads();
  }
  auto store = [&](int r, int c, double x) {
    const long long i = r * g.ldc + c;
    if (g.alpha != 1.0) x *= g.alpha;
    if (g.sub != nullptr) x -= __ldcg(g.sub + i);
    if (g.mul != nullptr) x *= __ldcg(g.mul + i);
    C[i] = x;
  };
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int r = m0 + wm + (lane >> 2) + 8 * (i >> 1), c = n0 + wn + 2 * (lane & 3) + (i & 1);
    if (r >= g.M || c >= g.N) continue;
    if (kc > 1)
      P[(((long long)z * gridDim.z / kc + b) * g.M + r) * g.N + c] = out[i];
    else
      store(r, c, out[i]);
  }
  if (kc == 1) return;
  // split K: the tile's last CTA to arrive adds the kc sums in order
  __threadfence();
  __syncthreads();
  const int tile_id = b * gridDim.x + blockIdx.x;
  if (tid == 0) s_last = atomicAdd(tcnt + tile_id, 1) == kc - 1;
  __syncthreads();
  if (!s_last) return;
  __threadfence();
  const int batch = gridDim.z / kc;
#pragma unroll
  for (int i = 0; i < MT * NT / THR; ++i) {
    const int r = m0 + (tid + i * THR) / NT, c = n0 + (tid + i * THR) % NT;
    if (r >= g.M || c >= g.N) continue;
    double sum = 0.0;
#pragma unroll 8
    for (int zz = 0; zz < kc; ++zz)
      sum += __ldcg(P + (((long long)zz * batch + b) * g.M + r) * g.N + c);
    store(r, c, sum);
  }
  if (tid == 0) tcnt[tile_id] = 0;
}

// ------------------------------------------------ 128 x 128 products
// The generator's exponential and its derivative are chains of 128 x 128
// products; each launch is one link:
//   v_h  = f sum_{i < passes} op(A[h][i]) B[h][i],  h = 0, 1 (halves of a CTA)
//   out0 = v_0 + v_1 + diag I + sum_{j < 4} cy[j] Y[j]            (out[1] null)
//   out0 = v_0, out1 = v_1, P = diag I + cy[0] Y[0] + cy[1] Y[1]
//          + cy[2] v_0 + cy[3] v_1                            (out[1] given)
// with f = 2^-(fs *s), s the device-decided number of squarings.  In digit
// products as above, over the whole depth of 128 under one exponent.
//
// What bounds it: the chain, 26 to 32 links per Adam step, so a link's latency
// (launch, one load, the split, 88 mma per warp, the sum over the four warps
// that share the depth).  16 x 16 tiles on 64 CTAs of one or two halves (256
// threads each) take 7.2 us (10.4 with two products); with seven digits 6.6, where
// 32 x 32 tiles of the kernel above, 16 of them in two chunks, took 9.4 us a
// product.
constexpr int kMT = 16;
constexpr int kMaxSquare = 16;  // norms up to 2^15

struct MatOp {
  const double *A[2][2], *B[2][2];
  int passes, tA;
  double* out[2];
  double* P;
  const double* Y;  // four consecutive matrices
  double cy[4], diag;
  int* s;
  int gate;   // >= 0: nothing is done when gate >= *s
  int fs;     // f = 2^-(fs *s)
  int sel_b;  // B[0][0] is the *s-th of consecutive matrices
  // first link (A = B = S, unscaled): *s is set here, the smallest with
  // max(norm) 2^-s <= 1/2, at most s_max, and X = 2^-s S is written
  const double* norm;
  int s_max;
  double* X;
  unsigned* err;
};

struct MatHalf {
  __half d[2][kDigits][kMT][kCD];  // as in GemmTile
  DigitSum part[4][kMT][kMT];      // sums of the four depth slices
  float mag[4][kMT][kMT];
  int emax[kMT][17];
  int e[2][kMT];
  double v[kMT][kMT];
};

template <int H>
__global__ void __launch_bounds__(256 * H) mat_product_kernel(MatOp o) {
  extern __shared__ __align__(16) unsigned char gsm_[];
  __shared__ unsigned long long s_norm[4];
  const int half = threadIdx.x >> 8, tid = threadIdx.x & 255, warp = tid >> 5, lane = tid & 31;
  MatHalf& S = reinterpret_cast<MatHalf*>(gsm_)[half];
  const int m0 = (blockIdx.x >> 3) * kMT, n0 = (blockIdx.x & 7) * kMT;
  pdl_wait();
  pdl_trigger();
  int s = 0;
  if (o.norm != nullptr) {
    // Non-negative doubles compare as their bits, here plus 1.  A NaN is 0, the
    // smallest: a generator with NaN in some rows gives NaN results, one with NaN
    // in all of them is out of range.
    if (threadIdx.x < kCD) {
      unsigned long long b = __double_as_longlong(__ldcg(o.norm + threadIdx.x));
      b = b > 0x7ff0000000000000ull ? 0 : b + 1;
#pragma unroll
      for (int i = 16; i > 0; i >>= 1) {
        const unsigned long long u = __shfl_xor_sync(0xffffffffu, b, i);
        b = u > b ? u : b;
      }
      if (lane == 0) s_norm[threadIdx.x >> 5] = b;
    }
    __syncthreads();
    unsigned long long b = s_norm[0];
#pragma unroll
    for (int i = 1; i < 4; ++i) b = s_norm[i] > b ? s_norm[i] : b;
    double nrm = __longlong_as_double(b - 1);  // (0: all bits set, a NaN)
    while (nrm > 0.5 && s < o.s_max) {
      nrm *= 0.5;
      ++s;
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) {
      if (!(nrm <= 0.5)) atomicOr(o.err, OPTR_DEVERR_CALIB_RANGE);
      *o.s = s;
    }
  } else if (o.s != nullptr) {
    s = __ldcg(o.s);
  }
  if (o.gate >= s && o.gate >= 0) return;
  const int ra = tid >> 4, ka = tid & 15, rb = tid & 15, kb = tid >> 4;
  const int wn = warp & 1, ws = warp >> 1;  // 16 x 8 outputs, depth slice of 32
  const int r = tid >> 4, c = tid & 15;
  double v = 0.0;
  for (int ps = 0; ps < o.passes; ++ps) {
    const double* A = o.A[half][ps];
    const double* B = o.B[half][ps] + (o.sel_b ? s * kCD * kCD : 0);
    double xa[8], xb[8];
    int ea = 0, eb = 0;
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const int k = ka + 16 * i;  // piece p holds k = p, p + 16, ..
      xa[i] = __ldcg(o.tA ? A + k * kCD + m0 + ra : A + (m0 + ra) * kCD + k);
    }
#pragma unroll
    for (int i = 0; i < 8; ++i) xb[i] = __ldcg(B + (kb + 16 * i) * kCD + n0 + rb);
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      ea = max(ea, field(xa[i]));
      eb = max(eb, field(xb[i]));
    }
#pragma unroll
    for (int i = 8; i > 0; i >>= 1) ea = max(ea, __shfl_xor_sync(0xffffffffu, ea, i));
    S.emax[rb][kb] = eb;
    __syncthreads();
#pragma unroll
    for (int i = 0; i < 16; ++i) eb = max(eb, S.emax[rb][i]);
    ea = row_exponent(ea);
    eb = row_exponent(eb);
    store_digits(S.d[0], ra, ka, xa, ea);
    store_digits(S.d[1], rb, kb, xb, eb);
    if (ka == 0) S.e[0][ra] = ea;
    if (kb == 0) S.e[1][rb] = eb;
    __syncthreads();
    float acc[kWeights][4], mag[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
    for (int d = 0; d < kWeights; ++d)
#pragma unroll
      for (int i = 0; i < 4; ++i) acc[d][i] = 0.f;
#pragma unroll
    for (int ks = 0; ks < 2; ++ks)
      digits_step(acc, mag, S.d[0], S.d[1], 0, 8 * wn, 4 * ws + 2 * ks, lane);
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int ri = (lane >> 2) + 8 * (i >> 1), ci = 8 * wn + 2 * (lane & 3) + (i & 1);
      S.part[ws][ri][ci] = digits_sum(acc, i);
      S.mag[ws][ri][ci] = mag[i];
    }
    __syncthreads();
    DigitSum t = S.part[0][r][c];
    float m = S.mag[0][r][c];
#pragma unroll
    for (int i = 1; i < 4; ++i) {
      t.hi += S.part[i][r][c].hi;
      t.lo += S.part[i][r][c].lo;
      m += S.mag[i][r][c];
    }
    const bool lost = digits_lost(m, S.e[0][r], S.e[1][c]);
    if (!lost) v = digits_add(v, t, S.e[0][r], S.e[1][c], o.fs * s);
    if (__any_sync(0xffffffffu, lost)) {
      double x = 0.0;
      float64_sums(lost, o.tA ? A + m0 + r : A + (m0 + r) * kCD, o.tA ? kCD : 1, B + n0 + c, kCD,
                   kCD, x);
      v += ldexp(x, -o.fs * s);
    }
  }
  const int idx = (m0 + r) * kCD + n0 + c;
  const double dg = m0 + r == n0 + c ? o.diag : 0.0;
  if (H == 2) {
    if (half == 1) S.v[r][c] = v;
    __syncthreads();
    if (half == 1) return;
    const double v1 = reinterpret_cast<MatHalf*>(gsm_)[1].v[r][c];
    if (o.out[1] != nullptr) {
      o.out[0][idx] = v;
      o.out[1][idx] = v1;
      if (o.P != nullptr)
        o.P[idx] = dg + (o.cy[0] * __ldcg(o.Y + idx) + (o.cy[1] * __ldcg(o.Y + kCD * kCD + idx) +
                                                        (o.cy[2] * v + o.cy[3] * v1)));
      return;
    }
    v += v1;
  }
  if (o.Y != nullptr) {
    double y = 0.0;
#pragma unroll
    for (int j = 3; j >= 0; --j)
      if (o.cy[j] != 0.0) y += o.cy[j] * __ldcg(o.Y + j * kCD * kCD + idx);
    v = (v + y) + dg;
  }
  o.out[0][idx] = v;
  if (o.norm != nullptr) o.X[idx] = ldexp(__ldcg(o.A[0][0] + idx), -s);
}

// ------------------------------------------------------- small kernels

// mu[c] = mean over T of K[t][c]; blocks of 256 threads, four channels (a
// sector) each, 64 rows at a time
__global__ void __launch_bounds__(256) col_mean_kernel(const double* __restrict__ K, int T,
                                                       double* __restrict__ mu) {
  __shared__ double sh[64][4];
  const int c = threadIdx.x & 3, r = threadIdx.x >> 2;
  double s = 0.0;
  for (int t = r; t < T; t += 64) s += K[(long long)t * kCD + 4 * blockIdx.x + c];
  sh[r][c] = s;
  for (int w = 32; w > 0; w >>= 1) {
    __syncthreads();
    if (r < w) sh[r][c] += sh[r + w][c];
  }
  if (r == 0) mu[4 * blockIdx.x + c] = sh[0][c] / (double)T;
}

// qp[j][t] = q[t][j] (rows of d): the query rows in the order of the logits
__global__ void permute_kernel(const double* __restrict__ q, int nt, int g,
                               double* __restrict__ qp) {
  const long long row = blockIdx.x;  // j nt + t
  const long long j = row / nt, t = row % nt;
  qp[row * kCD + threadIdx.x] = q[(t * g + j) * kCD + threadIdx.x];
}

// Kc = K - mu (rows of d)
__global__ void center_kernel(const double* __restrict__ K,
                              const double* __restrict__ mu, long long n,
                              double* __restrict__ Kc) {
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n;
       i += (long long)gridDim.x * blockDim.x)
    Kc[i] = K[i] - mu[i % kCD];
}

// Sum over a block of 128 threads of v, on thread 0.
__device__ __forceinline__ double row_sum128(double v) {
  __shared__ double sh[4];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = v;
  __syncthreads();
  return (sh[0] + sh[1]) + (sh[2] + sh[3]);
}

// S = X - X^T (d x d; X the (*s & 1)-th of two when s is given) and, when
// given, norm[i] = sum_j |S[i][j]|: the largest is both |S|_1 and |S|_inf.
__global__ void __launch_bounds__(kCD) skew_kernel(const double* X, const int* s, double* S,
                                                   double* norm) {
  const int i = blockIdx.x, j = threadIdx.x;
  pdl_wait();
  pdl_trigger();
  if (s != nullptr) X += (__ldcg(s) & 1) * kCD * kCD;
  const double v = __ldcg(X + i * kCD + j) - __ldcg(X + j * kCD + i);
  S[i * kCD + j] = v;
  if (norm == nullptr) return;
  const double n = row_sum128(fabs(v));
  if (j == 0) norm[i] = n;
}

// normalised Sylvester-Hadamard matrix: (-1)^popcount(i & j) / sqrt(d)
__global__ void hadamard_kernel(double* __restrict__ H) {
  const int i = blockIdx.x, j = threadIdx.x;
  H[i * kCD + j] = (__popc(i & j) & 1 ? -1.0 : 1.0) / sqrt((double)kCD);
}

__global__ void fill_kernel(double* __restrict__ x, long long n, double v) {
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n;
       i += (long long)gridDim.x * blockDim.x)
    x[i] = v;
}

__global__ void copy_kernel(const double* __restrict__ x, long long n,
                            double* __restrict__ y) {
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n;
       i += (long long)gridDim.x * blockDim.x)
    y[i] = x[i];
}

__global__ void neg_kernel(const double* __restrict__ x, long long n, double* __restrict__ y) {
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n;
       i += (long long)gridDim.x * blockDim.x)
    y[i] = -x[i];
}

__device__ __forceinline__ bool is_window(int s, int t, int sink, int recent) {
  return s < sink || s > t - recent;
}

// Q2 (Sec. 3.1: group-wise asymmetric INT2 with clipping ratio c, fp16 scale
// and min; the cache quantizer's rule) with the straight-through indicator
// (Sec. 4.5): per row and group of G channels of Z, mn = c min, mx = c max,
// r = mx - mn, u = (clamp(z, mn, mx) - mn) * 3 / r, code = clamp(rint(u), 0,
// 3), zh = code * fp16(r / 3) + fp16(mn) (fp16 values of the float32
// rounding), inside = mn <= z <= mx.  Degenerate groups (r <= 1e-30): code
// 0, scale 0.  One warp per 256 consecutive channels (8 groups of 32 or 2 of
// 128).  What bounds it: float64 operations, 2 per clock and SM.  Comparisons
// are made on integers and a warp's groups share one evaluation of the scalars
// (two divisions), each on its own lanes: 5 float64 operations per value; with
// one group per warp 2048 rows took 15.8 us, now 5.9.
__device__ __forceinline__ long long order_key(double z) {
  long long b = __double_as_longlong(z);
  if ((unsigned long long)b == 0x8000000000000000ull) b = 0;  // -0 = 0
  return b < 0 ? b ^ 0x7fffffffffffffffll : b;
}
__device__ __forceinline__ double key_value(long long k) {
  return __longlong_as_double(k < 0 ? k ^ 0x7fffffffffffffffll : k);
}
template <int NG>  // groups per warp: 8 (of 32 channels) or 2 (of 128)
__global__ void __launch_bounds__(256) q2_kernel(const double* Z, long long n, double clip,
                                                 double* Zh, double* inside) {
  constexpr int PER = 8 / NG;  // channels of a group per lane
  const int lane = threadIdx.x & 31;
  const long long wid = (blockIdx.x * 256ll + threadIdx.x) >> 5;
  pdl_wait();
  pdl_trigger();
  const long long base = wid * 256 + lane;  // group i, channel e: base + (i PER + e) 32
  if (wid * 256 >= n) return;  // n is a multiple of 128: the last warp may be half full
  const long long kInf = 0x7ff0000000000000ll;
  long long key[8], lo[NG], hi[NG];
  double z[8];
#pragma unroll
  for (int i = 0; i < 8; ++i) z[i] = base + 32 * i < n ? __ldcg(Z + base + 32 * i) : 0.0;
#pragma unroll
  for (int i = 0; i < NG; ++i) {
    lo[i] = kInf;
    hi[i] = order_key(__longlong_as_double(kInf | (long long)0x8000000000000000ull));
#pragma unroll
    for (int e = 0; e < PER; ++e) {
      const long long k = key[i * PER + e] = order_key(z[i * PER + e]);
      const bool nan = (__double_as_longlong(z[i * PER + e]) & 0x7fffffffffffffffll) > kInf;
      lo[i] = !nan && k < lo[i] ? k : lo[i];
      hi[i] = !nan && k > hi[i] ? k : hi[i];
    }
  }
  // halving exchange: lane bits 4, 3, .. pick the group whose range it ends with
  int o = 16;
#pragma unroll
  for (int n = NG; n > 1; n >>= 1, o >>= 1) {
    const bool up = lane & o;
#pragma unroll
    for (int i = 0; i < n / 2; ++i) {
      const long long l = __shfl_xor_sync(0xffffffffu, up ? lo[i] : lo[i + n / 2], o);
      const long long h = __shfl_xor_sync(0xffffffffu, up ? hi[i] : hi[i + n / 2], o);
      const long long l0 = up ? lo[i + n / 2] : lo[i], h0 = up ? hi[i + n / 2] : hi[i];
      lo[i] = l < l0 ? l : l0;
      hi[i] = h > h0 ? h : h0;
    }
  }
#pragma unroll
  for (; o > 0; o >>= 1) {
    const long long l = __shfl_xor_sync(0xffffffffu, lo[0], o);
    const long long h = __shfl_xor_sync(0xffffffffu, hi[0], o);
    lo[0] = l < lo[0] ? l : lo[0];
    hi[0] = h > hi[0] ? h : hi[0];
  }
  const double mn = clip * key_value(lo[0]), mx = clip * key_value(hi[0]);
  const double r = mx - mn;
  const bool deg = !(r > 1e-30);
  const double inv = deg ? 0.0 : 3.0 / r;
  const double scale = deg ? 0.0 : (double)__half2float(__float2half_rn(__double2float_rn(r / 3.0)));
  const double mn16 = (double)__half2float(__float2half_rn(__double2float_rn(mn)));
#pragma unroll
  for (int i = 0; i < NG; ++i) {
    const int src = i * (32 / NG);  // first lane of group i
    const double gmn = __shfl_sync(0xffffffffu, mn, src), gmx = __shfl_sync(0xffffffffu, mx, src);
    const double ginv = __shfl_sync(0xffffffffu, inv, src);
    const double gsc = __shfl_sync(0xffffffffu, scale, src);
    const double g16 = __shfl_sync(0xffffffffu, mn16, src);
    const long long kmn = order_key(gmn), kmx = order_key(gmx);
#pragma unroll
    for (int e = 0; e < PER; ++e) {
      const long long k = key[i * PER + e];
      const bool ge = k >= kmn, le = k <= kmx;
      const double u = ((ge ? (le ? z[i * PER + e] : gmx) : gmn) - gmn) * ginv;
      const int c = min(max(__double2int_rn(u), 0), 3);
      // 0, 1, 2, 3 as float64 bits
      const double code = __hiloint2double(c == 0 ? 0 : 0x3ff00000 + (c >> 1) * 0x100000 +
                                                          (c == 3 ? 0x80000 : 0), 0);
      const long long j = base + 32 * (i * PER + e);
      if (j >= n) continue;
      Zh[j] = __dadd_rn(__dmul_rn(code, gsc), g16);
      inside[j] = ge && le ? 1.0 : 0.0;
    }
  }
}

// Row (j, t) of [g][nt][T]: logits x (the row of X, or of Xc at the BF16-window
// pairs when windows; scaled already), masked to s <= t_pos[t]; the softmax goes
// to P.  With Pref: D = P - Pref and rowv[row] = KL(Pref || P) =
// sum_s pref (logpref - log max(p, 1e-300)), log p = x - m - log(sum) (below
// 1e-300 the clamp); without: that log p goes to logP.  One block of 256
// threads per row; exp(x - m) is stored in the sum pass and normalised in the
// last.  What bounds it: float64 operations, about 20 of them in exp; the
// maximum is taken on integers and the quotient by a product and one exact
// correction (with a division per element, and D by a pass of its own, 256 rows
// of 2048 took 54 us, now 36).
__device__ __forceinline__ double block_reduce(double v, double* sh) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  __syncthreads();  // sh free from an earlier reduction
  if (lane == 0) sh[w] = v;
  __syncthreads();
  double r = sh[0];
  for (int i = 1; i < 8; ++i) r += sh[i];
  return r;
}

__global__ void __launch_bounds__(256) softmax_rows_kernel(
    const double* X, const double* Xc, int nt, int T, const int32_t* __restrict__ t_pos,
    int sink, int recent, double* P, const double* Pref, double* logP, double* D, double* rowv) {
  __shared__ double sh[8];
  __shared__ long long shk[8];
  pdl_wait();
  pdl_trigger();
  const long long row = blockIdx.x;
  const int t = t_pos[row % nt];
  const bool win = Xc != nullptr;
  const double* x = X + row * (long long)T;
  const double* xc = win ? Xc + row * (long long)T : nullptr;
  auto logit = [&](int s) {
    return __ldcg((win && is_window(s, t, sink, recent)) ? xc + s : x + s);
  };
  // a NaN is passed over here and reaches the sum below
  long long k = order_key(__longlong_as_double((long long)0xfff0000000000000ull));
  for (int s = threadIdx.x; s < T; s += 256)
    if (s <= t) {
      const double v = logit(s);
      const long long kv = order_key(v);
      const bool nan = (__double_as_longlong(v) & 0x7fffffffffffffffll) > 0x7ff0000000000000ll;
      k = !nan && kv > k ? kv : k;
    }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const long long u = __shfl_xor_sync(0xffffffffu, k, o);
    k = u > k ? u : k;
  }
  if ((threadIdx.x & 31) == 0) shk[threadIdx.x >> 5] = k;
  __syncthreads();
  for (int i = 0; i < 8; ++i) k = shk[i] > k ? shk[i] : k;
  const double m = key_value(k);
  double* p = P + row * (long long)T;
  double sum = 0.0;
  for (int s = threadIdx.x; s < T; s += 256) {
    const double e = s <= t ? exp(logit(s) - m) : 0.0;
    p[s] = e;
    sum += e;
  }
  sum = block_reduce(sum, sh);
  const double lsum = log(sum), inv = 1.0 / sum, lmin = log(1e-300);
  double kl = 0.0;
  for (int s = threadIdx.x; s < T; s += 256) {
    const long long i = row * (long long)T + s;
    const double e = p[s];
    double v = e * inv;
    v = fma(fma(-v, sum, e), inv, v);  // e / sum
    p[s] = v;
    const double lp = v > 1e-300 ? (logit(s) - m) - lsum : lmin;
    if (Pref != nullptr) {
      const double pr = __ldcg(Pref + i);
      D[i] = v - pr;
      kl += pr * (__ldcg(logP + i) - lp);
    } else {
      logP[i] = lp;
    }
  }
  if (Pref != nullptr) {
    kl = block_reduce(kl, sh);
    if (threadIdx.x == 0) rowv[row] = kl;
  }
}

// Gradient of the key loss with respect to the raw logits x of row (j, t)
// (l = scale x): G[s] = coef * (D + pk (gv - sum_s pk gv)), D = pk - p, at the
// causal non-window pairs, 0 elsewhere.  In place over GV.  One block per row
// (8 rows per block left most SMs idle: 68 us for 256 rows of 2048, now 9).
__global__ void __launch_bounds__(256) key_row_grad_kernel(
    const double* PK, const double* D, double* GV, int nt, int T,
    const int32_t* __restrict__ t_pos, double coef, int sink, int recent, int win) {
  __shared__ double sh[8];
  pdl_wait();
  pdl_trigger();
  const long long row = blockIdx.x;
  const int t = t_pos[row % nt];
  const double* pk = PK + row * (long long)T;
  const double* d = D + row * (long long)T;
  double* gv = GV + row * (long long)T;
  double gbar = 0.0;
  for (int s = threadIdx.x; s < T; s += 256) gbar += __ldcg(pk + s) * __ldcg(gv + s);
  gbar = block_reduce(gbar, sh);
  for (int s = threadIdx.x; s < T; s += 256) {
    double gsum = 0.0;
    if (s <= t && !(win && is_window(s, t, sink, recent)))
      gsum = coef * (__ldcg(d + s) + __ldcg(pk + s) * (__ldcg(gv + s) - gbar));
    gv[s] = gsum;
  }
}

// Zero the BF16-window pairs of rows (j, t) of [g][nt][T].
__global__ void zero_window_kernel(double* __restrict__ P, int rows, int nt, int T,
                                   const int32_t* __restrict__ t_pos, int sink,
                                   int recent) {
  const int lane = threadIdx.x & 31;
  const long long row = (blockIdx.x * (long long)blockDim.x + threadIdx.x) >> 5;
  if (row >= rows) return;
  const int t = t_pos[row % nt];
  for (int s = lane; s < T; s += 32)
    if (is_window(s, t, sink, recent)) P[row * (long long)T + s] = 0.0;
}

// rowv[row] = (add ? rowv[row] : 0) + lam * (sum_c E[row][c]^2) / dm
__global__ void row_sqsum_kernel(const double* E, int rows, int dm, double lam, int add,
                                 double* rowv) {
  const int lane = threadIdx.x & 31;
  const long long row = (blockIdx.x * (long long)blockDim.x + threadIdx.x) >> 5;
  pdl_wait();
  pdl_trigger();
  if (row >= rows) return;
  double s = 0.0;
  for (int c = lane; c < dm; c += 32) {
    const double e = __ldcg(E + row * (long long)dm + c);
    s += e * e;
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  if (lane == 0) {
    const double v = lam * s / (double)dm;
    rowv[row] = add ? __ldcg(rowv + row) + v : v;
  }
}

// out = (sum_i rowv[i]) / n, one block of 256 threads, fixed order
__global__ void __launch_bounds__(256) loss_reduce_kernel(const double* rowv, int rows, double n,
                                                          double* out) {
  __shared__ double sh[8];
  pdl_wait();
  pdl_trigger();
  double s = 0.0;
  for (int i = threadIdx.x; i < rows; i += 256) s += __ldcg(rowv + i);
  s = block_reduce(s, sh);
  if (threadIdx.x == 0) *out = s / n;
}

// Adam (Kingma & Ba), in the order m = b1 m + (1 - b1) g,
// v = b2 v + ((1 - b2) g) g, x -= (lr mh) / (sqrt(vh) + eps), mh = m / bc1,
// vh = v / bc2; separate roundings (no contraction).
// The gradient g = dA = L^T - L comes from the derivative buffers L (the
// (*s & 1)-th of two).  It is skew to the last bit, and so is x when it starts
// from 0: S = x - x^T = 2 x, written with its row norms for the next rotation.
// One block per row: at 2 float64 FMAs per clock and SM one SM alone would take
// 50 us for the norms.
__global__ void __launch_bounds__(kCD) adam_kernel(double* x, const double* L, const int* s,
                                                   double* m, double* v, double* S,
                                                   double* norm, double lr, double b1,
                                                   double omb1, double b2, double omb2,
                                                   double bc1, double bc2, double eps) {
  pdl_wait();
  pdl_trigger();
  const int i = blockIdx.x * kCD + threadIdx.x;
  L += (__ldcg(s) & 1) * kCD * kCD;
  const double gi = __ldcg(L + threadIdx.x * kCD + blockIdx.x) - __ldcg(L + i);
  const double mi = __dadd_rn(__dmul_rn(b1, __ldcg(m + i)), __dmul_rn(omb1, gi));
  const double vi = __dadd_rn(__dmul_rn(b2, __ldcg(v + i)), __dmul_rn(__dmul_rn(omb2, gi), gi));
  m[i] = mi;
  v[i] = vi;
  const double mh = __ddiv_rn(mi, bc1), vh = __ddiv_rn(vi, bc2);
  const double xi = __dsub_rn(
      __ldcg(x + i), __ddiv_rn(__dmul_rn(lr, mh), __dadd_rn(__dsqrt_rn(vh), eps)));
  x[i] = xi;
  S[i] = 2.0 * xi;
  const double n = row_sum128(fabs(2.0 * xi));
  if (threadIdx.x == 0) norm[blockIdx.x] = n;
}

// Held-out selection: keep R when its score is the first or a lower one.
__global__ void select_kernel(const double* __restrict__ score,
                              double* __restrict__ best, int first,
                              const double* __restrict__ R,
                              double* __restrict__ bestR) {
  __shared__ int take;
  if (threadIdx.x == 0) {
    take = first || *score < *best;
    if (take) *best = *score;
  }
  __syncthreads();
  if (take)
    for (int i = threadIdx.x; i < kCD * kCD; i += blockDim.x) bestR[i] = R[i];
}

}  // namespace

// ------------------------------------------------------------ host side

namespace {

// blocks of 256 threads for one warp per row (no grid-stride loop)
inline int nwarp_blocks(long long rows) { return (int)((rows * 32 + 255) / 256); }

inline int nblk(long long n, int t = 256) {
  long long b = (n + t - 1) / t;
  return (int)(b < 4096 ? (b > 0 ? b : 1) : 4096);
}

constexpr int kGSplit = 160;  // K is split up to this many CTAs, about one per SM
constexpr int kGSmall = 76;   // fewer tiles x chunks of 64 x 32: 32 x 16 instead
constexpr long long kGemmScratch = 1 << 21;  // split-K doubles (16 MiB)
constexpr int kGemmTiles = 512;  // K is split only while a call has fewer tiles

struct GemmCall {
  cudaStream_t s;
  double* scratch;        // split-K partial sums
  long long scratch_len;  // doubles
  int* tcnt;              // split-K arrival counters, one per output tile (0)
  static Gemm args(int M, int N, int K, const double* A, long long lda, bool tA,
                   const double* B, long long ldb, bool tB, double* C, long long ldc) {
    Gemm g{};
    g.M = M; g.N = N; g.K = K;
    g.A = A; g.lda = lda; g.tA = tA;
    g.B = B; g.ldb = ldb; g.tB = tB;
    g.C = C; g.ldc = ldc;
    g.alpha = 1.0;
    return g;
  }
  void operator()(int M, int N, int K, const double* A, long long lda, bool tA,
                  const double* B, long long ldb, bool tB, double* C, long long ldc,
                  double alpha = 1.0, int batch = 1, long long sA = 0, long long sB = 0,
                  long long sC = 0) const {
    Gemm g = args(M, N, K, A, lda, tA, B, ldb, tB, C, ldc);
    g.alpha = alpha;
    g.sA = sA;
    g.sB = sB;
    g.sC = sC;
    run(g, batch);
  }
  void run(const Gemm& g, int batch) const {
    const long long tiles = (long long)((g.M + 63) / 64) * ((g.N + 31) / 32) * batch;
    const int chunks = (g.K + kGK - 1) / kGK * (g.A2 != nullptr ? 2 : 1);
    if (tiles * chunks < kGSmall) launch<32, 16>(g, batch);
    else launch<64, 32>(g, batch);
  }
  template <int MT, int NT>
  void launch(const Gemm& g, int batch) const {
    const int tm = (g.M + MT - 1) / MT, tn = (g.N + NT - 1) / NT;
    const long long tiles = (long long)tm * tn * batch;
    // split K while the CTAs do not fill the SMs
    int kc = 1;
    const int chunks = (g.K + kGK - 1) / kGK * (g.A2 != nullptr ? 2 : 1);
    while (tiles <= kGemmTiles && tiles * kc * 2 <= kGSplit && 2 * kc <= chunks &&
           (long long)(2 * kc) * batch * g.M * g.N <= scratch_len)
      kc *= 2;
    launch_pdl(&gemm_digits_kernel<MT, NT>, dim3(tn * tm, 1, batch * kc),
               dim3(GemmTile<MT, NT>::kThreads), sizeof(GemmTile<MT, NT>), s, g, kc, scratch, tcnt);
  }
};

// One trace: the inputs and what stays fixed over the Adam steps.
struct Trace {
  const double *q, *K, *V;
  const int32_t* tpos;
  int T, nt;
  double *Kc;       // [T][d]     K - mu
  double *qp;       // [g][nt][d] the query rows
  double *Pref;     // [g][nt][T] softmax of the BF16 logits
  double *logPref;  // [g][nt][T] log max(Pref, 1e-300)
  double *Lc;       // [g][nt][T] window logits scale q (K - mu)^T (windows only)
  double *Phat;     // [g][nt][T] key-phase attention, window pairs zeroed
};

struct Calib {
  optr_calib_config c;
  int windows;
  double scale;  // 1 / sqrt(d)
  Trace tr[2];   // calibration, held-out
  // working buffers (sized for the larger trace)
  double *Z, *Zh, *inside, *Kt, *dKt, *dZh;  // [T][d]
  double *X, *PK, *GV, *DP;                  // [g][nt][T]
  double *rowv;                              // [g][nt]
  double *DV, *U;                            // [g][nt][d]
  double *Eo;                                // [g][nt][d_model]
  // d x d
  double *R0[2], *A, *m, *v, *dA, *S, *R, *dR, *best;
  double *Y, *dY;        // powers X .. X^4 of the scaled generator, and derivatives
  double *P, *dP[2];     // P3, P2, P1 of the polynomial; derivatives
  double *F;             // exp(X)^(2^i) - I, i = 0 .. kMaxSquare
  double *L;             // derivative of F[i], two buffers, i & 1
  double *norm;          // row norms of S
  int squares;           // squarings launched: a bound on *s_dev
  double* scal;  // [0] training loss scratch, [1] score, [2] best score
  int* s_dev;
  unsigned* err;
  const double* W;  // [g][d_model][d]
  double* gsc;      // split-K scratch of the GEMMs
  int* gcnt;        // split-K arrival counters (kGemmTiles, zero between calls)
  cudaStream_t st;
  GemmCall gemm() const { return GemmCall{st, gsc, kGemmScratch, gcnt}; }
};

struct Layout {
  size_t off = 0;
  char* base = nullptr;
  template <typename T>
  T* take(size_t n) {
    T* p = base ? reinterpret_cast<T*>(base + off) : nullptr;
    off += (n * sizeof(T) + 255) & ~(size_t)255;
    return p;
  }
};

// Carves the workspace (base == nullptr: only sizes it).
size_t carve(Calib& C, char* base) {
  const optr_calib_config& c = C.c;
  Layout L;
  L.base = base;
  const int Th = c.T_held > 0 ? c.T_held : c.T, nh = c.T_held > 0 ? c.nt_held : c.nt;
  const long long Tm = c.T > Th ? c.T : Th, nm = c.nt > nh ? c.nt : nh;
  const long long g = c.g, D = kCD, D2 = kCD * kCD;
  C.err = L.take<unsigned>(1);
  C.s_dev = L.take<int>(1);
  C.scal = L.take<double>(8);
  for (int k = 0; k < 2; ++k) {
    const long long T = k ? Th : c.T, nt = k ? nh : c.nt;
    Trace& t = C.tr[k];
    t.Kc = L.take<double>(T * D);
    t.qp = L.take<double>(g * nt * D);
    t.Pref = L.take<double>(g * nt * T);
    t.logPref = L.take<double>(g * nt * T);
    t.Lc = C.windows ? L.take<double>(g * nt * T) : nullptr;
    t.Phat = L.take<double>(g * nt * T);
  }
  C.Z = L.take<double>(Tm * D);
  C.Zh = L.take<double>(Tm * D);
  C.inside = L.take<double>(Tm * D);
  C.Kt = L.take<double>(Tm * D);
  C.dKt = L.take<double>(Tm * D);
  C.dZh = L.take<double>(Tm * D);
  C.X = L.take<double>(g * nm * Tm);
  C.PK = L.take<double>(g * nm * Tm);
  C.GV = L.take<double>(g * nm * Tm);
  C.DP = L.take<double>(g * nm * Tm);
  C.rowv = L.take<double>(g * nm);
  C.DV = L.take<double>(g * nm * D);
  C.U = L.take<double>(g * nm * D);
  C.Eo = L.take<double>(g * nm * c.d_model);
  C.gsc = L.take<double>(kGemmScratch);
  C.gcnt = L.take<int>(kGemmTiles);
  double** dd[] = {&C.R0[0], &C.R0[1], &C.A, &C.m, &C.v, &C.dA, &C.S, &C.R, &C.dR, &C.best,
                   &C.dP[0], &C.dP[1]};
  for (double** p : dd) *p = L.take<double>(D2);
  C.Y = L.take<double>(4 * D2);
  C.dY = L.take<double>(4 * D2);
  C.P = L.take<double>(3 * D2);
  C.F = L.take<double>((kMaxSquare + 1) * D2);
  C.L = L.take<double>(2 * D2);
  C.norm = L.take<double>(kCD);
  return L.off;
}

// One link of the 128 x 128 chain on C.st.
void link(Calib& C, int halves, const MatOp& o) {
  auto k = halves == 2 ? &mat_product_kernel<2> : &mat_product_kernel<1>;
  launch_pdl(k, dim3(64), dim3(256 * halves), halves * sizeof(MatHalf), C.st, o);
}
MatOp product(const double* A, const double* B, double* out) {
  MatOp o{};
  o.A[0][0] = A;
  o.B[0][0] = B;
  o.passes = 1;
  o.out[0] = out;
  o.gate = -1;
  return o;
}
MatOp& plus(MatOp& o, const double* A, const double* B) {
  o.A[1][0] = A;
  o.B[1][0] = B;
  return o;
}

constexpr int kD2 = kCD * kCD;

// 1 / k!
double inv_fact(int k) {
  double f = 1.0;
  for (int i = 2; i <= k; ++i) f *= i;
  return 1.0 / f;
}
void taylor(MatOp& o, const double* Y, int k0, int n, bool constant) {
  o.Y = Y;
  o.diag = constant ? inv_fact(k0) : 0.0;
  for (int j = 0; j < 4; ++j) o.cy[j] = j < n ? inv_fact(k0 + 1 + j) : 0.0;
}

// I + F[s] = exp(S) with X = S 2^-s, |X| <= 1/2: the Taylor polynomial of degree
// 16 (remainder 2e-20) in Paterson and Stockmeyer's form ("On the number of
// nonscalar multiplications necessary to evaluate polynomials", 1973),
//   P3 = sum_{j <= 4} X^j / (12 + j)!,  P_i = X^4 P_{i+1} + sum_{j < 4} X^j / (4 i + j)!,
// F[0] = P0 - I, then s squarings (I + F)^2 = I + (2 F + F^2); 5 dependent links
// and the squarings, where Horner's rule has 18.  F rather than I + F is kept
// because each squaring doubles the relative error, and entries of F round at
// their own size, not at 1: the gradient's relative error against quad precision
// is 1e-15 to 6e-15 for entries of A of 0.005 to 0.4 (FMA chain, Horner:
// 3e-15 to 9e-14; this chain with I + F: 2e-15 to 2e-13).
// 20 + 20 Adam steps 86.5 -> 27.5 ms (Horner and one launch per product before).
// C.squares squarings are launched, those past s do nothing.  The powers, P_i
// and F[i] stay for generator_grad.
void expm(Calib& C) {
  MatOp o = product(C.S, C.S, C.Y + kD2);
  o.s = C.s_dev;
  o.fs = 2;
  o.norm = C.norm;
  o.s_max = C.squares;
  o.X = C.Y;
  o.err = C.err;
  link(C, 1, o);
  o = product(C.Y, C.Y + kD2, C.Y + 2 * kD2);
  plus(o, C.Y + kD2, C.Y + kD2);
  o.out[1] = C.Y + 3 * kD2;
  o.P = C.P;
  taylor(o, C.Y, 12, 4, true);
  link(C, 2, o);
  for (int i = 2; i >= 0; --i) {
    o = product(C.Y + 3 * kD2, C.P + (2 - i) * kD2, i ? C.P + (3 - i) * kD2 : C.F);
    taylor(o, C.Y, 4 * i, 3, i > 0);
    link(C, 1, o);
  }
  for (int i = 0; i < C.squares; ++i) {
    o = product(C.F + i * kD2, C.F + i * kD2, C.F + (i + 1) * kD2);
    o.Y = C.F + i * kD2;
    o.cy[0] = 2.0;
    o.s = C.s_dev;
    o.gate = i;
    link(C, 1, o);
  }
}

// R = R0 exp(S) into C.R, S = A - A^T and its row norms given
void rotation(Calib& C, const double* R0) {
  expm(C);
  MatOp o = product(R0, C.F, C.R);  // R0 + R0 F
  o.Y = R0;
  o.cy[0] = 1.0;
  o.s = C.s_dev;
  o.sel_b = 1;
  link(C, 1, o);
}

// dS^T = L_exp(S, dR^T R0) into C.L[*s & 1] (dA = dS - dS^T): the chain of
// expm() differentiated, two products per link.
void generator_grad(Calib& C, const double* R0) {
  MatOp o = product(C.dR, R0, C.dY);  // H = 2^-s dR^T R0
  o.tA = 1;
  o.s = C.s_dev;
  o.fs = 1;
  link(C, 1, o);
  o = product(C.dY, C.Y, C.dY + kD2);  // d(X^2) = H X + X H
  link(C, 2, plus(o, C.Y, C.dY));
  o = product(C.dY, C.Y + kD2, C.dY + 2 * kD2);  // d(X^3) = H X^2 + X d(X^2)
  plus(o, C.dY + kD2, C.Y + kD2);                // d(X^4) = d(X^2) X^2 + X^2 d(X^2)
  o.passes = 2;
  o.A[0][1] = C.Y;
  o.B[0][1] = C.dY + kD2;
  o.A[1][1] = C.Y + kD2;
  o.B[1][1] = C.dY + kD2;
  o.out[1] = C.dY + 3 * kD2;
  o.P = C.dP[0];
  taylor(o, C.dY, 12, 4, false);
  link(C, 2, o);
  for (int i = 2; i >= 0; --i) {  // dP_i = d(X^4) P_{i+1} + X^4 dP_{i+1} + ..
    o = product(C.dY + 3 * kD2, C.P + (2 - i) * kD2, i ? C.dP[(i + 1) & 1] : C.L);
    plus(o, C.Y + 3 * kD2, C.dP[i & 1]);
    taylor(o, C.dY, 4 * i, 3, false);
    link(C, 2, o);
  }
  for (int i = 0; i < C.squares; ++i) {
    double *L0 = C.L + (i & 1) * kD2, *L1 = C.L + ((i + 1) & 1) * kD2;
    o = product(C.F + i * kD2, L0, L1);  // 2 L + F L + L F
    plus(o, L0, C.F + i * kD2);
    o.Y = L0;
    o.cy[0] = 2.0;
    o.s = C.s_dev;
    o.gate = i;
    link(C, 2, o);
  }
}

// Squarings that t Adam steps from A = 0 can need.  A step moves an entry by
// at most lr |mh| / sqrt(vh), and by Cauchy and Schwarz
//   mh^2 <= vh (1-b1)^2 / (1-b2) (bc2 / bc1^2) sum_{j < t} (b1^2 / b2)^j;
// a row of S = 2 A has 127 entries.
int adam_squares(double reach) {
  double n = 2.0 * (kCD - 1) * reach * (1.0 + 1e-6);
  int s = 0;
  while (n > 0.5 && s < kMaxSquare) {
    n *= 0.5;
    ++s;
  }
  return s;
}
double adam_reach(double lr, double b1, double b2, int t) {
  const double q = b1 * b1 / b2;
  const double bc1 = 1.0 - pow(b1, (double)t), bc2 = 1.0 - pow(b2, (double)t);
  return lr * (1.0 - b1) / bc1 * sqrt(bc2 / (1.0 - b2) * (1.0 - pow(q, (double)t)) / (1.0 - q));
}

}  // namespace

namespace {

// Inputs that stay fixed over the steps: K - mu, the query rows by head, the
// BF16 reference attention p and log p, the window logits.
void trace_setup(Calib& C, Trace& t, const double* mu) {
  GemmCall gm = C.gemm();
  const int g = C.c.g, D = kCD;
  const long long nT = (long long)t.T * D, r = (long long)g * t.nt, nD = (long long)t.nt * D;
  center_kernel<<<nblk(nT), 256, 0, C.st>>>(t.K, mu, nT, t.Kc);
  permute_kernel<<<(unsigned)r, kCD, 0, C.st>>>(t.q, t.nt, g, t.qp);
  // BF16 logits scale q_j K^T into X, softmax into Pref
  gm(t.nt, t.T, D, t.qp, D, false, t.K, D, true, C.X, t.T, C.scale, g, nD, 0,
     (long long)t.nt * t.T);
  launch_pdl(&softmax_rows_kernel, dim3((unsigned)r), dim3(256), 0, C.st, C.X, nullptr, t.nt, t.T,
             t.tpos, 0, 0, t.Pref, nullptr, t.logPref, nullptr, nullptr);
  if (C.windows)
    gm(t.nt, t.T, D, t.qp, D, false, t.Kc, D, true, t.Lc, t.T, C.scale, g, nD, 0,
       (long long)t.nt * t.T);
}

// Effective rotated-and-back rows Q2(X R) R^T, less `sub` when given, into C.Kt
// (Zh, inside kept).
void q2_roundtrip(Calib& C, const double* X, int T, double clip, const double* sub) {
  GemmCall gm = C.gemm();
  gm(T, kCD, kCD, X, kCD, false, C.R, kCD, false, C.Z, kCD);
  const long long n = (long long)T * kCD;
  launch_pdl(C.c.group == 32 ? &q2_kernel<8> : &q2_kernel<2>, dim3(nwarp_blocks((n + 255) / 256)),
             dim3(256), 0, C.st, C.Z, n, clip, C.Zh, C.inside);
  Gemm k = gm.args(T, kCD, kCD, C.Zh, kCD, false, C.R, kCD, true, C.Kt, kCD);
  k.sub = sub;
  gm.run(k, 1);
}

// e_j = DV_j W_j^T into Eo, rowv[j, t] (+)= lam ||e_j||^2 / d_model.  (||e||^2 as
// DV (W^T W) DV^T, with W^T W once per call, took 0.1 ms less per Adam step at
// d_model = 4096, but its error grows with the square of W's condition number:
// 4e-6 of the term at 1e6, and below zero for a rank-deficient W.)
void output_error(Calib& C, Trace& t, double lam, int add) {
  const int g = C.c.g, D = kCD, dm = C.c.d_model, r = g * t.nt;
  C.gemm()(t.nt, dm, D, C.DV, D, false, C.W, D, true, C.Eo, dm, 1.0, g, (long long)t.nt * D,
           (long long)dm * D, (long long)t.nt * dm);
  launch_pdl(&row_sqsum_kernel, dim3(nwarp_blocks(r)), dim3(256), 0, C.st, C.Eo, r, dm, lam, add,
             C.rowv);
}

// U0 = e_j W_j (after output_error on the same trace)
void output_grad(Calib& C, Trace& t) {
  const int g = C.c.g, D = kCD, dm = C.c.d_model;
  C.gemm()(t.nt, D, dm, C.Eo, dm, false, C.W, D, false, C.U, D, 1.0, g, (long long)t.nt * dm,
           (long long)dm * D, (long long)t.nt * D);
}

void loss_mean(Calib& C, int rows, double* out) {
  launch_pdl(&loss_reduce_kernel, dim3(1), dim3(256), 0, C.st, C.rowv, rows, (double)rows, out);
}

// L_K of trace t under C.R into *out; leaves PK, DP and the output error's
// buffers for the backward.
void key_forward(Calib& C, Trace& t, double* out) {
  GemmCall gm = C.gemm();
  const int g = C.c.g, D = kCD;
  const long long r = (long long)g * t.nt, nTT = (long long)t.nt * t.T, nD = (long long)t.nt * D;
  q2_roundtrip(C, t.Kc, t.T, C.c.clip_k, nullptr);
  gm(t.nt, t.T, D, t.qp, D, false, C.Kt, D, true, C.X, t.T, C.scale, g, nD, 0, nTT);
  launch_pdl(&softmax_rows_kernel, dim3((unsigned)r), dim3(256), 0, C.st, C.X,
             C.windows ? t.Lc : nullptr, t.nt, t.T, t.tpos, C.c.sink, C.c.recent, C.PK, t.Pref,
             t.logPref, C.DP, C.rowv);
  // DV_j = (pk - p) V
  gm(t.nt, D, t.T, C.DP, t.T, false, t.V, D, false, C.DV, D, 1.0, g, nTT, 0, nD);
  output_error(C, t, C.c.lam, 1);
  loss_mean(C, (int)r, out);
}

// dR = dKt^T Zh + X^T (inside * (dKt R))
void rotation_grad(Calib& C, int T, const double* X) {
  GemmCall gm = C.gemm();
  const int D = kCD;
  Gemm z = gm.args(T, D, D, C.dKt, D, false, C.R, D, false, C.dZh, D);
  z.mul = C.inside;
  gm.run(z, 1);
  Gemm d = gm.args(D, D, T, C.dKt, D, true, C.Zh, D, false, C.dR, D);
  d.A2 = X;
  d.B2 = C.dZh;
  gm.run(d, 1);
}

// dR of L_K (after key_forward on the same trace and rotation).
void key_backward(Calib& C, Trace& t) {
  GemmCall gm = C.gemm();
  const int g = C.c.g, D = kCD;
  const long long r = (long long)g * t.nt, nTT = (long long)t.nt * t.T;
  // GV_j = (2 lambda / d_model) U0_j V^T
  output_grad(C, t);
  gm(t.nt, t.T, D, C.U, D, false, t.V, D, true, C.GV, t.T, 2.0 * C.c.lam / C.c.d_model, g,
     (long long)t.nt * D, 0, nTT);
  launch_pdl(&key_row_grad_kernel, dim3((unsigned)r), dim3(256), 0, C.st, C.PK, C.DP, C.GV, t.nt,
             t.T, t.tpos, C.scale / (double)r, C.c.sink, C.c.recent, C.windows);
  // dKt = sum_j dl_j^T q_j
  gm(t.T, D, (int)r, C.GV, t.T, true, t.qp, D, false, C.dKt, D);
  rotation_grad(C, t.T, t.Kc);
}

// Phat of trace t: the key-phase attention under C.R (the selected R_K),
// window pairs zeroed (their values are exact, so they add no error).
void value_setup(Calib& C, Trace& t) {
  key_forward(C, t, C.scal + 3);
  const long long r = (long long)C.c.g * t.nt;
  copy_kernel<<<nblk(r * t.T), 256, 0, C.st>>>(C.PK, r * t.T, t.Phat);
  if (C.windows)
    zero_window_kernel<<<nwarp_blocks(r), 256, 0, C.st>>>(t.Phat, (int)r, t.nt, t.T,
                                                        t.tpos, C.c.sink, C.c.recent);
}

// L_V of trace t under C.R (the value rotation) into *out.
void value_forward(Calib& C, Trace& t, double* out) {
  const int g = C.c.g, D = kCD;
  const long long r = (long long)g * t.nt, nTT = (long long)t.nt * t.T;
  q2_roundtrip(C, t.V, t.T, C.c.clip_v, t.V);
  C.gemm()(t.nt, D, t.T, t.Phat, t.T, false, C.Kt, D, false, C.DV, D, 1.0, g, nTT, 0,
           (long long)t.nt * D);
  output_error(C, t, 1.0, 0);
  loss_mean(C, (int)r, out);
}

// dR of L_V (after value_forward on the same trace and rotation).
void value_backward(Calib& C, Trace& t) {
  const int D = kCD;
  const long long r = (long long)C.c.g * t.nt;
  output_grad(C, t);
  C.gemm()(t.T, D, (int)r, t.Phat, t.T, true, C.U, D, false, C.dKt, D,
           2.0 / ((double)C.c.d_model * r));
  rotation_grad(C, t.T, t.V);
}

// One Adam run of the appendix algorithm on generator A (from 0) for the
// key (kind 0) or value (kind 1) objective; the best-scoring rotation on
// the held-out trace (scored at step 0, every select_every steps and after
// the last step) ends in C.best; hist[i] = the training loss at step i.
void adam_run(Calib& C, int kind, const double* R0, double* hist) {
  const optr_calib_config& c = C.c;
  const int n = kCD * kCD;
  fill_kernel<<<nblk(n), 256, 0, C.st>>>(C.A, n, 0.0);
  fill_kernel<<<nblk(n), 256, 0, C.st>>>(C.m, n, 0.0);
  fill_kernel<<<nblk(n), 256, 0, C.st>>>(C.v, n, 0.0);
  skew_kernel<<<kCD, kCD, 0, C.st>>>(C.A, nullptr, C.S, C.norm);
  const double b1 = 0.9, b2 = 0.999, eps = 1e-8;
  double reach = 0.0;  // bound on |A| after i steps
  for (int i = 0; i <= c.steps; ++i) {
    C.squares = adam_squares(reach);
    rotation(C, R0);
    if (i % c.select_every == 0 || i == c.steps) {
      if (kind == 0) key_forward(C, C.tr[1], C.scal + 1);
      else value_forward(C, C.tr[1], C.scal + 1);
      select_kernel<<<1, 256, 0, C.st>>>(C.scal + 1, C.scal + 2, i == 0, C.R, C.best);
    }
    if (i == c.steps) break;
    if (kind == 0) {
      key_forward(C, C.tr[0], hist + i);
      key_backward(C, C.tr[0]);
    } else {
      value_forward(C, C.tr[0], hist + i);
      value_backward(C, C.tr[0]);
    }
    generator_grad(C, R0);
    const int t = i + 1;
    launch_pdl(&adam_kernel, dim3(kCD), dim3(kCD), 0, C.st, C.A, C.L, C.s_dev, C.m, C.v, C.S,
               C.norm, c.lr, b1, 1.0 - b1, b2, 1.0 - b2, 1.0 - pow(b1, (double)t),
               1.0 - pow(b2, (double)t), eps);
    reach += adam_reach(c.lr, b1, b2, t);
  }
}

}  // namespace

namespace {

bool calib_config_ok(const optr_calib_config* c) {
  if (!c) return false;
  const bool held = c->T_held > 0;
  // tokens and query rows: launch grids stay within their limits
  const double lim = 4000000.0;
  return c->g >= 1 && c->g <= 64 && c->d_model >= 1 && c->d_model <= (1 << 20) &&
         c->T >= 1 && c->T <= lim && c->nt >= 1 &&
         (double)c->g * c->nt <= lim && c->T_held >= 0 &&
         (!held || (c->nt_held >= 1 && c->T_held <= lim &&
                    (double)c->g * c->nt_held <= lim)) &&
         c->steps >= 0 && c->steps <= 100000 && c->select_every >= 1 &&
         (c->group == 32 || c->group == 128) && c->sink >= 0 && c->recent >= 0 &&
         c->clip_k > 0.0 && c->clip_k <= 1.0 && c->clip_v > 0.0 && c->clip_v <= 1.0 &&
         c->lr > 0.0 && c->lr < 1e6 && c->lam >= 0.0 && c->lam < 1e12;
}

bool calib_init(Calib& C, const optr_calib_config* c, void* ws, const double* W_O,
                cudaStream_t s) {
  C = Calib{};
  const struct {
    const void* kernel;
    size_t bytes;
  } need[] = {{reinterpret_cast<const void*>(&gemm_digits_kernel<64, 32>),
               sizeof(GemmTile<64, 32>)},
              {reinterpret_cast<const void*>(&gemm_digits_kernel<32, 16>),
               sizeof(GemmTile<32, 16>)},
              {reinterpret_cast<const void*>(&mat_product_kernel<1>), sizeof(MatHalf)},
              {reinterpret_cast<const void*>(&mat_product_kernel<2>), 2 * sizeof(MatHalf)}};
  for (const auto& k : need)
    if (ensure_dynamic_smem(k.kernel, k.bytes) != cudaSuccess) return false;
  C.c = *c;
  C.windows = c->sink > 0 || c->recent > 0;
  C.scale = 1.0 / sqrt((double)kCD);
  carve(C, static_cast<char*>(ws));
  C.W = W_O;
  C.st = s;
  return true;
}

optr_status calib_finish(Calib& C) {
  if (cudaGetLastError() != cudaSuccess) return OPTR_ERR_CUDA;
  unsigned e = 0;
  if (cudaMemcpyAsync(&e, C.err, sizeof(unsigned), cudaMemcpyDeviceToHost, C.st) !=
          cudaSuccess ||
      cudaStreamSynchronize(C.st) != cudaSuccess)
    return OPTR_ERR_CUDA;
  return e ? OPTR_ERR_OUT_OF_RANGE : OPTR_OK;
}

}  // namespace
}  // namespace optr

using namespace optr;

extern "C" size_t optr_calib_workspace_size(const optr_calib_config* c) {
  if (!calib_config_ok(c)) return 0;
  Calib C{};
  C.c = *c;
  C.windows = c->sink > 0 || c->recent > 0;
  return carve(C, nullptr);
}

extern "C" optr_status optr_calibrate_head(
    const optr_calib_config* c, const double* q, const double* K, const double* V,
    const int32_t* t_pos, const double* W_O, const double* q_held,
    const double* K_held, const double* V_held, const int32_t* t_pos_held,
    const double* R0_K, const double* R0_V, double* R_K, double* R_V, double* mu,
    double* hist_k, double* hist_v, void* workspace, size_t ws_bytes,
    cudaStream_t stream) {
  if (!calib_config_ok(c)) return OPTR_ERR_INVALID_ARG;
  if (!q || !K || !V || !t_pos || !W_O || !R_K || !R_V || !mu) return OPTR_ERR_INVALID_ARG;
  if (c->steps > 0 && (!hist_k || !hist_v)) return OPTR_ERR_INVALID_ARG;
  const bool held = c->T_held > 0;
  if (held && (!q_held || !K_held || !V_held || !t_pos_held)) return OPTR_ERR_INVALID_ARG;
  const size_t need = optr_calib_workspace_size(c);
  if (!workspace || ws_bytes < need || (reinterpret_cast<uintptr_t>(workspace) & 255))
    return OPTR_ERR_WORKSPACE;
  Calib C;
  if (!calib_init(C, c, workspace, W_O, stream)) return OPTR_ERR_CUDA;
  const int n = kCD * kCD;
  if (cudaMemsetAsync(C.err, 0, sizeof(unsigned), stream) != cudaSuccess ||
      cudaMemsetAsync(C.gcnt, 0, sizeof(int) * kGemmTiles, stream) != cudaSuccess)
    return OPTR_ERR_CUDA;
  col_mean_kernel<<<kCD / 4, 256, 0, stream>>>(K, c->T, mu);
  const double* r0[2] = {R0_K, R0_V};
  for (int k = 0; k < 2; ++k) {
    if (r0[k]) copy_kernel<<<nblk(n), 256, 0, stream>>>(r0[k], n, C.R0[k]);
    else hadamard_kernel<<<kCD, kCD, 0, stream>>>(C.R0[k]);
  }
  C.tr[0].q = q; C.tr[0].K = K; C.tr[0].V = V; C.tr[0].tpos = t_pos;
  C.tr[0].T = c->T; C.tr[0].nt = c->nt;
  trace_setup(C, C.tr[0], mu);
  if (held) {
    C.tr[1].q = q_held; C.tr[1].K = K_held; C.tr[1].V = V_held;
    C.tr[1].tpos = t_pos_held; C.tr[1].T = c->T_held; C.tr[1].nt = c->nt_held;
    trace_setup(C, C.tr[1], mu);
  } else {
    C.tr[1] = C.tr[0];
  }
  adam_run(C, 0, C.R0[0], hist_k);
  copy_kernel<<<nblk(n), 256, 0, stream>>>(C.best, n, R_K);
  copy_kernel<<<nblk(n), 256, 0, stream>>>(C.best, n, C.R);
  value_setup(C, C.tr[0]);
  if (held) value_setup(C, C.tr[1]);
  adam_run(C, 1, C.R0[1], hist_v);
  copy_kernel<<<nblk(n), 256, 0, stream>>>(C.best, n, R_V);
  return calib_finish(C);
}

extern "C" optr_status optr_calib_loss_grad(
    const optr_calib_config* c, int which, const double* q, const double* K,
    const double* V, const int32_t* t_pos, const double* W_O, const double* mu,
    const double* R_K, const double* R0, const double* A, double* loss, double* dA,
    void* workspace, size_t ws_bytes, cudaStream_t stream) {
  if (!calib_config_ok(c) || (which != 0 && which != 1)) return OPTR_ERR_INVALID_ARG;
  if (!q || !K || !V || !t_pos || !W_O || !mu || !R0 || !A || !loss)
    return OPTR_ERR_INVALID_ARG;
  if (which == 1 && !R_K) return OPTR_ERR_INVALID_ARG;
  const size_t need = optr_calib_workspace_size(c);
  if (!workspace || ws_bytes < need || (reinterpret_cast<uintptr_t>(workspace) & 255))
    return OPTR_ERR_WORKSPACE;
  Calib C;
  if (!calib_init(C, c, workspace, W_O, stream)) return OPTR_ERR_CUDA;
  const int n = kCD * kCD;
  if (cudaMemsetAsync(C.err, 0, sizeof(unsigned), stream) != cudaSuccess ||
      cudaMemsetAsync(C.gcnt, 0, sizeof(int) * kGemmTiles, stream) != cudaSuccess)
    return OPTR_ERR_CUDA;
  C.tr[0].q = q; C.tr[0].K = K; C.tr[0].V = V; C.tr[0].tpos = t_pos;
  C.tr[0].T = c->T; C.tr[0].nt = c->nt;
  trace_setup(C, C.tr[0], mu);
  if (which == 1) {
    copy_kernel<<<nblk(n), 256, 0, stream>>>(R_K, n, C.R);
    value_setup(C, C.tr[0]);
  }
  copy_kernel<<<nblk(n), 256, 0, stream>>>(A, n, C.A);
  skew_kernel<<<kCD, kCD, 0, stream>>>(C.A, nullptr, C.S, C.norm);
  C.squares = kMaxSquare;
  rotation(C, R0);
  if (which == 0) key_forward(C, C.tr[0], loss);
  else value_forward(C, C.tr[0], loss);
  if (dA) {
    if (which == 0) key_backward(C, C.tr[0]);
    else value_backward(C, C.tr[0]);
    generator_grad(C, R0);
    // dA = L^T - L
    skew_kernel<<<kCD, kCD, 0, stream>>>(C.L, C.s_dev, C.dA, nullptr);
    neg_kernel<<<nblk(n), 256, 0, stream>>>(C.dA, n, dA);
  }
  return calib_finish(C);
}
