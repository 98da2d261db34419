// Elimination of a block by a warp, or by a CTA's warps (bigblock.cu), in 64-bit fixed point:
// panels of eight columns in integer arithmetic, the updates between panels on the tensor cores.
//
// On GB300 a warp's FP64 instruction holds its sub-partition's pipe for 64 cycles; at m = 60
// the elimination's 1,270 of them per location were the kernels' bound (FP64 pipe 81-85%
// busy).  A multiply-accumulate of 31-bit limbs takes about 16 cycles of the integer pipes,
// an mma.m16n8k16 (half precision, FP32 accumulation) 7.4 for 2,048 products.  So the block
// is factored without FP64, as a left-looking Cholesky A = Lc Lc^T:
//   - entries below the diagonal, and Schur complements, in units of 2^-60 (they are at most
//     1 in magnitude), the diagonal (up to 1 + gamma) in units of 2^(2f - 60), f =
//     floor(log2(1 + gamma) / 2);
//   - V = Lc 2^62.  Off-diagonal entries of Lc are at most 2^-f in magnitude: a Schur
//     complement of R + gamma I is gamma I plus a positive semidefinite matrix with diagonal
//     at most 1, hence Lc_rk^2 <= 1 / (1 + gamma);
//   - the data row y stays in FP64 (data have no common scale: one outlier, or a rough field under
//     a smooth covariance, would cost a row of integers its digits): each column's
//     z_c = y_c / sqrt(d_c) and y_r -= Lc_rc z_c, one conversion and one FMA a row and column on the
//     pipe that the integers leave idle.  (A row of integers in units chosen from sigma and the largest
//     datum, built again with larger ones where z outgrew them, took 3% less time with the gradient at m =
//     60 and 7% less without where it fitted, and 60% and 85% more where it did not: n = 100k, white data
//     under nu = 3/2, no nugget, 13.7 and 10.6 ms against 8.53 and 5.70.)
// FP64's column-by-column update rounds entries of size 1 to 2^-54 at every step; here every
// entry carries an absolute error of about 2^-58.
//
// Updates between panels: A_rc -= sum_{k < c0} Lc_rk Lc_ck, for the eight columns of the next
// panel at once, as exact products of integers.  V is stored as its eight bytes, V +
// 0x8080808080808080 = sum_i b_i 256^(7-i): digits d_i = b_i - 128, each a half exactly.  The
// products d_i d'_j of one diagonal i + j = s add up to integers, which an FP32 accumulator holds
// exactly below 2^24.  With c0 columns a pair of digits adds up to at most 2^14 c0, or, where one is d_0 =
// 64 Lc rounded (a row's squares add up to at most 1), 2^13 sqrt(c0); of the eight pairs of s = 7, six of
// the first kind.  Up to m = 150 (c0 <= 144) that is 2^23.8, so every sum is exact.  Up to 63 (c0 <=
// 56) the sums to s = 5 stay below 2^22 too: they start at 1.5 2^23, so that the integer is read off the
// accumulator's bits, without a conversion (all converted: n = 100k, m = 60 with the gradient 8.57 -> 8.69
// ms).  Kept are the pairs i + j <= 7; the dropped ones add up to a few units of 2^-60.
//
// The bytes take the factor entries' own places: the four entries (r, 4w .. 4w+3) of a row
// become eight words, one per digit plane, each with the digit of the four columns; so the
// panels need no memory of their own (12 locations an SM, as with FP64).  A lane's four k of
// a k16 step are the four columns of one word group (the MMA's k order is free as long as
// both operands share it), so a fragment register is one byte permute (1024 + b as a half)
// and one packed subtraction.
//
// All loops over columns and rows stay rolled: the phases of a location then run from the
// instruction cache (unrolled over a panel's columns, instruction fetch was the largest
// stall and the kernel 1.5 times slower).
#pragma once

#include "common.cuh"
#include "fixtable.cuh"
#include "matern.cuh"

namespace vecchia {

constexpr int kPanelCols = 8;
constexpr int kPanelWords = kPanelCols / 4;
constexpr unsigned long long kByteBias = 0x8080808080808080ull;
// A pivot, or s_i / sigma2, at or below 2^-53 of the variance (in units of 2^-60) counts as zero: the block is not
// positive definite.  Two coincident points without a nugget leave a Schur complement that is exactly 0; the
// rows are eliminated alike but for where a column's products are summed, on the tensor cores or in a
// panel, so what is left of it is the rounding of one panel's fourteen mixed products (28 units at
// most, 6 as a rule), of the dropped digits (some 3) and of V (2).  The smallest nugget that
// FP64 tells from none leaves twice the threshold.
constexpr long long kSmallestPivot = 128;
// Blocks that are eliminated in FP64 all the same.  The factor's absolute errors are as good as FP64's relative
// ones while its entries and data are of ordinary size; not
//  - where a few data tower over the others, whose small weights' errors they multiply: fewer than half
//    of the block's data (zeros left aside) within 2^6 (by exponent) of the largest.  Of 61 normal variates 58 are;
//  - where the location is barely correlated with any neighbour and what is wanted is as small: a prediction
//    (rho < 2^-8), or derivatives (rho < 2^-12: they are double-float, to 2^-46).  The nearest neighbour's u
//    says so (looked up in the table at every location: n = 50k on the sphere, m = 60 5.26 -> 5.52 ms);
//  - where the nugget is 2^16 times the variance or more (f >= 8).
// They cost what FP64 costs (n = 100k, m = 60, value and with the gradient, ms: every block 8.97 and 11.1; one
// datum in 60 a million times larger 7.81 and 11.3; none 5.83 and 8.54).
constexpr int kEvenBits = 6;
constexpr int kMostShift = 7;
constexpr float kAccZero = 12582912.0f;  // 1.5 2^23
constexpr unsigned kAccZeroBits = 0x4B400000u;

__device__ __forceinline__ unsigned exponent_field(double x) {
  return (unsigned)(__double_as_longlong(x) >> 52) & 0x7FFu;
}

// 2^k, -1022 <= k <= 1023 (clamped).
__device__ __forceinline__ double pow2_double(int k) {
  return __longlong_as_double((long long)(min(max(k, -1022), 1023) + 1023) << 52);
}

__device__ __forceinline__ void mma_f16(float (&c)[4], const unsigned (&a)[4], const unsigned (&b)[2]) {
  asm("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b[0]), "r"(b[1]));
}

// Two digits (bytes of w picked by sel) as a pair of halves.
__device__ __forceinline__ unsigned digit_pair(unsigned w, unsigned sel) {
  const unsigned p = __byte_perm(w, 0x64646464u, sel);  // 1024 + b
  unsigned r;
  asm("sub.rn.f16x2 %0, %1, %2;" : "=r"(r) : "r"(p), "r"(0x64806480u));  // - 1152
  return r;
}

// Digit planes of four columns' integers.
__device__ __forceinline__ void digit_planes(const long long (&v)[4], unsigned (&out)[8]) {
  unsigned lo[4], hi[4];
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const unsigned long long b = (unsigned long long)v[k] + kByteBias;
    lo[k] = (unsigned)b;
    hi[k] = (unsigned)(b >> 32);
  }
  const unsigned a = __byte_perm(lo[0], lo[1], 0x5140), b = __byte_perm(lo[2], lo[3], 0x5140);  // bytes 0, 1
  const unsigned c = __byte_perm(lo[0], lo[1], 0x7362), d = __byte_perm(lo[2], lo[3], 0x7362);  // bytes 2, 3
  out[7] = __byte_perm(a, b, 0x5410);
  out[6] = __byte_perm(a, b, 0x7632);
  out[5] = __byte_perm(c, d, 0x5410);
  out[4] = __byte_perm(c, d, 0x7632);
  const unsigned e = __byte_perm(hi[0], hi[1], 0x5140), f = __byte_perm(hi[2], hi[3], 0x5140);
  const unsigned g = __byte_perm(hi[0], hi[1], 0x7362), h = __byte_perm(hi[2], hi[3], 0x7362);
  out[3] = __byte_perm(e, f, 0x5410);
  out[2] = __byte_perm(e, f, 0x7632);
  out[1] = __byte_perm(g, h, 0x5410);
  out[0] = __byte_perm(g, h, 0x7632);
}

// Integer of column x (0..3) from the digit planes of its word.
__device__ __forceinline__ long long planes_value(const unsigned (&w)[8], int x) {
  const unsigned s2 = ((4 + x) << 4) | x;
  const unsigned lo = __byte_perm(__byte_perm(w[7], w[6], s2), __byte_perm(w[5], w[4], s2), 0x5410);
  const unsigned hi = __byte_perm(__byte_perm(w[3], w[2], s2), __byte_perm(w[1], w[0], s2), 0x5410);
  return (long long)((((unsigned long long)hi << 32) | lo) - kByteBias);
}

// Slots of the entries (row, k0 .. k0 + 3): slot of (row, k) is tri_off(K, k) + row - k.
struct WordSlots {
  int e[4];
  __device__ __forceinline__ WordSlots(int K, int k0) {  // of row 0; add the row
    e[0] = tri_off(K, k0) - k0;
#pragma unroll
    for (int i = 1; i < 4; ++i) e[i] = e[i - 1] - (K - k0 - i + 1) - 1;
  }
};

// 1/sqrt(d) of a positive d < 2^62: with d 2^(2q) in [2^60, 2^62), 2^31 / sqrt(d 2^(2q)) =
// R 2^-60, in (1, 2].  FP32 seed y, then one third-order step y (1 + e/2 + 3
// e^2/8), e = 1 - d y^2 in units of 2^-60 (|e| < 2^-20: the omitted 5 e^3/16 is below 2^-61).
__device__ __forceinline__ long long rsqrt_fixed(long long d, int& q) {
  q = (__clzll(d) - 2) >> 1;
  const long long dn = d << (2 * q);
  const float g = __int2float_rn((int)(dn >> 32)) * 0x1p-30f;  // d 2^(2q) / 2^62 in [1/4, 1]
  float r;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(g));
  r = fminf(fmaxf(r, 1.0f), 0x1.fffffep0f);
  const int Y = (int)(((__float_as_uint(r) & 0x7FFFFFu) | 0x800000u) << 7);  // y 2^30
  const long long t = (long long)(int)(dn >> 31) * Y + (((long long)((int)dn & 0x7FFFFFFF) * Y) >> 31);
  const long long w = (long long)(int)(t >> 31) * Y + (((long long)((int)t & 0x7FFFFFFF) * Y) >> 31);
  const long long e = (1LL << 60) - w;
  const int e32 = (int)(e >> 8);
  const int s = (int)(((long long)e32 * e32) >> 32);  // e^2 2^72
  const long long de = e + ((3LL * s) >> 14);         // (e/2 + 3 e^2/8) 2^61
  const long long R = ((long long)Y << 30) + (long long)Y * (int)(de >> 31) +
                      (((long long)Y * ((int)de & 0x7FFFFFFF)) >> 31);
  return R;
}

// Whether a pivot (a double) counts as zero.
__device__ __forceinline__ bool zero_pivot(double d) { return __double2hiint(d) <= (1023 - 53) << 20; }

// Whether a datum of exponent field e counts as large in a block whose largest has top.
__device__ __forceinline__ bool large_datum(int e, int top) { return e >= top - kEvenBits; }

// A finite positive double times 2^sh as a 64-bit integer, rounded to nearest; the result must stay
// below 2^62.
__device__ __forceinline__ long long fixed_from_double(double x, int sh) {
  const long long b = __double_as_longlong(x);
  const int ef = (int)((b >> 52) & 0x7FF);
  const unsigned long long mant = (unsigned long long)((b & 0xFFFFFFFFFFFFFLL) | (ef ? 0x10000000000000LL : 0LL)) << 9;
  const int r = 9 - ((ef ? ef : 1) - 1075 + sh);  // x 2^sh = (mant << 9) >> r
  return r <= 0 ? (long long)mant : r < 63 ? (long long)((mant + (1ull << (r - 1))) >> r) : 0LL;
}

// R 2^k for rsqrt_fixed's R in (2^60, 2^61], rounded to nearest; the pivot d 2^(2f - 60) has the
// reciprocal square root R 2^(q - f - 61).
__device__ __forceinline__ double pivot_scale(long long R, int k) {
  return __longlong_as_double(((R + 128) >> 8) + ((long long)(1022 + 60 + k) << 52));
}

// x 2^k for any int k, by exact powers of two.
__device__ __forceinline__ double mul_pow2(double x, int k) {
  k = min(max(k, -2400), 2400);
  const int k1 = k / 3, k2 = (k - k1) / 2, k3 = k - k1 - k2;
  return x * pow2_double(k1) * pow2_double(k2) * pow2_double(k3);
}

// c + (a b >> 32), one instruction.
__device__ __forceinline__ int mad_hi(int a, int b, int c) {
  int r;
  asm("mad.hi.s32 %0, %1, %2, %3;" : "=r"(r) : "r"(a), "r"(b), "r"(c));
  return r;
}

// |a| >> 32, roughly (one below for negative a).
__device__ __forceinline__ int top_magnitude(long long a) { return (int)(a >> 32) ^ (int)(a >> 63); }

// A Schur complement's entry times its column's pivot reciprocal: V.
__device__ __forceinline__ long long scaled_entry(long long a, int q, int rh, int rl, int f) {
  const long long n = a << q;
  const int ch = (int)(n >> 31), cl = (int)n & 0x7FFFFFFF;
  const long long mid = (long long)ch * rl + (long long)cl * rh;
  const long long v = ((long long)ch * rh << 3) + (mid >> 28);
  return f ? v >> min(f, 63) : v;
}

// f of the diagonal's units (see above).
__device__ __forceinline__ int panel_shift(double gamma1) { return max(((int)exponent_field(gamma1) - 1023) >> 1, 0); }

// A_rc -= sum_{k < c0} Lc_rk Lc_ck for the columns [c0, pe) of the panel and the sixteen rows
// from rt on; WIDE where c0 may exceed 56.  (Two row tiles at a time, which share the column operand's conversion, cost
// more in registers and code than they save.)
template <bool WIDE>
__device__ __forceinline__ void update_tile(int K, long long* __restrict__ A, int rt, int c0, int pe, int f, int lane) {
  const int g = lane >> 2, t = lane & 3;
  const uint2* __restrict__ D = reinterpret_cast<const uint2*>(A);
  const int R = K - 1;            // the last row, the location's
  const int rb = min(c0 + g, R);  // the panel's own rows: the MMA's columns
  const int r0 = min(rt + g, R), r1 = min(rt + g + 8, R);
  float d[8][4];
#pragma unroll
  for (int s = 0; s < 8; ++s)
#pragma unroll
    for (int v = 0; v < 4; ++v) d[s][v] = WIDE || s > 5 ? 0.0f : kAccZero;
#pragma unroll 1
  for (int kb = 0; kb < c0; kb += 16) {
    const int k0 = kb + 4 * t;  // this lane's four columns; past the last panel: zeros
    uint2 x[4], y[4], z[4];
    if (k0 < c0) {
      const WordSlots w(K, k0);
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        x[i] = D[w.e[i] + r0];
        y[i] = D[w.e[i] + r1];
        z[i] = D[w.e[i] + rb];
      }
    } else {
#pragma unroll
      for (int i = 0; i < 4; ++i) x[i] = y[i] = z[i] = make_uint2(0x80808080u, 0x80808080u);
    }
    unsigned bf[8][2];
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      const unsigned v = j & 1 ? z[j >> 1].y : z[j >> 1].x;
      bf[j][0] = digit_pair(v, 0x4140);
      bf[j][1] = digit_pair(v, 0x4342);
    }
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const unsigned u = i & 1 ? x[i >> 1].y : x[i >> 1].x, v = i & 1 ? y[i >> 1].y : y[i >> 1].x;
      const unsigned af[4] = {digit_pair(u, 0x4140), digit_pair(v, 0x4140), digit_pair(u, 0x4342), digit_pair(v, 0x4342)};
#pragma unroll
      for (int j = 0; j < 8; ++j)
        if (i + j < 8) mma_f16(d[i + j], af, bf[j]);
    }
  }
  // sum_s acc_s 2^(48 - 8s), in units of 2^-60
#pragma unroll
  for (int v = 0; v < 4; ++v) {
    int a[8];
#pragma unroll
    for (int s = 0; s < 7; ++s)
      a[s] = WIDE || s > 5 ? __float2int_rn(d[s][v]) : (int)(__float_as_uint(d[s][v]) - kAccZeroBits);
    a[7] = (int)(__float_as_uint(__fadd_rn(d[7][v], 256.0f * kAccZero)) - kAccZeroBits - (8u << 23));  // to units of 2^8
    const unsigned T = (unsigned)a[0] * 65536u + (unsigned)a[1] * 256u + (unsigned)a[2];
    long long sum = (long long)((unsigned long long)T << 32) + (long long)a[3] * (1 << 24) + (long long)a[4] * (1 << 16) +
                    (long long)a[5] * 256 + (a[6] + a[7]);
    const int row = rt + g + 8 * (v >> 1), c = c0 + 2 * t + (v & 1);
    if (row <= R && c < pe && row >= c) {
      const int e = tri_off(K, c) + row - c;
      if (f && row == c) sum >>= min(2 * f, 63);
      A[e] -= sum;
    }
  }
}

// The columns [c0, min(c0 + 8, K - 1)) of a panel, left-looking, a row per lane and slot (rows
// c0 + lane and c0 + lane + 32): A becomes V there.  C_mm is returned in corner when column
// m = K - 1 lies in the panel.  The high limbs' products are summed in 64
// bits, the mixed ones in units of 2^-58 (each rounded down, half a unit on average, which
// the start values give back; a row's entries have squares that add up to at most 1, so that seven
// columns' stay below 2^31).  The data of the lane's rows (slots (K, r) of the triangle) take each
// column's z_c times the row's entry off, and column c's own slot is left z_c / sqrt(d_c), the unit factor's
// entry.  Returns whether the block can still be positive definite.
// With CTA only the panel's own rows (of the last panel: all) and not the data, and the pivots' reciprocals are
// left in piv for panel_row and panel_solve.
template <bool GRAD, bool CTA>
__device__ __forceinline__ bool panel_columns(int K, long long* __restrict__ A, float2* __restrict__ RJ,
                                              int4* __restrict__ piv, int c0, int f, long long& corner, int lane) {
  const int R = K - 1;
  const int rmax = CTA && c0 + kPanelCols < K ? c0 + kPanelCols - 1 : R;
  const int last = K - 1 - c0;    // panel position of column m
  const int jn = min(last + 1, kPanelCols);
  const int r0 = c0 + lane, r1 = r0 + 32;
  const bool two = !CTA && c0 + 32 <= R;  // warp-uniform
  int over = 0;
  bool ok = true;
  const int2* __restrict__ V = reinterpret_cast<const int2*>(A);
  double* __restrict__ Y = reinterpret_cast<double*>(A);
  const int y0s = tri_off(K, min(r0, R)) + K - min(r0, R), y1s = tri_off(K, min(r1, R)) + K - min(r1, R);
  // The data: column j's z_j goes round (through the triangle's unused slot 0) after its V, and is taken off
  // the rows in the next column, where the FP64 pipe's latency hides behind the integers.
  double y0 = CTA ? 0.0 : Y[y0s], y1 = two ? Y[y1s] : 0.0;
  double v0 = 0.0, v1 = 0.0, z = 0.0, scale = 0.0;
#pragma unroll 1
  for (int j = 0; j < jn; ++j) {
    const int oj = tri_off(K, c0 + j) - (c0 + j);
    const int q0 = min(max(r0, c0 + j), rmax), q1 = min(r1, R);
    long long s0 = 0, s1 = 0;
    int m0 = j, m1 = j;
    int ok_ = tri_off(K, c0) - c0, step = K - c0;  // slot of (row 0, column c0 + k)
#pragma unroll 1
    for (int k = 0; k < j; ++k) {
      const int2 p = V[ok_ + c0 + j], x = V[ok_ + q0];
      const int lp = (int)((unsigned)p.x >> 2);
      s0 += (long long)x.y * p.y;
      m0 = mad_hi(x.y, lp, m0);
      m0 = mad_hi((int)((unsigned)x.x >> 2), p.y, m0);
      if (two) {
        const int2 y = V[ok_ + q1];
        s1 += (long long)y.y * p.y;
        m1 = mad_hi(y.y, lp, m1);
        m1 = mad_hi((int)((unsigned)y.x >> 2), p.y, m1);
      }
      ok_ -= step + 1;
      --step;
    }
    if (!CTA) y0 = fma(-v0, z, y0);
    if (two) y1 = fma(-v1, z, y1);
    s0 += (long long)m0 * 4;
    if (f && lane == j) s0 >>= min(2 * f, 63);
    const long long a0 = r0 >= c0 + j && r0 <= rmax ? A[oj + q0] - s0 : 0;
    if (j == last) {
      corner = __shfl_sync(0xffffffffu, a0, j);
      break;
    }
    long long d = __shfl_sync(0xffffffffu, a0, j);
    if (d <= kSmallestPivot) {  // a failed block runs on (values unused)
      ok = false;
      d = 1LL << 60;
    }
    int q;
    const long long pr = rsqrt_fixed(d, q);
    const int rh = (int)(pr >> 31), rl = (int)pr & 0x7FFFFFFF;
    if (CTA && lane == 0) piv[j] = make_int4(q, rh, rl, 0);
    const double rs = pivot_scale(pr, q - f - 61 - 62);  // 2^-62 / sqrt(d)
    const double zj = y0 * rs;  // lane j: z_j 2^-62
    if (GRAD && lane == j) scale = rs;
    // V of this lane's rows; |V| >= 2^62 2^-f: not a positive definite block
    const int lim = max(29 - q, 0);
    __syncwarp();  // the pivot row's entries of this column are read
    if (GRAD) v0 = 0.0;  // (without, the eliminated rows' data are not used again)
    if (lane > j && r0 <= rmax) {
      over |= top_magnitude(a0) >> lim;
      const long long v = scaled_entry(a0, q, rh, rl, f);
      A[oj + r0] = v;
      if (!CTA) v0 = (double)v;
    }
    if (two) {
      s1 += (long long)m1 * 4;
      const long long a1 = A[oj + q1] - s1;
      if (r1 <= R) {
        over |= top_magnitude(a1) >> lim;
        const long long v = scaled_entry(a1, q, rh, rl, f);
        A[oj + r1] = v;
        v1 = (double)v;
      }
    }
    if (!CTA && lane == j) Y[0] = zj;
    __syncwarp();
    if (!CTA) z = Y[0];
  }
  if (CTA) return ok && !__any_sync(0xffffffffu, over != 0);
  if (c0 + kPanelCols <= R) {  // (the last panel's last column takes nothing off)
    y0 = fma(-v0, z, y0);
    if (two) y1 = fma(-v1, z, y1);
  }
  if (r0 <= rmax) {
    if (r0 >= c0 + kPanelCols || r0 == R) Y[y0s] = y0;
    else if (GRAD) Y[y0s] = y0 * (scale * 0x1p62) * (scale * 0x1p62);
    if (GRAD && r0 < min(c0 + kPanelCols, R)) RJ[r0] = d2f_trunc(scale);
  }
  if (two && r1 <= R) Y[y1s] = y1;
  __syncwarp();
  return ok && !__any_sync(0xffffffffu, over != 0);
}

// Row r below the panel [c0, c0 + 8), by one thread: its eight entries of the factor, from the
// panel's own rows and pivots, and then their digits, in place; and (DATA) its datum.
template <bool DATA>
__device__ __forceinline__ void panel_row(int K, long long* __restrict__ A, const int4* __restrict__ piv,
                                          const double* __restrict__ zs, int c0, int f, int r, int& over) {
  const int2* __restrict__ V = reinterpret_cast<const int2*>(A);
  double* __restrict__ Y = reinterpret_cast<double*>(A) + tri_off(K, r) + K - r;
  double y = DATA ? *Y : 0.0, v0 = 0.0, z = 0.0;  // a column's part is taken off in the next one
#pragma unroll 1
  for (int j = 0; j < kPanelCols; ++j) {
    long long s0 = 0;
    int m0 = j;
    int ok_ = tri_off(K, c0) - c0, step = K - c0;  // slot of (row 0, column c0 + k)
#pragma unroll 1
    for (int k = 0; k < j; ++k) {
      const int2 p = V[ok_ + c0 + j], x = V[ok_ + r];
      s0 += (long long)x.y * p.y;
      m0 = mad_hi(x.y, (int)((unsigned)p.x >> 2), m0);
      m0 = mad_hi((int)((unsigned)x.x >> 2), p.y, m0);
      ok_ -= step + 1;
      --step;
    }
    if (DATA) y = fma(-v0, z, y);
    const int4 pv = piv[j];
    const long long a = A[ok_ + r] - s0 - (long long)m0 * 4;
    over |= top_magnitude(a) >> max(29 - pv.x, 0);
    const long long v = scaled_entry(a, pv.x, pv.y, pv.z, f);
    A[ok_ + r] = v;
    if (DATA) {
      v0 = (double)v;
      z = zs[j];
    }
  }
  if (DATA) *Y = fma(-v0, z, y);
#pragma unroll 1
  for (int k0 = 0; k0 < kPanelCols; k0 += 4) {
    const WordSlots w(K, c0 + k0);
    long long v[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) v[i] = A[w.e[i] + r];
    unsigned pl[8];
    digit_planes(v, pl);
#pragma unroll
    for (int i = 0; i < 4; ++i) reinterpret_cast<uint2*>(A)[w.e[i] + r] = make_uint2(pl[2 * i], pl[2 * i + 1]);
  }
}

// The data of panel [c0, c0 + 8)'s own rows, all earlier columns taken off, by one warp: z_c 2^-62 to zs, the unit
// factor's entries z_c / sqrt(d_c) and (GRAD) 2^-62 / sqrt(d_c); row m's datum, in the last panel, becomes the
// residual.
template <bool GRAD>
__device__ __forceinline__ void panel_solve(int K, long long* __restrict__ A, float2* __restrict__ RJ,
                                            const int4* __restrict__ piv, double* __restrict__ zs, int c0, int f, int lane) {
  const int R = K - 1, jn = min(kPanelCols, R - c0), r = min(c0 + lane, R);
  double* __restrict__ Y = reinterpret_cast<double*>(A) + tri_off(K, r) + K - r;
  const int4 pv = piv[min(lane, max(jn - 1, 0))];
  const double rs = pivot_scale(((long long)pv.y << 31) + pv.z, pv.x - f - 61 - 62);
  double y = *Y;
#pragma unroll 1
  for (int j = 0; j < jn; ++j) {
    const double v = r > c0 + j ? (double)A[tri_off(K, c0 + j) + r - c0 - j] : 0.0;
    const double z = __shfl_sync(0xffffffffu, y * rs, j);
    if (lane == j) zs[j] = z;
    if (r > c0 + j) y = fma(-v, z, y);
  }
  __syncwarp();
  if (lane < jn) {
    if (GRAD) {
      *Y = y * (rs * 0x1p62) * (rs * 0x1p62);
      RJ[r] = d2f_trunc(rs);
    }
  } else if (c0 + lane == R && lane < kPanelCols) {
    *Y = y;
  }
  __syncwarp();
}

// Panel [c0, c0 + 8)'s columns taken off the datum of row r below it, from the digits.
__device__ __forceinline__ void panel_row_data(int K, long long* __restrict__ A, const double* __restrict__ zs, int c0, int r) {
  double* __restrict__ Y = reinterpret_cast<double*>(A) + tri_off(K, r) + K - r;
  double y = *Y;
#pragma unroll 1
  for (int k0 = 0; k0 < kPanelCols; k0 += 4) {
    const WordSlots ws(K, c0 + k0);
    unsigned w[8];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const uint2 x = reinterpret_cast<const uint2*>(A)[ws.e[i] + r];
      w[2 * i] = x.x;
      w[2 * i + 1] = x.y;
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) y = fma(-(double)planes_value(w, i), zs[k0 + i], y);
  }
  *Y = y;
}

// The panel's factor entries of the rows below it as digits, in place.
__device__ __forceinline__ void panel_to_digits(int K, long long* __restrict__ A, int c0, int lane) {
  const int r0 = c0 + kPanelCols;
#pragma unroll 1
  for (int u = lane; u < kPanelWords * (K - r0); u += 32) {  // (row, word)
    const int r = r0 + u / kPanelWords, k0 = c0 + 4 * (u % kPanelWords);
    const WordSlots w(K, k0);
    long long v[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) v[i] = A[w.e[i] + r];
    unsigned pl[8];
    digit_planes(v, pl);
#pragma unroll
    for (int i = 0; i < 4; ++i) reinterpret_cast<uint2*>(A)[w.e[i] + r] = make_uint2(pl[2 * i], pl[2 * i + 1]);
  }
  __syncwarp();
}

// Cholesky over the neighbour columns.  Returns whether the block is positive definite.
template <bool GRAD>
__device__ __forceinline__ bool panels_eliminate(int K, long long* __restrict__ A, float2* __restrict__ RJ, int f,
                                                 long long& corner, int lane) {
  bool ok = true;
#pragma unroll 1
  for (int c0 = 0; c0 < K; c0 += kPanelCols) {
    const int pe = min(c0 + kPanelCols, K);
    if (c0 > 0) {
#pragma unroll 1
      for (int rt = c0; rt < K; rt += 16) update_tile<false>(K, A, rt, c0, pe, f, lane);
      __syncwarp();
    }
    const bool o = panel_columns<GRAD, false>(K, A, RJ, nullptr, c0, f, corner, lane);
    ok = ok && o;
    if (pe < K) panel_to_digits(K, A, c0, lane);
  }
  return ok;
}

// V 2^-62 / sqrt(d) as a float pair, rj = 2^-62 / sqrt(d).
__device__ __forceinline__ float2 unit_pair(long long v, float2 rj) {
  // v = a 2^39 + b 2^23 + c, each an exact float
  const float fa = __int2float_rn((int)(v >> 39)) * 0x1p39f;
  const float fb = __int2float_rn((int)(v >> 23) & 0xFFFF) * 0x1p23f;
  const float fc = __int2float_rn((int)((unsigned)v & 0x7FFFFFu));
  float vh, vl;
  float2 o;
  fast_two_sum(fa, fb, vh, vl);
  df_mul(vh, __fadd_rn(vl, fc), rj.x, rj.y, o.x, o.y);
  return o;
}

// After the elimination, for the adjoint: every entry of the factor below the diagonal
// (neighbour columns) becomes a float pair of the unit factor in its place, those of the data row too.
// By nth threads.
__device__ __forceinline__ void panels_to_pairs(int K, long long* __restrict__ A, const float2* __restrict__ RJ, int tid,
                                                int nth) {
  float2* __restrict__ P = reinterpret_cast<float2*>(A);
  for (int c = tid; c < K - 1; c += nth) {
    const int e = tri_off(K, c) + K - c;
    P[e] = d2f_trunc(reinterpret_cast<const double*>(A)[e]);
  }
#pragma unroll 1
  for (int c0 = 0; c0 < K - 1; c0 += kPanelCols) {
    // below the panel: digits, one (row, word) per lane; in it (and all of the last panel): V
    const bool lastp = c0 + kPanelCols >= K;
    const int rb = lastp ? K : c0 + kPanelCols;
#pragma unroll 1
    for (int u = tid; u < kPanelWords * (K - c0); u += nth) {
      const int r = c0 + u / kPanelWords, k0 = c0 + 4 * (u % kPanelWords);
      const WordSlots ws(K, k0);
      unsigned w[8];
      if (r >= rb) {
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const uint2 x = reinterpret_cast<const uint2*>(A)[ws.e[i] + r];
          w[2 * i] = x.x;
          w[2 * i + 1] = x.y;
        }
      }
#pragma unroll
      for (int x = 0; x < 4; ++x) {
        const int c = k0 + x;
        if (r > c && c < K - 1) {
          const long long v = r >= rb ? planes_value(w, x) : A[ws.e[x] + r];
          P[ws.e[x] + r] = unit_pair(v, RJ[c]);
        }
      }
    }
  }
}

}  // namespace vecchia
