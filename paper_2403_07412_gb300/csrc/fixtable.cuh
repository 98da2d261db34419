// The covariance table of the likelihood kernels: rho(u) by way of 64-bit fixed point and
// h(u) = u rho'(u) as a float pair, from u = uh + ul as a float pair.
//
// u in [2^e (1 + j/32), 2^e (1 + (j+1)/32)), e in [kELo, kEHi), t = 32 u / 2^e - 32 - j in
// [0, 1), rho 2^E ~ P(t) = sum_{k<=7} c_k t^k, where E is 0 down to rho = 2^-7 and brings the
// smaller ones to 2^-7 .. 2^-6, so that a correlation has its leading 50 bits however small it is
// (down to 2^-970 or so; E costs nothing: the exponent that is subtracted with it was a constant
// before).  rho is completely monotone in u (both
// families), so the c_k alternate in sign and, up to u = 2^12, each |c_k| is at least
// |c_{k+1} + c_{k+2} t + ...|: a Horner step can add its two parts with the three-
// instruction form of the error-free sum (fast_two_sum), which wants the larger one first.
// (Beyond, rho is below 2^-90 and changes by more than 2 within an interval: the polynomial
// itself is then off by 2^-22 and more.)  A step does not renormalise its pair either: nine instructions
// where the general double-float step (df_horner) takes fifteen.  Twice the intervals of
// the general table (matern.cuh), whose t runs over [-1, 1), keep the coefficients as small.
// Words of interval idx (kFixWords float4 each), every c_k for k >= 1 times 2^S:
//   w0: c1 hi, c1 lo, c2 hi, c2 lo       w1: c3 hi, c3 lo, c4 hi, c4 lo
//   w2: c5, c6, c7, (62 + E) 2^20 (int)  w3: c0 in units of 2^-62 (int64, low word first),
//   w4: 3c3 hi, 3c3 lo, 5c5, 6c6              2^(36-S), 2^(-S-E)
// (Five words: with an odd number the gathers of a warp spread over all banks.)
#pragma once

#include "common.cuh"
#include "matern.cuh"

namespace vecchia {

__host__ __device__ __forceinline__ double* fix_const(double* tab) { return tab + 2 * kFixWords * kFixInt; }
__device__ __forceinline__ const double* fix_const(const double* tab) { return tab + 2 * kFixWords * kFixInt; }

// After the small-u constants: the least u, by intervals, from which on rho is below 2^-kWeakPrediction and
// 2^-kWeakGradient (E two and six; to within a factor of two).
constexpr int kWeakPrediction = 8, kWeakGradient = 12;
constexpr int kConstWeakPrediction = 6, kConstWeakGradient = 7;

// s + e = a + b exactly for |a| >= |b| (or a = 0).
__device__ __forceinline__ void fast_two_sum(float a, float b, float& s, float& e) {
  s = __fadd_rn(a, b);
  e = __fsub_rn(b, __fsub_rn(s, a));
}

// (ph, pl) <- (ch, cl) + (ph, pl) (th, tl) for |c| >= |p t|.
__device__ __forceinline__ void fix_horner(float& ph, float& pl, float th, float tl, float ch, float cl) {
  float xh, xl, s, e;
  df_mul(ph, pl, th, tl, xh, xl);
  fast_two_sum(ch, xh, s, e);
  ph = s;
  pl = __fadd_rn(e, __fadd_rn(xl, cl));
}

struct FixArg {
  int idx, ex;
  float th, tl, mh;  // t = th + tl, u 2^(5-e) = mh + tl
};

__device__ __forceinline__ FixArg fix_arg(float uh, float ul) {
  FixArg a;
  const unsigned ub = __float_as_uint(uh);
  a.ex = (int)(ub >> 23) - 127;  // u >= 0
  const int ec = min(max(a.ex, kELo), kEHi - 1);
  a.idx = ((ec - kELo) << kFixSub) | (int)((ub >> (23 - kFixSub)) & ((1u << kFixSub) - 1));
  const float sc = __uint_as_float((unsigned)(127 + kFixSub - ec) << 23);
  a.th = __uint_as_float(0x3F800000u | ((ub << kFixSub) & 0x7FFFFFu)) - 1.0f;
  a.tl = __fmul_rn(ul, sc);
  a.mh = __fmul_rn(uh, sc);
  return a;
}

// A correlation v 2^-(sh / 2^20): |v| <= 2^62, sh >= 61 2^20.
struct FixRho {
  long long v;
  int sh;
};

// t (c1 + ...) is a float pair below 2^-6 in magnitude: its multiple of 2^-36 and the rest (below
// 2^-26: q tl), in units of 2^-56, go to integers by conversion.  The integer re-enters FP64 by
// one conversion (64 cycles of the FP64 pipe; two additions before).
__device__ __forceinline__ FixRho rho_table62(float uh, float ul, const double* __restrict__ tab) {
  const FixArg a = fix_arg(uh, ul);
  const float4* __restrict__ w = reinterpret_cast<const float4*>(tab) + a.idx * kFixWords;
  const float4 w0 = __ldg(w), w1 = __ldg(w + 1), w2 = __ldg(w + 2), w3 = __ldg(w + 3);
  float s, l, xh, xl;
  fast_two_sum(w1.z, __fmul_rn(fmaf(fmaf(w2.z, a.th, w2.y), a.th, w2.x), a.th), s, l);
  l = __fadd_rn(l, w1.w);
  fix_horner(s, l, a.th, a.tl, w1.x, w1.y);
  fix_horner(s, l, a.th, a.tl, w0.z, w0.w);
  fix_horner(s, l, a.th, a.tl, w0.x, w0.y);
  df_mul(s, l, a.th, a.tl, xh, xl);
  xl = fmaf(l, a.tl, xl);  // up to 2^-48 here
  const float fs = w3.z;  // 2^(36 - S)
  const float y = __fmul_rn(xh, fs);
  const int n1 = __float2int_rn(y);
  const float r = fmaf(xl, fs, __fsub_rn(y, __int2float_rn(n1)));
  const int n2 = __float2int_rn(r * 0x1p20f);
  const long long c0 = (long long)(((unsigned long long)__float_as_uint(w3.y) << 32) | __float_as_uint(w3.x));
  return {c0 + (long long)n1 * (1 << 26) + (long long)n2 * 64, __float_as_int(w2.w)};
}

// Whether u lies outside the table.
__device__ __forceinline__ bool fix_outside(float uh) {
  return __float_as_uint(uh) - ((unsigned)(kELo + 127) << 23) >= (unsigned)(kEHi - kELo) << 23;
}

// rho(u) there, exactly as FP64 has it (0 below 2^-1022).
__device__ __forceinline__ FixRho rho_outside62(float uh, float ul, const MaternConst& mc) {
  double rho = 0.0, h = 0.0;
  rho_fix(df_to_double(uh, ul), mc, rho, h);
  const long long b = __double_as_longlong(rho);
  const int ef = (int)((b >> 52) & 0x7FF);
  const long long mant = ((b & 0xFFFFFFFFFFFFFLL) | 0x10000000000000LL) << 9;
  return {ef == 0 ? 0LL : mant, (1084 - ef) << 20};
}

// (Rare; the constants by value, which keeps them in registers.)
static __device__ __noinline__ FixRho rho_outside62_call(float uh, float ul, int kind, double nu, double a1, double G,
                                                         double b0, double b1) {
  return rho_outside62(uh, ul, MaternConst{kind, nu, a1, G, b0, b1});
}

// rho(u) of one pair.
__device__ __forceinline__ FixRho rho_fixed62(float uh, float ul, const double* __restrict__ tab, const MaternConst& mc) {
  const FixRho r = rho_table62(uh, ul, tab);
  return fix_outside(uh) ? rho_outside62(uh, ul, mc) : r;
}

// rho(u) of two pairs: one branch for both keeps their instructions together (n = 100k, m = 10
// 162 -> 156 us, m = 60 5.39 -> 5.33 ms; the FP64 gradient kernels take more registers with it).
__device__ __forceinline__ void rho_fixed62(float u0h, float u0l, float u1h, float u1l, const double* __restrict__ tab,
                                            const MaternConst& mc, FixRho& r0, FixRho& r1) {
  r0 = rho_table62(u0h, u0l, tab);
  r1 = rho_table62(u1h, u1l, tab);
  if (fix_outside(u0h) || fix_outside(u1h)) {
    if (fix_outside(u0h)) r0 = rho_outside62_call(u0h, u0l, mc.kind, mc.nu, mc.a1, mc.G, mc.b0, mc.b1);
    if (fix_outside(u1h)) r1 = rho_outside62_call(u1h, u1l, mc.kind, mc.nu, mc.a1, mc.G, mc.b0, mc.b1);
  }
}

// In FP64: one conversion, and the power of two on the exponent field.  (A conversion holds the FP64 pipe
// for 64 cycles; integer operations in its place, some 25, gave 2% at m = 30 and took 2% at m = 10.)
__device__ __forceinline__ double fixed_to_double(FixRho r) {
  const double d = (double)r.v;
  return __hiloint2double(__double2hiint(d) - (r.v != 0 ? r.sh : 0), __double2loint(d));
}

// In units of 2^-60.
__device__ __forceinline__ long long fixed60(FixRho r) { return r.v >> min((r.sh >> 20) - 60, 63); }

// h(u) outside the table, as a float pair (rare).
static __device__ __noinline__ float2 h_outside(float uh, float ul, int kind, double nu, double a1, double G, double b0,
                                                double b1) {
  const MaternConst mc{kind, nu, a1, G, b0, b1};
  double r = 0.0, h = 0.0;
  rho_fix(df_to_double(uh, ul), mc, r, h);
  const float hi = __double2float_rn(h);
  return make_float2(hi, __double2float_rn(h - (double)hi));
}

// h(u) as a float pair (CALL: the rare path in a function, in the fixed-point kernels: n = 100k, m =
// 60 8.33 -> 8.26 ms).
template <bool CALL>
__device__ __forceinline__ void h_fixed(float uh, float ul, const double* __restrict__ tab, const MaternConst& mc,
                                        float& hh, float& hl) {
  const FixArg a = fix_arg(uh, ul);
  const float4* __restrict__ w = reinterpret_cast<const float4*>(tab) + a.idx * kFixWords;
  const float4 w0 = __ldg(w), w1 = __ldg(w + 1), w2 = __ldg(w + 2), w4 = __ldg(w + 4);
  const float inv = __ldg(reinterpret_cast<const float*>(w + 3) + 3);
  float s, l;
  fast_two_sum(4.0f * w1.z, __fmul_rn(fmaf(fmaf(7.0f * w2.z, a.th, w4.w), a.th, w4.z), a.th), s, l);
  l = fmaf(4.0f, w1.w, l);
  fix_horner(s, l, a.th, a.tl, w4.x, w4.y);
  fix_horner(s, l, a.th, a.tl, 2.0f * w0.z, 2.0f * w0.w);
  fix_horner(s, l, a.th, a.tl, w0.x, w0.y);
  df_mul(s, l, a.mh, a.tl, hh, hl);
  hh *= inv;
  hl *= inv;
  if (fix_outside(uh)) {
    if constexpr (CALL) {
      const float2 h = h_outside(uh, ul, mc.kind, mc.nu, mc.a1, mc.G, mc.b0, mc.b1);
      hh = h.x;
      hl = h.y;
    } else {
      double r = 0.0, h = 0.0;
      rho_fix(df_to_double(uh, ul), mc, r, h);
      const float hi = __double2float_rn(h);
      hh = hi;
      hl = __double2float_rn(h - (double)hi);
    }
  }
}

}  // namespace vecchia
