// Construction of the per-nu Matérn correlation table and the stand-alone covariance
// evaluator (vecchia_matern).
//
// rho(u) = 2^{1-nu}/Gamma(nu) x^nu K_nu(x), u = x^2, is computed at the table nodes from
// the integral representation K_nu(z) = (z/2)^nu / 2 int_0^inf exp(-t - z^2/(4t)) t^{-nu-1} dt
// (DLMF 10.32.10).  Substituting t = z^2/(4s) and s = e^tau gives
//   rho(u) = I(u) / I(0),   I(u) = int_R exp(nu tau - e^tau - (u/4) e^{-tau}) dtau,
// (I(0) = Gamma(nu)).  The integrand is analytic in the strip |Im tau| < pi/2 and decays
// double-exponentially, so the trapezoidal rule converges geometrically; the step is
// set from the curvature at the peak and from nu, and terms are summed with Neumaier
// compensation until they fall below e^-45 of the peak.
// Each interval's polynomial is the degree-kDeg Chebyshev interpolant at the
// first-kind Chebyshev points, converted to monomials in t and stored in the split
// FP64/FP32 layout that matern.cuh evaluates.
#include <algorithm>
#include <cmath>
#include <cstring>
#include <limits>
#include <mutex>
#include <vector>

#include "common.cuh"
#include "fixtable.cuh"
#include "matern.cuh"

namespace vecchia {

// I(u) by the trapezoidal rule, computed by a whole warp: lane l takes nodes k = k0 + l
// of each chunk of 32 on either side of the peak; a side ends after the first chunk that
// reaches a node below e^-45 of the peak (the log-integrand is concave, so the tail only
// falls from there).  Each lane keeps a compensated sum; the lanes' sums are merged by a
// fixed shuffle tree and lane 0's result is returned on every lane.  (One FP64
// instruction costs a warp as much with 1 lane active as with 32, so a single thread's
// serial loop would take 32 times longer.)  All 32 lanes must call it together.
__device__ double quad_I_warp(double u, double nu) {
  const int lane = threadIdx.x & 31;
  const double a = 0.25 * u;
  const double et = 0.5 * (nu + sqrt(nu * nu + 4.0 * a));  // e^tau at the peak
  const double tc = log(et);
  const double curv = et + a / et;                          // -(log integrand)'' at the peak
  const double h = fmin(0.2, fmin(0.6 / sqrt(curv), 0.3 / fmax(nu, 1.0)));
  const double lpeak = nu * tc - et - a / et;
  Neumaier acc;
  for (int side = 0; side < 2; ++side) {
    for (int k0 = side; k0 < 200000; k0 += 32) {
      const int k = k0 + lane;
      const double tau = side == 0 ? tc + k * h : tc - k * h;
      const double e = exp(tau);
      const double lv = nu * tau - e - a / e;
      acc.add(exp(lv - lpeak));
      if (__any_sync(0xffffffffu, lv - lpeak < -45.0 && k > 3)) break;
    }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const double s2 = __shfl_down_sync(0xffffffffu, acc.s, o);
    const double c2 = __shfl_down_sync(0xffffffffu, acc.c, o);
    acc.merge(s2, c2);
  }
  return __shfl_sync(0xffffffffu, acc.value(), 0) * h * exp(lpeak);
}

// One warp: I(0) and the small-u expansion constants (family Matérn), or the exponent
// (power exponential).
__global__ void matern_const_kernel(double nu, int family, double* c) {
  if (blockIdx.x != 0 || threadIdx.x >= 32) return;
  const double I0 = family == kFamilyPowExp ? 1.0 : quad_I_warp(0.0, nu);
  if (threadIdx.x != 0) return;
  if (family == kFamilyPowExp) {
    c[0] = __longlong_as_double(3LL);
    c[1] = nu;
    c[2] = c[3] = c[4] = c[5] = 0.0;
    c[6] = 1.0;
    c[7] = 0.0;
    return;
  }
  const bool integer = (nu == floor(nu));
  long long kind = integer ? (nu == 1.0 ? 1 : 2) : 0;
  c[0] = __longlong_as_double(kind);
  c[1] = nu;
  if (integer) {
    c[2] = nu == 1.0 ? 0.0 : -0.25 / (nu - 1.0);
    c[3] = c[4] = c[5] = 0.0;
  } else {
    c[2] = 0.25 / (1.0 - nu);
    c[3] = tgamma(1.0 - nu);
    c[4] = 1.0 / tgamma(1.0 + nu);
    c[5] = 0.25 / tgamma(2.0 + nu);
  }
  c[6] = I0;
  c[7] = 0.0;
}

// One block per interval, a warp per Chebyshev node.  Node values: the Matérn quadrature,
// or the power exponential exp(-u^(alpha/2)) (u = (d / beta^(1/alpha))^2) evaluated directly.
// One interval's coefficients in the layout of matern.cuh: c0 in FP64; c1..c4 and
// 3 c3 as float pairs (hi = nearest float, lo = nearest float to the rest); c5..c8,
// 5 c5, 6 c6 as floats; all floats scaled by 2^S, |max(c1..c4)| 2^S in [1/2, 1), so
// that they keep their relative precision wherever rho is small.
__device__ void split_float(double x, float* hl) {
  hl[0] = (float)x;
  hl[1] = (float)(x - (double)hl[0]);
}

__device__ void write_interval(const double* mono, float* w) {
  double top = 0.0;
  for (int k = 1; k <= 4; ++k) top = fmax(top, fabs(mono[k]));
  int S = 0;
  if (top > 0.0) {
    frexp(top, &S);
    S = -S;
  }
  double c[kDeg + 1];
  for (int k = 1; k <= kDeg; ++k) c[k] = ldexp(mono[k], S);
  split_float(c[1], w + 0);
  split_float(c[2], w + 2);
  split_float(c[3], w + 4);
  split_float(c[4], w + 6);
  for (int k = 5; k <= 8; ++k) w[8 + k - 5] = (float)c[k];
  const unsigned long long d0 = (unsigned long long)__double_as_longlong(mono[0]);
  w[12] = __uint_as_float((unsigned)(d0 & 0xFFFFFFFFULL));
  w[13] = __uint_as_float((unsigned)(d0 >> 32));
  w[14] = __int_as_float(S);
  w[15] = 0.0f;
  split_float(3.0 * c[3], w + 16);
  w[18] = (float)(5.0 * c[5]);
  w[19] = (float)(6.0 * c[6]);
}

// One CTA of kFitThreads (a warp per node) per interval.
constexpr int kFitThreads = 32 * (kDeg + 1);

__global__ void __launch_bounds__(kFitThreads) matern_fit_kernel(double nu, int family, double* tab) {
  constexpr int N = kDeg + 1;
  __shared__ double f[N], cheb[N], mono[N], tm[N][N];
  const int idx = blockIdx.x;
  const int e = kELo + (idx >> kSub);
  const int j = idx & ((1 << kSub) - 1);
  const int tid = threadIdx.x;
  const double I0 = tab[2 * kIntWords * kNInt + 6];
  const double scale = ldexp(1.0, e);
  const double mid = scale * (1.0 + (2.0 * j + 1.0) / (2.0 * (1 << kSub)));
  const double hw = scale / (2.0 * (1 << kSub));
  {  // node w = warp w: the first-kind Chebyshev point cos(pi (w + 1/2) / N)
    const int w = tid >> 5;
    const double tn = cospi((w + 0.5) / N);
    const double u = mid + hw * tn;
    const double v = family == kFamilyPowExp ? exp(-exp(0.5 * nu * log(u))) : quad_I_warp(u, nu) / I0;
    if ((tid & 31) == 0) f[w] = v;
  }
  if (tid == 0) {
    // Monomial coefficients of T_0..T_kDeg (exact small integers).
    for (int k = 0; k < N; ++k)
      for (int q = 0; q < N; ++q) tm[k][q] = 0.0;
    tm[0][0] = 1.0;
    tm[1][1] = 1.0;
    for (int k = 2; k < N; ++k)
      for (int q = 0; q < N; ++q)
        tm[k][q] = (q > 0 ? 2.0 * tm[k - 1][q - 1] : 0.0) - tm[k - 2][q];
  }
  __syncthreads();
  if (tid < N) {
    double s = 0.0;
    for (int q = 0; q < N; ++q) s += f[q] * cospi(tid * (q + 0.5) / N);
    cheb[tid] = (tid == 0 ? 1.0 : 2.0) * s / N;
  }
  __syncthreads();
  if (tid < N) {
    double a = 0.0;
    for (int k = N - 1; k >= 0; --k) a += cheb[k] * tm[k][tid];
    mono[tid] = a;
  }
  __syncthreads();
  if (tid == 0) write_interval(mono, reinterpret_cast<float*>(tab) + (size_t)idx * 4 * kIntWords);
}

// ------------------------------------------------------------------ likelihood table
// The likelihood kernels' table (fixtable.cuh) is wanted to 2^-60 or so of rho(0) = 1, and where rho
// is small to 2^-50 of itself, and an optimiser that moves nu builds one at every step, so it is
// built in 64-bit integers, which cost a warp 2 to 5 cycles an instruction where FP64 costs 64:
//   rho(u) = sum_k exp(-(x_k + u G_k)),  x_k = e^tau_k - nu tau_k + log Gamma(nu) - log h,
// G_k = e^-tau_k / 4, the trapezoidal rule for I(u) on one grid for all u; an interval whose
// values are small takes exp(E ln 2 - x_k - u G_k).  h = ln 2 / p, so
// that e^tau_k is a power of two times one of p numbers in [1, 2).  h <= 0.6 / sqrt(nu + 47)
// resolves the integrand's peak (width (nu^2 + u)^(-1/4)) to a relative 2^-50 up to sqrt(u) = 67,
// beyond which the polynomials' own relative error (2^-30 there) grows faster.  The integrand falls
// below e^-44 of its peak within acosh(1 + 44 / R) above the peak t* = (nu + R) / 2, R =
// sqrt(nu^2 + u): with s = tau - log t* it is exp(-R (cosh s - 1) - nu (sinh s - s)) of the peak.
// The grid ends where that has happened at the largest u, and where x_k, or 2^kELo G_k, exceeds 44.
// A fresh nu took 350 us beside the call's own work with a quadrature in FP64 of each
// interval's Chebyshev values.
struct FixSetup {
  int family, p, klo, n;
  unsigned long long lnp;    // ln 2 / p in units of 2^-64
  double nu, norm, norm_lo;  // log Gamma(nu) - log h as a pair
  float stirling;            // Stirling's log Gamma(nu), to order 1 / nu^0, less log Gamma(nu)
  double c[kNConst];         // small-u constants (matern.cuh)
  FixSetup(int family_, double nu_) : family(family_), nu(nu_) {
    p = 1;
    klo = n = 0;
    lnp = 0;
    norm = norm_lo = 0.0;
    stirling = 0.0f;
    for (double& v : c) v = 0.0;
    c[1] = nu;
    c[kConstWeakPrediction] = c[kConstWeakGradient] = std::numeric_limits<double>::infinity();
    const bool integer = nu == std::floor(nu);
    const long long kind = family == kFamilyPowExp ? 3 : integer ? (nu == 1.0 ? 1 : 2) : 0;
    std::memcpy(&c[0], &kind, sizeof(kind));
    if (family == kFamilyPowExp) return;
    if (integer) {
      c[2] = nu == 1.0 ? 0.0 : -0.25 / (nu - 1.0);
    } else {
      c[2] = 0.25 / (1.0 - nu);
      c[3] = std::tgamma(1.0 - nu);
      c[4] = 1.0 / std::tgamma(1.0 + nu);
      c[5] = 0.25 / std::tgamma(2.0 + nu);
    }
    constexpr double kLn2 = 0.693147180559945309417;
    const double R = std::sqrt(nu * nu + std::ldexp(1.0, kEHi));
    const double hi = std::max(std::log(60.0 + nu + std::min(nu, 14.0 * std::sqrt(nu))),
                               std::log(0.5 * (nu + R)) + std::acosh(1.0 + 44.0 / R));
    const double lo = std::max(std::log(nu) - 45.0 / nu - std::sqrt(120.0 / nu), -26.5);
    const double most = (kFixNodes - 3) * kLn2 / (hi - lo);
    p = (int)std::max(1.0, std::min(std::ceil(kLn2 * std::sqrt(nu + 47.0) / 0.6), std::min(std::floor(most), 1e6)));
    klo = (int)std::floor(lo * p / kLn2);
    n = std::min(kFixNodes, (int)std::ceil(hi * p / kLn2) - klo + 1);
    lnp = 0xB17217F7D1CF79ACull / p;
    const long double lg = std::lgamma((long double)nu);
    const long double v = lg - std::log(0.693147180559945309417232121458L / p);
    norm = (double)v;
    norm_lo = (double)(v - norm);
    stirling = (float)(nu * std::log((long double)nu) - nu - 0.5L * std::log(nu / 6.283185307179586477L) - lg);
  }
};

// exp(-x 2^-58) in units of 2^-63, for x < 44 2^58: x = n ln 2 + 16 z; d = 1 - e^-z by its
// Taylor polynomial of degree 9 (z < 0.0434; the terms from z^7 on in 32 bits), then four
// times 1 - d <- (1 - d)^2.  Its error is a few units.
__device__ __forceinline__ unsigned long long fix_exp(unsigned long long x) {
  const unsigned n = __umulhi((unsigned)(x >> 32), 0xB8AA3B29u) >> 25;  // log2(e) 2^31
  const unsigned long long z = ((x << 5) - n * 0x58B90BFBE8E7BCD6ull) >> 3;  // units of 2^-64
  const unsigned zh = (unsigned)(z >> 32);
  unsigned t = ~0u - __umulhi(zh, 0xFFFFFFFFu / 9);
  t = ~0u - __umulhi(__umulhi(zh, 0xFFFFFFFFu / 8), t);
  t = ~0u - __umulhi(__umulhi(zh, 0xFFFFFFFFu / 7), t);
  constexpr unsigned long long one = ~0ull;
  unsigned long long a = __umul64hi(one / 720, (unsigned long long)t << 32);
  a = one / 120 - __umul64hi(z, a);
  a = one / 24 - __umul64hi(z, a);
  a = one / 6 - __umul64hi(z, a);
  a = one / 2 - __umul64hi(z, a);
  unsigned long long d = z - __umul64hi(z, __umul64hi(z, a));
#pragma unroll
  for (int i = 0; i < 4; ++i) d = 2 * d - __umul64hi(d, d);
  return (0x8000000000000000ull - (d >> 1)) >> n;
}

// 2^-tau/ln2 at node k: 2^q times 2^(b/p), 0 <= b < p.
__device__ __forceinline__ void fix_node_power(const FixSetup& s, int k, int& q, int& b) {
  const int K = -(s.klo + k);
  q = K >= 0 ? K / s.p : -((s.p - 1 - K) / s.p);
  b = K - q * s.p;
}

// Nodes (after the constants): x_k modulo 64 in units of 2^-58, and 2^(b/p - 1) in units of 2^-63;
// then x_k as floats.
__global__ void fix_nodes_kernel(const FixSetup s, double* tab) {
  double* c = fix_const(tab);
  const int k = blockIdx.x * 32 + threadIdx.x;
  if (k < kNConst) c[k] = s.c[k];
  if (k >= s.n) return;
  int q, b;
  fix_node_power(s, k, q, b);
  const unsigned long long bl = b * s.lnp;
  const unsigned long long et = fix_exp(bl >> 6);  // e^tau = et 2^(-63 - q)
  const long long tau = -q * 0x162E42FEFA39EF3ll - (long long)(bl >> 7);  // units of 2^-57; and q ln 2's rest
  const double th = (double)tau, tl = (double)(tau - (long long)th) - 0.34375 * q;
  const double ph = s.nu * th, pl = fma(s.nu, tl, fma(s.nu, th, -ph));
  const double sc = __longlong_as_double((long long)(1023 - 63 - q) << 52);
  const double eh = (double)et, el = (double)(long long)(et - (unsigned long long)eh);
  // x = norm - nu tau + e^tau >= 0, as a pair
  Neumaier x;
  x.add(s.norm);
  x.add(-ph * 0x1p-57);
  x.add(eh * sc);
  x.add(s.norm_lo - pl * 0x1p-57 + el * sc);
  const double xt = x.s + x.c, xl = (x.s - xt) + x.c;
  const double xm = xt < 1024.0 ? xt - 64.0 * floor(xt * 0x1p-6) : 0.0;  // beyond, the float says enough
  const unsigned long long xi = __double2ull_rz(xm * 0x1p58) + (unsigned long long)__double2ll_rn(xl * 0x1p58);
  const unsigned long long mant = fix_exp(((s.p - b) * s.lnp) >> 6);
  ulonglong2* nodes = reinterpret_cast<ulonglong2*>(c + kNConst);
  nodes[k] = make_ulonglong2(xi, mant);
  reinterpret_cast<float*>(nodes + kFixNodes)[k] = (float)xt;
}

// v 2^sh modulo 2^64.
__device__ __forceinline__ unsigned long long fix_shift(unsigned long long v, int sh) {
  return sh >= 0 ? (sh < 64 ? v << sh : 0) : (sh > -64 ? v >> -sh : 0);
}

// cos(i pi / 16)
constexpr double kCos16[9] = {1.0,
                              0.98078528040323044913,
                              0.92387953251128675613,
                              0.83146961230254523708,
                              0.70710678118654752440,
                              0.55557023301960222474,
                              0.38268343236508977173,
                              0.19509032201612826785,
                              0.0};
constexpr double cos16(int i) {
  i &= 31;
  if (i > 16) i = 32 - i;
  return i <= 8 ? kCos16[i] : -kCos16[16 - i];
}
static_assert(kFixDeg == 7, "the interpolation nodes are those of degree 7");
// Interpolation at the eight Chebyshev points t_q = (1 + cos((2q + 1) pi / 16)) / 2: the
// coefficient of T_j(2t - 1) is sum_q cheb[j][q] f(t_q), that of t^k sum_j mono[j][k] (it); t_q
// in units of 2^-64.  (The product of the two matrices has entries up to 10^4 of either sign:
// FP64 sums with it lose the small coefficients.)
struct FixInterp {
  double cheb[8][8], mono[8][8];
  unsigned long long t[8];
  constexpr FixInterp() : cheb(), mono(), t() {
    mono[0][0] = 1.0;
    mono[1][0] = -1.0;
    mono[1][1] = 2.0;
    for (int j = 2; j < 8; ++j)
      for (int k = 0; k < 8; ++k)
        mono[j][k] = 2.0 * ((k > 0 ? 2.0 * mono[j - 1][k - 1] : 0.0) - mono[j - 1][k]) - mono[j - 2][k];
    for (int q = 0; q < 8; ++q) {
      for (int j = 0; j < 8; ++j) cheb[j][q] = (j ? 0.25 : 0.125) * cos16(j * (2 * q + 1));
      t[q] = (unsigned long long)((0.5 + 0.5 * cos16(2 * q + 1)) * 0x1p64);
    }
  }
};
__device__ const FixInterp kFixInterp = FixInterp();

// One CTA per kFixGroup = 8 intervals [2^e (1 + j/32), ...) of an octave, 64 values u = 2^e
// (1 + (j + t)/32).  exp(-u G) is the product of a factor for j, which takes x_k and the
// interval's E too, and one for t: 16 exponentials a node for the 64 values, and a 64-bit product each (some 30
// cycles of a warp; an exponential some 350, 1,400 in FP64).  The sum x_k + u G_k - E ln 2 is formed
// modulo 64, and beside it in floats, which say whether it exceeds 44 (and the term is left out).
// E comes from rho's estimate by Laplace's method at the interval's lower end, (nu / t*)^-nu
// exp(nu - R) sqrt(nu / R) over Stirling's error: within 2% for nu >= 0.05 where rho < 2^-7.  Then the eight values of an
// interval give its monomials: integer differences from one of them, exact, times the
// matrix above in FP64, a thread per coefficient.
constexpr int kFixGroup = 8;
constexpr int kFixThreads = 256;
constexpr int kFixChunk = 64;  // nodes at a time
constexpr int kFixMostE = 960;  // (62 + E) 2^20 is subtracted from an exponent field

__global__ void __launch_bounds__(kFixThreads) fix_table_kernel(const FixSetup s, double* tab) {
  __shared__ unsigned long long ea[kFixChunk][kFixGroup], eb[kFixChunk][8], part[4][64];
  __shared__ int scale[kFixGroup + 1];  // E; the last one the interval's before the group
  const int tid = threadIdx.x;
  const int e = kELo + (blockIdx.x * kFixGroup >> kFixSub);
  const int j0 = blockIdx.x * kFixGroup & ((1 << kFixSub) - 1);
  const float nu = (float)s.nu;
  if (tid <= kFixGroup) {
    const float u = tid < kFixGroup ? ldexpf((float)(32 + j0 + tid), e - kFixSub)
                                    : j0 > 0 ? ldexpf((float)(31 + j0), e - kFixSub) : ldexpf(63.0f, e - 1 - kFixSub);
    float bits;  // -log2 rho
    if (s.family == kFamilyPowExp) {
      bits = 1.442695041f * expf(0.5f * nu * logf(u));
    } else {
      const float R = sqrtf(fmaf(nu, nu, u)), d = u / (R + nu);  // R - nu
      bits = 1.442695041f * (d - nu * log1pf(0.5f * d / nu) - 0.5f * logf(nu / R) - s.stirling);
    }
    scale[tid] = (int)fminf(fmaxf(floorf(bits) - 6.0f, 0.0f), (float)kFixMostE);
  }
  __syncthreads();
  if (tid < kFixGroup) {
    const int E = scale[tid], before = tid ? scale[tid - 1] : scale[kFixGroup];
    const double u = ldexp((double)(32 + j0 + tid), e - kFixSub);
    if (E >= kWeakPrediction - 6 && before < kWeakPrediction - 6) fix_const(tab)[kConstWeakPrediction] = u;
    if (E >= kWeakGradient - 6 && before < kWeakGradient - 6) fix_const(tab)[kConstWeakGradient] = u;
  }
  if (s.family == kFamilyPowExp) {
    if (tid < 64) {
      const double t = (double)kFixInterp.t[tid & 7] * 0x1p-64;
      const double u = ldexp(1.0 + (j0 + (tid >> 3) + t) / (1 << kFixSub), e);
      const double x = exp(0.5 * s.nu * log(u)) - 0.693147180559945309417 * scale[tid >> 3];
      part[0][tid] = __double2ull_rn(exp(-x) * 0x1p63);
    }
  } else {
    const ulonglong2* __restrict__ nodes = reinterpret_cast<const ulonglong2*>(fix_const(tab) + kNConst);
    const float* __restrict__ xf = reinterpret_cast<const float*>(nodes + kFixNodes);
    // outside [k0, k1) a term is below e^-44
    const float eln2 = 0.6931472f * (float)scale[kFixGroup - 1], u1 = ldexpf(1.0f, e + 1);
    const int k0 = max(0, (int)(((float)e - log2f(4.0f * (44.0f + eln2))) * s.p) - s.klo - 2);
    const float R1 = sqrtf(fmaf(nu, nu, u1));
    const float top = logf(0.5f * (nu + R1)) + acoshf(1.0f + 44.0f / R1);
    const int k1 = min(s.n, max(k0, (int)(1.442695041f * top * s.p) - s.klo + 3));
    unsigned long long acc = 0;
    unsigned terms = 0;
    const int out = tid & 63, slice = tid >> 6;
    for (int kc = k0; kc < k1; kc += kFixChunk) {
      const int kk = tid & (kFixChunk - 1), k = kc + kk, r = 2 * (tid / kFixChunk);
      ulonglong2 w = make_ulonglong2(0, 0);
      float x = INFINITY, g = 0.0f;
      int q = 0, b;
      if (k < k1) {
        w = nodes[k];
        x = xf[k];
        fix_node_power(s, k, q, b);
        g = ldexpf(__ull2float_rn(w.y), e + q - 64 - kFixSub);  // 2^e G / 32 = mant 2^(e + q - 1) / 32
      }
#pragma unroll
      for (int i = 0; i < 2; ++i) {
        const int E = scale[r + i];
        const float about = fmaf(g, (float)(32 + j0 + r + i), x) - 0.6931472f * (float)E;
        unsigned long long xa = w.x + fix_shift((w.y >> 6) * (32 + j0 + r + i), e + q - 5) -
                                (unsigned long long)E * 0x2C5C85FDF473DE7ull;
        if (about < 1.0f && (long long)xa < 0) xa = 0;  // rounded below 0
        ea[kk][r + i] = about < 44.0f ? min(2 * fix_exp(xa), 0xFFFFFFFFFFFFFFFEull) : 0;
        const unsigned long long xb = fix_shift(__umul64hi(w.y, kFixInterp.t[r + i]), e + q - 11);
        eb[kk][r + i] = g < 44.0f ? fix_exp(xb) : 0;
      }
      __syncthreads();
#pragma unroll 4
      for (int i = slice * (kFixChunk / 4); i < (slice + 1) * (kFixChunk / 4); ++i) {
        const unsigned long long x1 = ea[i][out >> 3];
        acc += __umul64hi(x1, eb[i][out & 7]);
        terms += x1 != 0;
      }
      __syncthreads();
    }
    part[slice][out] = acc + terms / 2;  // the products are rounded down
  }
  __syncthreads();
  if (tid >= 64) return;
  if (s.family != kFamilyPowExp) part[0][tid] += part[1][tid] + part[2][tid] + part[3][tid];
  __syncwarp();
  const int k = tid & 7;
  const unsigned long long* __restrict__ f = part[0] + (tid & ~7);
  double a = 0.0, m = 0.0;
#pragma unroll 1
  for (int q = 0; q < 8; ++q) a = fma(kFixInterp.cheb[k][q], (double)(long long)(f[q] - f[4]) * 0x1p-63, a);
#pragma unroll 1
  for (int j = 7; j >= 0; --j) m = fma(kFixInterp.mono[j][k], __shfl_sync(0xffffffffu, a, j, 8), m);
  // S = -exponent of the largest of c1..c4
  int top = k >= 1 && k <= 4 ? (int)((__double_as_longlong(m) >> 52) & 0x7FF) : 0;
#pragma unroll
  for (int o = 4; o > 0; o >>= 1) top = max(top, __shfl_xor_sync(0xffffffffu, top, o, 8));
  const int S = top > 0 ? 1022 - top : 0;
  const double ms = m * __longlong_as_double((long long)(1023 + S) << 52);
  const int E = scale[tid >> 3];
  float* w = reinterpret_cast<float*>(tab) + (size_t)(blockIdx.x * kFixGroup + (tid >> 3)) * 4 * kFixWords;
  if (k == 0) {
    const long long c0 = (long long)((f[4] + 1) >> 1) + __double2ll_rn(m * 0x1p62);
    w[12] = __int_as_float((int)(unsigned)((unsigned long long)c0 & 0xFFFFFFFFull));
    w[13] = __int_as_float((int)(c0 >> 32));
    w[14] = ldexpf(1.0f, 36 - S);
    w[15] = ldexpf(1.0f, -S - E);
  } else if (k <= 4) {
    split_float(ms, w + 2 * (k - 1));
    if (k == 3) split_float(3.0 * ms, w + 16);
  } else {
    w[8 + k - 5] = (float)ms;
    if (k == 5) w[18] = (float)(5.0 * ms);
    if (k == 6) w[19] = (float)(6.0 * ms);
    if (k == 7) w[11] = __int_as_float((62 + E) << 20);
  }
}

// ------------------------------------------------------------------ table cache
// Tables are cached per (device, kind, family, nu), at most kMaxTables of a kind per process; a call that
// needs a table not in the cache builds it on its own stream.  Every launch that reads a
// table records a use event on its stream afterwards (cov_table_used; one event per
// stream that used the table).  When the cache is full, the least recently used table
// that no call is between look-up and launch of is rebuilt in place: the building stream
// first waits on that table's use events, so the new contents are written only after
// every earlier reader has finished.  Nothing synchronises the device or frees memory.
namespace {
struct TableUse {
  cudaStream_t stream;
  cudaEvent_t done;
};
struct TableEntry {
  int device = -1;
  bool fixed = false;  // the likelihood kernels' table
  int family = 0;
  double nu = 0.0;
  double* d_tab = nullptr;
  cudaEvent_t ready = nullptr;  // recorded after the build
  std::vector<TableUse> uses;   // recorded after each launch that read the table
  int pending = 0;              // calls between get_cov_table and cov_table_used
  unsigned long long last_use = 0;
};
std::mutex g_mu;
std::vector<TableEntry> g_tables;
unsigned long long g_clock = 0;
constexpr size_t kMaxTables = 32;
constexpr size_t kMaxUseStreams = 8;

void launch_cov_table(int family, double nu, double* tab, cudaStream_t stream, bool fixed) {
  if (fixed) {
    const FixSetup q(family, nu);
    fix_nodes_kernel<<<kFixNodes / 32, 32, 0, stream>>>(q, tab);
    fix_table_kernel<<<kFixInt / kFixGroup, kFixThreads, 0, stream>>>(q, tab);
    return;
  }
  matern_const_kernel<<<1, 32, 0, stream>>>(nu, family, tab + 2 * kIntWords * kNInt);
  matern_fit_kernel<<<kNInt, kFitThreads, 0, stream>>>(nu, family, tab);
}
}  // namespace

// Returns (building on `stream` if needed) the device table for (family, nu), the likelihood
// kernels' (fixed) or the covariance evaluator's, on the
// current device, and makes `stream` wait until it is built.  The caller launches its
// kernels and then calls cov_table_used(table, stream).
int get_cov_table(int family, double nu, cudaStream_t stream, const double** out, bool fixed) {
  int dev = 0;
  VECCHIA_CUDA_TRY(cudaGetDevice(&dev));
  std::lock_guard<std::mutex> lk(g_mu);
  for (auto& t : g_tables) {
    if (t.device == dev && t.fixed == fixed && t.family == family && t.nu == nu) {
      VECCHIA_CUDA_TRY(cudaStreamWaitEvent(stream, t.ready, 0));
      t.last_use = ++g_clock;
      t.pending += 1;
      *out = t.d_tab;
      return VECCHIA_OK;
    }
  }
  TableEntry* slot = nullptr;
  TableEntry* victim = nullptr;
  size_t of_kind = 0;
  for (auto& t : g_tables) of_kind += t.fixed == fixed;
  for (auto& t : g_tables)  // least recently used table of this device not pinned by a call
    if (t.device == dev && t.fixed == fixed && t.pending == 0 && (!victim || t.last_use < victim->last_use)) victim = &t;
  if (of_kind >= kMaxTables && victim) {
    // Rebuild in place once every earlier reader of the old contents has finished.
    for (const TableUse& u : victim->uses) {
      VECCHIA_CUDA_TRY(cudaStreamWaitEvent(stream, u.done, 0));
      cudaEventDestroy(u.done);
    }
    victim->uses.clear();
    slot = victim;
  } else {
    double* d = nullptr;
    if (cudaMalloc(&d, fixed ? kFixTableBytes : kTableBytes) != cudaSuccess) return VECCHIA_ENOMEM;
    cudaEvent_t ev;
    if (cudaEventCreateWithFlags(&ev, cudaEventDisableTiming) != cudaSuccess) {
      cudaFree(d);
      return VECCHIA_ECUDA;
    }
    g_tables.emplace_back();
    slot = &g_tables.back();
    slot->d_tab = d;
    slot->ready = ev;
  }
  launch_cov_table(family, nu, slot->d_tab, stream, fixed);
  VECCHIA_CUDA_TRY(cudaGetLastError());
  VECCHIA_CUDA_TRY(cudaEventRecord(slot->ready, stream));
  slot->device = dev;
  slot->fixed = fixed;
  slot->family = family;
  slot->nu = nu;
  slot->pending = 1;
  slot->last_use = ++g_clock;
  *out = slot->d_tab;
  return VECCHIA_OK;
}

// Records that the kernels enqueued on `stream` so far have read `tab` (from
// get_cov_table), and releases the call's pin on it.
void cov_table_used(const double* tab, cudaStream_t stream) {
  std::lock_guard<std::mutex> lk(g_mu);
  for (auto& t : g_tables) {
    if (t.d_tab != tab) continue;
    if (t.pending > 0) t.pending -= 1;
    for (TableUse& u : t.uses)
      if (u.stream == stream) {
        cudaEventRecord(u.done, stream);
        return;
      }
    if (t.uses.size() >= kMaxUseStreams) {  // fold the oldest stream's use into this one
      cudaStreamWaitEvent(stream, t.uses.front().done, 0);
      cudaEventDestroy(t.uses.front().done);
      t.uses.erase(t.uses.begin());
    }
    cudaEvent_t ev;
    if (cudaEventCreateWithFlags(&ev, cudaEventDisableTiming) != cudaSuccess) return;
    cudaEventRecord(ev, stream);
    t.uses.push_back({stream, ev});
    return;
  }
}

// Builds the likelihood kernels' Matérn table for nu into caller-provided device memory
// (kFixTableBytes, 16-byte aligned) on `stream`, without touching the cache.
int launch_matern_table(double nu, double* tab, cudaStream_t stream) {
  launch_cov_table(kFamilyMatern, nu, tab, stream, true);
  VECCHIA_CUDA_TRY(cudaGetLastError());
  return VECCHIA_OK;
}

// ------------------------------------------------------------------ vecchia_matern
// C(d) and dC/dbeta from the evaluators' table.  u = (d * inv_len)^2 with the
// family's length scale (beta for the Matérn, beta^(1/alpha) for the power
// exponential), and dC/dbeta = dcoef h(u), dcoef = -2 sigma2 / (beta a), a = 1 or alpha.
__global__ void matern_eval_kernel(const double* __restrict__ d, int64_t count, double sigma2,
                                   double beta, int family, const double* __restrict__ tab,
                                   double* __restrict__ c, double* __restrict__ dc) {
  const MaternConst mc = load_matern_const(tab);
  const double inv_len = family == kFamilyPowExp ? exp(-log(beta) / mc.nu) : 1.0 / beta;
  const double dcoef = -2.0 * sigma2 / (beta * (family == kFamilyPowExp ? mc.nu : 1.0));
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < count;
       i += (int64_t)gridDim.x * blockDim.x) {
    const double x = d[i] * inv_len;
    const double u = x * x;
    double rho, h;
    rho_eval<true>(u, tab, mc, rho, h);
    c[i] = sigma2 * rho;
    if (dc) dc[i] = dcoef * h;
  }
}

bool theta_ok(const double* th) {
  if (!th) return false;
  for (int k = 0; k < 4; ++k)
    if (!std::isfinite(th[k])) return false;
  return th[0] > 0.0 && th[1] > 0.0 && th[2] > 0.0 && th[3] >= 0.0;
}

// theta valid for the family: the power exponential needs 0 < alpha <= 2.
bool theta_ok_family(const double* th, int family) {
  return theta_ok(th) && (family != kFamilyPowExp || th[2] <= 2.0);
}

static int covariance(int family, const double* d_dev, int64_t count, const double* theta, double* c_dev,
                      double* dcdbeta_dev, cudaStream_t s) {
  if (count < 0 || (count > 0 && (!d_dev || !c_dev)) || !theta_ok_family(theta, family)) return VECCHIA_EINVAL;
  if (count == 0) return VECCHIA_OK;
  const double* tab = nullptr;
  int rc = get_cov_table(family, theta[2], s, &tab, false);
  if (rc) return rc;
  const int64_t blocks = std::min<int64_t>((count + 255) / 256, 4096);
  matern_eval_kernel<<<(int)blocks, 256, 0, s>>>(d_dev, count, theta[0], theta[1], family, tab, c_dev,
                                                 dcdbeta_dev);
  cov_table_used(tab, s);
  VECCHIA_CUDA_TRY(cudaGetLastError());
  return VECCHIA_OK;
}

}  // namespace vecchia

extern "C" int vecchia_matern(const double* d_dev, int64_t count, const double theta[4], double* c_dev,
                              double* dcdbeta_dev, void* stream) {
  return vecchia::covariance(vecchia::kFamilyMatern, d_dev, count, theta, c_dev, dcdbeta_dev,
                             (cudaStream_t)stream);
}

extern "C" int vecchia_covariance(int kernel, const double* d_dev, int64_t count, const double theta[4],
                                  double* c_dev, double* dcdbeta_dev, void* stream) {
  if (kernel != VECCHIA_KERNEL_MATERN && kernel != VECCHIA_KERNEL_POWEXP) return VECCHIA_EINVAL;
  return vecchia::covariance(kernel, d_dev, count, theta, c_dev, dcdbeta_dev, (cudaStream_t)stream);
}
