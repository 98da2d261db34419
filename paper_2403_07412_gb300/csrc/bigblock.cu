// Large conditioning sets (m > VECCHIA_MAX_M_WARP): one CTA per location.
//
// The paper runs m up to 150 (Sec. VI-D).  A 151-row bordered block is 93 KB, too much for
// a warp's share of shared memory, so here a CTA of two to eight warps owns one location at a
// time and eliminates its block in fixed point, as the full-warp kernels do (mmapanel.cuh):
// panels of eight columns, updates on the tensor cores, the trailing 2x2 corner s_i / sigma2
// and y_i - mu_i.  (In FP64, four columns a CTA-wide pass, the FP64 pipe was its bound: n =
// 50,000, m = 120 took 36.2 ms with the gradient.)  What bounds it now is latency: a location's
// phases, and the panels' serial columns most of all, leave a warp issuing one instruction in
// four cycles, and shared memory holds three locations an SM at m = 120, two at 150.  The
// (row, column) of a pair index is decoded arithmetically (a triangular-number inverse)
// instead of from schedule tables, to keep that many.  The adjoint's two backward solves run
// on the first two warps, one each, on vectors in shared memory; everything else is spread
// over all threads.
#include <algorithm>
#include <cmath>
#include <cstdlib>
#include <mutex>
#include <vector>

#include "block.cuh"
#include "common.cuh"
#include "matern.cuh"
#include "mmapanel.cuh"

namespace vecchia {

constexpr int kCtaThreadsMax = 256;  // two to eight warps (big_config)

struct BigArgs {
  const double* __restrict__ xy;
  const double* __restrict__ yf;
  const int32_t* __restrict__ nbr;
  const int32_t* __restrict__ self;
  const double* __restrict__ tab;
  int64_t n;
  int m;
  int family;
  double sigma2, beta, nu, tau2;
  double* partial;  // [gridDim.x][4]
  double* terms;
  unsigned long long* errloc;
  const double* __restrict__ xyz;  // n x 3 unit vectors (sphere plans)
  int metric;                      // 0 plane, 1 sphere
  double radius;
  int64_t i0, i1;                  // ordered locations [i0, i1) are evaluated
};

// Largest w with w(w+1)/2 <= e (e < 2^24).
__device__ __forceinline__ int tri_root(int e) {
  int w = (int)((sqrtf(8.0f * (float)e + 1.0f) - 1.0f) * 0.5f);
  if ((w + 1) * (w + 2) / 2 <= e) ++w;
  if (w * (w + 1) / 2 > e) --w;
  return w;
}

__device__ __forceinline__ double block_sum(double v, double* red) {
  v = warp_sum(v);
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  __syncthreads();
  if (lane == 0) red[wid] = v;
  __syncthreads();
  double s = 0.0;
  for (int k = 0; k < (int)(blockDim.x >> 5); ++k) s += red[k];
  return s;
}

// Cholesky over the neighbour columns.  A panel's own eight rows are a serial chain of eight
// columns, and warp 0 runs ahead with it: it takes the sixteen rows below a panel through the
// panel's columns (panel_row, a row per lane), updates them for the next panel and factors
// that panel's rows, while the other warps take the rows further down through the first
// panel's columns and, once warp 0's sixteen rows are in (barrier 1), update them.  The data are the other
// warps' work too, a panel behind: warp 1 solves for the first panel's z (barrier 2), each row's datum goes
// with the row, and warp 1 takes the sixteen rows' from their digits.  (On warp 0, in the panels' columns:
// n = 20k, m = 130 16.0 ms with the gradient and 12.3 without; so 15.0 and 11.6.)
template <bool GRAD>
__device__ __forceinline__ bool cta_eliminate(int K, long long* __restrict__ A, float2* __restrict__ RJ, int4* __restrict__ piv,
                                              double* __restrict__ zs, int f, long long* corner, int tid, int NTH) {
  const int lane = tid & 31, wid = tid >> 5;
  int over = 0, c1 = 0;
  // piv holds those of this panel and the next
#pragma unroll 1
  for (int c0 = -kPanelCols; c0 + kPanelCols < K; c0 += kPanelCols) {
    c1 = c0 + kPanelCols;
    const int pe = min(c1 + kPanelCols, K);
    const int4* __restrict__ pv = piv + (c0 & kPanelCols);
    if (wid == 0) {
      if (c0 >= 0) {
        if (lane < 16 && c1 + lane < K) panel_row<false>(K, A, pv, zs, c0, f, c1 + lane, over);
        __threadfence_block();
        asm volatile("bar.arrive 1, %0;" ::"r"(NTH) : "memory");
        __syncwarp();
        update_tile<true>(K, A, c1, c1, pe, f, lane);
        __syncwarp();
      }
      long long cr = 0;
      if (!panel_columns<GRAD, true>(K, A, RJ, piv + (c1 & kPanelCols), c1, f, cr, lane)) over = 1;
      if (pe == K && lane == 0) *corner = cr;
    } else if (c0 >= 0) {
      if (wid == 1) panel_solve<GRAD>(K, A, RJ, pv, zs, c0, f, lane);
      asm volatile("bar.sync 2, %0;" ::"r"(NTH - 32) : "memory");
#pragma unroll 1
      for (int r = c1 + 16 + tid - 32; r < K; r += NTH - 32) panel_row<true>(K, A, pv, zs, c0, f, r, over);
      asm volatile("bar.sync 1, %0;" ::"r"(NTH) : "memory");
      if (wid == 1 && lane < 16 && c1 + lane < K) panel_row_data(K, A, zs, c0, c1 + lane);
#pragma unroll 1
      for (int rt = c1 + 16 * wid; rt < K; rt += (NTH - 32) / 2) update_tile<true>(K, A, rt, c1, pe, f, lane);
    }
    __syncthreads();
  }
  if (wid == 1) panel_solve<GRAD>(K, A, RJ, piv + (c1 & kPanelCols), zs, c1, f, lane);
  return __syncthreads_or(over) == 0;
}

// B columns j..j+B-1 of the bordered L D L^T, CTA-wide.  Each column in turn is scaled by
// its pivot's reciprocal (its unscaled entries kept in TVs[q]) and applied to the later
// columns of the group; then one pass over the remaining prefix [1, o_{j+B-1}) applies
// all B columns to each slot in column order, fma(-L_q T_q, .) for q = 0..B-1.  Every
// slot sees the same roundings in the same order as with single-column steps, while the
// trailing matrix is read and written once per B columns.  Returns false (uniformly over
// the CTA) at a pivot outside rcp_fixed's domain or that counts as zero.
template <int B>
__device__ __forceinline__ bool cta_columns(double* A, double* const* TVs, int K, int j, int tid, int NTH) {
  int o[B];
#pragma unroll
  for (int q = 0; q < B; ++q) o[q] = tri_off(K, j + q);
#pragma unroll
  for (int q = 0; q < B; ++q) {
    const double d = A[o[q]];
    if (!pivot_in_range(d) || zero_pivot(d)) return false;  // every thread reads the same pivot
    const double inv = rcp_fixed(d);
    double* T = TVs[q];
    for (int r = j + q + 1 + tid; r <= K; r += NTH) {
      const double tv = A[o[q] + r - j - q];
      T[r] = tv;
      A[o[q] + r - j - q] = tv * inv;
    }
    __syncthreads();
    if (q + 1 < B) {
      const double* Lq = A + o[q] - j - q;
#pragma unroll
      for (int p = q + 1; p < B; ++p) {
        const double tp = T[j + p];
        for (int r = j + p + tid; r <= K; r += NTH) {
          const int e = o[p] + r - j - p;
          A[e] = fma(-Lq[r], tp, A[e]);
        }
      }
      __syncthreads();
    }
  }
  const double* L[B];
#pragma unroll
  for (int q = 0; q < B; ++q) L[q] = A + o[q] - j - q;
  constexpr int U = 8 / B;
  const int end = o[B - 1];
  const int nfull = (end - 1) / (NTH * U);
  const int tail0 = 1 + NTH * U * nfull;
  for (int bt = 0; bt < nfull; ++bt) {
    const int base = 1 + tid + NTH * U * bt;
    double av[U];
    int rr[U], cc[U];
#pragma unroll
    for (int k = 0; k < U; ++k) {
      const int e = base + NTH * k;
      const int w = tri_root(e);
      cc[k] = K - w;
      rr[k] = cc[k] + (e - w * (w + 1) / 2);
      av[k] = A[e];
    }
#pragma unroll
    for (int q = 0; q < B; ++q)
#pragma unroll
      for (int k = 0; k < U; ++k) av[k] = fma(-L[q][rr[k]], TVs[q][cc[k]], av[k]);
#pragma unroll
    for (int k = 0; k < U; ++k) A[base + NTH * k] = av[k];
  }
  for (int e = tail0 + tid; e < end; e += NTH) {
    const int w = tri_root(e);
    const int c = K - w, r = c + (e - w * (w + 1) / 2);
    double a = A[e];
#pragma unroll
    for (int q = 0; q < B; ++q) a = fma(-L[q][r], TVs[q][c], a);
    A[e] = a;
  }
  __syncthreads();
  return true;
}

// The block in FP64 (mmapanel.cuh says which blocks): assembly, L D L^T four columns at a time, then two, then
// one, and (GRAD) the factor as float pairs, as panels_to_pairs leaves it.  Returns whether the neighbours'
// block is positive definite; s_i / sigma2 and y_i - mu_i are in A[1] and A[2].  The data are in the border
// row; TV and the vectors before and after it are column buffers.  (A function of its own, for the registers
// of its caller.)
template <bool GRAD, bool SPHERE>
static __device__ __noinline__ bool cta_fp64_block(int K, int mi, double* A, const float2* CX, const float2* CY,
                                                   const float2* CZ, double* TV, int stride, double gamma1, float2 k2,
                                                   double k2d, const double* __restrict__ tab) {
  const int m = K - 1, NP = K * (K - 1) / 2, tid = threadIdx.x, NTH = blockDim.x;
  const MaternConst mc = matern_const_at(fix_const(tab));
  FieldView F;
  F.k2 = k2;
  F.k2d = k2d;
  for (int c = tid; c < K; c += NTH) {
    const int o = tri_off(K, c);
    A[o] = (c >= mi && c < m) ? 1.0 : gamma1;
  }
#pragma unroll 1
  for (int q = tid; q < NP; q += NTH) {
    const int v = tri_root(q), c = K - 2 - v, r = c + 1 + (q - v * (v + 1) / 2);
    float uh, ul;
    pair_u<SPHERE>(F, CX, CY, CZ, r, c, uh, ul);
    A[tri_off(K, c) + r - c] = c < mi && (r < mi || r == m) ? fixed_to_double(rho_fixed62(uh, ul, tab, mc)) : 0.0;
  }
  __syncthreads();
  double* TVs[4] = {TV, TV - stride, TV + stride, TV + 2 * stride};
  bool ok = true;
  int j = 0;
  for (; ok && j + 4 <= mi; j += 4) ok = cta_columns<4>(A, TVs, K, j, tid, NTH);  // (pads' columns are the identity's)
  for (; ok && j + 2 <= mi; j += 2) ok = cta_columns<2>(A, TVs, K, j, tid, NTH);
  if (ok && j + 1 <= mi) ok = cta_columns<1>(A, TVs, K, j, tid, NTH);
  if (GRAD) {
    for (int e = 3 + tid; e < (K + 1) * (K + 2) / 2; e += NTH) {
      const int w = tri_root(e);
      if (e > w * (w + 1) / 2) reinterpret_cast<float2*>(A)[e] = d2f_trunc(A[e]);
    }
    __syncthreads();
  }
  return ok;
}

template <bool GRAD, bool SPHERE>
__global__ void __launch_bounds__(kCtaThreadsMax) vecchia_big_kernel(const BigArgs a) {
  asm volatile("griddepcontrol.launch_dependents;");  // the reduction of the records
  extern __shared__ __align__(16) unsigned char smem[];
  const int m = a.m, K = m + 1;
  const int NTd = (K + 1) * (K + 2) / 2, NP = K * (K - 1) / 2;
  double* A = reinterpret_cast<double*>(smem);
  constexpr bool sphere = SPHERE;
  float2* CX = reinterpret_cast<float2*>(A + align_up(NTd, 2));
  float2* CY = CX + align_up(K + 1, 2);
  float2* CZ = sphere ? CY + align_up(K + 1, 2) : CY;
  double* YV = reinterpret_cast<double*>(CY + (sphere ? 2 : 1) * align_up(K + 1, 2));
  double* TV = YV + align_up(K + 1, 2);
  double* WH = TV + align_up(K + 1, 2);
  double* GV = WH + align_up(K + 1, 2);
  double* red = GV + align_up(K + 1, 2);
  long long* corner = reinterpret_cast<long long*>(red + 32);
  double* coef = reinterpret_cast<double*>(corner + 2);
  int4* piv = reinterpret_cast<int4*>(coef + 4);
  double* zs = reinterpret_cast<double*>(piv + 2 * kPanelCols);
  long long* AF = reinterpret_cast<long long*>(A);
  float2* WHf = reinterpret_cast<float2*>(WH);  // w^ and g as float pairs for the beta sums
  float2* GVf = reinterpret_cast<float2*>(GV);
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  const int NTH = blockDim.x;
  const MaternConst mc = matern_const_at(fix_const(a.tab));
  ThetaConst tc;
  tc.set(a.sigma2, a.beta, a.tau2, a.family, a.nu);
  tc.weak_u = (float)fix_const(a.tab)[kConstWeakGradient];
  const int f = panel_shift(tc.gamma1);
  const double2* __restrict__ xy2 = reinterpret_cast<const double2*>(a.xy);
  FieldView F;  // the distance fields pair_u reads
  F.sphere = sphere;
  F.xyz = a.xyz;
  if constexpr (SPHERE) {
    const double k = 2.0 * a.radius * tc.inv_len;
    F.k2d = k * k;
    F.k2 = d2f_pair(F.k2d);
  }
  Accum acc;
  for (int64_t i = a.i0 + blockIdx.x; i < a.i1; i += gridDim.x) {
    const int mi = i < m ? (int)i : m;
    const int32_t* __restrict__ row = a.nbr + i * m;
    bool bad_idx = false;  // bounds-checked builds only: an index outside [0, n)
    int js = a.self[i];
    if (kChecked && (unsigned long long)(int64_t)js >= (unsigned long long)a.n) {
      bad_idx = true;
      js = 0;
    }
    const double2 ps = xy2[js];
    // ---- gather: centred, 1/beta-scaled coordinates as float pairs, and data
#pragma unroll 1
    for (int p = tid; p < m; p += NTH) {
        double xv = 0.0, yv = 0.0, zv = 0.0, fv = 0.0;
        if (p < mi) {
          int j = row[p];
          if (kChecked && (unsigned long long)(int64_t)j >= (unsigned long long)a.n) {
            bad_idx = true;
            j = 0;
          }
          if constexpr (SPHERE) {
            xv = a.xyz[3 * j] - a.xyz[3 * js];
            yv = a.xyz[3 * j + 1] - a.xyz[3 * js + 1];
            zv = a.xyz[3 * j + 2] - a.xyz[3 * js + 2];
          } else {
            const double2 q = xy2[j];
            xv = (q.x - ps.x) * tc.inv_len;
            yv = (q.y - ps.y) * tc.inv_len;
          }
          fv = a.yf[j];
        }
        YV[p] = fv;
        CX[p] = d2f_pair(xv);
        CY[p] = d2f_pair(yv);
        if constexpr (SPHERE) CZ[p] = d2f_pair(zv);
    }
    if (tid == 0) {
      CX[m] = make_float2(0.0f, 0.0f);
      CY[m] = make_float2(0.0f, 0.0f);
      if constexpr (SPHERE) CZ[m] = make_float2(0.0f, 0.0f);
      YV[m] = a.yf[js];
    }
    if (kChecked) bad_idx = __syncthreads_or(bad_idx) != 0;
    __syncthreads();
    // whether few of the data are large (each warp for itself)
    int top = lane == 0 ? (int)exponent_field(YV[m]) : 0, count = 0;  // twice the large ones, less all but the zeros
    for (int p = lane; p < mi; p += 32) top = max(top, (int)exponent_field(YV[p]));
    top = __reduce_max_sync(0xffffffffu, top);
    for (int p = lane; p <= m; p += 32) {
      const int e = p < mi || p == m ? (int)exponent_field(YV[p]) : 0;
      if (e > 0) count += large_datum(e, top) ? 1 : -1;
    }
    bool exact = f > kMostShift || __reduce_add_sync(0xffffffffu, count) < 0;  // the block goes to cta_fp64_block
    if (GRAD) {
      unsigned near = 0x7F800000u;  // u of the nearest neighbour
      for (int p = lane; p < mi; p += 32) near = min(near, __float_as_uint(near_u<SPHERE>(F, CX, CY, CZ, p)));
      near = __reduce_min_sync(0xffffffffu, near);
      exact = exact || (__uint_as_float(near) >= tc.weak_u && mi > 0);
    }
    // ---- assemble, in fixed point (mmapanel.cuh)
    for (int c = tid; c < K; c += NTH) {
      const int o = tri_off(K, c);
      AF[o] = fixed_from_double(tc.gamma1, 60 - 2 * f);  // a pad's is any positive number
      A[o + K - c] = YV[c];
    }
    if (tid == 0) AF[0] = 0;
    for (int q0 = exact ? NP : tid; q0 < NP; q0 += 2 * NTH) {
      const int q1 = q0 + NTH;
      const bool has1 = q1 < NP;
      const int v0 = tri_root(q0), v1 = tri_root(has1 ? q1 : q0);
      const int c0 = K - 2 - v0, r0 = c0 + 1 + (q0 - v0 * (v0 + 1) / 2);
      const int qq1 = has1 ? q1 : q0;
      const int c1 = K - 2 - v1, r1 = c1 + 1 + (qq1 - v1 * (v1 + 1) / 2);
      const bool ok0 = c0 < mi && (r0 < mi || r0 == m);
      const bool ok1 = has1 && c1 < mi && (r1 < mi || r1 == m);
      float u0h, u0l, u1h, u1l;
      pair_u<SPHERE>(F, CX, CY, CZ, r0, c0, u0h, u0l);
      pair_u<SPHERE>(F, CX, CY, CZ, r1, c1, u1h, u1l);
      FixRho val0, val1;
      rho_fixed62(u0h, u0l, u1h, u1l, a.tab, mc, val0, val1);
      AF[tri_off(K, c0) + r0 - c0] = ok0 ? fixed60(val0) : 0LL;
      if (has1) AF[tri_off(K, c1) + r1 - c1] = ok1 ? fixed60(val1) : 0LL;
    }
    __syncthreads();
    const bool ok = exact ? cta_fp64_block<GRAD, SPHERE>(K, mi, A, CX, CY, CZ, TV, align_up(K + 1, 2), tc.gamma1, F.k2, F.k2d, a.tab)
                          : cta_eliminate<GRAD>(K, AF, reinterpret_cast<float2*>(TV), piv, zs, f, corner, tid, NTH);
    // ---- the term, on warp 0 (FP64)
    const double nan = __longlong_as_double(0x7FF8000000000000LL);
    if (wid == 0) {
      double st = A[1];
      st = exact ? (zero_pivot(st) ? 0.0 : st) : *corner > kSmallestPivot ? mul_pow2((double)*corner, 2 * f - 60) : 0.0;
      const double rr = A[2];
      const bool pd = ok && positive_finite(st);  // a non-finite rr with pd: non-finite data
      const bool good = pd && finite_bits(rr) && !bad_idx;
      const double s = tc.sigma2 * st;
      const double inv_s = rcp_newton(s);
      const double q = rr * rr * inv_s;
      if (good) {
        acc.Q.add(q);
        acc.mul_s(s);
        acc.count += 1;
      } else {
        acc.Q.add(nan);
        if (tid == 0) atomicMin(a.errloc, err_code(i, bad_idx ? kErrIndex : (pd ? kErrData : kErrNotPD)));
      }
      const double rs = rr * inv_s;
      if (a.terms && tid == 0) {
        const double li = good ? -0.5 * q - 0.5 * log(s) - 0.91893853320467274178 : nan;
        a.terms[GRAD ? 4 * i : i] = li;
      }
      if (GRAD && tid == 0) {
        coef[0] = 0.5 * (rs * rs - inv_s);
        coef[1] = rs * tc.inv_sigma2;
        coef[2] = good ? 0.5 * (rr * rs - 1.0) : nan;
      }
    }
    __syncthreads();
    if (!GRAD) continue;
    // ---- adjoint: the two backward solves on warps 0 (w) and 1 (alpha~) at once, then
    // the pair pass on all threads
    const double cb = coef[0], rsa = coef[1], sS = coef[2];
    const bool good = finite_bits(sS);
    if (!exact) panels_to_pairs(K, AF, reinterpret_cast<const float2*>(TV), tid, NTH);
    __syncthreads();
    const float2* __restrict__ L = reinterpret_cast<const float2*>(A);  // the unit factor
    double pT = 0.0;
    if (wid < 2 && good) {
      // Double-float solves on the FP32 pipe, as in the warp kernels: each step of the
      // serial chain would otherwise wait behind the other CTAs' FP64 work.  Warp 0
      // solves with row m of the factor (w) in TV, warp 1 with row K (alpha~) in YV (both
      // free after the elimination).  The vectors live in shared memory, not registers:
      // held in registers they took the kernel from 80 to 122 registers per thread and
      // one CTA per SM of occupancy at m = 90 and 120.
      float2* V = reinterpret_cast<float2*>(wid == 0 ? TV : YV);
      const int row = wid == 0 ? m : K;
      for (int c = lane; c < K - 1; c += 32) V[c] = L[tri_off(K, c) + row - c];
      __syncwarp();
      for (int c = K - 2; c >= 1; --c) {
        const float2 vc = V[c];  // final since the previous step (__syncwarp below)
        for (int cc = lane; cc < c; cc += 32) {
          const float2 l = L[tri_off(K, cc) + c - cc];
          float2 v = V[cc];
          df_fms(v.x, v.y, l, vc);
          V[cc] = v;
        }
        __syncwarp();
      }
    }
    __syncthreads();
    if (wid == 0 && good) {
      const float2* Vw = reinterpret_cast<const float2*>(TV);
      const float2* Va = reinterpret_cast<const float2*>(YV);
      for (int c = lane; c < K - 1; c += 32) {
        const double w = f2d_scaled(Vw[c].x, 0) + f2d_scaled(Vw[c].y, 0);
        const double al = f2d_scaled(Va[c].x, 0) + f2d_scaled(Va[c].y, 0);
        const double wh = -w, gv = fma(rsa, al, cb * wh);
        WHf[c] = d2f_pair(wh);
        GVf[c] = d2f_pair(gv);
        pT = fma(wh, gv, pT);
      }
      if (lane == 0) {
        WHf[m] = make_float2(1.0f, 0.0f);
        GVf[m] = d2f_pair(cb);
        pT += cb;
      }
    }
    __syncthreads();
    float pbh = 0.0f, pbl = 0.0f;
    if (good) {  // one pair per iteration (two took more registers, no less time)
      for (int q0 = tid; q0 < NP; q0 += NTH) {
        const int v0 = tri_root(q0);
        const int c0 = K - 2 - v0, r0 = c0 + 1 + (q0 - v0 * (v0 + 1) / 2);
        float u0h, u0l, h0h, h0l;
        pair_u<SPHERE>(F, CX, CY, CZ, r0, c0, u0h, u0l);
        h_fixed<true>(u0h, u0l, a.tab, mc, h0h, h0l);
        beta_pair_add(WHf[r0], WHf[c0], GVf[r0], GVf[c0], h0h, h0l, pbh, pbl);
      }
    }
    const double pB = f2d_scaled(pbh, 0) + f2d_scaled(pbl, 0);
    if (a.terms) {
      const double tB = block_sum(pB, red), tT = block_sum(pT, red);
      if (tid == 0) {
        double* o = a.terms + i * 4;
        o[1] = good ? (sS - tc.tau2 * tT) * tc.inv_sigma2 : nan;
        o[2] = good ? tc.dbeta_coef * tB : nan;
        o[3] = good ? tT : nan;
      }
    }
    if (wid == 0) acc.S += sS;  // a failed term's is NaN, and so every output
    acc.B += good ? pB : nan;
    acc.T += good ? pT : nan;
    __syncthreads();
  }
  const double B = block_sum(acc.B, red);
  const double T = block_sum(acc.T, red);
  if (tid == 0) {
    double* o = a.partial + (int64_t)blockIdx.x * 4;
    o[0] = acc.loglik();
    o[1] = acc.S;
    o[2] = B;
    o[3] = T;
  }
}

// Shared memory of the CTA kernel for block size K.
int big_smem_bytes(int K, bool sphere) {
  const int NTd = (K + 1) * (K + 2) / 2;
  return 8 * (align_up(NTd, 2) + (sphere ? 7 : 6) * align_up(K + 1, 2) + 32 + 6 + 5 * kPanelCols);
}

// CTA size: the W warps with the largest c W / (W + 2), c the CTAs of that size resident on an SM
// (at most the ones `count` > 0 locations give it): a location's serial part, the panels' own
// columns on warp 0, is worth about two warps' shares of the rest.  Ties go to the larger W.  n =
// 20,000 with the gradient, ms: m = 64 (8 CTAs of 2 warps, 5 of 3, 4 of 4) 2.86, 3.33, 3.47; m =
// 90 (6, 5, 4) 6.02, 5.49, 5.58; m = 120 (3 of any up to 5 warps, 2 of 6) 14.4, 11.7, 10.9, 10.6
// and 13.1; m = 150 (2) 27.4, 22.4, 20.2, 19.9, 18.4.  VECCHIA_CTA_THREADS, a multiple of 32 from
// 64 to 256, forces one.
struct BigShape {
  int dev, K, grad, sphere;
  int per_sm[kCtaThreadsMax / 32 + 1];
};
std::mutex g_big_mu;
std::vector<BigShape> g_big_shapes;  // the occupancy queries cost tens of microseconds

int big_config(int K, bool grad, int* blocks, int* threads, int* smem, bool sphere, int64_t count) {
  int dev = 0, sms = 0;
  VECCHIA_CUDA_TRY(cudaGetDevice(&dev));
  VECCHIA_CUDA_TRY(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
  *smem = big_smem_bytes(K, sphere);
  auto kern = grad ? (sphere ? vecchia_big_kernel<true, true> : vecchia_big_kernel<true, false>)
                   : (sphere ? vecchia_big_kernel<false, true> : vecchia_big_kernel<false, false>);
  VECCHIA_CUDA_TRY(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, *smem));
  BigShape shape{dev, K, (int)grad, (int)sphere, {}};
  {
    std::lock_guard<std::mutex> lk(g_big_mu);
    bool known = false;
    for (const BigShape& e : g_big_shapes)
      if (e.dev == dev && e.K == K && e.grad == (int)grad && e.sphere == (int)sphere) {
        shape = e;
        known = true;
        break;
      }
    if (!known) {
      for (int w = 2; w <= kCtaThreadsMax / 32; ++w)
        VECCHIA_CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&shape.per_sm[w], kern, 32 * w, *smem));
      g_big_shapes.push_back(shape);
    }
  }
  const char* e = getenv("VECCHIA_CTA_THREADS");
  const int forced = e ? atoi(e) : 0;
  const int64_t share = count > 0 ? (count + sms - 1) / sms : shape.per_sm[2];
  int W = 0;
  double best = 0.0;
  for (int w = 2; w <= kCtaThreadsMax / 32; ++w) {
    if (forced % 32 == 0 && forced >= 64 && forced <= kCtaThreadsMax && 32 * w != forced) continue;
    const double score = (double)std::min<int64_t>(shape.per_sm[w], share) * w / (w + 2);
    if (shape.per_sm[w] > 0 && score >= best) {
      best = score;
      W = w;
    }
  }
  if (W == 0) return VECCHIA_EINVAL;
  *blocks = shape.per_sm[W] * sms;
  if (count > 0) *blocks = (int)std::min<int64_t>(*blocks, count);
  *threads = 32 * W;
  return VECCHIA_OK;
}

void launch_big(bool grad, int blocks, int threads, int smem, const BigArgs& a, cudaStream_t s) {
  const bool sph = a.metric == 1;
  if (grad) {
    if (sph) vecchia_big_kernel<true, true><<<blocks, threads, smem, s>>>(a);
    else vecchia_big_kernel<true, false><<<blocks, threads, smem, s>>>(a);
  } else {
    if (sph) vecchia_big_kernel<false, true><<<blocks, threads, smem, s>>>(a);
    else vecchia_big_kernel<false, false><<<blocks, threads, smem, s>>>(a);
  }
}

}  // namespace vecchia
