// Many independent (field, theta) log-likelihood evaluations in a few persistent launches.
//
// The paper batches only over the locations of one field (Sec. V-B).  Here the unit of
// work is an item = (field, theta, tile of consecutive ordered locations); a persistent
// grid of warps takes items from a global counter, evaluates each location with the same
// per-location code as the single-field kernel (block.cuh), and writes one partial-sum
// record per item.  Fields may differ in n and m: the fields whose blocks run the same way
// (lanes per location, FP64 or fixed point) form a class, and each class is one launch of its own
// kernel, with a shared-memory layout sized for its largest block.  (One kernel for all of
// them held every variant's code and the largest variant's registers and area: n = 20,000, m
// = 60 / 30 / 10 took 102 / 30.0 / 6.5 ns a location.)  Each theta picks its covariance
// table by smoothness nu among the tables prepared with vecchia_batched_prepare.  Items are
// laid out so the most expensive fields (largest m) are handed out first.  A last kernel
// reduces each (field, theta)'s records in item order, so results do not depend on
// scheduling.  The launch sequence (two memsets, a kernel per class and the last one)
// allocates nothing and never waits on the host, so it can be captured in a CUDA graph once
// the work layout has been cached by a first call.
#include <algorithm>
#include <cmath>
#include <cstring>
#include <mutex>
#include <vector>

#include "block.cuh"
#include "common.cuh"
#include "matern.cuh"

namespace vecchia {

int launch_matern_table(double nu, double* tab, cudaStream_t stream);
bool theta_ok(const double* th);
int lanes_for(int K, bool grad, int64_t count);

// Locations an item gives each group of a warp: up to kMostSteps, fewer where the class has
// not kItemsPerWarp such items for each resident warp, more where it has kManyItems times as many, so
// that a class's records (32 bytes an item) stay at some kManyItems kItemsPerWarp for each resident warp,
// 4 MB or so, however large the batch.  A full-warp location of m = 60 takes
// a warp some 75 us: eight make an item long enough to hide its hand-out (an atomic, the
// field search, the constants: a few us).  Items of 256 locations took 19 ms each there, a
// batch of two fields of n = 20,000, two thetas, 44 ms where its work takes 7; with eight for
// every size, two fields of n = 700 took 1.40 ms, and 64 fields under 32 thetas kept 413 MB of records.
constexpr int kMostSteps = 8;
constexpr int kItemsPerWarp = 4;
constexpr int kManyItems = 16;
constexpr int kMaxNu = 8;        // prepared smoothness values
constexpr int kMaxDistinctK = 4; // distinct block sizes per batch, and so most classes

struct FieldDesc {
  const double2* xy;
  const double* yf;
  const int32_t* nbr;
  const int32_t* self;
  int64_t n;
  int32_t m;
  int32_t kidx;       // index of this field's block size in its class's K list
  int32_t orig;       // position in the caller's field list
  int32_t tile;       // locations per item
  int32_t tiles;      // ceil(n / tile)
  int64_t item_base;  // first item of this field
};

struct BatchArgs {
  const FieldDesc* fields;
  int first_field, last_field;  // the class's
  int ntheta;
  const double* thetas;  // [nfields][ntheta][4], caller order
  const double* nus;     // [kMaxNu]
  const double* const* tabs;
  int nnu;
  bool regather;                    // 8 lanes, gradient: see WarpArea
  int64_t first_item, total_items;  // the class's
  unsigned long long* counter;
  unsigned long long* errloc;
  double* partial;  // [total_items][4]
  int nk;
  int kval[kMaxDistinctK];
  int sched_off[kMaxDistinctK];
  int pairs_off[kMaxDistinctK];
  int area_off;
  int area_doubles;
};

// One item with G lanes per location: the 32/G groups of the warp take the tile's
// locations in turn.
template <bool GRAD, int G, bool FIXED>
__device__ __forceinline__ void run_item(const FieldDesc& fd, int64_t tile, const unsigned char* smem,
                                         const BatchArgs& a, double* base, const double* tab,
                                         const MaternConst& mc, const ThetaConst& tc, double* out, int lane) {
  constexpr int NL = 32 / G;
  const int grp = lane / G, sub = lane % G;
  FieldView F;
  F.xy = fd.xy;
  F.yf = fd.yf;
  F.nbr = fd.nbr;
  F.self = fd.self;
  F.n = fd.n;
  F.m = fd.m;
  F.nidx = fd.n;
  const int K = fd.m + 1;
  const SchedSize S(K);
  const uint16_t* sched = reinterpret_cast<const uint16_t*>(smem + a.sched_off[fd.kidx]);
  const uint32_t* pairs = reinterpret_cast<const uint32_t*>(smem + a.pairs_off[fd.kidx]);
  const WarpArea area(base + grp * group_doubles(K, GRAD, G, false, a.regather), K, GRAD, G, false, a.regather);
  Accum acc;
  const int64_t i0 = tile * fd.tile;
  const int64_t i1 = min(fd.n, i0 + fd.tile);
  for (int64_t b = i0; b < i1; b += NL) {
    const int64_t i = b + grp;
    const bool active = i < i1;
    process_location<GRAD, G, false, FIXED>(active ? i : b, active, F, S, sched, pairs, area, tab, mc, tc, acc, false,
                                            nullptr, a.errloc, sub);
  }
  write_partial<G>(acc, out, lane);
}

template <bool GRAD, int G, int FIXED>
__global__ void __launch_bounds__(lik_threads(GRAD, G, FIXED))
    vecchia_batched_kernel(const BatchArgs a) {
  extern __shared__ __align__(16) unsigned char smem[];
  for (int k = 0; k < a.nk; ++k)
    build_schedules(a.kval[k], reinterpret_cast<uint16_t*>(smem + a.sched_off[k]),
                    reinterpret_cast<uint32_t*>(smem + a.pairs_off[k]));
  __syncthreads();
  const int lane = threadIdx.x & 31;
  const int wib = threadIdx.x >> 5;
  double* base = reinterpret_cast<double*>(smem + a.area_off) + wib * a.area_doubles;
  while (true) {
    unsigned long long item = 0;
    if (lane == 0) item = atomicAdd(a.counter, 1ULL);
    item = __shfl_sync(0xffffffffu, item, 0);
    if ((int64_t)item >= a.total_items) break;
    item += a.first_item;
    // field of this item: fields are stored in item order
    int lo = a.first_field, hi = a.last_field;
    while (lo < hi) {
      const int mid = (lo + hi + 1) >> 1;
      if (a.fields[mid].item_base <= (int64_t)item) lo = mid; else hi = mid - 1;
    }
    const FieldDesc fd = a.fields[lo];
    const int64_t rel = (int64_t)item - fd.item_base;
    const int t = (int)(rel / fd.tiles);
    const int64_t tile = rel % fd.tiles;
    if (kChecked && (t >= a.ntheta || tile >= fd.tiles || tile < 0)) {
      if (lane == 0) {  // a work item outside the layout: record it and skip it
        atomicMin(a.errloc, err_code((int64_t)item, kErrIndex));
      }
      continue;
    }
    const double* th = a.thetas + ((int64_t)fd.orig * a.ntheta + t) * 4;
    const double s2 = th[0], beta = th[1], nu = th[2], t2 = th[3];
    const double* tab = nullptr;
    for (int k = 0; k < a.nnu; ++k)
      if (__double_as_longlong(a.nus[k]) == __double_as_longlong(nu)) tab = a.tabs[k];
    double* out = a.partial + item * 4;
    const bool theta_valid = s2 > 0.0 && beta > 0.0 && t2 >= 0.0 && isfinite(s2) && isfinite(beta) &&
                             isfinite(t2);
    if (!tab || !theta_valid) {
      if (lane == 0) {
        out[0] = out[1] = out[2] = out[3] = __longlong_as_double(0x7FF8000000000000LL);
        atomicMin(a.errloc, err_code(0, kErrData));
      }
      continue;
    }
    const MaternConst mc = matern_const_at(fix_const(tab));
    ThetaConst tc;
    tc.set(s2, beta, t2, kFamilyMatern, nu);
    if (FIXED) tc.weak_u = (float)fix_const(tab)[GRAD ? kConstWeakGradient : kConstWeakPrediction];
    run_item<GRAD, G, FIXED != 0>(fd, tile, smem, a, base, tab, mc, tc, out, lane);
    __syncwarp();
  }
}

// One CTA per (field, theta): the field's item records, each thread a strided subset in
// item order (compensated), merged by a fixed shuffle tree and warp order, so the result
// depends only on the field's item count.  (A compensated sum costs a warp some 1,800
// cycles of the FP64 pipe per 32 records: four sub-partitions share them.)
constexpr int kFinalWarps = 4;

__global__ void __launch_bounds__(32 * kFinalWarps)
    vecchia_batched_finalize(const FieldDesc* __restrict__ fields, int ntheta, const double* __restrict__ thetas,
                             const double* __restrict__ partial, int want_grad, double* out) {
  __shared__ Neumaier sums[kFinalWarps][4];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int fs = (int)(blockIdx.x / ntheta), t = (int)(blockIdx.x % ntheta);
  const FieldDesc fd = fields[fs];
  Neumaier acc[4];
  const double* p = partial + (fd.item_base + (int64_t)t * fd.tiles) * 4;
  for (int k = threadIdx.x; k < fd.tiles; k += 32 * kFinalWarps)
    for (int c = 0; c < 4; ++c) acc[c].add(p[(int64_t)k * 4 + c]);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1)
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      const double s2 = __shfl_down_sync(0xffffffffu, acc[c].s, o);
      const double c2 = __shfl_down_sync(0xffffffffu, acc[c].c, o);
      acc[c].merge(s2, c2);
    }
  if (lane == 0)
    for (int c = 0; c < 4; ++c) sums[warp][c] = acc[c];
  __syncthreads();
  if (threadIdx.x != 0) return;
  for (int w = 1; w < kFinalWarps; ++w)
    for (int c = 0; c < 4; ++c) acc[c].merge(sums[w][c].s, sums[w][c].c);
  const int64_t o = (int64_t)fd.orig * ntheta + t;
  if (!want_grad) {
    out[o] = acc[0].value();
    return;
  }
  const double* th = thetas + o * 4;
  double* r = out + o * 4;
  r[0] = acc[0].value();
  r[1] = (acc[1].value() - th[3] * acc[3].value()) / th[0];
  r[2] = -2.0 * th[0] / th[1] * acc[2].value();
  r[3] = acc[3].value();
}

// ------------------------------------------------------------------ host state
namespace {

struct PreparedNu {
  int device = -1;
  int nnu = 0;
  double nus[kMaxNu] = {};
  double* tabs[kMaxNu] = {};
  double* d_nus = nullptr;
  double** d_tabs = nullptr;
};

using BatchKernel = void (*)(const BatchArgs);

template <bool GRAD>
BatchKernel batch_kernel(int lanes, int fixed) {
  if (lanes == 4) return vecchia_batched_kernel<GRAD, 4, 0>;
  if (lanes == 8) return vecchia_batched_kernel<GRAD, 8, 0>;
  if (lanes == 16) return vecchia_batched_kernel<GRAD, 16, 0>;
  if (fixed == 0) return vecchia_batched_kernel<GRAD, 32, 0>;
  if constexpr (!GRAD)
    if (fixed == 2) return vecchia_batched_kernel<GRAD, 32, 2>;
  return vecchia_batched_kernel<GRAD, 32, 1>;
}

struct BatchClass {
  BatchArgs args{};
  BatchKernel kern = nullptr;
  int W = 0, per_sm = 0, blocks = 0, smem = 0;
};

struct BatchState {
  int device = -1;
  std::vector<const void*> plans;
  std::vector<const double*> ys;
  int ntheta = 0;
  int want_grad = 0;
  FieldDesc* d_fields = nullptr;
  double* d_partial = nullptr;
  unsigned long long* d_counter = nullptr;  // a work counter per class, then the error slot
  std::vector<BatchClass> classes;
};

std::mutex g_mu;
std::vector<PreparedNu> g_prepared;
std::vector<BatchState*> g_batches;

void free_batch(BatchState* b) {
  cudaFree(b->d_fields);
  cudaFree(b->d_partial);
  cudaFree(b->d_counter);
  delete b;
}

PreparedNu* prepared_for(int dev) {
  for (auto& p : g_prepared)
    if (p.device == dev) return &p;
  return nullptr;
}

// The class's warps per CTA with the most resident warps per SM (at most 16) and a grid of
// one wave, with the coordinates gathered twice where that gives a fifth more warps (as in
// the single-field launch).
int class_shape(BatchClass* c, const int* areas, int fixed_bytes, bool fixed) {
  int dev = 0, sms = 0, optin = 0;
  VECCHIA_CUDA_TRY(cudaGetDevice(&dev));
  VECCHIA_CUDA_TRY(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
  VECCHIA_CUDA_TRY(cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev));
  cudaFuncAttributes fa;
  VECCHIA_CUDA_TRY(cudaFuncGetAttributes(&fa, c->kern));
  // one limit for every batch: cached ones are launched again in any order
  VECCHIA_CUDA_TRY(cudaFuncSetAttribute(c->kern, cudaFuncAttributeMaxDynamicSharedMemorySize, optin - (int)fa.sharedSizeBytes));
  int best[2] = {-1, -1}, W[2] = {}, per[2] = {};
  for (int r = 0; r < 2; ++r)
    for (int w : {13, 12, 11, 10, 9, 8, 6, 4, 2, 1}) {
      const int bytes = fixed_bytes + w * areas[r] * 8;
      if (areas[r] == 0 || bytes > optin - (int)fa.sharedSizeBytes || 32 * w > fa.maxThreadsPerBlock) continue;
      int per_sm = 0;
      VECCHIA_CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, c->kern, w * 32, bytes));
      int warps = std::min(per_sm * w, 16);
      if (fixed && warps > 1 && warps % 4 == 1) warps -= 2;  // as in the single-field launch
      if (per_sm > 0 && warps > best[r]) {
        best[r] = warps;
        W[r] = w;
        per[r] = per_sm;
      }
    }
  const int r = best[1] > 0 && 5 * best[1] >= 6 * best[0] ? 1 : 0;
  if (best[r] <= 0) return VECCHIA_EINVAL;
  c->W = W[r];
  c->per_sm = per[r];
  c->blocks = per[r] * sms;
  c->smem = fixed_bytes + W[r] * areas[r] * 8;
  c->args.regather = r == 1;
  c->args.area_doubles = areas[r];
  return VECCHIA_OK;
}

int build_batch(const Plan* const* plans, const double* const* ys, int nfields, int ntheta, int want_grad,
                int dev, cudaStream_t stream, BatchState** out) {
  BatchState* b = new BatchState();
  b->device = dev;
  b->ntheta = ntheta;
  b->want_grad = want_grad;
  const bool grad = want_grad != 0;
  // fields by class, the wider groups (larger blocks) first, and by m within one
  auto lanes = [&](int f) {
    int64_t count = 0;
    for (int g = 0; g < nfields; ++g)
      if (plans[g]->m == plans[f]->m) count += plans[g]->n * ntheta;
    return lanes_for(plans[f]->m + 1, grad, count);
  };
  auto key = [&](int f) { return 2 * lanes(f) + (fixed_point_block(plans[f]->m + 1, grad, lanes(f)) ? 1 : 0); };
  std::vector<int> order(nfields);
  for (int f = 0; f < nfields; ++f) order[f] = f;
  std::stable_sort(order.begin(), order.end(), [&](int x, int y) {
    return key(x) != key(y) ? key(x) > key(y) : plans[x]->m > plans[y]->m;
  });
  std::vector<FieldDesc> fd(nfields);
  int64_t items = 0;
  int distinct = 0;
  for (int s = 0; s < nfields;) {
    BatchClass c;
    BatchArgs& a = c.args;
    const int k0 = key(order[s]), L = lanes(order[s]);
    c.kern = grad ? batch_kernel<true>(L, k0 & 1) : batch_kernel<false>(L, 2 * (k0 & 1));
    a.ntheta = ntheta;
    a.first_field = s;
    a.first_item = items;
    int areas[2] = {0, 0};
    int64_t steps = 0;
    for (; s < nfields && key(order[s]) == k0; ++s) {
      const Plan* p = plans[order[s]];
      FieldDesc& d = fd[s];
      d.xy = reinterpret_cast<const double2*>(p->d_xy);
      d.yf = ys[order[s]];
      d.nbr = p->d_nbr;
      d.self = p->d_self;
      d.n = p->n;
      d.m = p->m;
      d.orig = order[s];
      const int K = p->m + 1;
      if (a.nk == 0 || a.kval[a.nk - 1] != K) {
        if (distinct++ == kMaxDistinctK) { delete b; return VECCHIA_EINVAL; }
        a.kval[a.nk++] = K;
        for (int r = 0; r < (regather_capable(grad, L) ? 2 : 1); ++r)  // a warp holds 32/L blocks
          areas[r] = std::max(areas[r], (32 / L) * group_doubles(K, grad, L, false, r == 1));
      }
      d.kidx = a.nk - 1;
      steps += (d.n + 32 / L - 1) / (32 / L) * ntheta;
    }
    a.last_field = s - 1;
    int off = 0;
    for (int k = 0; k < a.nk; ++k) {
      const SchedSize S(a.kval[k]);
      a.sched_off[k] = off;
      off += S.sched_bytes;
      a.pairs_off[k] = off;
      off += S.pairs_bytes;
    }
    a.area_off = off;
    int rc = class_shape(&c, areas, off, k0 & 1);
    if (!rc && !grad && (k0 & 1) && c.W * c.per_sm < 16) {  // not room for 16 warps: the other form
      c.kern = batch_kernel<false>(L, 1);
      rc = class_shape(&c, areas, off, true);
    }
    if (rc) { delete b; return rc; }
    const int64_t share = steps / ((int64_t)kItemsPerWarp * c.blocks * c.W);
    for (int k = a.first_field; k <= a.last_field; ++k) {
      FieldDesc& d = fd[k];
      const int64_t step = std::max<int64_t>({1, std::min<int64_t>(kMostSteps, share), share / kManyItems});
      d.tile = (32 / L) * (int)std::min<int64_t>(step, (d.n + 32 / L - 1) / (32 / L));
      d.tiles = (int)((d.n + d.tile - 1) / d.tile);
      d.item_base = items;
      items += (int64_t)d.tiles * ntheta;
    }
    a.total_items = items - a.first_item;
    b->classes.push_back(c);
  }
  for (int s = 0; s < nfields; ++s) {
    b->plans.push_back(plans[s]);
    b->ys.push_back(ys[s]);
  }
  const int ncls = (int)b->classes.size();
  if (cudaMalloc(&b->d_fields, sizeof(FieldDesc) * nfields) != cudaSuccess ||
      cudaMalloc(&b->d_partial, sizeof(double) * 4 * std::max<int64_t>(items, 1)) != cudaSuccess ||
      cudaMalloc(&b->d_counter, sizeof(unsigned long long) * (ncls + 1)) != cudaSuccess) {
    free_batch(b);
    return VECCHIA_ENOMEM;
  }
  // on the caller's stream (it may not wait for the legacy default stream), and finished before
  // the layout is cached, where a call on another stream may find it
  if (cudaMemcpyAsync(b->d_fields, fd.data(), sizeof(FieldDesc) * nfields, cudaMemcpyHostToDevice, stream) != cudaSuccess ||
      cudaStreamSynchronize(stream) != cudaSuccess) {
    free_batch(b);
    return VECCHIA_ECUDA;
  }
  for (int k = 0; k < ncls; ++k) {
    BatchArgs& a = b->classes[k].args;
    a.fields = b->d_fields;
    a.partial = b->d_partial;
    a.counter = b->d_counter + k;
    a.errloc = b->d_counter + ncls;
  }
  *out = b;
  return VECCHIA_OK;
}

}  // namespace

// Drops cached batch layouts that reference `plan` (called by vecchia_plan_destroy).
void forget_plan_in_batches(const void* plan) {
  std::lock_guard<std::mutex> lk(g_mu);
  for (size_t k = 0; k < g_batches.size();) {
    BatchState* b = g_batches[k];
    if (std::find(b->plans.begin(), b->plans.end(), plan) != b->plans.end()) {
      free_batch(b);
      g_batches.erase(g_batches.begin() + k);
    } else {
      ++k;
    }
  }
}

}  // namespace vecchia

extern "C" int vecchia_batched_prepare(const double* nus, int32_t nnu, void* stream) {
  using namespace vecchia;
  if (!nus || nnu < 1 || nnu > kMaxNu) return VECCHIA_EINVAL;
  for (int k = 0; k < nnu; ++k)
    if (!std::isfinite(nus[k]) || !(nus[k] > 0.0)) return VECCHIA_EINVAL;
  int dev = 0;
  VECCHIA_CUDA_TRY(cudaGetDevice(&dev));
  cudaStream_t s = (cudaStream_t)stream;
  std::lock_guard<std::mutex> lk(g_mu);
  PreparedNu* p = prepared_for(dev);
  if (!p) {
    g_prepared.emplace_back();
    p = &g_prepared.back();
    p->device = dev;
    if (cudaMalloc(&p->d_nus, sizeof(double) * kMaxNu) != cudaSuccess ||
        cudaMalloc(&p->d_tabs, sizeof(double*) * kMaxNu) != cudaSuccess)
      return VECCHIA_ENOMEM;
    for (int k = 0; k < kMaxNu; ++k)
      if (cudaMalloc(&p->tabs[k], kFixTableBytes) != cudaSuccess) return VECCHIA_ENOMEM;
  }
  VECCHIA_CUDA_TRY(cudaStreamSynchronize(s));
  for (int k = 0; k < nnu; ++k) {
    p->nus[k] = nus[k];
    int rc = launch_matern_table(nus[k], p->tabs[k], s);
    if (rc) return rc;
  }
  p->nnu = nnu;
  VECCHIA_CUDA_TRY(cudaMemcpyAsync(p->d_nus, p->nus, sizeof(double) * kMaxNu, cudaMemcpyHostToDevice, s));
  VECCHIA_CUDA_TRY(cudaMemcpyAsync(p->d_tabs, p->tabs, sizeof(double*) * kMaxNu, cudaMemcpyHostToDevice, s));
  VECCHIA_CUDA_TRY(cudaStreamSynchronize(s));
  return VECCHIA_OK;
}

extern "C" int vecchia_loglik_batched(const vecchia_plan_t* plans, const double* const* y_devs, int32_t nfields,
                                      const double* thetas_dev, int32_t ntheta, int want_grad, double* out_dev,
                                      void* stream) {
  using namespace vecchia;
  if (!plans || !y_devs || nfields < 1 || ntheta < 1 || !thetas_dev || !out_dev) return VECCHIA_EINVAL;
  for (int f = 0; f < nfields; ++f)
    if (!plans[f] || !y_devs[f] || plans[f]->family != kFamilyMatern || plans[f]->m > kMaxMWarp ||
        plans[f]->metric != 0)
      return VECCHIA_EINVAL;
  want_grad = want_grad ? 1 : 0;
  int dev = 0;
  VECCHIA_CUDA_TRY(cudaGetDevice(&dev));
  cudaStream_t s = (cudaStream_t)stream;
  std::lock_guard<std::mutex> lk(g_mu);
  PreparedNu* pn = prepared_for(dev);
  if (!pn || pn->nnu == 0) return VECCHIA_EINVAL;
  BatchState* b = nullptr;
  for (BatchState* c : g_batches) {
    if (c->device != dev || c->ntheta != ntheta || c->want_grad != want_grad || (int)c->plans.size() != nfields)
      continue;
    bool same = true;
    for (int f = 0; f < nfields && same; ++f)
      same = c->plans[f] == (const void*)plans[f] && c->ys[f] == y_devs[f];
    if (same) { b = c; break; }
  }
  if (!b) {
    // First call for this set of fields: lay out the work (allocates; not capturable).
    cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
    VECCHIA_CUDA_TRY(cudaStreamIsCapturing(s, &cs));
    if (cs != cudaStreamCaptureStatusNone) return VECCHIA_EINVAL;
    std::vector<const Plan*> pp(nfields);
    for (int f = 0; f < nfields; ++f) pp[f] = plans[f];
    int rc = build_batch(pp.data(), y_devs, nfields, ntheta, want_grad, dev, s, &b);
    if (rc) return rc;
    g_batches.push_back(b);
  }
  const size_t ncls = b->classes.size();
  VECCHIA_CUDA_TRY(cudaMemsetAsync(b->d_counter, 0, sizeof(unsigned long long) * ncls, s));
  VECCHIA_CUDA_TRY(cudaMemsetAsync(b->d_counter + ncls, 0xFF, sizeof(unsigned long long), s));
  for (const BatchClass& c : b->classes) {
    BatchArgs a = c.args;
    a.thetas = thetas_dev;
    a.nus = pn->d_nus;
    a.tabs = pn->d_tabs;
    a.nnu = pn->nnu;
    c.kern<<<c.blocks, c.W * 32, c.smem, s>>>(a);
    VECCHIA_CUDA_TRY(cudaGetLastError());
  }
  const int64_t pairs = (int64_t)nfields * ntheta;
  vecchia_batched_finalize<<<(unsigned)pairs, 32 * kFinalWarps, 0, s>>>(b->d_fields, ntheta, thetas_dev, b->d_partial,
                                                                      want_grad, out_dev);
  VECCHIA_CUDA_TRY(cudaGetLastError());
  return VECCHIA_OK;
}
