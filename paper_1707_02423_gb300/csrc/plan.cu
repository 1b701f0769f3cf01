// a7 (batch scheduler), device side: validate the pair list, classify every
// pair into an execution class, order the pairs by cost (largest first, two
// buckets per octave) into one queue per class, and compute the output offsets
// x_off[p] = sum_{q<p} n_a n_b and m_off[p] = sum_{q<p} n_a.
//
// Up to kPlanSmall pairs: one launch of one CTA (plan_small_kernel), which also
// clears the workspace header.  More: a memset and three small launches --
// count (per-pair class/bucket histogram and per-block offset sums), scan (one
// CTA: bucket cursors and block offsets), scatter (queue positions and per-pair
// offsets).  No host round trip, so the whole call can be replayed from a CUDA
// graph.
//
// The plan is latency: the memset and the three launches take 15 us more of a call
// on 28 pairs than the one launch.
#include <algorithm>

#include "device_common.cuh"
#include "device_state.h"
#include "kernels.h"

namespace cfsim {

namespace {

struct PlanCtx {
  PackView A, B;
  int P;
  const int32_t* pairs;
  WsHeader* hdr;
  uint32_t* queue;
  int64_t* x_off;
  int64_t* m_off;
  int64_t* bsum;  // [2][plan_blocks]
  int nblk;
};

__device__ __forceinline__ PlanCtx plan_ctx(const CallArgs& a) {
  PlanCtx c;
  c.A = load_pack(a.pack_a);
  c.B = load_pack(a.pack_b);
  c.P = a.P;
  c.pairs = a.pairs;
  WsLayout L = ws_layout(a.P);
  c.hdr = reinterpret_cast<WsHeader*>(a.ws + L.hdr);
  c.queue = reinterpret_cast<uint32_t*>(a.ws + L.queue);
  c.x_off = reinterpret_cast<int64_t*>(a.ws + L.x_off);
  c.m_off = reinterpret_cast<int64_t*>(a.ws + L.m_off);
  c.bsum = reinterpret_cast<int64_t*>(a.ws + L.bsum);
  c.nblk = L.plan_blocks;
  return c;
}

struct PairFacts {
  bool valid;
  int na, nb, ea, eb;
  int cls, bucket;
  int n_row, ld;  // resident matrix shape (classify)
};

__device__ __forceinline__ PairFacts pair_facts(const PlanCtx& c, int p, const ClassCfg& cc) {
  PairFacts f{};
  int pa = __ldg(c.pairs + 2 * p), pb = __ldg(c.pairs + 2 * p + 1);
  f.valid = pa >= 0 && pa < c.A.n_cfgs && pb >= 0 && pb < c.B.n_cfgs;
  if (!f.valid) {
    f.cls = kClassSkip;
    return f;
  }
  f.na = __ldg(c.A.node_off + pa + 1) - __ldg(c.A.node_off + pa);
  f.nb = __ldg(c.B.node_off + pb + 1) - __ldg(c.B.node_off + pb);
  const int ea = __ldg(c.A.edge_off + pa + 1) - __ldg(c.A.edge_off + pa);
  const int eb = __ldg(c.B.edge_off + pb + 1) - __ldg(c.B.edge_off + pb);
  f.ea = ea;
  f.eb = eb;
  Shape s = classify(f.na, f.nb, ea, eb, cc, __ldg(c.A.xdeg + pa), __ldg(c.B.xdeg + pb));
  f.cls = s.cls;
  f.n_row = s.n_row;
  f.ld = s.ld;
  // per-iteration work: every entry is written once, every edge pair gathered twice
  int64_t cost = (int64_t)f.na * f.nb + 2 * (int64_t)ea * eb;
  // the global class is split over teams by cost: a CTA's shared memory also
  // limits the rows of its slab (about 2,000)
  const int64_t rows = team_tr(f.na, f.nb) ? f.nb : f.na;
  if (f.cls == kClassGlobal && cc.bwd != 2 && cost < kTeamRowCost * rows) cost = kTeamRowCost * rows;
  f.bucket = cost_bucket(cost);
  return f;
}

// Exclusive block scan of two int64 values (NT threads).
template <int NT>
__device__ __forceinline__ void block_scan2(int64_t& x, int64_t& m, int64_t& tx, int64_t& tm) {
  __shared__ int64_t sx[NT / 32], sm[NT / 32];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  int64_t ix = x, im = m;  // inclusive within warp
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    int64_t ux = __shfl_up_sync(0xffffffffu, ix, o);
    int64_t um = __shfl_up_sync(0xffffffffu, im, o);
    if (lane >= o) {
      ix += ux;
      im += um;
    }
  }
  if (lane == 31) {
    sx[w] = ix;
    sm[w] = im;
  }
  __syncthreads();
  int64_t bx = 0, bm = 0;
  tx = 0;
  tm = 0;
#pragma unroll
  for (int k = 0; k < NT / 32; ++k) {
    if (k < w) {
      bx += sx[k];
      bm += sm[k];
    }
    tx += sx[k];
    tm += sm[k];
  }
  x = bx + ix - x;  // exclusive
  m = bm + im - m;
  __syncthreads();
}

// What the workspace header keeps of a pair, beside its queue place.
struct PairNeeds {
  unsigned long long slot, bwd_slot, bwd_big;
};
__device__ __forceinline__ PairNeeds pair_needs(const PairFacts& f, const ClassCfg& cc, int K, int F_pad) {
  const bool large = f.cls == kClassGlobal || f.cls == kClassCluster;  // both use a scratch slot
  PairNeeds n{};
  if (large) n.slot = global_slot_bytes(f.na, f.nb);
  n.bwd_slot = bwd_slot_bytes(f.na, f.nb, f.ea, f.eb, K, F_pad);
  // the adjoint's per-team slots of pairs not resident in one CTA: the
  // full-matrix layout of the cluster tier, or the global tier's own
  if (cc.bwd && large) n.bwd_big = f.cls == kClassCluster ? bwd_res_slot_bytes(f.n_row, f.ld, K) : n.bwd_slot;
  return n;
}
__device__ __forceinline__ void max_needs(WsHeader* h, const PairNeeds& n) {
  if (n.slot) atomicMax(reinterpret_cast<unsigned long long*>(&h->slot_need), n.slot);
  if (n.bwd_slot) atomicMax(reinterpret_cast<unsigned long long*>(&h->bwd_slot_need), n.bwd_slot);
  if (n.bwd_big) atomicMax(reinterpret_cast<unsigned long long*>(&h->bwd_big_need), n.bwd_big);
}

// The queue order: class by class; within a class, costliest bucket first.
// hist [class][bucket] (shared) -> the buckets' first positions, in place, and
// the classes' sizes; the first 512 threads of the CTA work, all must call.
// (One thread walking the 448 counts in global memory, a load after a store
// each time, took most of the plan's time.)
constexpr int kSlots = kNumClasses * kBuckets;
static_assert(kSlots <= 512 && kBuckets == 64, "one thread per bucket");
__device__ __forceinline__ void queue_order(uint32_t* hist, uint32_t* n_class) {
  __shared__ uint32_t part[16];
  const int t = threadIdx.x, lane = t & 31, w = t >> 5;
  const int cls = t / kBuckets, at = cls * kBuckets + (kBuckets - 1 - t % kBuckets);
  const uint32_t v = t < kSlots ? hist[at] : 0u;
  uint32_t s = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t u = __shfl_up_sync(0xffffffffu, s, o);
    if (lane >= o) s += u;
  }
  if (w < 16 && lane == 31) part[w] = s;
  __syncthreads();
  if (t < kSlots) {
    uint32_t before = 0;
    for (int k = 0; k < w; ++k) before += part[k];
    hist[at] = before + s - v;
    if (t % kBuckets == 0) n_class[cls] = part[w] + part[w + 1];  // a class is two warps
  }
  __syncthreads();
}

// Team levels of the global class (the queue's first): the queue position
// each level ends at, from the class's counts (one thread; cnt: per bucket).
__device__ __forceinline__ void team_levels(const uint32_t* cnt, uint32_t ng, int n_cta, bool match, uint32_t* lvl_end) {
  // a bucket's middle cost: 2 to 3, or 3 to 4, times 2^(b / 2)
  auto mid = [](int b) { return (int64_t)((b & 1) ? 7 : 5) << (b / 2) >> 1; };
  int64_t total = 0;
  int lo = kBuckets, hi = -1;
  for (int b = 0; b < kBuckets; ++b) {
    total += cnt[b] * mid(b);
    if (cnt[b]) {
      lo = min(lo, b);
      hi = b;
    }
  }
  const bool even = hi - lo <= 1;  // within an octave
  uint32_t seen = 0;
  uint32_t end[kTeamLevels] = {};
  int level = 0;
  for (int b = kBuckets - 1; b >= 0 && seen < ng; --b) {
    if (cnt[b] == 0) continue;
    level = max(level, team_level(mid(b), total, n_cta, match, even));
    seen += cnt[b];
#pragma unroll
    for (int L = 0; L < kTeamLevels; ++L)
      if (L >= level) end[L] = seen;
  }
#pragma unroll
  for (int L = 0; L < kTeamLevels; ++L) lvl_end[L] = end[L];
}

// matching policy 3: the deferred-steps area at the end of the workspace, if
// it fits beside one scratch slot (when any pair needs one).  Under tune 0 it
// must leave every slot that the workspace was sized for, and pairs must be
// large enough on average for the second kernel to pay (kDeferCells).
__device__ __forceinline__ void defer_area(WsHeader* h, const CallArgs& a, int ranked, int64_t x_total, uint32_t n_large,
                                           size_t slot_need) {
  if (ranked != 3) return;
  const WsLayout L = ws_layout(a.P);
  const size_t need = defer_bytes(a.P, x_total);
  const size_t avail = a.ws_bytes > L.scratch ? a.ws_bytes - L.scratch : 0;
  size_t slots = n_large > 0 ? 1 : 0;
  if (a.defer_auto) {
    if (!defer_pays(a.P, x_total)) return;
    slots = n_large < 2u * (uint32_t)a.n_cta ? n_large : 2u * (uint32_t)a.n_cta;
  }
  if (need + slots * slot_need <= avail) {
    h->defer = 1;
    h->defer_off = (a.ws_bytes - need + kAlign - 1) / kAlign * kAlign;
  }
}

// The whole plan of up to kPlanSmall pairs by one CTA: two pairs per thread,
// counts and cursors in shared memory.
constexpr int kPlanSmallNT = 1024;

__global__ void __launch_bounds__(kPlanSmallNT) plan_small_kernel(CallArgs a, ClassCfg cc) {
  constexpr int kPer = kPlanSmall / kPlanSmallNT;
  __shared__ uint32_t hist[kSlots], s_class[kNumClasses], s_glob[kBuckets];
  PlanCtx c = plan_ctx(a);
  const int t = threadIdx.x;
  for (int i = t; i < (int)(sizeof(WsHeader) / 4); i += kPlanSmallNT) reinterpret_cast<uint32_t*>(c.hdr)[i] = 0u;
  if (t < kSlots) hist[t] = 0u;
  __syncthreads();
  PairFacts f[kPer];
  int64_t xc = 0, mc = 0;
#pragma unroll
  for (int k = 0; k < kPer; ++k) {
    const int p = kPer * t + k;
    f[k].valid = false;
    if (p >= c.P) continue;
    f[k] = pair_facts(c, p, cc);
    if (!f[k].valid) {
      set_status(c.hdr, 1 /* CF_ERR_INVALID_ARG */, p);
      continue;
    }
    atomicAdd(&hist[f[k].cls * kBuckets + f[k].bucket], 1u);
    max_needs(c.hdr, pair_needs(f[k], cc, a.K, c.A.F_pad));
    xc += (int64_t)f[k].na * f[k].nb;
    mc += f[k].na;
  }
  int64_t tx, tm;
  block_scan2<kPlanSmallNT>(xc, mc, tx, tm);
  if (t < kBuckets) s_glob[t] = hist[kClassGlobal * kBuckets + t];
  __syncthreads();
  queue_order(hist, s_class);
#pragma unroll
  for (int k = 0; k < kPer; ++k) {
    const int p = kPer * t + k;
    if (p >= c.P) continue;
    c.x_off[p] = xc;
    c.m_off[p] = mc;
    if (!f[k].valid) continue;
    c.queue[atomicAdd(&hist[f[k].cls * kBuckets + f[k].bucket], 1u)] = (uint32_t)p;
    xc += (int64_t)f[k].na * f[k].nb;
    mc += f[k].na;
  }
  if (t < kNumClasses) c.hdr->n_class[t] = s_class[t];
  if (t == 0) {
    c.hdr->x_total = tx;
    c.hdr->m_total = tm;
    c.x_off[c.P] = tx;
    c.m_off[c.P] = tm;
    defer_area(c.hdr, a, cc.ranked, tx, s_class[kClassGlobal] + s_class[kClassCluster],
               (size_t)*reinterpret_cast<volatile uint64_t*>(&c.hdr->slot_need));
    if (s_class[kClassGlobal] > 0)
      team_levels(s_glob, s_class[kClassGlobal], a.n_cta, cc.bwd == 2, c.hdr->team.lvl_end);
  }
}

__global__ void __launch_bounds__(kPlanThreads) plan_count_kernel(CallArgs a, ClassCfg cc) {
  PlanCtx c = plan_ctx(a);
  const int p = blockIdx.x * kPlanThreads + threadIdx.x;
  int64_t xc = 0, mc = 0;
  if (p < c.P) {
    PairFacts f = pair_facts(c, p, cc);
    if (!f.valid) {
      set_status(c.hdr, 1 /* CF_ERR_INVALID_ARG */, p);
    } else {
      atomicAdd(&c.hdr->hist[f.cls][f.bucket], 1u);
      max_needs(c.hdr, pair_needs(f, cc, a.K, c.A.F_pad));
      xc = (int64_t)f.na * f.nb;
      mc = f.na;
    }
  }
  int64_t tx, tm;
  block_scan2<kPlanThreads>(xc, mc, tx, tm);
  if (threadIdx.x == 0) {
    c.bsum[blockIdx.x] = tx;
    c.bsum[c.nblk + blockIdx.x] = tm;
  }
}

constexpr int kScanNT = 512;

__global__ void __launch_bounds__(kScanNT) plan_scan_kernel(CallArgs a, int ranked, bool match) {
  __shared__ uint32_t hist[kSlots], s_class[kNumClasses], s_glob[kBuckets];
  PlanCtx c = plan_ctx(a);
  const int t = threadIdx.x;
  if (t < kSlots) hist[t] = reinterpret_cast<const uint32_t*>(c.hdr->hist)[t];
  __syncthreads();
  if (t < kBuckets) s_glob[t] = hist[kClassGlobal * kBuckets + t];
  __syncthreads();
  queue_order(hist, s_class);
  if (t < kSlots) reinterpret_cast<uint32_t*>(c.hdr->cursor)[t] = hist[t];
  if (t < kNumClasses) c.hdr->n_class[t] = s_class[t];
  // exclusive scan of the per-block offset sums (chunked over the threads)
  const int per = ceil_div(c.nblk, kScanNT);
  const int b0 = t * per, b1 = min(c.nblk, b0 + per);
  int64_t sx = 0, sm = 0;
  for (int b = b0; b < b1; ++b) {
    sx += c.bsum[b];
    sm += c.bsum[c.nblk + b];
  }
  int64_t tx, tm;
  block_scan2<kScanNT>(sx, sm, tx, tm);
  for (int b = b0; b < b1; ++b) {
    int64_t vx = c.bsum[b], vm = c.bsum[c.nblk + b];
    c.bsum[b] = sx;
    c.bsum[c.nblk + b] = sm;
    sx += vx;
    sm += vm;
  }
  if (t == 0) {
    c.hdr->x_total = tx;
    c.hdr->m_total = tm;
    c.x_off[c.P] = tx;
    c.m_off[c.P] = tm;
    defer_area(c.hdr, a, ranked, tx, s_class[kClassGlobal] + s_class[kClassCluster], (size_t)c.hdr->slot_need);
    // (the levels' table takes the histogram's place)
    team_levels(s_glob, s_class[kClassGlobal], a.n_cta, match, c.hdr->team.lvl_end);
  }
}

__global__ void __launch_bounds__(kPlanThreads) plan_scatter_kernel(CallArgs a, ClassCfg cc) {
  PlanCtx c = plan_ctx(a);
  const int p = blockIdx.x * kPlanThreads + threadIdx.x;
  int64_t xc = 0, mc = 0;
  if (p < c.P) {
    PairFacts f = pair_facts(c, p, cc);
    if (f.valid) {
      uint32_t pos = atomicAdd(&c.hdr->cursor[f.cls][f.bucket], 1u);
      c.queue[pos] = (uint32_t)p;
      xc = (int64_t)f.na * f.nb;
      mc = f.na;
    }
  }
  int64_t tx, tm;
  block_scan2<kPlanThreads>(xc, mc, tx, tm);
  if (p < c.P) {
    c.x_off[p] = c.bsum[blockIdx.x] + xc;
    c.m_off[p] = c.bsum[c.nblk + blockIdx.x] + mc;
  }
}

}  // namespace

cudaError_t launch_plan(const CallArgs& args, const ClassCfg& cc, cudaStream_t s) {
  CallArgs a = args;
  int dev = 0;
  const cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  a.n_cta = std::min(std::max(sm_count_of(dev), 1), kTeamMaxCta);
  if (a.P <= kPlanSmall) {
    plan_small_kernel<<<1, kPlanSmallNT, 0, s>>>(a, cc);
    return cudaGetLastError();
  }
  const cudaError_t z = cudaMemsetAsync(a.ws, 0, sizeof(WsHeader), s);
  if (z != cudaSuccess) return z;
  WsLayout L = ws_layout(a.P);
  plan_count_kernel<<<L.plan_blocks, kPlanThreads, 0, s>>>(a, cc);
  plan_scan_kernel<<<1, kScanNT, 0, s>>>(a, cc.ranked, cc.bwd == 2);
  plan_scatter_kernel<<<L.plan_blocks, kPlanThreads, 0, s>>>(a, cc);
  return cudaGetLastError();
}

}  // namespace cfsim
