// Small kernels: pack edge-weight update from user-order weights, and the
// per-row top-k of the query workload (a9).
#include "device_common.cuh"
#include "kernels.h"

namespace cfsim {

namespace {

__global__ void zero_w_kernel(CfAdj* out_adj, int64_t n) {
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < n; e += (int64_t)gridDim.x * blockDim.x)
    out_adj[e].w = 0.f;
}

// Duplicate user edges add into their one distinct edge.
__global__ void add_w_kernel(CfAdj* out_adj, const int32_t* u2c, const float* w_user, int64_t n_user) {
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < n_user; e += (int64_t)gridDim.x * blockDim.x)
    atomicAdd(&out_adj[u2c[e]].w, w_user[e]);
}

__global__ void in_w_kernel(CfAdj* in_adj, const int32_t* in_eid, const CfAdj* out_adj, int64_t n) {
  for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < n; k += (int64_t)gridDim.x * blockDim.x)
    in_adj[k].w = out_adj[in_eid[k]].w;
}

// Order-preserving map of a float to uint32 (larger float -> larger key).
__device__ __forceinline__ uint32_t float_key(float v) {
  uint32_t u = __float_as_uint(v);
  return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}

// Warp maximum of 64-bit keys.
__device__ __forceinline__ uint64_t warp_max_u64(uint64_t v) {
  const uint32_t hi = __reduce_max_sync(0xffffffffu, (uint32_t)(v >> 32));
  const uint32_t lo = __reduce_max_sync(0xffffffffu, (uint32_t)(v >> 32) == hi ? (uint32_t)v : 0u);
  return ((uint64_t)hi << 32) | lo;
}

constexpr int kTopkMax = 1024;              // largest k
constexpr int kTopkCand = 256 + 2 * kTopkMax;  // candidates, 256 + 2 k of them are ranked

// One CTA per row.  Elements are compared by 64-bit keys (score key << 32 |
// ~column), all different, so ties go to the smaller column and the result is
// exact and deterministic.  Thread t owns the columns t + NT m.
//   1  the best key of each group of threads (a warp or a part of one, so that
//      there are at least 1.5 k groups, as far as the threads go: 1,024 groups
//      at most, 256 up to 2,048 columns); the k-th best of these is a bound
//      that at least k elements reach, in random order little more than k;
//   2  the elements that reach the bound are collected and ranked by counting.
// Two reads of the row and three barriers for any k.  A row whose best elements
// crowd into few groups has too many candidates: it goes by rounds, each the
// block's maximum of the threads' best keys, after which the warp of the
// winner's thread finds that thread's next best.
// What bounds it: the latency of a read of the row and of the barriers.  (k
// rounds over the row: 24.9 us a call for the best 16 of 32 x 10,000, against
// 7.3, of which 7 is the launch; 1.30 ms against 0.60 for the best 1,024.)
template <int NT>
__global__ void __launch_bounds__(NT) topk_kernel(const float* scores, int C, int k, int g, float* top, int32_t* idx) {
  __shared__ uint64_t s_key[kTopkCand];  // the groups' best keys, then the candidates
  __shared__ uint64_t s_bound;
  __shared__ int s_n;
  const int q = blockIdx.x, t = threadIdx.x, lane = t & 31, wid = t >> 5;
  const float* row = scores + (size_t)q * C;
  auto key_of = [](float v, int c) { return ((uint64_t)float_key(v) << 32) | (uint32_t)(~(uint32_t)c); };
  uint64_t best = 0;
  for (int64_t c0 = t; c0 < C; c0 += 8 * NT) {
    float v[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) v[u] = c0 + u * NT < C ? row[c0 + u * NT] : 0.f;
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      const uint64_t key = c0 + u * NT < C ? key_of(v[u], (int)(c0 + u * NT)) : 0u;
      best = key > best ? key : best;
    }
  }
  uint64_t gb = best;
  if (g == 32) {
    gb = warp_max_u64(gb);
  } else {
    for (int o = g >> 1; o > 0; o >>= 1) {
      const uint64_t w = __shfl_xor_sync(0xffffffffu, gb, o);
      gb = w > gb ? w : gb;
    }
  }
  const int G = NT / g;
  if (t % g == 0) s_key[t / g] = gb;
  if (t == 0) {
    s_bound = 1;  // fewer than k groups hold an element: every element
    s_n = 0;
  }
  __syncthreads();
  if (t < G && s_key[t]) {
    const uint64_t mine = s_key[t];
    int r = 0;
    for (int j = 0; j < G; ++j) r += s_key[j] > mine;
    if (r == k - 1) s_bound = mine;
  }
  __syncthreads();
  const uint64_t bound = s_bound;
  const int limit = 256 + 2 * k;
  if (best >= bound)
    for (int64_t c = t; c < C; c += NT) {
      const uint64_t key = key_of(row[c], (int)c);
      if (key >= bound) {
        const int at = atomicAdd(&s_n, 1);
        if (at < limit) s_key[at] = key;
      }
    }
  __syncthreads();
  const int n = s_n;
  if (n <= limit) {
    for (int i = t; i < n; i += NT) {
      const uint64_t mine = s_key[i];
      int r = 0;
      for (int j = 0; j < n; ++j) r += s_key[j] > mine;
      if (r < k) {
        const int c = (int)(~(uint32_t)mine);
        idx[(size_t)q * k + r] = c;
        top[(size_t)q * k + r] = row[c];
      }
    }
    return;
  }
  for (int r = 0; r < k; ++r) {
    const uint64_t wb = warp_max_u64(best);
    if (lane == 0) s_key[(r & 1) * 32 + wid] = wb;
    __syncthreads();
    const uint64_t win = warp_max_u64(lane < NT / 32 ? s_key[(r & 1) * 32 + lane] : 0u);
    const int c = (int)(~(uint32_t)win), owner = c % NT;
    if (t == owner) {
      idx[(size_t)q * k + r] = c;
      top[(size_t)q * k + r] = row[c];
    }
    if (owner >> 5 == wid) {  // the owner's best key below the winner
      uint64_t next = 0;
      for (int64_t e = owner + (int64_t)NT * lane; e < C; e += 32 * NT) {
        const uint64_t key = key_of(row[e], (int)e);
        if (key < win && key > next) next = key;
      }
      next = warp_max_u64(next);
      if (t == owner) best = next;
    }
  }
}

// The pair list of the winners: pairs[2 (q k + r)] = rows ? rows[q] : q, and
// pairs[2 (q k + r) + 1] = idx[q k + r], for every query q and rank r.
__global__ void topk_pairs_kernel(const int32_t* idx, int Q, int k, const int32_t* rows, int32_t* pairs) {
  const int64_t n = (int64_t)Q * k;
  for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < n; t += (int64_t)gridDim.x * blockDim.x) {
    const int q = (int)(t / k);
    pairs[2 * t] = rows ? rows[q] : q;
    pairs[2 * t + 1] = idx[t];
  }
}

}  // namespace

cudaError_t launch_topk_pairs(const int32_t* idx, int Q, int k, const int32_t* rows, int32_t* pairs, cudaStream_t s) {
  const int64_t n = (int64_t)Q * k;
  const int g = (int)((n + 255) / 256 < 1024 ? (n + 255) / 256 : 1024);
  if (n > 0) topk_pairs_kernel<<<g, 256, 0, s>>>(idx, Q, k, rows, pairs);
  return cudaGetLastError();
}

cudaError_t launch_set_weights(CfAdj* out_adj, CfAdj* in_adj, const int32_t* in_eid, const int32_t* u2c,
                               int64_t n_user_edges, int64_t n_edges, const float* w_user, cudaStream_t s) {
  const int nt = 256;
  const int g1 = (int)((n_edges + nt - 1) / nt > 0 ? (n_edges + nt - 1) / nt : 1);
  const int g2 = (int)((n_user_edges + nt - 1) / nt > 0 ? (n_user_edges + nt - 1) / nt : 1);
  if (n_edges > 0) zero_w_kernel<<<g1 < 4096 ? g1 : 4096, nt, 0, s>>>(out_adj, n_edges);
  if (n_user_edges > 0) add_w_kernel<<<g2 < 4096 ? g2 : 4096, nt, 0, s>>>(out_adj, u2c, w_user, n_user_edges);
  if (n_edges > 0) in_w_kernel<<<g1 < 4096 ? g1 : 4096, nt, 0, s>>>(in_adj, in_eid, out_adj, n_edges);
  return cudaGetLastError();
}

cudaError_t launch_topk(const float* scores, int Q, int C, int k, float* top, int32_t* idx, cudaStream_t s) {
  // a thread per 8 columns or fewer up to 2,048 columns, then all a CTA can have
  const int nt = C <= 2048 ? 256 : 1024;
  int g = 32;
  while (g > 1 && 2 * (nt / g) < 3 * k) g >>= 1;
  if (nt == 256)
    topk_kernel<256><<<Q, 256, 0, s>>>(scores, C, k, g, top, idx);
  else
    topk_kernel<1024><<<Q, 1024, 0, s>>>(scores, C, k, g, top, idx);
  return cudaGetLastError();
}

}  // namespace cfsim
