// Ward clustering of CFGs by their similarity profiles (Sec. 5.3: Ward's
// minimum-variance method on squared Euclidean distances), and the scatter of
// pair scores into the dense score matrix whose rows are those profiles.
//
// ward_dist_kernel: D[i][j] = |X_i - X_j|^2 for all point pairs (D[i][i] = +inf).
// ward_merge_kernel (one CTA): n - 1 merges.  Each step takes the active pair
// (a < b) of smallest D (ties: smaller a, then smaller b), records it in
// scipy's linkage convention (cluster ids, height sqrt(D), size), keeps the
// union in slot a and retires slot b, and updates row / column a by the
// Lance-Williams recurrence for Ward,
//   D(a u b, k) = ((n_a + n_k) D(a, k) + (n_b + n_k) D(b, k) - n_k D(a, b))
//                 / (n_a + n_b + n_k).
#include <algorithm>
#include <cstdio>

#include "../../include/cfsim.h"
#include "device_common.cuh"
#include "device_state.h"
#include "kernels.h"

namespace cfsim {

void set_error_detail(const char* msg);

namespace {

constexpr int kWardNT = 1024;
constexpr int kWardMaxN = 16384;
constexpr size_t kWardSmem = 230400;  // dynamic shared memory of the merge kernel, at most

struct WardLayout {
  size_t hdr, D, total;
};

WardLayout ward_layout(int n) {
  WardLayout L{};
  L.hdr = 0;
  L.D = align_up(64, kAlign);
  L.total = align_up(L.D + 4 * (size_t)n * n, kAlign);
  return L;
}

// A 16 x 16 tile of D per CTA, a thread per entry; the points' rows pass
// through shared memory in chunks of 32, the next chunk's loads in flight.  The
// sum runs along k in one chain, so D is symmetric to the bit.  (Straight out of
// global memory a warp's loads were a point apart from lane to lane.)
__global__ void __launch_bounds__(256) ward_dist_kernel(const float* __restrict__ X, int n, int dim,
                                                        float* __restrict__ D) {
  __shared__ float xi[16][33], xj[16][33];
  const int t = threadIdx.x, tx = t & 15, ty = t >> 4;
  const int i0 = blockIdx.y * 16, j0 = blockIdx.x * 16;
  const int lr = t >> 5, lk = t & 31;  // this thread loads rows lr and lr + 8 of both tiles
  float pi[2], pj[2];
  auto fetch = [&](int k0) {
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      const int r = lr + 8 * u, k = k0 + lk;
      pi[u] = i0 + r < n && k < dim ? __ldg(X + (size_t)(i0 + r) * dim + k) : 0.f;
      pj[u] = j0 + r < n && k < dim ? __ldg(X + (size_t)(j0 + r) * dim + k) : 0.f;
    }
  };
  fetch(0);
  float s = 0.f;
  for (int k0 = 0; k0 < dim; k0 += 32) {
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      xi[lr + 8 * u][lk] = pi[u];
      xj[lr + 8 * u][lk] = pj[u];
    }
    __syncthreads();
    if (k0 + 32 < dim) fetch(k0 + 32);
    const int kn = min(32, dim - k0);
    if (kn == 32) {
#pragma unroll
      for (int k = 0; k < 32; ++k) {
        const float d = xi[ty][k] - xj[tx][k];
        s = fmaf(d, d, s);
      }
    } else {
      for (int k = 0; k < kn; ++k) {
        const float d = xi[ty][k] - xj[tx][k];
        s = fmaf(d, d, s);
      }
    }
    __syncthreads();
  }
  const int i = i0 + ty, j = j0 + tx;
  if (i < n && j < n) D[(size_t)i * n + j] = i == j ? CUDART_INF_F : s;
}

// Unsigned order of floats that are not NaN; -0 equals +0.
__device__ __forceinline__ uint32_t dist_key(float v) {
  if (v == 0.f) v = 0.f;
  const uint32_t b = __float_as_uint(v);
  return (b & 0x80000000u) ? ~b : (b | 0x80000000u);
}
__device__ __forceinline__ float key_dist(uint32_t k) {
  return __uint_as_float((k & 0x80000000u) ? (k & 0x7fffffffu) : ~k);
}
constexpr uint32_t kInfKey = 0xff800000u;  // dist_key(+inf)

// Smallest entry of a row (ties: smaller column; neither +inf nor NaN), by one
// warp: its key and column, kInfKey or more if there is none.
__device__ __forceinline__ uint32_t warp_row_min(const float* row, int n, int lane, int& arg) {
  float bv = CUDART_INF_F;
  int bj = 0x7fffffff;
  for (int j0 = lane; j0 < n; j0 += 256) {
    float v[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) v[u] = j0 + 32 * u < n ? row[j0 + 32 * u] : CUDART_INF_F;
#pragma unroll
    for (int u = 0; u < 8; ++u)
      if (v[u] < bv) {  // lanes scan increasing columns: ties keep the smaller one
        bv = v[u];
        bj = j0 + 32 * u;
      }
  }
  const uint32_t k = dist_key(bv), mk = __reduce_min_sync(0xffffffffu, k);
  arg = (int)__reduce_min_sync(0xffffffffu, k == mk ? (uint32_t)bj : 0x7fffffffu);
  return mk;
}

// Thread t owns rows t + kWardNT m: the smallest entry of the row's pairs
// (rmin, rarg) and the cluster's size stay in its registers.  A merge needs one
// block barrier, the one of the arg-min over the rows:
//   - thread k updates D(a, k) and its own row's column a, and puts +inf into
//     its own row's column b, so a scan of a row asks for no flags;
//   - a row whose minimum was at a or b is rescanned: its entries are its own
//     thread's writes of this step and writes of earlier steps;
//   - row a is not rescanned: every pair (a, k) was just compared with row k's
//     minimum, so row a only has to stand for pairs with rows merged later,
//     which compare themselves with it (a pair is always held by one of its
//     two rows, with its value and the smaller column at ties, so the minimum
//     over the rows is the pair of the order above).
// With D in shared memory (kShared, up to 238 points) a rescan is done by the row's own warp;
// else D stays in global memory (L1 / L2) and the rescans are shared by all
// warps through a list, for two more barriers.
// What bounds it: the chain of a merge, two redux.sync rounds, the barrier, the
// update's loads and division and a rescan.  (D and all state in global memory
// and five barriers a merge: the call 907 us at 200 points, against 194; 3.33 ms
// against 0.80 at 400, 12.1 against 2.31 at 800, 747 against 183 at 6,000.)
template <int R, bool kShared>
__global__ void __launch_bounds__(kWardNT, 1) ward_merge_kernel(int32_t* hdr, float* Dg, int n, int32_t* merge,
                                                                float* height, int32_t* size_out) {
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ uint2 s_best[2][32];
  __shared__ int s_cnt[2];
  const int t = threadIdx.x, lane = t & 31, wid = t >> 5;
  const int ld = kShared ? n | 1 : n;
  float* res_v = reinterpret_cast<float*>(smem);  // rows' scans: value, column
  float* Ds = res_v + n;                          // kShared
  uint16_t* res_j = reinterpret_cast<uint16_t*>(kShared ? Ds + (size_t)n * ld : Ds);
  uint16_t* list = res_j + n;
  uint16_t* csize = list + n;
  uint16_t* cid = csize + n;  // < 2 n - 1
  float* D = kShared ? Ds : Dg;
  if (kShared)
    for (int i = wid; i < n; i += kWardNT / 32)
      for (int j = lane; j < n; j += 32) D[i * ld + j] = Dg[(size_t)i * n + j];
  for (int i = t; i < n; i += kWardNT) {
    csize[i] = 1;
    cid[i] = (uint16_t)i;
  }
  if (t < 2) s_cnt[t] = 0;
  __syncthreads();
  for (int i = wid; i < n; i += kWardNT / 32) {
    int j;
    const uint32_t k = warp_row_min(D + (size_t)i * ld, n, lane, j);
    if (lane == 0) {
      res_v[i] = key_dist(k);
      res_j[i] = (uint16_t)(k < kInfKey ? j : 0xffff);
    }
  }
  __syncthreads();
  // with D in shared memory only the warps that own rows go on, and one that
  // writes the linkage beside them
  const int nw = kShared ? (n + 31) >> 5 : kWardNT / 32, n_sync = 32 * (kShared ? nw + 1 : nw);
  if (kShared && wid > nw) return;
  const bool recorder = t == (kShared ? 32 * nw : 0);
  float rmin[R];
  int rarg[R], nk[R];  // nk 0: retired
#pragma unroll
  for (int m = 0; m < R; ++m) {
    const int k = t + kWardNT * m;
    nk[m] = k < n ? 1 : 0;
    rmin[m] = k < n ? res_v[k] : CUDART_INF_F;
    rarg[m] = k < n && res_j[k] != 0xffff ? (int)res_j[k] : -1;
  }
  int la = -1, ls = 0;  // the last merge's slot and size (csize[la] is written a step later)
  for (int step = 0; step < n - 1; ++step) {
    const int par = step & 1;
    uint32_t bk = 0xffffffffu, bp = 0xffffffffu;
#pragma unroll
    for (int m = 0; m < R; ++m)
      if (rarg[m] >= 0) {
        const int k = t + kWardNT * m;
        const uint32_t q = dist_key(rmin[m]), pr = ((uint32_t)min(k, rarg[m]) << 16) | (uint32_t)max(k, rarg[m]);
        if (q < bk || (q == bk && pr < bp)) {
          bk = q;
          bp = pr;
        }
      }
    uint32_t mk = __reduce_min_sync(0xffffffffu, bk);
    uint32_t mp = __reduce_min_sync(0xffffffffu, bk == mk ? bp : 0xffffffffu);
    if (lane == 0) s_best[par][wid] = make_uint2(mk, mp);
    bar_sync(1, n_sync);
    const uint2 best = lane < nw ? s_best[par][lane] : make_uint2(0xffffffffu, 0xffffffffu);
    mk = __reduce_min_sync(0xffffffffu, best.x);
    mp = __reduce_min_sync(0xffffffffu, best.x == mk ? best.y : 0xffffffffu);
    if (mk >= kInfKey) {  // no finite distance left: NaN or overflow in the points
      if (recorder && atomicCAS(&hdr[0], 0, 6 /* CF_ERR_NUMERIC */) == 0) hdr[1] = step;
      return;
    }
    const int a = (int)(mp >> 16), b = (int)(mp & 0xffffu);
    const float dab = key_dist(mk);
    const int na = a == la ? ls : csize[a], nb = b == la ? ls : csize[b];
    float* Da = D + (size_t)a * ld;
    const float* Db = D + (size_t)b * ld;
    unsigned flags = 0;
#pragma unroll
    for (int m = 0; m < R; ++m) {
      const int k = t + kWardNT * m;
      if (nk[m] == 0) continue;
      if (k == a || k == b) {
        if (k == a) Da[b] = CUDART_INF_F;
        nk[m] = k == a ? na + nb : 0;
        rmin[m] = CUDART_INF_F;
        rarg[m] = -1;
        continue;
      }
      const float fk = (float)nk[m];
      const float dak = Da[k], dbk = Db[k];
      const float v = (((float)na + fk) * dak + ((float)nb + fk) * dbk - fk * dab) / ((float)(na + nb) + fk);
      Da[k] = v;
      D[(size_t)k * ld + a] = v;
      D[(size_t)k * ld + b] = CUDART_INF_F;
      if (rarg[m] == a || rarg[m] == b) {
        flags |= 1u << m;  // its minimum may have moved
      } else if (v < rmin[m] || (v == rmin[m] && a < rarg[m])) {
        rmin[m] = v;
        rarg[m] = a;
      }
    }
    if (recorder) {
      if (la >= 0) csize[la] = (uint16_t)ls;
      const int ca = cid[a], cb = cid[b];
      cid[a] = (uint16_t)(n + step);
      merge[2 * step] = min(ca, cb);
      merge[2 * step + 1] = max(ca, cb);
      height[step] = sqrtf(fmaxf(dab, 0.f));
      size_out[step] = na + nb;
    }
    la = a;
    ls = na + nb;
    if constexpr (kShared) {
      static_assert(R == 1, "a row per thread");
      __syncwarp();
      for (unsigned rows = __ballot_sync(0xffffffffu, flags != 0); rows; rows &= rows - 1) {
        const int l = __ffs(rows) - 1;
        int j;
        const uint32_t k = warp_row_min(D + (32 * wid + l) * ld, n, lane, j);
        if (lane == l) {
          rmin[0] = key_dist(k);
          rarg[0] = k < kInfKey ? j : -1;
        }
      }
    } else {
      int at[R];
#pragma unroll
      for (int m = 0; m < R; ++m)
        if (flags >> m & 1u) {
          at[m] = atomicAdd(&s_cnt[par], 1);
          list[at[m]] = (uint16_t)(t + kWardNT * m);
        }
      if (t == 0) s_cnt[par ^ 1] = 0;  // last read before this step's first barrier
      __syncthreads();
      const int cnt = s_cnt[par];
      if (cnt == 0) continue;
      for (int q = wid; q < cnt; q += kWardNT / 32) {
        int j;
        const uint32_t k = warp_row_min(D + (size_t)list[q] * ld, n, lane, j);
        if (lane == 0) {
          res_v[q] = key_dist(k);
          res_j[q] = (uint16_t)(k < kInfKey ? j : 0xffff);
        }
      }
      __syncthreads();
#pragma unroll
      for (int m = 0; m < R; ++m)
        if (flags >> m & 1u) {
          rmin[m] = res_v[at[m]];
          rarg[m] = res_j[at[m]] != 0xffff ? (int)res_j[at[m]] : -1;
        }
    }
  }
}

size_t ward_smem(int n, bool shared) {
  return 12 * (size_t)n + (shared ? 4 * (size_t)n * (n | 1) : 0);
}

cudaError_t launch_ward(int32_t* hdr, const float* points, int n, int dim, float* D, int32_t* merge, float* height,
                        int32_t* size, cudaStream_t st) {
  static DeviceOnce once;
  int dev = 0;
  const cudaError_t e = once.run([](int) {
    cudaError_t r = cudaSuccess;
    for (const void* f : {(const void*)ward_merge_kernel<1, true>, (const void*)ward_merge_kernel<1, false>,
                          (const void*)ward_merge_kernel<4, false>, (const void*)ward_merge_kernel<16, false>})
      if (r == cudaSuccess) r = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kWardSmem);
    return r;
  }, &dev);
  if (e != cudaSuccess) return e;
  const unsigned tiles = (unsigned)((n + 15) / 16);
  ward_dist_kernel<<<dim3(tiles, tiles), 256, 0, st>>>(points, n, dim, D);
  const bool shared = ward_smem(n, true) <= kWardSmem;
  const size_t sm = ward_smem(n, shared);
  if (shared)
    ward_merge_kernel<1, true><<<1, kWardNT, sm, st>>>(hdr, D, n, merge, height, size);
  else if (n <= kWardNT)
    ward_merge_kernel<1, false><<<1, kWardNT, sm, st>>>(hdr, D, n, merge, height, size);
  else if (n <= 4 * kWardNT)
    ward_merge_kernel<4, false><<<1, kWardNT, sm, st>>>(hdr, D, n, merge, height, size);
  else
    ward_merge_kernel<16, false><<<1, kWardNT, sm, st>>>(hdr, D, n, merge, height, size);
  return cudaGetLastError();
}

// S[a][b] = score of pair (a, b), and S[b][a] when symmetric; S zeroed first.
__global__ void zero_kernel(float* S, size_t m) {
  for (size_t e = (size_t)blockIdx.x * blockDim.x + threadIdx.x; e < m; e += (size_t)gridDim.x * blockDim.x) S[e] = 0.f;
}

__global__ void scatter_scores_kernel(const int32_t* pairs, const float* scores, int P, int n_rows, int n_cols,
                                      int symmetric, float* S, int32_t* bad) {
  const int p = blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= P) return;
  const int a = pairs[2 * p], b = pairs[2 * p + 1];
  if (a < 0 || a >= n_rows || b < 0 || b >= n_cols || (symmetric && (b >= n_rows || a >= n_cols))) {
    atomicCAS(bad, 0, p + 1);
    return;
  }
  S[(size_t)a * n_cols + b] = scores[p];
  if (symmetric) S[(size_t)b * n_cols + a] = scores[p];
}

void set_err(const char* m) { set_error_detail(m); }

}  // namespace

}  // namespace cfsim

using namespace cfsim;

extern "C" {

cf_status cf_ward_ws_size(int32_t n, size_t* bytes) {
  if (!bytes || n < 1 || n > kWardMaxN) {
    set_err("cf_ward_ws_size: need 1 <= n <= 16384 and bytes");
    return CF_ERR_INVALID_ARG;
  }
  *bytes = ward_layout(n).total;
  set_err("");
  return CF_OK;
}

cf_status cf_ward(const float* d_points, int32_t n, int32_t dim, int32_t* d_merge, float* d_height, int32_t* d_size,
                  void* d_ws, size_t ws_bytes, cf_stream_t stream) {
  if (n < 1 || n > kWardMaxN || dim < 1 || !d_points || !d_ws || (n > 1 && (!d_merge || !d_height || !d_size))) {
    set_err("cf_ward: need 1 <= n <= 16384, dim >= 1 and non-NULL buffers");
    return CF_ERR_INVALID_ARG;
  }
  const WardLayout L = ward_layout(n);
  if (ws_bytes < L.total) {
    set_err("cf_ward: workspace too small (see cf_ward_ws_size)");
    return CF_ERR_WORKSPACE;
  }
  cudaStream_t st = (cudaStream_t)stream;
  char* base = static_cast<char*>(d_ws);
  int32_t* hdr = reinterpret_cast<int32_t*>(base + L.hdr);
  cudaError_t e = cudaMemsetAsync(hdr, 0, 64, st);
  if (e == cudaSuccess && n > 1)
    e = launch_ward(hdr, d_points, n, dim, reinterpret_cast<float*>(base + L.D), d_merge, d_height, d_size, st);
  if (e != cudaSuccess) {
    char buf[256];
    snprintf(buf, sizeof buf, "cf_ward: %s", cudaGetErrorString(e));
    set_err(buf);
    return CF_ERR_CUDA;
  }
  set_err("");
  return CF_OK;
}

cf_status cf_score_matrix(const int32_t* d_pairs, const float* d_scores, int32_t P, int32_t n_rows, int32_t n_cols,
                          int32_t symmetric, float* d_S, int32_t* d_status, cf_stream_t stream) {
  if (P < 0 || n_rows < 1 || n_cols < 1 || !d_S || !d_status || (P > 0 && (!d_pairs || !d_scores)) ||
      (symmetric && n_rows != n_cols)) {
    set_err("cf_score_matrix: bad sizes or NULL buffer (symmetric needs n_rows == n_cols)");
    return CF_ERR_INVALID_ARG;
  }
  cudaStream_t st = (cudaStream_t)stream;
  const size_t m = (size_t)n_rows * n_cols;
  cudaError_t e = cudaMemsetAsync(d_status, 0, sizeof(int32_t), st);
  if (e == cudaSuccess) {
    zero_kernel<<<(unsigned)std::min<size_t>((m + 255) / 256, 4096), 256, 0, st>>>(d_S, m);
    if (P > 0) scatter_scores_kernel<<<(P + 255) / 256, 256, 0, st>>>(d_pairs, d_scores, P, n_rows, n_cols, symmetric, d_S, d_status);
    e = cudaGetLastError();
  }
  if (e != cudaSuccess) {
    char buf[256];
    snprintf(buf, sizeof buf, "cf_score_matrix: %s", cudaGetErrorString(e));
    set_err(buf);
    return CF_ERR_CUDA;
  }
  set_err("");
  return CF_OK;
}

}  // extern "C"
