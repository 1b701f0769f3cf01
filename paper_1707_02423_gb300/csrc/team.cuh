// The team tier: pairs too large for one CTA's shared memory, each on a team
// of the persistent kernel's CTAs.
//
// A pair's iterates live in a scratch slot of the workspace (L2, or HBM
// beyond it); the team's CTAs each own a slab of consecutive rows and meet at
// one barrier per iteration, which also carries the norm.  What bounds the
// tier is the traffic of the gathers (L1 and L2), so
//   - a pair is given enough CTAs that few pairs are in flight and their
//     iterates stay in L2: with one CTA per pair, 152 pairs of 1,250 blocks
//     hold 2.9 GB and every iteration streams HBM;
//   - the columns are stored in an order of their own: first the blocks with
//     at most one out- and one in-neighbour (about 70 % of a CFG's blocks),
//     then those with at most two, then the busy ones.  A warp's 32 columns
//     then need the same number of loads, two per entry instead of the eight
//     of the padded 2 x 2 gather where row and column are both of the first
//     kind.  Rows need no order in memory: a warp's lanes share a row, so the
//     sweep takes each slab's rows kind by kind;
//   - each column's lists are staged once per pair, each slab's row records
//     too, so a gather is one load at a known address.
#pragma once

#include "device_common.cuh"
#include "iterate.cuh"

namespace cfsim {

namespace {

// Chunks of 32 columns and the wpr warps of a row: warp cw owns the chunks cw,
// cw + wpr, ... of the columns in order of kind (so that every warp has its
// share of the dearer ones), and they are stored side by side: first the warps
// that own one chunk fewer, then the others, so that there is no gap and the
// last chunk, which may be partly filled, comes last.
__host__ __device__ __forceinline__ int chunk_first(int cw, int nch, int wpr) {
  const int most = (nch + wpr - 1) / wpr, full = nch - wpr * (most - 1);  // `full` warps own `most`
  return cw >= full ? (cw - full) * (most - 1) : (wpr - full) * (most - 1) + cw * most;
}
// How the consumer warps share a row of nch chunks: CH chunks per warp, rg rows
// at a time -- the least (fixed cost of a row + its chunks) / rows, the fixed
// cost (the row's records, the step's barriers) being about that of a chunk.
__host__ __device__ __forceinline__ void team_split(int nch, int NC, int& CH, int& wpr, int& rg) {
  int best = 0x7fffffff;
  CH = wpr = rg = 1;
  for (int c = 1; c <= 8; ++c) {
    const int p = (nch + c - 1) / c;
    if (p > NC) continue;
    const int g = NC / p, cost = 64 * (c + 1) / g;
    if (cost < best) {
      best = cost;
      CH = c;
      wpr = p;
      rg = g;
    }
    if (c >= 4) break;  // more chunks per warp only where a row needs them
  }
  if (best == 0x7fffffff) {
    CH = (nch + NC - 1) / NC;
    wpr = (nch + CH - 1) / CH;
    rg = NC / wpr;
  }
}

// What the sweep needs of a pair (in shared memory).  Addresses of shared
// memory are 32-bit (ld.shared, not generic loads).
struct TeamStage {
  const int4* cA;         // per column in order of kind: {4 out 0, weight, 4 in 0, weight} (positions), in the
                          // ring's place until the warps have read them
  const int4* brow;       // per busy row of the whole row graph: its out- and in-ranges in redge
  const uint32_t* browo;  // its 4 ld row
  const int2* redge;      // {4 ld neighbour, weight}
  uint16_t* src;          // per copy: its first row, bit 15: of E
  uint16_t* buf;          // its first buffer
  uint16_t* cnt;          // its rows
  uint16_t* req;          // steps that must be done before it
  uint16_t* stp;          // the step that needs it first
  uint16_t* first;        // per step (and the end): its first copy
  uint16_t* rows;         // per step: rows its copies bring
  uint32_t blane;         // per lane of the busy columns' warps: {column, first entry (byte address), entries |
                          // direction << 8, lanes of the column from this one on}
  int blanes;             // lanes in use (0: the lists are walked)
  uint32_t cb;            // second neighbours by column in order of kind (from the first chunk that has any on)
  uint32_t bran;          // per busy column: its out- and in-ranges in cedge (byte addresses)
  uint32_t cedge;         // {4 position, weight}
  uint32_t rec;           // per slab row that is not busy, 48 bytes: buffers {out 0, in 0, out 1, in 1} (byte
                          // addresses), their weights, {buffer of its E row, 4 ld row}
  uint32_t full;          // mbarriers of the steps: their rows have arrived
  uint32_t empty;         // and: every warp is past them
  uint32_t ring;
  uint32_t rowb;          // bytes of a row buffer
  int S;                  // buffers
  int n0, nnb, nb;        // columns of the first kind, not busy, busy
  int nr;                 // the slab's rows that are not busy
  int nbr;                // busy rows of the row graph
  int rps, nsteps, ncopy; // rows per step, steps, copies of an iteration
  int nch, wpr, rg;       // column chunks, consumer warps per row, rows at a time
};

// Per-CTA state of the team tier.
struct TeamSh {
  float redw[64];  // per-warp partials (two parities for the fallback matching's sums)
  int redi[64];
  float tot;
  uint32_t gen;    // level << kTeamGenBits | barriers passed in it
  int fail;        // a wait ran out: the CTA waits no more and leaves the kernel
  uint64_t wait;   // longest wait (team_wait_ns)
  int n0, nb, tb, tbp;           // columns: first kind, busy, list entries of the busy ones
  int nbs, nbr, tr, trp;         // busy rows, their list entries
  uint64_t red[32];      // per-warp maxima
  uint2 step[2][8];      // per-warp best heads of a matching step: key, low word
  int pre[8][32];        // per-warp counts of the listed rows
  int bin, nl, ids;
  uint32_t mine[16][8];  // per consumer warp and chunk: the busy rows it does
  TeamStage st;
};

constexpr int kTeamGenBits = 28;
struct Team {
  int c, T;         // this CTA's index in the team, CTAs of the team
  uint64_t* slots;  // barrier words of the team's CTAs, parity 0 (parity 1: kTeamMaxCta words on)
  WsHeader* hdr;
};

__device__ __forceinline__ uint64_t ld_relaxed_u64(const uint64_t* p) {
  uint64_t v;
  asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ void st_release_u64(uint64_t* p, uint64_t v) {
  asm volatile("st.release.gpu.global.u64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}
__device__ __forceinline__ void fence_gpu() { asm volatile("fence.acq_rel.gpu;" ::: "memory"); }
__device__ __forceinline__ uint64_t global_ns() {
  uint64_t t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

// Waits are bounded: for another CTA of the team (the CTAs are co-resident, the
// kernel being launched cooperatively) by team_wait_over, within the CTA by the
// same time.  One that runs out sets CF_ERR_TIMEOUT; the CTA then takes no
// further part, as what it read may be unfinished: it leaves the pair without
// using any of it as an index, and the kernel.

// Sum of v over every thread of the team, the same bits on every thread, and
// a barrier: what any thread of the team wrote before is visible to all of
// them after.  Each CTA publishes {barrier number, its sum} in one 64-bit
// word and reads every other CTA's: one trip through L2, no counter.  The
// words alternate by parity; a CTA writes its next word of the same parity
// only after all have passed the barrier in between.
__device__ __forceinline__ float team_sum(const Team& tm, TeamSh& sh, float v) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, NW = blockDim.x >> 5;
  v = warp_sum(v);
  if (lane == 0) sh.redw[w] = v;
  __syncthreads();
  if (w == 0) {
    float x = warp_sum(lane < NW ? sh.redw[lane] : 0.f);
    if (tm.T > 1) {
      const uint32_t want = sh.gen + 1;
      uint64_t* s = tm.slots + (size_t)(want & 1) * kTeamMaxCta;
      if (lane == 0) {
        fence_gpu();
        st_release_u64(s + tm.c, ((uint64_t)want << 32) | __float_as_uint(x));
      }
      x = 0.f;
      for (int k = lane; k < tm.T; k += 32) {
        uint64_t got = ld_relaxed_u64(s + k);
        if ((uint32_t)(got >> 32) != want && !sh.fail) {
          TeamWait wait{global_ns(), got};
          for (uint32_t n = 0;; ++n) {
            got = ld_relaxed_u64(s + k);
            if ((uint32_t)(got >> 32) == want) break;
            if ((n & 255u) == 255u && team_wait_over(wait, global_ns(), got, sh.wait)) {
              set_status(tm.hdr, 5 /* CF_ERR_TIMEOUT */, tm.c);
              sh.fail = 1;
              break;
            }
          }
        }
        x += __uint_as_float((uint32_t)got);
      }
      fence_gpu();
      x = warp_sum(x);
      __syncwarp();
      if (lane == 0) sh.gen = want;
    }
    if (lane == 0) sh.tot = x;
  }
  __syncthreads();
  return sh.tot;
}

// Largest a and largest b over the CTA, as a << 32 | b.
template <int NW>
__device__ __forceinline__ uint64_t block_max2(TeamSh& sh, uint32_t a, uint32_t b, int lane, int w) {
  a = __reduce_max_sync(0xffffffffu, a);
  b = __reduce_max_sync(0xffffffffu, b);
  __syncthreads();
  if (lane == 0) sh.red[w] = ((uint64_t)a << 32) | b;
  __syncthreads();
  const uint64_t v = lane < NW ? sh.red[lane] : 0ull;
  a = __reduce_max_sync(0xffffffffu, (uint32_t)(v >> 32));
  b = __reduce_max_sync(0xffffffffu, (uint32_t)v);
  return ((uint64_t)a << 32) | b;
}

// Largest v over the CTA.
template <int NW>
__device__ __forceinline__ uint64_t block_max_u64(TeamSh& sh, uint64_t v, int lane, int w) {
  uint32_t hi = __reduce_max_sync(0xffffffffu, (uint32_t)(v >> 32));
  uint32_t lo = __reduce_max_sync(0xffffffffu, (uint32_t)(v >> 32) == hi ? (uint32_t)v : 0u);
  __syncthreads();
  if (lane == 0) sh.red[w] = ((uint64_t)hi << 32) | lo;
  __syncthreads();
  v = lane < NW ? sh.red[lane] : 0ull;
  hi = __reduce_max_sync(0xffffffffu, (uint32_t)(v >> 32));
  lo = __reduce_max_sync(0xffffffffu, (uint32_t)(v >> 32) == hi ? (uint32_t)v : 0u);
  return ((uint64_t)hi << 32) | lo;
}

// A team's last barrier on a level: afterwards its CTAs may join other teams.
// No value is read, so a word that its CTA has already moved on with, which is
// larger, counts as well.
__device__ __forceinline__ void team_leave(const Team& tm, TeamSh& sh) {
  const int lane = threadIdx.x & 31;
  __syncthreads();
  if (tm.T > 1 && threadIdx.x < 32) {
    const uint32_t want = sh.gen + 1;
    uint64_t* s = tm.slots + (size_t)(want & 1) * kTeamMaxCta;
    if (lane == 0) {
      fence_gpu();
      st_release_u64(s + tm.c, (uint64_t)want << 32);
    }
    for (int k = lane; k < tm.T; k += 32) {
      uint64_t got = ld_relaxed_u64(s + k);
      TeamWait wait{global_ns(), got};
      while ((uint32_t)(got >> 32) < want && !*reinterpret_cast<volatile int*>(&sh.fail)) {
        if (team_wait_over(wait, global_ns(), got, sh.wait)) {
          set_status(tm.hdr, 5 /* CF_ERR_TIMEOUT */, tm.c);
          *reinterpret_cast<volatile int*>(&sh.fail) = 1;
        }
        got = ld_relaxed_u64(s + k);
      }
    }
    __syncwarp();
  }
  __syncthreads();
}

// Exclusive prefix counts of two bit masks over `words` words (warp 0), and
// their totals.
__device__ __forceinline__ void mask_prefix(const uint32_t* m0, const uint32_t* mb, uint32_t* p0, uint32_t* pb,
                                            int words, int lane, int* t0, int* tb) {
  uint32_t r0 = 0, rb = 0;
  for (int k = 0; k < words; k += 32) {
    const bool in = k + lane < words;
    uint32_t a = in ? __popc(m0[k + lane]) : 0u, b = in ? __popc(mb[k + lane]) : 0u;
    const uint32_t a0 = a, b0 = b;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t ua = __shfl_up_sync(0xffffffffu, a, o), ub = __shfl_up_sync(0xffffffffu, b, o);
      if (lane >= o) {
        a += ua;
        b += ub;
      }
    }
    if (in) {
      p0[k + lane] = r0 + a - a0;
      pb[k + lane] = rb + b - b0;
    }
    r0 += __shfl_sync(0xffffffffu, a, 31);
    rb += __shfl_sync(0xffffffffu, b, 31);
  }
  if (lane == 0) {
    *t0 = (int)r0;
    *tb = (int)rb;
  }
}

// Bit masks of the row graph's busy rows (more than two out- or in-neighbours),
// twice.
template <int NW>
__device__ __forceinline__ void row_masks(const Geo& g, int n_row, int words, uint32_t* m0, uint32_t* mb, int lane,
                                          int w) {
  for (int wd = w; wd < words; wd += NW) {
    const int i = 32 * wd + lane;
    const bool busy = i < n_row && (__ldg(g.r_optr + i + 1) - __ldg(g.r_optr + i) > 2 ||
                                    __ldg(g.r_iptr + i + 1) - __ldg(g.r_iptr + i) > 2);
    const unsigned m = __ballot_sync(0xffffffffu, busy);
    if (lane == 0) m0[wd] = mb[wd] = m;
  }
}

// ---- the sweep: rows through a ring in shared memory -----------------------
//
// A slab's rows are swept in order, and every row they gather from comes
// through a ring of row buffers that one warp keeps filling with bulk copies
// (cp.async.bulk, whole rows, up to the ring's depth in flight).  The gathers
// then read shared memory at known addresses, and no warp ever waits for L2 or
// HBM itself: with the gathers going to global memory the sweep kept too few
// loads in flight (1.0 entries per ns and SM, issue slots 25 % used, half the
// stalls on loads).
//   - The order of the copies and the buffer each gather reads are worked out
//     once per pair (team_schedule): copy l goes to buffer l mod S; a row still
//     in the ring is not copied again (row i is needed at rows i - 1 and i + 1,
//     so most are copied once).
//   - Consumer warps own 32-column chunks, whose lists they hold in registers
//     for the whole pair.  After each step (one row, or several where a row has
//     few chunks) a warp publishes its progress; the copying warp reuses a
//     buffer when every warp is past the last step that reads it.
//   - Consecutive rows that go to consecutive buffers are one copy.
//   - Busy columns (lists of up to dozens of neighbours) have warps of their
//     own: a lane keeps up to four entries of one column's list in registers
//     for the whole pair, and a column's lanes add up by shuffles.  (Walking the
//     lists in shared memory at every row took 1.5 us a row, four times the
//     other warps' row, and held up the ring.)
//   - Busy rows (the STOP block collects an edge from every early return) are
//     shared out over the team chunk by chunk and gather from global memory,
//     while the ring fills.  (Left to their slab's CTA, the STOP x STOP entry
//     alone, 2,200 terms, took most of a 45 us iteration of a 1,371 x 1,998
//     pair.)
constexpr int kBusyWarps = 3;
constexpr int kBusyPer = 4;      // list entries of a busy column per lane
template <int NT>
constexpr int kConsumers = NT / 32 - kBusyWarps - 1 < 16 ? NT / 32 - kBusyWarps - 1 : 16;
constexpr int kMaxChunks = 8;    // chunks a consumer warp may own
constexpr int kMinRing = 12;     // row buffers (one row per step needs at most five at a time)
constexpr int kMaxRing = 256;
constexpr int kStepRing = 32;    // step barriers

__device__ __forceinline__ float ldb(const float* Y, uint32_t off) {
  return *reinterpret_cast<const float*>(reinterpret_cast<const char*>(Y) + off);
}
__device__ __forceinline__ void stb(float* Y, uint32_t off, float v) {
  *reinterpret_cast<float*>(reinterpret_cast<char*>(Y) + off) = v;
}
__device__ __forceinline__ float lds32(uint32_t a) {
  float v;
  asm volatile("ld.shared.f32 %0, [%1];" : "=f"(v) : "r"(a));
  return v;
}
__device__ __forceinline__ void fence_async() { asm volatile("fence.proxy.async;" ::: "memory"); }
// Records, written before the sweep starts: no ordering needed.
__device__ __forceinline__ int4 lds_rec4(uint32_t a) {
  int4 v;
  asm("ld.shared.v4.b32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(a));
  return v;
}
__device__ __forceinline__ int2 lds_rec2(uint32_t a) {
  int2 v;
  asm("ld.shared.v2.b32 {%0, %1}, [%2];" : "=r"(v.x), "=r"(v.y) : "r"(a));
  return v;
}
__device__ __forceinline__ bool mbar_try(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(bar), "r"(parity)
      : "memory");
  return ok != 0;
}
// (does not suspend the thread, as a try_wait may)
__device__ __forceinline__ bool mbar_test(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\tmbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(bar), "r"(parity)
      : "memory");
  return ok != 0;
}

// A place in the steps: barrier of the next one and its parity.
struct RingPos {
  uint32_t at, parity;
  __device__ __forceinline__ void next() {
    if (++at == (uint32_t)kStepRing) {
      at = 0;
      parity ^= 1u;
    }
  }
};

// Waits (bounded) until the copies of the next step have arrived.
__device__ __noinline__ void ring_slow_wait(TeamSh& sh, WsHeader* hdr, uint32_t bar, uint32_t parity) {
  const uint64_t t0 = global_ns();
  for (uint32_t n = 0; !mbar_try(bar, parity); ++n) {
    if (*reinterpret_cast<volatile int*>(&sh.fail)) break;
    if ((n & 255u) == 255u && global_ns() - t0 > sh.wait) {
      set_status(hdr, 5 /* CF_ERR_TIMEOUT */, -2);
      *reinterpret_cast<volatile int*>(&sh.fail) = 1;
      break;
    }
  }
}
__device__ __forceinline__ void ring_wait(TeamSh& sh, WsHeader* hdr, uint32_t full, const RingPos& p) {
  if (!mbar_try(full + 8u * p.at, p.parity)) ring_slow_wait(sh, hdr, full + 8u * p.at, p.parity);
}
// (an arrival, not a released flag: a store with release order waited for the
// step's global stores)
__device__ __forceinline__ void ring_done(uint32_t empty, RingPos& p, int lane) {
  __syncwarp();
  if (lane == 0) asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(empty + 8u * p.at) : "memory");
  p.next();
}

// The copying warp's iteration: Y = the iterate gathered from; fill / done =
// the next step to bring and the next to be done, over all iterations.
__device__ __forceinline__ void ring_fill(const TeamStage& st, TeamSh& sh, WsHeader* hdr, const float* Y,
                                          const float* eb, uint32_t base, RingPos& dp, int lane) {
  fence_async();  // the rows were written through the generic proxy
  uint64_t t0 = 0;
  uint32_t spins = 0;
  const int ncopy = st.ncopy, nsteps = st.nsteps;
  const uint32_t rowb = st.rowb, full = st.full, empty = st.empty;
  int done = 0;
  for (int at = 0; at < ncopy;) {
    while (done < nsteps && __all_sync(0xffffffffu, mbar_test(empty + 8u * dp.at, dp.parity))) {
      ++done;
      dp.next();
    }
    const int l = at + lane, step = l < ncopy ? st.stp[l] : 0;
    const bool ok = l < ncopy && (int)st.req[l] <= done && step - kStepRing + 1 <= done;
    const unsigned m = __ballot_sync(0xffffffffu, ok);
    const int n = m == 0xffffffffu ? 32 : __ffs(~m) - 1;  // in order
    if (n > 0) {
      const uint32_t bar = full + 8u * ((base + (uint32_t)step) % (uint32_t)kStepRing);
      if (lane < n && st.first[step] == l) {
        const uint32_t bytes = (uint32_t)st.rows[step] * rowb;
        asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
      }
      __syncwarp();
      if (lane < n) {
        const uint32_t dst = st.ring + (uint32_t)st.buf[l] * rowb, s = st.src[l];
        const char* from = reinterpret_cast<const char*>(s & 0x8000u ? eb : Y) + (size_t)(s & 0x7fffu) * rowb;
        asm volatile(
            "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst),
            "l"(from), "r"((uint32_t)st.cnt[l] * rowb), "r"(bar)
            : "memory");
      }
      __syncwarp();
      at += n;
      spins = 0;
    } else {
      if (spins == 0) t0 = global_ns();
      if ((++spins & 1023u) == 0u && global_ns() - t0 > sh.wait && lane == 0) {
        set_status(hdr, 5 /* CF_ERR_TIMEOUT */, -3);
        *reinterpret_cast<volatile int*>(&sh.fail) = 1;
      }
      __syncwarp();
      if (__any_sync(0xffffffffu, *reinterpret_cast<volatile int*>(&sh.fail))) break;
    }
  }
  __syncwarp();
  for (; done < nsteps; ++done) {  // the steps still being done
    if (!mbar_try(empty + 8u * dp.at, dp.parity)) ring_slow_wait(sh, hdr, empty + 8u * dp.at, dp.parity);
    dp.next();
  }
}

// The rows an iteration brings into the ring, in the order the steps need
// them, the buffers each row reads, and the copies (one warp).  A step's E rows
// come first, a lane per row; then, row by row, lanes 1..4 look at its
// neighbours out 0, in 0, out 1, in 1.  last: per row of the row graph the
// newest place it was brought to, -1 at first.  A row brought earlier is read
// again only if it is recent (a third of the ring): an older one would keep
// the ring from running ahead (rows of 2,000 entries: 1.2 us instead of
// 0.3 us each), and at most S - 5 rps places old, so that nothing the step
// brings takes its buffer.
__device__ __forceinline__ void team_schedule(TeamStage& st, int4* rec, int16_t* last, uint16_t* use,
                                              uint16_t* what, int lane) {
  int next = 0, copies = 0;
  const int S = st.S, rps = st.rps, nr = st.nr, nsteps = st.nsteps;
  for (int step = 0; step < nsteps; ++step) {
    // places below this one may be gone, or would hold up the copies to come:
    // a place read at this step keeps the copy S places on waiting
    const int keep = max(next + 5 * rps - S, next - max(S / 3, 5 * rps));
    const int r0 = step * rps, r1 = min(nr, r0 + rps), start = next;
    if (lane < r1 - r0) {
      const int l = next + lane;
      what[l] = (uint16_t)(0x8000 | rec[3 * (r0 + lane) + 2].x);
      use[l] = (uint16_t)step;
      rec[3 * (r0 + lane) + 2].x = (int)(st.ring + (uint32_t)(l % S) * st.rowb);
    }
    next += r1 - r0;
    for (int r = r0; r < r1; ++r) {
      // rows as left by the staging: neighbours (-1: none) in the buffers' place
      const int u = lane >= 1 && lane < 5 ? reinterpret_cast<const int*>(rec + 3 * r)[lane - 1] : -1;
      const unsigned same = __match_any_sync(0xffffffffu, u);
      int l = u >= 0 ? last[u] : -1;
      const bool fresh = u >= 0 && l < max(keep, 0) && __ffs(same) - 1 == lane;
      const unsigned m = __ballot_sync(0xffffffffu, fresh);
      if (fresh) {
        l = next + __popc(m & ((1u << lane) - 1u));
        what[l] = (uint16_t)u;
        last[u] = (int16_t)l;
      }
      l = __shfl_sync(0xffffffffu, l, __ffs(same) - 1);
      next += __popc(m);
      if (u >= 0) use[l] = (uint16_t)step;
      if (lane >= 1 && lane < 5)  // a missing neighbour (weight 0) reads the row's E
        reinterpret_cast<int*>(rec + 3 * r)[lane - 1] =
            u >= 0 ? (int)(st.ring + (uint32_t)(l % S) * st.rowb) : rec[3 * r + 2].x;
      __syncwarp();
    }
    // runs of consecutive rows in consecutive buffers become one copy
    if (lane == 0) {
      st.first[step] = (uint16_t)copies;
      st.rows[step] = (uint16_t)(next - start);
    }
    for (int l0 = start; l0 < next; l0 += 32) {
      const int l = l0 + lane;
      const bool in = l < next;
      const int me = in ? what[l] : 0, before = in && l > start ? what[l - 1] : -2;
      const bool head = in && (me != before + 1 || l % S == 0);
      const unsigned m = __ballot_sync(0xffffffffu, head);
      if (head) {
        const int c = copies + __popc(m & ((1u << lane) - 1u));
        st.src[c] = (uint16_t)me;
        st.buf[c] = (uint16_t)(l % S);
        st.cnt[c] = (uint16_t)l;  // its first place, for now
        st.stp[c] = (uint16_t)step;
      }
      copies += __popc(m);
    }
    __syncwarp();
  }
  if (lane == 0) {
    st.first[nsteps] = (uint16_t)copies;
    st.ncopy = copies;
  }
  __syncwarp();
  for (int c0 = 0; c0 < copies; c0 += 32) {
    const int c = c0 + lane;
    int l = 0, n = 0, q = 0;
    if (c < copies) {
      l = st.cnt[c];
      n = (c + 1 < copies ? st.cnt[c + 1] : next) - l;
      for (int p = max(l - S, 0); p < l + n - S; ++p) q = max(q, use[p] + 1);
    }
    __syncwarp();
    if (c < copies) {
      st.cnt[c] = (uint16_t)n;
      st.req[c] = (uint16_t)q;
    }
    __syncwarp();
  }
}

// The busy columns' lists dealt out to the lanes of their warps (one warp):
// kBusyPer entries of one direction per lane, a column's lanes side by side in
// one warp.  blanes = 0 if they do not fit.
__device__ __forceinline__ void busy_lanes(TeamStage& st, const int4* bran, int4* blane, int lane) {
  int at = 0;
  for (int j = 0; j < st.nb; ++j) {
    const int4 R = bran[j];
    const int no = (R.y - R.x) / 8, ni = (R.w - R.z) / 8;
    const int lo = ceil_div(no, kBusyPer), n = lo + ceil_div(ni, kBusyPer);
    if (n > 32 - (at & 31)) {  // the next warp; unused lanes have no entries
      const int end = (at + 31) & ~31;
      if (at + lane < end && at + lane < 32 * kBusyWarps) blane[at + lane] = make_int4(0, 0, 0, 1);
      at = end;
    }
    if (n > 32 || at + n > 32 * kBusyWarps) {
      if (lane == 0) st.blanes = 0;
      return;
    }
    if (lane < n) {
      const bool in = lane >= lo;
      const int e = kBusyPer * (in ? lane - lo : lane), left = (in ? ni : no) - e;
      blane[at + lane] = make_int4(j, (in ? R.z : R.x) + 8 * e, min(left, kBusyPer) | (in ? 256 : 0),
                                   (n - lane) | (lane == 0 ? 256 : 0));
    }
    at += n;
  }
  if (lane == 0) st.blanes = at;
}

// A lane's column: its first out- and in-neighbour, positions times four; a
// missing neighbour has weight 0.  The second ones stay in shared memory ({out,
// weight, in, weight}): held in registers too, four chunks of 32 columns spilled.
struct ColRec {
  uint32_t vo, vi;
  float wo, wi;
};

// sum over a busy row's neighbours -- redge [e0, em) out, [em, e1) in -- at
// this lane's column: the loads of U rows in flight.
template <bool C2, int U>
__device__ __forceinline__ float team_busy_row(const float* Y, const int2* redge, int e0, int em, int e1,
                                               const ColRec& c, const int4 B) {
  float s = 0.f;
  for (int e = e0; e < e1; e += U) {
    float a[U], b[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int q = min(e + u, e1 - 1);
      const uint32_t o = (uint32_t)redge[q].x;
      a[u] = ldb(Y, o + (q < em ? c.vo : c.vi));
      if (C2) b[u] = ldb(Y, o + (uint32_t)(q < em ? B.x : B.z));
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int q = min(e + u, e1 - 1);
      const float wt = e + u < e1 ? __int_as_float(redge[q].y) : 0.f;
      const float w0 = q < em ? c.wo : c.wi, w1 = __int_as_float(q < em ? B.y : B.w);
      s = fmaf(wt, C2 ? fmaf(w1, b[u], w0 * a[u]) : w0 * a[u], s);
    }
  }
  return s;
}

// The same at a busy column: the warp's lanes take the column's neighbours.
__device__ __forceinline__ float team_busy_pair(const float* Y, const int2* redge, int e0, int e1, uint32_t f0,
                                                uint32_t f1, int lane) {
  float s = 0.f;
  for (uint32_t f = f0 + 8u * lane; f < f1; f += 256u) {
    const int2 v = lds_rec2(f);
    float z = 0.f;
    for (int e = e0; e < e1; e += 8) {
      float a[8], wt[8];
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        const int2 r = redge[min(e + u, e1 - 1)];
        wt[u] = e + u < e1 ? __int_as_float(r.y) : 0.f;
        a[u] = ldb(Y, (uint32_t)r.x + (uint32_t)v.x);
      }
#pragma unroll
      for (int u = 0; u < 8; ++u) z = fmaf(wt[u], a[u], z);
    }
    s = fmaf(__int_as_float(v.y), z, s);
  }
  return s;
}

// Two rows (ra, rb; two: rb is one of its own) at a busy column's lanes.
__device__ __forceinline__ float busy_cols(uint32_t rec, int ra, int rb, bool two,
                                           bool in, bool head, int len, int span, const uint32_t (&bv)[kBusyPer],
                                           const float (&bw)[kBusyPer], uint32_t p, float* nxt, float ca, float cbi) {
  const uint32_t q0 = rec + 48u * ra, q1 = rec + 48u * rb;
  const int4 A0 = lds_rec4(q0), W0 = lds_rec4(q0 + 16u), A1 = lds_rec4(q1), W1 = lds_rec4(q1 + 16u);
  const int2 E0 = lds_rec2(q0 + 32u), E1 = lds_rec2(q1 + 32u);
  const uint32_t x0 = in ? A0.y : A0.x, x1 = in ? A1.y : A1.x;
  float y0[kBusyPer], y1[kBusyPer];
#pragma unroll
  for (int u = 0; u < kBusyPer; ++u) {
    y0[u] = lds32(x0 + bv[u]);
    y1[u] = lds32(x1 + bv[u]);
  }
  const float e0 = lds32((uint32_t)E0.x + p), e1 = lds32((uint32_t)E1.x + p);
  float s0 = 0.f, s1 = 0.f;
#pragma unroll
  for (int u = 0; u < kBusyPer; ++u) {
    s0 = fmaf(bw[u], y0[u], s0);
    s1 = fmaf(bw[u], y1[u], s1);
  }
  s0 *= __int_as_float(in ? W0.y : W0.x);
  s1 *= __int_as_float(in ? W1.y : W1.x);
  if ((W0.z | W0.w | W1.z | W1.w) != 0) {
    const uint32_t z0 = in ? A0.w : A0.z, z1 = in ? A1.w : A1.z;
    float t0 = 0.f, t1 = 0.f;
#pragma unroll
    for (int u = 0; u < kBusyPer; ++u) {
      t0 = fmaf(bw[u], lds32(z0 + bv[u]), t0);
      t1 = fmaf(bw[u], lds32(z1 + bv[u]), t1);
    }
    s0 = fmaf(__int_as_float(in ? W0.w : W0.z), t0, s0);
    s1 = fmaf(__int_as_float(in ? W1.w : W1.z), t1, s1);
  }
  for (int o = span >> 1; o > 0; o >>= 1) {
    const float t0 = __shfl_down_sync(0xffffffffu, s0, o), t1 = __shfl_down_sync(0xffffffffu, s1, o);
    if (o < len) {
      s0 += t0;
      s1 += t1;
    }
  }
  float ss = 0.f;
  if (head) {
    const float y = fmaf(ca, s0, cbi * e0);
    stb(nxt, (uint32_t)E0.y + p, y);
    ss = y * y;
    if (two) {
      const float v = fmaf(ca, s1, cbi * e1);
      stb(nxt, (uint32_t)E1.y + p, v);
      ss = fmaf(v, v, ss);
    }
  }
  return ss;
}

// One step of a consumer warp: RR rows (every rg-th from r on) x its CH chunks
// of 32 columns, side by side.  Every load that does not depend on a row's
// or chunk's kind is issued before any value is used.
template <int RR, int CH>
__device__ __forceinline__ float team_step(uint32_t rec, int r, int rg, int nr, int nq, const ColRec (&c)[CH],
                                           uint32_t cb, uint32_t cbs, uint32_t p4, bool last_act, int n_one,
                                           char* nxt, float ca, float cbi) {
  int4 A[RR], W[RR];
  int2 Eo[RR];
#pragma unroll
  for (int j = 0; j < RR; ++j) {
    const uint32_t q = rec + 48u * (uint32_t)min(r + j * rg, nr - 1);
    A[j] = lds_rec4(q);
    W[j] = lds_rec4(q + 16u);
    Eo[j] = lds_rec2(q + 32u);
  }
  int4 Bk[CH];  // kept over the rows of a step of several
  if (RR > 1) {
#pragma unroll
    for (int q = 0; q < CH; ++q) Bk[q] = q >= n_one && q < nq ? lds_rec4(cb + cbs * q) : make_int4(0, 0, 0, 0);
  }
  float e[RR][CH], so[RR][CH], si[RR][CH];
#pragma unroll
  for (int j = 0; j < RR; ++j)
#pragma unroll
    for (int q = 0; q < CH; ++q) {  // (a warp's last chunk may be missing: its lists are zero, the reads in bounds)
      e[j][q] = lds32((uint32_t)Eo[j].x + p4 + 128u * q);
      so[j][q] = lds32((uint32_t)A[j].x + c[q].vo);
      si[j][q] = lds32((uint32_t)A[j].y + c[q].vi);
    }
  float ss = 0.f;
#pragma unroll
  for (int j = 0; j < RR; ++j) {
    const bool r2 = (W[j].z | W[j].w) != 0;
    float z[CH];
#pragma unroll
    for (int q = 0; q < CH; ++q) {
      float o = c[q].wo * so[j][q], i = c[q].wi * si[j][q], o2 = 0.f, i2 = 0.f;
      if (r2) {
        o2 = c[q].wo * lds32((uint32_t)A[j].z + c[q].vo);
        i2 = c[q].wi * lds32((uint32_t)A[j].w + c[q].vi);
      }
      if (q >= n_one && q < nq) {  // a chunk with second neighbours
        const int4 B = RR > 1 ? Bk[q] : lds_rec4(cb + cbs * q);
        o = fmaf(__int_as_float(B.y), lds32((uint32_t)(A[j].x + B.x)), o);
        i = fmaf(__int_as_float(B.w), lds32((uint32_t)(A[j].y + B.z)), i);
        if (r2) {
          o2 = fmaf(__int_as_float(B.y), lds32((uint32_t)(A[j].z + B.x)), o2);
          i2 = fmaf(__int_as_float(B.w), lds32((uint32_t)(A[j].w + B.z)), i2);
        }
      }
      z[q] = __int_as_float(W[j].x) * o;
      so[j][q] = __int_as_float(W[j].y) * i;
      if (r2) {
        z[q] = fmaf(__int_as_float(W[j].z), o2, z[q]);
        so[j][q] = fmaf(__int_as_float(W[j].w), i2, so[j][q]);
      }
    }
    char* to = nxt + (uint32_t)Eo[j].y;
    const bool row = r + j * rg < nr;
#pragma unroll
    for (int q = 0; q < CH; ++q) {
      const float y = fmaf(ca, z[q] + so[j][q], cbi * e[j][q]);
      if (row && (q < nq - 1 || (q == nq - 1 && last_act))) {
        *reinterpret_cast<float*>(to + 128 * q) = y;
        ss = fmaf(y, y, ss);
      }
    }
  }
  return ss;
}

// The iterations, role by role: every warp of the CTA runs one of these loops
// (separate functions, so that each holds only its own registers), and all of
// them meet in team_sum.
struct TeamIter {
  float* eb;
  float* b0;
  float* b1;
  float alpha, s0, cbi;  // s0 = 1 / |E|_F
  int K, norm_mode;
};
__device__ __forceinline__ const float* iter_from(const TeamIter& it, int k) {
  return k == 0 ? it.eb : ((it.K - k) & 1) ? it.b1 : it.b0;  // Y_K ends up in b0
}
__device__ __forceinline__ float* iter_to(const TeamIter& it, int k) {
  return ((it.K - 1 - k) & 1) ? it.b1 : it.b0;
}
__device__ __forceinline__ float iter_end(const Team& tm, TeamSh& sh, const TeamIter& it, float ss) {
  fence_async();  // Y_{k+1} is read by bulk copies
  const float yy = team_sum(tm, sh, ss);
  return it.norm_mode == 0 ? 1.0f / sqrtf(yy) : 1.f;
}

// A consumer warp with CH chunks, RR rows per step.
template <int NT, int CH, int RR>
__device__ __noinline__ float team_consume(const Team& tm, TeamSh& sh, const TeamIter& it) {
  const TeamStage& st = sh.st;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int nch = st.nch, wpr = st.wpr, rg = st.rg, nr = st.nr, nsteps = st.nsteps, rps = st.rps;
  const int grp = w / wpr, cw = w % wpr;
  const int nq = (nch - cw + wpr - 1) / wpr;                             // chunks this warp owns: cw, cw + wpr, ...
  const int n_one = min(nq, max(0, (st.n0 / 32 - cw + wpr - 1) / wpr));  // of them, all columns of the first kind
  const uint32_t p4 = 4u * (uint32_t)(32 * chunk_first(cw, nch, wpr) + lane);
  const bool last_act = 32 * (cw + wpr * (nq - 1)) + lane < st.nnb;
  ColRec c[CH];
  // the team's busy rows this warp does at its chunks (bits; beyond 32 rows they are looked for)
  const int slots = tm.T * rg, slot = tm.c * rg + grp;  // the warps that own the same chunks, over the team
  uint32_t any = 0u;
#pragma unroll
  for (int q = 0; q < CH; ++q) {
    const int p = 32 * (cw + wpr * q) + lane;
    const int4 A = q < nq && p < st.nnb ? st.cA[p] : make_int4(0, 0, 0, 0);
    c[q] = ColRec{(uint32_t)A.x, (uint32_t)A.z, __int_as_float(A.y), __int_as_float(A.w)};
    uint32_t m = 0u;
    for (int b = 0; q < nq && b < min(st.nbr, 32); ++b)
      if ((5 * cw + b * CH + q) % slots == slot) m |= 1u << b;
    if (lane == 0) sh.mine[w][q] = m;
    any |= m;
  }
  const uint32_t cb = st.cb + 16u * (uint32_t)(32 * cw + lane), cbs = 512u * (uint32_t)wpr;
  __syncwarp();
  const uint32_t full = st.full, empty = st.empty, rec = st.rec;
  fence_async();  // the buffers' memory was the staging's: generic accesses before the copies
  __syncthreads();
  RingPos pos{0u, 0u};
  float sk = it.s0;
#pragma unroll 1
  for (int k = 0; k < it.K; ++k) {
    const float* Y = iter_from(it, k);
    float* nxt = iter_to(it, k);
    const float ca = 0.5f * it.alpha * sk, cbi = it.cbi;
    float ss = 0.f;
    if (any || st.nbr > 32) {
#pragma unroll
      for (int q = 0; q < CH; ++q) {
        auto busy_row = [&](int b) {
          const int4 R = st.brow[b];
          const uint32_t off = st.browo[b] + p4 + 128u * q;
          const bool act = q < nq - 1 || last_act;
          const float e = act ? ldb(it.eb, off) : 0.f;
          const float s = q >= n_one ? team_busy_row<true, CH < 4 ? 8 : 4>(Y, st.redge, R.x, R.y, R.w, c[q], lds_rec4(cb + cbs * q))
                                     : team_busy_row<false, CH < 4 ? 16 : 8>(Y, st.redge, R.x, R.y, R.w, c[q], make_int4(0, 0, 0, 0));
          if (act) {
            const float y = fmaf(ca, s, cbi * e);
            stb(nxt, off, y);
            ss = fmaf(y, y, ss);
          }
        };
        for (uint32_t m = sh.mine[w][q]; m; m &= m - 1) busy_row(__ffs(m) - 1);
        for (int b = 32; q < nq && b < st.nbr; ++b)
          if ((5 * cw + b * CH + q) % slots == slot) busy_row(b);
      }
    }
    char* to = reinterpret_cast<char*>(nxt) + p4;
    int r = grp;
#pragma unroll 1
    for (int step = 0; step < nsteps; ++step, r += rps) {
      ring_wait(sh, tm.hdr, full, pos);
      ss += team_step<RR, CH>(rec, r, rg, nr, nq, c, cb, cbs, p4, last_act, n_one, to, ca, cbi);
      ring_done(empty, pos, lane);
    }
    sk = iter_end(tm, sh, it, ss);
  }
  return sk;
}

// A busy columns' warp.
template <int NT>
__device__ __noinline__ float team_busy(const Team& tm, TeamSh& sh, const TeamIter& it) {
  constexpr int NC = kConsumers<NT>;
  const TeamStage& st = sh.st;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int nb = st.nb, nr = st.nr, nsteps = st.nsteps, rps = st.rps, nnb = st.nnb;
  const uint32_t full = st.full, empty = st.empty, rec = st.rec;
  // this lane's entries; few lanes per row: several rows side by side in a warp
  const int warps = max(1, ceil_div(st.blanes, 32));  // warps per row
  int side = 1;
  while (side < 8 && 2 * side * st.blanes <= 32) side *= 2;
  const int per = 32 / side, rows = kBusyWarps / warps * side;  // lanes per row, rows at a time
  const int grp = (w - NC) / warps * side + lane / per, at = warps > 1 ? 32 * ((w - NC) % warps) + lane : lane % per;
  int4 bl = make_int4(0, 0, 0, 0);
  if (grp < rows && at < st.blanes) bl = lds_rec4(st.blane + 16u * (uint32_t)at);
  uint32_t bv[kBusyPer];
  float bw[kBusyPer];
#pragma unroll
  for (int u = 0; u < kBusyPer; ++u) {
    const int2 v = u < (bl.z & 255) ? lds_rec2((uint32_t)bl.y + 8u * u) : make_int2(0, 0);
    bv[u] = (uint32_t)v.x;
    bw[u] = __int_as_float(v.y);
  }
  const bool in = (bl.z >> 8) != 0, head = (bl.w >> 8) != 0;
  const int len = bl.w & 255;
  int span = 1;  // lanes of the warp's longest column
  while (span < __reduce_max_sync(0xffffffffu, len)) span <<= 1;
  fence_async();
  __syncthreads();
  RingPos pos{0u, 0u};
  float sk = it.s0;
#pragma unroll 1
  for (int k = 0; k < it.K; ++k) {
    const float* Y = iter_from(it, k);
    float* nxt = iter_to(it, k);
    const float ca = 0.5f * it.alpha * sk, cbi = it.cbi;
    float ss = 0.f;
    // busy rows at busy columns: lists times lists, an entry per warp
    for (int q = (w - NC) * tm.T + tm.c; q < st.nbr * nb; q += kBusyWarps * tm.T) {
      const int b = q / nb, j = q - b * nb;
      const int4 R = st.brow[b], C = lds_rec4(st.bran + 16u * j);
      float s = team_busy_pair(Y, st.redge, R.x, R.y, (uint32_t)C.x, (uint32_t)C.y, lane) +
                team_busy_pair(Y, st.redge, R.z, R.w, (uint32_t)C.z, (uint32_t)C.w, lane);
      s = warp_sum(s);
      if (lane == 0) {
        const uint32_t off = st.browo[b] + 4u * (uint32_t)(nnb + j);
        const float y = fmaf(ca, s, cbi * ldb(it.eb, off));
        stb(nxt, off, y);
        ss = fmaf(y, y, ss);
      }
    }
    if (st.blanes > 0) {
      const uint32_t p = 4u * (uint32_t)(nnb + bl.x);
#pragma unroll 1
      for (int step = 0; step < nsteps; ++step) {
        ring_wait(sh, tm.hdr, full, pos);
        const int r0 = step * rps, r1 = min(nr, r0 + rps);
        if (rps == 1) {  // a row per step: the row groups take turns
          if (r0 % rows / side == (w - NC) / warps)
            ss += busy_cols(rec, r0, r0, false, in, head && r0 % rows == grp, len, span, bv, bw, p, nxt, ca,
                            cbi);
        } else {
          for (int rb = r0; rb < r1; rb += 2 * rows) {
            const int ra = rb + grp, rc = ra + rows;
            ss += busy_cols(rec, min(ra, r1 - 1), min(rc, r1 - 1), rc < r1, in, head && ra < r1, len, span,
                            bv, bw, p, nxt, ca, cbi);
          }
        }
        ring_done(empty, pos, lane);
      }
    } else {  // too many list entries for the lanes: eight lanes walk an entry's list
      const uint32_t l8 = lane & 7;
#pragma unroll 1
      for (int step = 0; step < nsteps; ++step) {
        ring_wait(sh, tm.hdr, full, pos);
        const int r0 = step * rps, items = min(rps, nr - r0) * nb;
        for (int q0 = 4 * (w - NC); q0 < items; q0 += 4 * kBusyWarps) {
          const int q = min(q0 + (lane >> 3), items - 1);
          const int r = r0 + q / nb, j = q % nb;
          const int4 R = lds_rec4(st.bran + 16u * j), A = lds_rec4(rec + 48u * r), W = lds_rec4(rec + 48u * r + 16u);
          float s = 0.f;
          for (uint32_t e = (uint32_t)R.x + 8u * l8; e < (uint32_t)R.y; e += 64u) {
            const int2 v = lds_rec2(e);
            s = fmaf(__int_as_float(v.y), fmaf(__int_as_float(W.z), lds32((uint32_t)A.z + v.x),
                                               __int_as_float(W.x) * lds32((uint32_t)A.x + v.x)), s);
          }
          for (uint32_t e = (uint32_t)R.z + 8u * l8; e < (uint32_t)R.w; e += 64u) {
            const int2 v = lds_rec2(e);
            s = fmaf(__int_as_float(v.y), fmaf(__int_as_float(W.w), lds32((uint32_t)A.w + v.x),
                                               __int_as_float(W.y) * lds32((uint32_t)A.y + v.x)), s);
          }
#pragma unroll
          for (int o = 4; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
          if (l8 == 0 && q0 + (lane >> 3) < items) {
            const int2 Eo = lds_rec2(rec + 48u * r + 32u);
            const uint32_t p = 4u * (uint32_t)(nnb + j);
            const float y = fmaf(ca, s, cbi * lds32((uint32_t)Eo.x + p));
            stb(nxt, (uint32_t)Eo.y + p, y);
            ss = fmaf(y, y, ss);
          }
        }
        ring_done(empty, pos, lane);
      }
    }
    sk = iter_end(tm, sh, it, ss);
  }
  return sk;
}

// The copying warp (fill), or a warp without work.
template <int NT>
__device__ __noinline__ float team_fill(const Team& tm, TeamSh& sh, const TeamIter& it, bool fill) {
  const TeamStage& st = sh.st;
  const int lane = threadIdx.x & 31;
  fence_async();
  __syncthreads();
  uint32_t base = 0;
  RingPos dp{0u, 0u};
  float sk = it.s0;
#pragma unroll 1
  for (int k = 0; k < it.K; ++k, base += (uint32_t)st.nsteps) {
    if (fill) ring_fill(st, sh, tm.hdr, iter_from(it, k), it.eb, base, dp, lane);
    sk = iter_end(tm, sh, it, 0.f);
  }
  return sk;
}

// All iterations of the slab; returns s_K.
template <int NT>
__device__ __forceinline__ float team_iterate(const Team& tm, TeamSh& sh, const TeamIter& it, int CH) {
  constexpr int NC = kConsumers<NT>;
  const int w = threadIdx.x >> 5;
  float sk;
  if (w < sh.st.wpr * sh.st.rg) {
    sk = CH == 1   ? team_consume<NT, 1, 2>(tm, sh, it)
         : CH == 2 ? team_consume<NT, 2, 1>(tm, sh, it)
         : CH == 3 ? team_consume<NT, 3, 1>(tm, sh, it)
         : CH == 4 ? team_consume<NT, 4, 1>(tm, sh, it)
                   : team_consume<NT, kMaxChunks, 1>(tm, sh, it);
  } else if (w >= NC && w < NC + kBusyWarps && sh.st.nb > 0) {
    sk = team_busy<NT>(tm, sh, it);
  } else {
    sk = team_fill<NT>(tm, sh, it, w == NC + kBusyWarps);
  }
  if (sh.fail) __nanosleep(1000000);  // copies still in flight land
  __syncthreads();
  if (threadIdx.x < 2 * kStepRing)  // full, then empty
    asm volatile("mbarrier.inval.shared::cta.b64 [%0];" ::"r"(sh.st.full + 8u * threadIdx.x) : "memory");
  __syncthreads();
  return sk;
}

// The iterations of a pair whose graphs cannot be staged (rows too long for a
// ring of them, about 3,800 columns and more): rows and column lists come from
// memory, columns in natural order.  What bounds an iteration is the loads in
// flight and the longest chain of list terms that one warp has, so
//   - a slab's rows with at most two neighbours either way are swept by strips,
//     32 columns and a run of rows a warp: the columns' first two neighbours
//     stay in registers, the rows' records come from shared memory, and kFarRows
//     rows' loads are issued before any is used;
//   - the other rows (the STOP block has an in-edge from every early return) are
//     shared out over the team's warps, 32 columns at a time;
//   - an entry at a column with more than kFarList neighbours is the whole
//     warp's, its lanes over the longer of the two lists.
// One pair of 4,400 x 4,800 blocks, in-degree of the STOP block 129, K = 40: 14.8
// ms; 152 pairs of 4,400-4,800: 2.59 s.  (Both lists read entry by entry, a lane
// per column whatever its list, so that one warp had the STOP row and one lane
// the entry at both STOP blocks: 542 ms and 77.5 s.  The busy rows shared out
// but no strips, a column's lists read again at every row: 31 ms and 5.1 s.  One
// CTA per pair: 3,400 ms and 4.7 s.)
constexpr int kFarRows = 4;
constexpr int kFarList = 16;
constexpr int kFarBlock = 1024;        // rows whose records are staged at a time
constexpr size_t kFarRecs = 1 << 16;   // their place, behind the list of the other rows

// sum_e sum_f w_e w_f Y[u_e, v_f] over two lists: this lane's part.
__device__ __forceinline__ float far_pair(const float* Y, uint32_t ld, const CfAdj* ra, int e0, int e1, const CfAdj* ca,
                                          int f0, int f1, int lane) {
  uint32_t sa = 1, sb = ld;  // strides: of the list over the lanes, of the other
  if (e1 - e0 > f1 - f0) {
    const CfAdj* a = ra;
    ra = ca;
    ca = a;
    int k = e0;
    e0 = f0;
    f0 = k;
    k = e1;
    e1 = f1;
    f1 = k;
    sa = ld;
    sb = 1;
  }
  float s = 0.f;
  for (int f = f0 + lane; f < f1; f += 32) {
    const CfAdj v = ldg_adj(ca + f);
    const float* y = Y + sa * (uint32_t)v.nbr;
    float z = 0.f;
#pragma unroll 8
    for (int e = e0; e < e1; ++e) {
      const CfAdj u = ldg_adj(ra + e);
      z = fmaf(u.w, y[sb * (uint32_t)u.nbr], z);
    }
    s = fmaf(v.w, z, s);
  }
  return s;
}

// The same at this lane's column, whose list is short.
__device__ __forceinline__ float far_lane(const float* Y, uint32_t ld, const CfAdj* ra, int e0, int e1, const CfAdj* ca,
                                          int f0, int f1) {
  float s = 0.f;
  for (int f = f0; f < f1; ++f) {
    const CfAdj v = ldg_adj(ca + f);
    float z = 0.f;
#pragma unroll 8
    for (int e = e0; e < e1; ++e) {
      const CfAdj u = ldg_adj(ra + e);
      z = fmaf(u.w, Y[(uint32_t)u.nbr * ld + (uint32_t)v.nbr], z);
    }
    s = fmaf(v.w, z, s);
  }
  return s;
}

// A lane's column: its lists' ranges and first two neighbours (a missing one
// has weight 0).
struct FarCol {
  int c0, c1, d0, d1;
  uint32_t vo0, vo1, vi0, vi1;
  float wo0, wo1, wi0, wi1;
};
__device__ __forceinline__ FarCol far_col(const Geo& g, int j, int n_col) {
  FarCol c{};
  if (j < n_col) {
    c.c0 = __ldg(g.c_optr + j);
    c.c1 = __ldg(g.c_optr + j + 1);
    c.d0 = __ldg(g.c_iptr + j);
    c.d1 = __ldg(g.c_iptr + j + 1);
    const CfAdj z{0, 0.f};
    const CfAdj a0 = c.c1 > c.c0 ? ldg_adj(g.c_oadj + c.c0) : z, a1 = c.c1 > c.c0 + 1 ? ldg_adj(g.c_oadj + c.c0 + 1) : z;
    const CfAdj b0 = c.d1 > c.d0 ? ldg_adj(g.c_iadj + c.d0) : z, b1 = c.d1 > c.d0 + 1 ? ldg_adj(g.c_iadj + c.d0 + 1) : z;
    c.vo0 = (uint32_t)a0.nbr;
    c.vo1 = (uint32_t)a1.nbr;
    c.vi0 = (uint32_t)b0.nbr;
    c.vi1 = (uint32_t)b1.nbr;
    c.wo0 = a0.w;
    c.wo1 = a1.w;
    c.wi0 = b0.w;
    c.wi1 = b1.w;
  }
  return c;
}

// Rows i0 + r .. of the staged records (r + kFarRows > r1: the last ones are
// left out) at the lanes' columns.  A record: {4 out 0, out 1, in 0, in 1: ld
// times the row}, their weights; x = ~0: not one of these rows.
__device__ __forceinline__ float far_rows(const Geo& g, const float* Y, float* nxt, const float* eb, uint32_t ld, int i0,
                                          const int4* rec, int r, int r1, const FarCol& c, bool big, int j, int n_col,
                                          float ca, float cbi, int lane) {
  int4 A[kFarRows], W[kFarRows];
  float s0[kFarRows], s1[kFarRows], t0[kFarRows], t1[kFarRows], e[kFarRows], z[kFarRows];
#pragma unroll
  for (int u = 0; u < kFarRows; ++u) {
    const int q = min(r + u, r1 - 1);
    A[u] = rec[2 * q];
    W[u] = rec[2 * q + 1];
    const uint32_t o = A[u].x == -1 ? 0u : (uint32_t)A[u].x;
    s0[u] = Y[o + c.vo0];
    s1[u] = Y[(uint32_t)A[u].z + c.vi0];
    t0[u] = Y[o + c.vo1];
    t1[u] = Y[(uint32_t)A[u].z + c.vi1];
    e[u] = j < n_col ? eb[(uint32_t)(i0 + q) * ld + (uint32_t)j] : 0.f;
  }
#pragma unroll
  for (int u = 0; u < kFarRows; ++u) {
    z[u] = __int_as_float(W[u].x) * fmaf(c.wo1, t0[u], c.wo0 * s0[u]) +
           __int_as_float(W[u].z) * fmaf(c.wi1, t1[u], c.wi0 * s1[u]);
    if ((W[u].y | W[u].w) != 0) {
      const float* y1 = Y + (uint32_t)A[u].y;
      const float* y2 = Y + (uint32_t)A[u].w;
      z[u] += __int_as_float(W[u].y) * fmaf(c.wo1, y1[c.vo1], c.wo0 * y1[c.vo0]) +
              __int_as_float(W[u].w) * fmaf(c.wi1, y2[c.vi1], c.wi0 * y2[c.vi0]);
    }
  }
  // further neighbours: the lane's, or over the warp
  auto terms = [&](const CfAdj v, bool in, float (&s)[kFarRows]) {
#pragma unroll
    for (int u = 0; u < kFarRows; ++u) {
      const uint32_t a = in ? (uint32_t)A[u].z : A[u].x == -1 ? 0u : (uint32_t)A[u].x, b = (uint32_t)(in ? A[u].w : A[u].y);
      const float wa = __int_as_float(in ? W[u].z : W[u].x), wb = __int_as_float(in ? W[u].w : W[u].y);
      float y = wa * Y[a + (uint32_t)v.nbr];
      if (wb != 0.f) y = fmaf(wb, Y[b + (uint32_t)v.nbr], y);
      s[u] = fmaf(v.w, y, s[u]);
    }
  };
  if (!big) {
    for (int f = c.c0 + 2; f < c.c1; ++f) terms(ldg_adj(g.c_oadj + f), false, z);
    for (int f = c.d0 + 2; f < c.d1; ++f) terms(ldg_adj(g.c_iadj + f), true, z);
  }
  for (unsigned m = __ballot_sync(0xffffffffu, big); m; m &= m - 1) {
    const int l = __ffs(m) - 1;
    const int f0 = __shfl_sync(0xffffffffu, c.c0, l) + 2, f1 = __shfl_sync(0xffffffffu, c.c1, l);
    const int h0 = __shfl_sync(0xffffffffu, c.d0, l) + 2, h1 = __shfl_sync(0xffffffffu, c.d1, l);
    float s[kFarRows] = {};
    for (int f = f0 + lane; f < f1; f += 32) terms(ldg_adj(g.c_oadj + f), false, s);
    for (int f = h0 + lane; f < h1; f += 32) terms(ldg_adj(g.c_iadj + f), true, s);
#pragma unroll
    for (int u = 0; u < kFarRows; ++u) {
      const float v = warp_sum(s[u]);
      if (lane == l) z[u] += v;
    }
  }
  float ss = 0.f;
#pragma unroll
  for (int u = 0; u < kFarRows; ++u)
    if (r + u < r1 && A[u].x != -1 && j < n_col) {
      const float y = fmaf(ca, z[u], cbi * e[u]);
      nxt[(uint32_t)(i0 + r + u) * ld + (uint32_t)j] = y;
      ss = fmaf(y, y, ss);
    }
  return ss;
}

// region: the rows of the row graph with more than two neighbours (nbr of
// them), then room for the records; i0, i1: this CTA's slab.  Returns s_K.
template <int NT>
__device__ __noinline__ float team_far(const Team& tm, TeamSh& sh, const TeamIter& it, const Geo& g, uint32_t ld, int i0,
                                       int i1, unsigned char* region, int nbr) {
  constexpr int NW = NT / 32;
  const int t = threadIdx.x, lane = t & 31, w = t >> 5, n_col = g.nb;
  const int nch = ceil_div(n_col, 32);
  const uint16_t* rows = reinterpret_cast<const uint16_t*>(region);
  int4* rec = reinterpret_cast<int4*>(region + kFarRecs);
  float sk = it.s0;
  for (int k = 0; k < it.K; ++k) {
    const float* Y = iter_from(it, k);
    float* nxt = iter_to(it, k);
    const float ca = 0.5f * it.alpha * sk;
    float ss = 0.f;
    // the longest first
    for (int64_t q = (int64_t)w * tm.T + tm.c; q < (int64_t)nbr * nch; q += NW * tm.T) {
      const int b = (int)(q / nch), j = 32 * (int)(q - (int64_t)b * nch) + lane, i = rows[b];
      const int o0 = __ldg(g.r_optr + i), o1 = __ldg(g.r_optr + i + 1);
      const int q0 = __ldg(g.r_iptr + i), q1 = __ldg(g.r_iptr + i + 1);
      int c0 = 0, c1 = 0, d0 = 0, d1 = 0;
      if (j < n_col) {
        c0 = __ldg(g.c_optr + j);
        c1 = __ldg(g.c_optr + j + 1);
        d0 = __ldg(g.c_iptr + j);
        d1 = __ldg(g.c_iptr + j + 1);
      }
      const bool big = c1 - c0 > kFarList || d1 - d0 > kFarList;
      float z = 0.f;
      if (!big)
        z = far_lane(Y, ld, g.r_oadj, o0, o1, g.c_oadj, c0, c1) + far_lane(Y, ld, g.r_iadj, q0, q1, g.c_iadj, d0, d1);
      for (unsigned m = __ballot_sync(0xffffffffu, big); m; m &= m - 1) {
        const int l = __ffs(m) - 1;
        const int f0 = __shfl_sync(0xffffffffu, c0, l), f1 = __shfl_sync(0xffffffffu, c1, l);
        const int h0 = __shfl_sync(0xffffffffu, d0, l), h1 = __shfl_sync(0xffffffffu, d1, l);
        const float v = warp_sum(far_pair(Y, ld, g.r_oadj, o0, o1, g.c_oadj, f0, f1, lane) +
                                 far_pair(Y, ld, g.r_iadj, q0, q1, g.c_iadj, h0, h1, lane));
        if (lane == l) z = v;
      }
      if (j < n_col) {
        const uint32_t at = (uint32_t)i * ld + (uint32_t)j;
        const float y = fmaf(ca, z, it.cbi * it.eb[at]);
        nxt[at] = y;
        ss = fmaf(y, y, ss);
      }
    }
    for (int b0 = i0; b0 < i1; b0 += kFarBlock) {
      const int nr = min(kFarBlock, i1 - b0);
      if (k == 0 || i1 - i0 > kFarBlock) {
        __syncthreads();
        for (int r = t; r < nr; r += NT) {
          const int o0 = __ldg(g.r_optr + b0 + r), o1 = __ldg(g.r_optr + b0 + r + 1);
          const int q0 = __ldg(g.r_iptr + b0 + r), q1 = __ldg(g.r_iptr + b0 + r + 1);
          const bool in = o1 - o0 <= 2 && q1 - q0 <= 2;
          const CfAdj z{0, 0.f};
          const CfAdj a0 = in && o1 > o0 ? ldg_adj(g.r_oadj + o0) : z, a1 = in && o1 > o0 + 1 ? ldg_adj(g.r_oadj + o0 + 1) : z;
          const CfAdj d0 = in && q1 > q0 ? ldg_adj(g.r_iadj + q0) : z, d1 = in && q1 > q0 + 1 ? ldg_adj(g.r_iadj + q0 + 1) : z;
          rec[2 * r] = make_int4(in ? (int)((uint32_t)a0.nbr * ld) : -1, (int)((uint32_t)a1.nbr * ld),
                                 (int)((uint32_t)d0.nbr * ld), (int)((uint32_t)d1.nbr * ld));
          rec[2 * r + 1] = make_int4(__float_as_int(a0.w), __float_as_int(a1.w), __float_as_int(d0.w), __float_as_int(d1.w));
        }
        __syncthreads();
      }
      // strips: every warp some, whatever the matrix's shape
      const int runs = min(ceil_div(nr, kFarRows), ceil_div(4 * NW, nch)), len = ceil_div(nr, runs);
      for (int q = w; q < nch * runs; q += NW) {
        const int h = q % nch, r0 = q / nch * len, r1 = min(nr, r0 + len), j = 32 * h + lane;
        const FarCol c = far_col(g, j, n_col);
        const bool big = c.c1 - c.c0 > kFarList || c.d1 - c.d0 > kFarList;
        for (int r = r0; r < r1; r += kFarRows)
          ss += far_rows(g, Y, nxt, it.eb, ld, b0, rec, r, r1, c, big, j, n_col, ca, it.cbi, lane);
      }
    }
    const float yy = team_sum(tm, sh, ss);
    sk = it.norm_mode == 0 ? 1.0f / sqrtf(yy) : 1.f;
  }
  return sk;
}

// ---------------------------------------------------------------------------
// The greedy matching of a team's pair, in phases.  X_K is close to rank one,
// so the sequential greedy takes its entries nearly one at a time, and rounds
// of locally dominant entries (greedy()) need hundreds of team barriers.  A
// phase takes about a hundred steps for three barriers:
//   1  every live row's best live value (all CTAs, a warp per row);
//   2  the rows of the largest best values, up to kTop; each of them lists its
//      best live columns in greedy order (value desc, column asc), up to kLen;
//   3  CTA 0 takes the sequential greedy's steps on those lists, a lane per
//      row: a row's head is its best live entry, the best head (value desc,
//      row asc) is the largest live entry.  The steps end when they reach the
//      best row that is not listed, or a row whose list is used up while it
//      has more live columns (it counts with its last listed value).
constexpr int kTop = 160;
constexpr int kLen = 96;
constexpr int kCand = 512;       // candidates a warp holds while it makes a list
constexpr int kTeamRowsPer = 8;  // rows a thread holds while the listed rows are chosen
constexpr int kBins = 256;
// pitches of the lists in shared memory ([entry][list]): odd in words, so that
// neither the copy in (along a list) nor the steps (along an entry) conflict
constexpr int kKeyPitch = kTop + 1, kColPitch = kTop + 2;

// Writes a row's m chosen entries (up to kLen, in column order, at the front of
// cand) in greedy order: each counts the ones before it.
__device__ __forceinline__ void rank_list(uint2* cand, int m, uint2* out, int lane) {
  // (c = lane + 32 q: the candidates of a block before block q come before
  // c where equal, those of a block after it do not)
  uint32_t* keys = reinterpret_cast<uint32_t*>(cand + kLen);  // past the chosen ones
  for (int d = lane; d < ((m + 31) & ~31); d += 32) keys[d] = d < m ? cand[d].x : 0u;
  __syncwarp();
  for (int q = 0; 32 * q < m; ++q) {
    const int c = lane + 32 * q;
    const uint2 a = c < m ? cand[c] : make_uint2(0xffffffffu, 0u);
    int rank = 0;
    for (int b = 0; 32 * b < m; ++b) {
      const uint4* kp = reinterpret_cast<const uint4*>(keys + 32 * b);
      if (b != q) {
        const uint32_t t = b < q ? a.x - 1u : a.x;
#pragma unroll
        for (int d = 0; d < 8; ++d) {
          const uint4 k = kp[d];
          rank += (k.x > t) + (k.y > t) + (k.z > t) + (k.w > t);
        }
      } else {
#pragma unroll
        for (int d = 0; d < 8; ++d) {
          const uint4 k = kp[d];
          rank += (k.x > a.x - (uint32_t)(4 * d < lane)) + (k.y > a.x - (uint32_t)(4 * d + 1 < lane)) +
                  (k.z > a.x - (uint32_t)(4 * d + 2 < lane)) + (k.w > a.x - (uint32_t)(4 * d + 3 < lane));
        }
      }
    }
    if (c < m) out[rank] = a;
  }
  __syncwarp();
}

// list_row where a row has too many candidates, or more than K entries of one
// value: over the row, the key hi that at most K entries reach while more than K
// reach the largest one below it, by halving between keys that occur; if few reach
// hi, the first entries of that one as well.  bound: a key that more than K entries
// reach, top: the largest.  (One entry after another over the row, 500 matrices of
// 13 x 5,000 with three values took 5.5 ms, near rank one 0.5; now 0.7.  A function
// of its own: in line it cost the other rows' lists 3 % of a call.)
__device__ __noinline__ int list_row_far(const float* x, int n_col, const unsigned char* dead, int K, uint32_t bound,
                                         uint32_t top, uint2* cand, uint2* out, int lane) {
  uint32_t lo = bound, hi = top + 1u;
  int gt = 0;
  auto key_at = [&](int j) -> uint32_t {
    const float v = j < n_col ? x[j] : 0.f;
    return j < n_col && !dead[j] && v > -CUDART_INF_F ? okey(v) : 0u;
  };
  while (hi - lo > 1u && 4 * gt < 3 * K) {
    const uint32_t mid = lo + (hi - lo) / 2;
    uint32_t up = 0xffffffffu, down = 0u;
    int c = 0;
    for (int j0 = 0; j0 < n_col; j0 += 256) {
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        const uint32_t k = key_at(j0 + 32 * u + lane);
        c += k >= mid;
        up = k >= mid ? min(up, k) : up;
        down = k >= mid ? down : max(down, k);
      }
    }
    c = __reduce_add_sync(0xffffffffu, c);
    if (c > K) {
      lo = __reduce_min_sync(0xffffffffu, up);
    } else {
      hi = __reduce_max_sync(0xffffffffu, down) + 1u;
      gt = c;
    }
  }
  const int eq = 4 * gt < 3 * K ? K - gt : 0;  // (hi is lo + 1)
  int m = 0, same = 0;
  for (int j0 = 0; j0 < n_col; j0 += 256) {
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      const int j = j0 + 32 * u + lane;
      const uint32_t k = key_at(j);
      const unsigned lt = (1u << lane) - 1u, ms = __ballot_sync(0xffffffffu, k == lo);
      const bool in = k >= hi || (k == lo && same + __popc(ms & lt) < eq);
      const unsigned mt = __ballot_sync(0xffffffffu, in);
      if (in) cand[m + __popc(mt & lt)] = make_uint2(k, (uint32_t)j);
      m += __popc(mt);
      same += __popc(ms);
    }
  }
  __syncwarp();
  rank_list(cand, m, out, lane);
  return m;
}

// The list of one row: x = its entries, dead = column flags (shared memory),
// cand = the warp's candidates.  Returns its length (bit 8: every live column
// is in it).
__device__ __forceinline__ int list_row(const float* x, int n_col, const unsigned char* dead, int K, uint2* cand,
                                        uint2* out, int lane) {
  // the lane's three largest live keys (0: none; neither NaN nor -inf is ever taken)
  uint32_t m1 = 0, m2 = 0, m3 = 0;
  for (int j0 = lane; j0 < n_col; j0 += 256) {
    float v[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) v[u] = j0 + 32 * u < n_col ? x[j0 + 32 * u] : 0.f;
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      const int j = j0 + 32 * u;
      const uint32_t k = j < n_col && !dead[j] && v[u] > -CUDART_INF_F ? okey(v[u]) : 0u;
      const uint32_t a = min(m1, k), b = min(m2, a);
      m1 = max(m1, k);
      m2 = max(m2, a);
      m3 = max(m3, b);
    }
  }
  // every lane has three entries >= the smallest third key, so at least 96
  // reach that bound; a lane with fewer live entries: every live entry
  const uint32_t low = __reduce_min_sync(0xffffffffu, m3), bound = max(1u, low);
  const uint32_t top = __reduce_max_sync(0xffffffffu, m1);
  int n = 0;
  for (int j0 = 0; j0 < n_col; j0 += 256) {
    float v[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) v[u] = j0 + 32 * u + lane < n_col ? x[j0 + 32 * u + lane] : 0.f;
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      const int j = j0 + 32 * u + lane;
      const uint32_t k = j < n_col && !dead[j] && v[u] > -CUDART_INF_F ? okey(v[u]) : 0u;
      const unsigned m = __ballot_sync(0xffffffffu, k >= bound);
      const int at = n + __popc(m & ((1u << lane) - 1u));
      if (k >= bound && at < kCand) cand[at] = make_uint2(k, (uint32_t)j);
      n += __popc(m);
    }
  }
  __syncwarp();
  if (n <= kCand) {
    // a key that at most K candidates reach, found by halving
    uint32_t thr = bound;
    int cnt = n;
    uint32_t lo = bound, hi = top;  // more than K reach lo
    for (int it = 0; it < 40 && cnt > K; ++it) {
      thr = hi - lo <= 1 ? hi : lo + (hi - lo) / 2;
      int c = 0;
      for (int d = lane; d < n; d += 32) c += cand[d].x >= thr;
      cnt = __reduce_add_sync(0xffffffffu, c);
      if (cnt > K) {
        if (thr == hi) break;  // more than K entries equal the largest
        lo = thr;
      } else if (4 * cnt < 3 * K && hi - lo > 1) {  // too few: try lower
        hi = thr;
        cnt = K + 1;
      }
    }
    if (cnt <= K) {
      // the chosen ones to the front (candidates are in column order)
      int m = 0;
      for (int d0 = 0; d0 < n; d0 += 32) {
        const uint2 a = d0 + lane < n ? cand[d0 + lane] : make_uint2(0u, 0u);
        const unsigned in = __ballot_sync(0xffffffffu, a.x >= thr);
        if (a.x >= thr) cand[m + __popc(in & ((1u << lane) - 1u))] = a;
        m += __popc(in);
        __syncwarp();
      }
      rank_list(cand, m, out, lane);
      return m | (low == 0u && m == n ? 256 : 0);
    }
  }
  return list_row_far(x, n_col, dead, K, bound, top, cand, out, lane);
}

// Step 3 of a phase, kTop threads (thread t: list t, row sel[t], rows
// ascending).  key / col [entry][list] of the nl lists, col as numbers of this
// phase's columns (idcol: their columns); inv [column][list]: the entry of the
// list that holds the column (0xff: none); okey / olist: the best row that is
// not listed comes before a head of a smaller key, or of key okey and list >=
// olist.  A lane keeps its live entries as a bit mask and its head in
// registers: when a column is taken, it drops the bit inv names, and if that
// was its head, the next set bit is the new one.  So a step is two warp
// maxima, an exchange of one word per warp over a barrier, and two dependent
// shared loads, whatever the lists hold.  (Lists walked past dead columns
// entry by entry: 0.32 to 0.9 us per step.)  Returns the matches made.
__device__ __forceinline__ int team_steps(TeamSh& sh, int nl, int left, const uint32_t* key, const uint16_t* col,
                                          const unsigned char* inv, const uint16_t* idcol, const int* len,
                                          const uint16_t* sel, uint32_t okey, int olist, int32_t* mrow,
                                          unsigned char* gdead) {
  constexpr int NWT = kTop / 32;
  static_assert(kLen == 96, "three words of live entries");
  const int t = threadIdx.x, lane = t & 31, w = t >> 5;
  const int n = t < nl ? len[t] & 255 : 0;
  const bool whole = t >= nl || (len[t] & 256) != 0;
  const uint32_t tie = (uint32_t)(255 - t) << 16;
  auto ones = [](int c) { return c >= 32 ? 0xffffffffu : c <= 0 ? 0u : (1u << c) - 1u; };
  uint32_t m0 = ones(n), m1 = ones(n - 32), m2 = ones(n - 64);
  // head: key hk, low word hl = blocked << 28 | (255 - list) << 16 | column number; its entry h
  uint32_t hk = 0u, hl = 0u;
  int h = 255;
  if (n > 0) {
    h = 0;
    hk = key[t];
    hl = tie | col[t];
  }
  int made = 0;
  for (; made < left; ++made) {
    uint32_t hi = __reduce_max_sync(0xffffffffu, hk);
    uint32_t lo = __reduce_max_sync(0xffffffffu, hk == hi ? hl : 0u);
    if (lane == 0) sh.step[made & 1][w] = make_uint2(hi, lo);
    bar_sync(1, kTop);
    uint2 v[NWT];
#pragma unroll
    for (int q = 0; q < NWT; ++q) v[q] = sh.step[made & 1][q];
    hi = 0u;
    lo = 0u;
#pragma unroll
    for (int q = 0; q < NWT; ++q) hi = max(hi, v[q].x);
#pragma unroll
    for (int q = 0; q < NWT; ++q) lo = max(lo, v[q].x == hi ? v[q].y : 0u);
    const int x = 255 - (int)((lo >> 16) & 0xffu);
    // nothing live, a used-up list or a row without a list is next
    if (hi == 0u || (lo >> 28) || hi < okey || (hi == okey && x >= olist)) break;
    const uint32_t c = lo & 0xffffu;
    if (t == x) {
      mrow[sel[t]] = (int32_t)idcol[c];
      gdead[idcol[c]] = 1;
      m0 = m1 = m2 = 0u;
      hk = hl = 0u;
      h = 255;
    } else {
      const int p = inv[c * kTop + t];
      const uint32_t bit = 1u << (p & 31);
      if (p < 32)
        m0 &= ~bit;
      else if (p < 64)
        m1 &= ~bit;
      else
        m2 &= p < 96 ? ~bit : 0xffffffffu;
      if (p == h && h != 255) {
        h = m0 ? __ffs(m0) - 1 : m1 ? 31 + __ffs(m1) : m2 ? 63 + __ffs(m2) : 255;
        if (h != 255) {
          hk = key[h * kKeyPitch + t];
          hl = tie | col[h * kColPitch + t];
        } else {
          hk = whole ? 0u : key[(n - 1) * kKeyPitch + t];
          hl = whole ? 0u : 1u << 28;
        }
      }
    }
  }
  return made;
}

// Shared memory of a phase: the listed rows and their lengths, then the larger
// of the column flags with the warps' candidates (or the bins) and, where those
// are no longer read, the lists with their column numbers.
constexpr int kIds = 680;  // columns a phase numbers; a list ends before its first column without a number
constexpr size_t kListBytes = kTop * (8 * (size_t)kLen + 4);  // scratch: the lists, their lengths
__device__ __forceinline__ size_t greedy_team_bytes(int n_col, int NT, bool wide) {
  const size_t a = align_up((size_t)n_col, 16) + sizeof(uint2) * kCand * (NT / 32);
  const size_t b = (4 * (size_t)kKeyPitch + 2 * (size_t)kColPitch) * kLen + kIds * (size_t)kTop + 2 * kIds +
                   (wide ? 0 : align_up(2 * (size_t)n_col, 16));
  return 2 * kTop + 4 * kTop + (a > b ? a : b);
}
// The forms of greedy_team: rows in registers and the columns' numbers in
// shared memory; beyond (5,120 rows, 10,616 columns: wide) the rows' best
// values are read where they are needed and the columns' numbers lie behind the
// lists.  Neither takes a matrix that is smaller than the lists' scratch: for
// the few thousand entries of a thin one greedy() is enough.
enum GreedyForm { kGreedySmall, kGreedyTeam, kGreedyWide };
__device__ __forceinline__ GreedyForm greedy_form(int n_row, int n_col, int NT, int region_bytes) {
  const bool wide = n_row > kTeamRowsPer * NT || greedy_team_bytes(n_col, NT, false) > (size_t)region_bytes;
  if (NT < kTop || greedy_team_bytes(n_col, NT, wide) > (size_t)region_bytes ||
      8 * (size_t)n_row * n_col < kListBytes + (wide ? 2 * (size_t)n_col : 0))
    return kGreedySmall;
  return wide ? kGreedyWide : kGreedyTeam;
}

// X: the pair's X_K (or a caller's matrix), row-major n_row x n_col, complete
// and visible to the team.  lists: scratch of 8 n_row n_col bytes; ms: n_row
// ints (row matches), then n_col bytes (column flags); best: n_row ints.  Ends
// with a team barrier.  Returns the score on every thread.
// (5,200 x 5,200 given, near rank one: 11.3 ms in the wide form, 5,000 x 5,200 9.2
// ms in the other; one CTA with greedy(), the team waiting, 7.6 s.  152 such pairs,
// a CTA each: 0.25 s in phases, 12.4 s with greedy().)
template <int NT, bool kWide>
__device__ __noinline__ float greedy_team(const Team& tm, TeamSh& sh, const float* X, int n_row, int n_col,
                                          uint2* lists, int32_t* ms, uint32_t* best, unsigned char* region,
                                          int32_t* mo, int pidx) {
  constexpr int NW = NT / 32;
  const int t = threadIdx.x, lane = t & 31, w = t >> 5;
  const int i0 = (int)((int64_t)n_row * tm.c / tm.T), i1 = (int)((int64_t)n_row * (tm.c + 1) / tm.T);
  int32_t* mrow = ms;
  unsigned char* gdead = reinterpret_cast<unsigned char*>(ms + n_row);
  int* glen = reinterpret_cast<int*>(lists + kTop * kLen);
  uint16_t* sel = reinterpret_cast<uint16_t*>(region);
  int* len = reinterpret_cast<int*>(sel + kTop);
  unsigned char* dead = reinterpret_cast<unsigned char*>(len + kTop);
  unsigned char* rest = dead + align_up((size_t)n_col, 16);
  int* pre = kWide ? reinterpret_cast<int*>(rest) + kBins : &sh.pre[0][0];  // [rows' block][warp]
  const int K = min(kLen, n_col), M = kWide ? ceil_div(n_row, NT) : kTeamRowsPer;
  for (int i = i0 + t; i < i1; i += NT) mrow[i] = -1;
  if (tm.c == 0)
    for (int j = t; j < n_col; j += NT) gdead[j] = 0;
  team_sum(tm, sh, 0.f);
  const int need = min(n_row, n_col);
  int matched = 0;
  while (matched < need) {
    for (int j = t; j < n_col; j += NT) dead[j] = gdead[j];
    int* bins = reinterpret_cast<int*>(rest);
    for (int q = t; q < kBins; q += NT) bins[q] = 0;
    __syncthreads();
    const int cw = ceil_div(n_col, 32), side = cw <= 2 ? 16 / cw : 0;
    // short rows: as many of them as give 16 loads in flight (for up to eight
    // chunks of columns in place of two, 2 % slower at 200 columns)
    if (side) {
      for (int i = i0 + w; i < i1; i += NW * side) {
        const int mine = i + NW * lane;
        const unsigned live = __ballot_sync(0xffffffffu, lane < side && mine < i1 && mrow[min(mine, i1 - 1)] < 0);
        float v[16];
#pragma unroll
        for (int u = 0, r = 0, c = 0; u < 16; ++u) {
          const int j = 32 * c + lane;
          v[u] = (live >> r & 1u) && j < n_col ? X[(size_t)(i + NW * r) * n_col + j] : -CUDART_INF_F;
          if (++c == cw) {
            c = 0;
            ++r;
          }
        }
        uint32_t k = 0;
#pragma unroll
        for (int u = 0, r = 0, c = 0; u < 16; ++u) {
          const int j = 32 * c + lane;
          if (v[u] > -CUDART_INF_F && !dead[j]) k = max(k, okey(v[u]));
          if (++c == cw) {
            k = __reduce_max_sync(0xffffffffu, k);
            if (lane == 0 && r < side && i + NW * r < i1) best[i + NW * r] = k;
            k = 0;
            c = 0;
            ++r;
          }
        }
      }
    }
    for (int i = i0 + w; !side && i < i1; i += NW) {
      uint32_t k = 0;
      if (mrow[i] < 0) {
        const float* x = X + (size_t)i * n_col;
        for (int j0 = lane; j0 < n_col; j0 += 512) {
          float v[16];
#pragma unroll
          for (int u = 0; u < 16; ++u) v[u] = j0 + 32 * u < n_col ? x[j0 + 32 * u] : 0.f;
#pragma unroll
          for (int u = 0; u < 16; ++u) {
            const int j = j0 + 32 * u;
            if (j < n_col && !dead[j] && v[u] > -CUDART_INF_F) k = max(k, okey(v[u]));
          }
        }
        k = __reduce_max_sync(0xffffffffu, k);
      }
      if (lane == 0) best[i] = k;
    }
    team_sum(tm, sh, 0.f);
    if (sh.fail) return 0.f;
    // the listed rows (every CTA finds the same ones): all rows down to a bin
    // of best values, at most kTop of them
    uint32_t v[kTeamRowsPer];
    if constexpr (!kWide) {
#pragma unroll
      for (int m = 0; m < kTeamRowsPer; ++m) v[m] = t + NT * m < n_row ? best[t + NT * m] : 0u;
    }
    auto value = [&](int m) -> uint32_t {
      if constexpr (kWide)
        return t + NT * m < n_row ? best[t + NT * m] : 0u;
      else
        return v[m];
    };
    uint32_t vmax = 0, vmin = 0xffffffffu;
#pragma unroll
    for (int m = 0; m < M; ++m) {
      const uint32_t k = value(m);
      vmax = max(vmax, k);
      if (k) vmin = min(vmin, k);
    }
    const uint64_t mm = block_max2<NW>(sh, vmax, ~vmin, lane, w);
    vmax = (uint32_t)(mm >> 32);
    if (vmax == 0u) break;  // no entry is left that can be taken
    vmin = ~(uint32_t)mm;
    int shift = max(0, 32 - __clz(vmax - vmin) - 8), bin;
    for (;;) {
#pragma unroll
      for (int m = 0; m < M; ++m) {
        const uint32_t k = value(m), q = (vmax - k) >> shift;
        if (k && q < (uint32_t)kBins) atomicAdd(&bins[q], 1);
      }
      __syncthreads();
      if (w == 0) {  // the last bin that keeps the count within kTop
        int run = 0, last = -1;
        for (int q0 = 0; q0 < kBins; q0 += 32) {
          int c = bins[q0 + lane];
#pragma unroll
          for (int o = 1; o < 32; o <<= 1) {
            const int u = __shfl_up_sync(0xffffffffu, c, o);
            if (lane >= o) c += u;
          }
          c += run;
          const unsigned ok = __ballot_sync(0xffffffffu, c <= kTop);
          if (ok) last = q0 + 31 - __clz(ok);  // counts do not fall: a prefix of the lanes
          run = __shfl_sync(0xffffffffu, c, 31);
          if (ok != 0xffffffffu) break;
        }
        if (lane == 0) sh.bin = last;
      }
      __syncthreads();
      bin = sh.bin;
      if (bin >= 0 || shift == 0) break;
      // the first bin alone holds more than kTop rows: its own range in bins
      shift = max(0, shift - 8);
      for (int q = t; q < kBins; q += NT) bins[q] = 0;
      __syncthreads();
    }
    // (more than kTop rows of the largest value: the first kTop of them by index)
    auto listed = [&](uint32_t k) { return k != 0u && (bin >= 0 ? (vmax - k) >> shift <= (uint32_t)bin : k == vmax); };
    uint64_t below = 0;  // the best row that is not listed
#pragma unroll
    for (int m = 0; m < M; ++m) {
      const unsigned b = __ballot_sync(0xffffffffu, listed(value(m)));
      if (lane == 0) pre[32 * m + w] = __popc(b);
    }
    __syncthreads();
    if (w == 0) {  // exclusive prefix over (m, warp)
      int run = 0;
      for (int e0 = 0; e0 < NW * ceil_div(n_row, NT); e0 += 32) {
        const int m = (e0 + lane) / NW, q = (e0 + lane) % NW;
        const int c = m < M ? pre[32 * m + q] : 0;
        int inc = c;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
          const int u = __shfl_up_sync(0xffffffffu, inc, o);
          if (lane >= o) inc += u;
        }
        if (m < M) pre[32 * m + q] = run + inc - c;
        run += __shfl_sync(0xffffffffu, inc, 31);
      }
      if (lane == 0) sh.nl = min(run, kTop);
    }
    __syncthreads();
#pragma unroll
    for (int m = 0; m < M; ++m) {
      const uint32_t k = value(m);
      const bool in = listed(k);
      const unsigned b = __ballot_sync(0xffffffffu, in);
      const int i = t + NT * m, at = in ? pre[32 * m + w] + __popc(b & ((1u << lane) - 1u)) : kTop;
      if (at < kTop) {
        sel[at] = (uint16_t)i;
      } else if (k) {
        const uint64_t q = ((uint64_t)k << 16) | (uint32_t)(0xffff - i);
        below = q > below ? q : below;
      }
    }
    const uint64_t out = block_max_u64<NW>(sh, below, lane, w);  // also: sel complete
    const int nl = sh.nl;
    uint2* cand = reinterpret_cast<uint2*>(rest) + w * kCand;
    for (int s = w * tm.T + tm.c; s < nl; s += NW * tm.T) {
      const int l = list_row(X + (size_t)sel[s] * n_col, n_col, dead, K, cand, lists + s * kLen, lane);
      if (lane == 0) glen[s] = l;
    }
    team_sum(tm, sh, 0.f);
    if (sh.fail) return 0.f;
    int made = 0;
    if (tm.c == 0) {
      uint32_t* key = reinterpret_cast<uint32_t*>(dead);  // the flags and candidates are done with
      uint16_t* col = reinterpret_cast<uint16_t*>(key + kKeyPitch * kLen);
      unsigned char* inv = reinterpret_cast<unsigned char*>(col + kColPitch * kLen);
      uint16_t* idcol = reinterpret_cast<uint16_t*>(inv + kIds * kTop);
      unsigned short* id = kWide ? reinterpret_cast<unsigned short*>(lists) + kListBytes / 2
                                 : reinterpret_cast<unsigned short*>(idcol + kIds);  // column -> number
      for (int s = t; s < nl; s += NT) len[s] = glen[s];
      for (int q = t; q < kIds * kTop / 16; q += NT)
        reinterpret_cast<uint4*>(inv)[q] = make_uint4(0xffffffffu, 0xffffffffu, 0xffffffffu, 0xffffffffu);
      for (int j = t; j < n_col; j += NT) id[j] = 0xffffu;
      if (t == 0) sh.ids = 0;
#pragma unroll 4
      for (int e = t; e < nl * kLen; e += NT) {  // entries past a list's length are not read
        const int s = e / kLen, k = e - s * kLen;
        const uint2 a = lists[e];
        key[k * kKeyPitch + s] = a.x;
        col[k * kColPitch + s] = (uint16_t)a.y;
      }
      __syncthreads();
      // number the columns: every list's first, then the others, best entries first
      for (int part = 0; part < 2; ++part) {
        for (int e = (part ? nl : 0) + t; e < (part ? nl * kLen : nl); e += NT) {
          const int k = e / nl, s = e - k * nl;
          if (k >= (len[s] & 255)) continue;
          const int j = col[k * kColPitch + s];
          if (id[j] == 0xffffu && atomicCAS(&id[j], (unsigned short)0xffffu, (unsigned short)0xfffeu) == 0xffffu) {
            const int q = atomicAdd(&sh.ids, 1);
            if (q < kIds) {
              idcol[q] = (uint16_t)j;
              id[j] = (unsigned short)q;  // 0xfffe: no number left
            }
          }
        }
        __syncthreads();
      }
      for (int s = t; s < nl; s += NT) {
        const int n = len[s] & 255;
        int k = 0;
        for (; k < n; ++k) {
          const int q = id[col[k * kColPitch + s]];
          if (q >= kIds) break;
          col[k * kColPitch + s] = (uint16_t)q;
          inv[q * kTop + s] = (unsigned char)k;
        }
        if (k < n) len[s] = k;
      }
      // the best row that is not listed, as the steps compare it
      const uint32_t okey_out = (uint32_t)(out >> 16);
      int olist = 0;
      if (t < kTop) {
        const int orow = 0xffff - (int)(out & 0xffffu);
        olist = __popc(__ballot_sync(0xffffffffu, t < nl && (int)sel[t] < orow));
        if (lane == 0) sh.redi[w] = olist;
      }
      __syncthreads();
      olist = 0;
      for (int q = 0; q < kTop / 32; ++q) olist += sh.redi[q];
      if (t < kTop)
        made = team_steps(sh, nl, need - matched, key, col, inv, idcol, len, sel, okey_out, olist, mrow, gdead);
    }
    const int got = (int)team_sum(tm, sh, t == 0 ? (float)made : 0.f);
    if (sh.fail) return 0.f;
    if (got <= 0) break;  // (not reached: a phase takes the largest live entry)
    matched += got;
  }
  if (matched < need && tm.c == 0 && t == 0) set_status(tm.hdr, 6 /* CF_ERR_NUMERIC */, pidx);
  float sc = 0.f;
  if (tm.c == 0) {
    for (int i = t; i < n_row; i += NT) {
      const int c = mrow[i];
      if (c >= 0) sc += X[(size_t)i * n_col + c];
      if (mo) mo[i] = c;
    }
  }
  return team_sum(tm, sh, sc);
}

// rounds_pay for a matrix in memory, by the CTA: of 16 lines of the shorter side,
// a warp each, four or more are the best of their best entry's other line; of
// four, three where that side is short (16 would be the whole matrix, and in a
// random one nearly all of them are).
template <int NT>
__device__ __forceinline__ bool rounds_pay_t(TeamSh& sh, const float* X, int n_row, int n_col) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  static_assert(NT >= 512, "a warp per line");
  const int S = min(n_row, n_col), L = max(n_row, n_col);
  const size_t sa = n_row <= n_col ? n_col : 1, sb = n_row <= n_col ? 1 : n_col;  // from line to line, along a line
  auto key_at = [&](int q, int e) -> uint32_t {
    const float v = q < S && e < L ? X[q * sa + e * sb] : -CUDART_INF_F;
    return v > -CUDART_INF_F ? okey(v) : 0u;
  };
  const int lines = S < 32 ? 4 : 16;
  if (w < lines) {
    const int line = (int)((int64_t)S * w / lines);
    uint32_t k = 0u;
    int at = 0;
    for (int e0 = lane; e0 < L; e0 += 256) {
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        const uint32_t q = key_at(line, e0 + 32 * u);
        if (q > k) {
          k = q;
          at = e0 + 32 * u;
        }
      }
    }
    const uint32_t best = __reduce_max_sync(0xffffffffu, k);
    at = __reduce_min_sync(0xffffffffu, k == best ? at : 0x7fffffff);
    bool less = best == 0u;
    for (int q0 = lane; q0 < S; q0 += 256) {
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        const int q = q0 + 32 * u;
        const uint32_t x = key_at(q, at);
        less |= x > best || (x == best && q < line);
      }
    }
    less = __any_sync(0xffffffffu, less);
    if (lane == 0) sh.redi[w] = !less;
  }
  __syncthreads();
  const int pay = __popc(__ballot_sync(0xffffffffu, lane < lines && sh.redi[lane]));
  __syncthreads();
  return pay >= (S < 32 ? 3 : 4);
}

// The matching of a team's pair: X row-major n_row x n_col, written by the team
// (or the caller's); lists: scratch of two matrices; the slot's state arrays.
// Ends with a team barrier.  kGiven: the caller's matrix, which need not be close
// to rank one; one CTA then takes it by rounds where they pay (a team's phases
// are the faster all the same).
template <int NT, bool kGiven>
__device__ __forceinline__ void match_pair_t(const Ctx& cx, const Geo& g, const Team& tm, TeamSh& sh, float* slot,
                                             const float* X, float* lists, unsigned char* region, int region_bytes) {
  const int t = threadIdx.x, n_row = g.na, n_col = g.nb;
  float* rn = slot + 3 * team_elems(n_row, n_col);
  int32_t* ms = reinterpret_cast<int32_t*>(rn + n_row + n_col);
  int32_t* mo = cx.match ? cx.match + cx.m_off[g.p] : nullptr;
  GreedyForm form = greedy_form(n_row, n_col, NT, region_bytes);
  if (kGiven && tm.T == 1 && form != kGreedySmall && rounds_pay_t<NT>(sh, X, n_row, n_col)) form = kGreedySmall;
  if (form != kGreedySmall) {
    uint2* ls = reinterpret_cast<uint2*>(lists);
    uint32_t* best = reinterpret_cast<uint32_t*>(rn);
    const float sc = form == kGreedyWide
                         ? greedy_team<NT, true>(tm, sh, X, n_row, n_col, ls, ms, best, region, mo, g.p)
                         : greedy_team<NT, false>(tm, sh, X, n_row, n_col, ls, ms, best, region, mo, g.p);
    if (cx.scores && tm.c == 0 && t == 0) cx.scores[g.p] = sc;
    return;
  }
  team_sum(tm, sh, 0.f);
  if (sh.fail) return;
  if (tm.c == 0) {
    const Group cta{t, NT, 0, sh.redw, sh.redi};
    int16_t* st = reinterpret_cast<int16_t*>(region);
    const float sc = greedy<int16_t, 8>(cta, X, n_col, n_row, n_col, 0, st, st + n_row, st + n_row + n_col, mo, cx.hdr,
                                        g.p);
    if (cx.scores && t == 0) cx.scores[g.p] = sc;
    __syncthreads();  // team_sum takes redw, which greedy's last sum was read from
  }
  team_sum(tm, sh, 0.f);
}

// One pair on a team.  Slot: [E | Y | Y'] (n_row rows of ld floats each, ld =
// n_col rounded up to 8: bulk copies take multiples of 16 bytes), row and
// column norms, matching state.  E holds the unscaled attribute term: Y_0 = E
// with s_0 = 1 / |E|_F, and (1 - alpha) Ehat = (1 - alpha) / |E|_F E, so no
// pass scales it.  A tall pair's matrices are kept transposed up to X_K.
template <int NT>
__device__ __noinline__ void run_pair_t(const Ctx& cx, const Geo& given, const Team& tm, TeamSh& sh, float* slot,
                                        unsigned char* region, int region_bytes) {
  constexpr int NW = NT / 32, NC = kConsumers<NT>;
  const int t = threadIdx.x, lane = t & 31, w = t >> 5;
  const bool tr = team_tr(given.na, given.nb);
  const Geo g = tr ? swapped(given) : given;
  const int n_row = g.na, n_col = g.nb;
  const uint32_t ld = (uint32_t)team_ld(n_col), ld4 = 4 * ld;
  const size_t E = (size_t)n_row * ld;
  float* eb = slot;
  float* b0 = eb + E;
  float* b1 = b0 + E;
  float* rn = b1 + E;
  const int i0 = (int)((int64_t)n_row * tm.c / tm.T), i1 = (int)((int64_t)n_row * (tm.c + 1) / tm.T);
  const int nr = i1 - i0, nr_max = ceil_div(n_row, tm.T);

  // the columns' kinds, the busy rows (both at the region's end for now: the
  // ring's place)
  const int words = ceil_div(max(n_col, n_row), 32);
  if (t == 0) {
    sh.tb = 0;
    sh.tbp = 0;
    sh.nbr = 0;
    sh.tr = 0;
    sh.trp = 0;
  }
  __syncthreads();
  const size_t tmp_bytes = align_up(16 * (size_t)words, 16);
  uint32_t* m0 = reinterpret_cast<uint32_t*>(region + region_bytes - tmp_bytes);
  uint32_t* mb = m0 + words;
  uint32_t* p0 = mb + words;
  uint32_t* pb = p0 + words;
  for (int i = t; i < n_row; i += NT) {
    const int od = __ldg(g.r_optr + i + 1) - __ldg(g.r_optr + i), id = __ldg(g.r_iptr + i + 1) - __ldg(g.r_iptr + i);
    if (od > 2 || id > 2) {
      atomicAdd(&sh.nbr, 1);
      atomicAdd(&sh.tr, od + id);
    }
  }
  for (int wd = w; wd < words; wd += NW) {
    const int j = 32 * wd + lane;
    int od = 0, id = 0;
    if (j < n_col) {
      od = __ldg(g.c_optr + j + 1) - __ldg(g.c_optr + j);
      id = __ldg(g.c_iptr + j + 1) - __ldg(g.c_iptr + j);
    }
    const bool busy = od > 2 || id > 2;
    const unsigned k0 = __ballot_sync(0xffffffffu, j < n_col && od <= 1 && id <= 1);
    const unsigned kb = __ballot_sync(0xffffffffu, busy);
    if (lane == 0) {
      m0[wd] = k0;
      mb[wd] = kb;
    }
    if (busy) atomicAdd(&sh.tb, od + id);
  }
  __syncthreads();
  if (w == 0) mask_prefix(m0, mb, p0, pb, words, lane, &sh.n0, &sh.nb);
  __syncthreads();
  const int n0 = sh.n0, nb = sh.nb, nnb = n_col - nb, nbr = sh.nbr, nch = ceil_div(nnb, 32);
  int CH, wpr, rg;
  team_split(max(nch, 1), NC, CH, wpr, rg);
  // what stays beside the ring; the same on every CTA of the team (the storage
  // order depends on whether it fits)
  const int e_row = __ldg(g.r_optr + n_row) - __ldg(g.r_optr);
  const size_t c16 = align_up(2 * (size_t)n_col, 16);
  // rows an iteration can bring: each row's E, and its neighbours at most
  const size_t most = (size_t)nr_max + (size_t)min((int64_t)4 * nr_max, (int64_t)2 * e_row);
  // a warp's missing last chunks are read all the same: room past the last buffer
  const size_t slack = 128 * (size_t)((CH <= 4 ? CH : kMaxChunks) - CH + 2);
  const int ps = n0 / 32 * 32;  // the second neighbours' first position
  const size_t cb_bytes = 16 * (size_t)max(0, 32 * nch - ps);
  const size_t keep = c16 + 16 * (size_t)nb + align_up(8 * (size_t)sh.tb, 16) + 20 * (size_t)nbr +
                      8 * (size_t)sh.tr + 16 + 48 * (size_t)nr_max + 5 * align_up(2 * most, 16) +
                      2 * align_up(2 * (size_t)nr_max + 2, 16) + 16 * 32 * kBusyWarps + 16 * kStepRing + 64 + slack +
                      cb_bytes;
  const size_t avail = (size_t)region_bytes > keep ? (size_t)region_bytes - keep : 0;
  // the staging's own needs, in the ring's place: column records and
  // positions, masks, and the schedule's tables
  const size_t stage = 16 * (size_t)n_col + 2 * c16 + 2 * (size_t)n_row + 2 * align_up(2 * most, 16) + tmp_bytes + 64;
  const int S = (int)min((size_t)kMaxRing, avail / ld4);
  const int rows_per_warp = CH == 1 ? 2 : 1;
  while (rg > 1 && S < 7 * rg * rows_per_warp) rg /= 2;  // a step's rows must leave room for the next ones
  const int rps = rg * rows_per_warp;
  const bool staged = CH <= kMaxChunks && nch > 0 && S >= max(kMinRing, 7 * rps) && stage <= avail && most < 32768 &&
                      n_row < 32768;
  if (staged) {
    unsigned char* at = region;
    auto take = [&](size_t bytes) {
      unsigned char* p = at;
      at += align_up(bytes, 16);
      return p;
    };
    uint16_t* cnat = reinterpret_cast<uint16_t*>(take(2 * (size_t)n_col));
    int4* bran = reinterpret_cast<int4*>(take(16 * (size_t)nb));
    int2* cedge = reinterpret_cast<int2*>(take(8 * (size_t)sh.tb));
    int4* brow = reinterpret_cast<int4*>(take(16 * (size_t)nbr));
    int2* redge = reinterpret_cast<int2*>(take(8 * (size_t)sh.tr));
    uint32_t* browo = reinterpret_cast<uint32_t*>(take(4 * (size_t)nbr));
    int4* rec = reinterpret_cast<int4*>(take(48 * (size_t)nr_max));
    uint16_t* src = reinterpret_cast<uint16_t*>(take(2 * most));
    uint16_t* buf = reinterpret_cast<uint16_t*>(take(2 * most));
    uint16_t* cnt = reinterpret_cast<uint16_t*>(take(2 * most));
    uint16_t* req = reinterpret_cast<uint16_t*>(take(2 * most));
    uint16_t* stp = reinterpret_cast<uint16_t*>(take(2 * most));
    uint16_t* first = reinterpret_cast<uint16_t*>(take(2 * (size_t)nr_max + 2));
    uint16_t* rows = reinterpret_cast<uint16_t*>(take(2 * (size_t)nr_max + 2));
    int4* blane = reinterpret_cast<int4*>(take(16 * 32 * kBusyWarps));
    const uint32_t full = (uint32_t)__cvta_generic_to_shared(take(16 * kStepRing));
    int4* cB = reinterpret_cast<int4*>(take(cb_bytes));
    int4* cA = reinterpret_cast<int4*>(at);
    uint16_t* cpos = reinterpret_cast<uint16_t*>(cA + n_col);
    uint16_t* corder = reinterpret_cast<uint16_t*>(reinterpret_cast<unsigned char*>(cpos) + c16);
    int16_t* last = reinterpret_cast<int16_t*>(reinterpret_cast<unsigned char*>(corder) + c16);
    uint16_t* use = reinterpret_cast<uint16_t*>(last + n_row);
    uint16_t* what = use + most;
    for (int j = t; j < n_col; j += NT) {
      const int wd = j >> 5;
      const uint32_t bit = 1u << (j & 31), lt = bit - 1u;
      const int r0 = (int)p0[wd] + __popc(m0[wd] & lt), rb = (int)pb[wd] + __popc(mb[wd] & lt);
      const int by = (m0[wd] & bit) ? r0 : (mb[wd] & bit) ? nnb + rb : n0 + j - r0 - rb;  // in order of kind
      const int ch = by >> 5;
      const int pos = by >= nnb ? by : 32 * (chunk_first(ch % wpr, nch, wpr) + ch / wpr) + (by & 31);
      cpos[j] = (uint16_t)pos;
      corder[j] = (uint16_t)by;
      cnat[pos] = (uint16_t)j;
    }
    for (int i = t; i < n_row; i += NT) last[i] = -1;
    for (int p = max(nnb, ps) + t; p < 32 * nch; p += NT) cB[p - ps] = make_int4(0, 0, 0, 0);
    if (t < 2 * kStepRing) {  // full: the copying warp's arrival; empty: every working warp's
      const int n = t < kStepRing ? 1 : wpr * rg + (nb > 0 ? kBusyWarps : 0);
      asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(full + 8u * t), "r"(n) : "memory");
    }
    __syncthreads();
    for (int j = t; j < n_col; j += NT) {
      const int by = corder[j];
      const int o0 = __ldg(g.c_optr + j), o1 = __ldg(g.c_optr + j + 1);
      const int q0 = __ldg(g.c_iptr + j), q1 = __ldg(g.c_iptr + j + 1);
      const CfAdj z{0, 0.f};
      const CfAdj a0 = o1 > o0 ? ldg_adj(g.c_oadj + o0) : z, a1 = o1 > o0 + 1 ? ldg_adj(g.c_oadj + o0 + 1) : z;
      const CfAdj d0 = q1 > q0 ? ldg_adj(g.c_iadj + q0) : z, d1 = q1 > q0 + 1 ? ldg_adj(g.c_iadj + q0 + 1) : z;
      cA[by] = make_int4(4 * cpos[a0.nbr], __float_as_int(a0.w), 4 * cpos[d0.nbr], __float_as_int(d0.w));
      if (by >= ps && by < nnb) cB[by - ps] = make_int4(4 * cpos[a1.nbr], __float_as_int(a1.w), 4 * cpos[d1.nbr], __float_as_int(d1.w));
      if (by >= nnb) {
        const int od = o1 - o0, id = q1 - q0;
        const int to = atomicAdd(&sh.tbp, od + id);
        const int b0a = (int)__cvta_generic_to_shared(cedge + to);  // byte addresses
        bran[by - nnb] = make_int4(b0a, b0a + 8 * od, b0a + 8 * od, b0a + 8 * (od + id));
        for (int e = 0; e < od; ++e) {
          const CfAdj a = ldg_adj(g.c_oadj + o0 + e);
          cedge[to + e] = make_int2(4 * cpos[a.nbr], __float_as_int(a.w));
        }
        for (int e = 0; e < id; ++e) {
          const CfAdj a = ldg_adj(g.c_iadj + q0 + e);
          cedge[to + od + e] = make_int2(4 * cpos[a.nbr], __float_as_int(a.w));
        }
      }
    }
    __syncthreads();
    // the row graph's busy rows, in index order
    row_masks<NW>(g, n_row, words, m0, mb, lane, w);
    __syncthreads();
    if (w == 0) mask_prefix(m0, mb, p0, pb, words, lane, &sh.nbs, &sh.nbs);
    __syncthreads();
    const int base = i0 - ((int)p0[i0 >> 5] + __popc(m0[i0 >> 5] & ((1u << (i0 & 31)) - 1u)));  // rows before, not busy
    for (int i = t; i < n_row; i += NT) {
      const uint32_t m = m0[i >> 5], bit = 1u << (i & 31);
      const int b = (int)p0[i >> 5] + __popc(m & (bit - 1u));
      const int o0 = __ldg(g.r_optr + i), o1 = __ldg(g.r_optr + i + 1);
      const int q0 = __ldg(g.r_iptr + i), q1 = __ldg(g.r_iptr + i + 1);
      if (m & bit) {
        const int od = o1 - o0, id = q1 - q0;
        const int to = atomicAdd(&sh.trp, od + id);
        brow[b] = make_int4(to, to + od, to + od, to + od + id);
        browo[b] = (uint32_t)i * ld4;
        for (int e = 0; e < od; ++e) {
          const CfAdj a = ldg_adj(g.r_oadj + o0 + e);
          redge[to + e] = make_int2((int)((uint32_t)a.nbr * ld4), __float_as_int(a.w));
        }
        for (int e = 0; e < id; ++e) {
          const CfAdj a = ldg_adj(g.r_iadj + q0 + e);
          redge[to + od + e] = make_int2((int)((uint32_t)a.nbr * ld4), __float_as_int(a.w));
        }
      } else if (i >= i0 && i < i1) {
        // the slab's rows: their neighbours for now (-1: none), the buffers after the schedule
        const int r = i - b - base;
        const CfAdj z{-1, 0.f};
        const CfAdj a0 = o1 > o0 ? ldg_adj(g.r_oadj + o0) : z, a1 = o1 > o0 + 1 ? ldg_adj(g.r_oadj + o0 + 1) : z;
        const CfAdj d0 = q1 > q0 ? ldg_adj(g.r_iadj + q0) : z, d1 = q1 > q0 + 1 ? ldg_adj(g.r_iadj + q0 + 1) : z;
        rec[3 * r] = make_int4(a0.nbr, d0.nbr, a1.nbr, d1.nbr);
        rec[3 * r + 1] = make_int4(__float_as_int(a0.w), __float_as_int(d0.w), __float_as_int(a1.w), __float_as_int(d1.w));
        rec[3 * r + 2] = make_int4(i, (int)((uint32_t)i * ld4), 0, 0);
      }
    }
    if (t == 0) {
      TeamStage& st = sh.st;
      const int li = i1 > i0 ? i1 - 1 : i0;  // rows of the slab that are not busy
      const uint32_t m = m0[li >> 5], bit = 1u << (li & 31);
      st.nr = i1 > i0 ? li - ((int)p0[li >> 5] + __popc(m & (bit - 1u))) - base + (m & bit ? 0 : 1) : 0;
      st.cA = cA;
      st.cb = (uint32_t)__cvta_generic_to_shared(cB) - 16u * (uint32_t)ps;
      st.brow = brow;
      st.browo = browo;
      st.redge = redge;
      st.src = src;
      st.buf = buf;
      st.cnt = cnt;
      st.rows = rows;
      st.blane = (uint32_t)__cvta_generic_to_shared(blane);
      st.req = req;
      st.stp = stp;
      st.first = first;
      st.bran = (uint32_t)__cvta_generic_to_shared(bran);
      st.cedge = (uint32_t)__cvta_generic_to_shared(cedge);
      st.rec = (uint32_t)__cvta_generic_to_shared(rec);
      st.full = full;
      st.empty = full + 8 * kStepRing;
      st.ring = (uint32_t)__cvta_generic_to_shared(at);
      st.rowb = ld4;
      st.S = S;
      st.n0 = n0;
      st.nnb = nnb;
      st.nb = nb;
      st.nbr = nbr;
      st.rps = rps;
      st.nsteps = ceil_div(st.nr, rps);
      st.ncopy = 0;
      st.nch = nch;
      st.wpr = wpr;
      st.rg = rg;
    }
    __syncthreads();
    if (w == NC + kBusyWarps) team_schedule(sh.st, rec, last, use, what, lane);
    if (w == NC) busy_lanes(sh.st, bran, blane, lane);
  }
  if (!staged) {  // the rows with more than two neighbours, in index order
    uint16_t* rows = reinterpret_cast<uint16_t*>(region);
    row_masks<NW>(g, n_row, words, m0, mb, lane, w);
    __syncthreads();
    if (w == 0) mask_prefix(m0, mb, p0, pb, words, lane, &sh.nbs, &sh.nbs);
    __syncthreads();
    for (int i = t; i < n_row; i += NT) {
      const uint32_t m = m0[i >> 5], bit = 1u << (i & 31);
      if (m & bit) rows[p0[i >> 5] + __popc(m & (bit - 1u))] = (uint16_t)i;
    }
  }
  const uint16_t* cnat = reinterpret_cast<const uint16_t*>(region);
  for (int i = i0 + t; i < i1; i += NT) rn[i] = attr_norm(g.r_attr + (size_t)i * cx.Fp, cx.om, cx.Fp);
  __syncthreads();

  // a3: E over the slab, four rows of a column at a time, and |E|_F
  float ss = 0.f;
  {
    const int nw = ceil_div(n_col, 32), nq = cx.Fp >> 2, groups = ceil_div(nr, 4);
    const float4* o4 = reinterpret_cast<const float4*>(cx.om);
    for (int q = w; q < nw * groups; q += NW) {
      const int gr = q / nw, p = 32 * (q - gr * nw) + lane;
      if (p >= n_col) continue;
      const int j = staged ? cnat[p] : p;
      const float4* cv = reinterpret_cast<const float4*>(g.c_attr + (size_t)j * cx.Fp);
      const int r0 = 4 * gr, m = min(4, nr - r0);
      float acc[4] = {0.f, 0.f, 0.f, 0.f}, nrm = 0.f;
      const float4* rv = reinterpret_cast<const float4*>(g.r_attr + (size_t)(i0 + r0) * cx.Fp);
      for (int f = 0; f < nq; ++f) {
        const float4 v = __ldg(cv + f), o = o4[f];
        nrm = fmaf(o.x * v.x, v.x, nrm);
        nrm = fmaf(o.y * v.y, v.y, nrm);
        nrm = fmaf(o.z * v.z, v.z, nrm);
        nrm = fmaf(o.w * v.w, v.w, nrm);
#pragma unroll
        for (int r = 0; r < 4; ++r) {
          const float4 u = __ldg(rv + (size_t)min(r, m - 1) * nq + f);
          acc[r] = fmaf(o.x * u.x, v.x, acc[r]);
          acc[r] = fmaf(o.y * u.y, v.y, acc[r]);
          acc[r] = fmaf(o.z * u.z, v.z, acc[r]);
          acc[r] = fmaf(o.w * u.w, v.w, acc[r]);
        }
      }
      const float cj = sqrtf(nrm);
#pragma unroll
      for (int r = 0; r < 4; ++r)
        if (r < m) {
          const float den = rn[i0 + r0 + r] * cj;
          const float e = den > 0.f ? acc[r] / den : 0.f;
          eb[(size_t)(i0 + r0 + r) * ld + p] = e;
          ss = fmaf(e, e, ss);
        }
    }
  }
  fence_async();
  const float tot = team_sum(tm, sh, ss);
  if (sh.fail) return;
  float inv = 1.f;
  if (tot > 0.f) {
    inv = 1.0f / sqrtf(tot);
  } else {
    const float uni = 1.0f / sqrtf((float)n_row * (float)n_col);
    for (size_t q = (size_t)i0 * ld + t; q < (size_t)i1 * ld; q += NT) eb[q] = uni;
    fence_async();
    team_sum(tm, sh, 0.f);
  }
  const float cbi = (1.f - cx.alpha) * inv;

  // a4: K renormalised iterations, one team barrier each
  float sk = inv;
  if (staged) {
    const TeamIter it{eb, b0, b1, cx.alpha, inv, cbi, cx.K, cx.norm_mode};
    sk = team_iterate<NT>(tm, sh, it, CH);
  } else {
    sk = team_far<NT>(tm, sh, TeamIter{eb, b0, b1, cx.alpha, inv, cbi, cx.K, cx.norm_mode}, g, ld, i0, i1,
                      region, nbr);
  }
  if (sh.fail) return;
  // X_K in the caller's column order (rows of n_col): to the output, and for
  // the matching into b1 (the matching's lists then take E and b0)
  const float* Yk = cx.K == 0 ? eb : b0;
  float* Xn = b1;
  const bool want = cx.scores || cx.match;
  float* xo = cx.X ? cx.X + cx.x_off[g.p] : nullptr;
  for (int i = i0 + w; i < i1; i += NW)
    for (int p = lane; p < n_col; p += 32) {
      const float x = Yk[(size_t)i * ld + p] * sk;
      const int j = staged ? cnat[p] : p;
      const size_t to = tr ? (size_t)j * n_row + i : (size_t)i * n_col + j;
      if (xo) xo[to] = x;
      if (want) Xn[to] = x;
    }
  if (!want) {
    team_sum(tm, sh, 0.f);  // the slot is free for the next pair
    return;
  }
  match_pair_t<NT, false>(cx, given, tm, sh, slot, Xn, eb, region, region_bytes);
}

}  // namespace

}  // namespace cfsim
