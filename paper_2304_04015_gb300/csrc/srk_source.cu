// The source side of a query (steps a2-a3): the source's walks, their
// Fisher-Yates shuffle, the walk pairs with their step caps, and the end nodes
// of the pairs for the lockstep walks (srk_lockstep.cu).
//
// The shuffle.  The permutation sigma of the sequential loop "for t = N-1 down
// to 1: swap(sigma[t], sigma[k_t])" is resolved in parallel.  Position t >= 1
// is final after step t and receives the value that position k_t held just
// before step t.  Position p (p <= t) was last written before step t by the step
// t' = min{t' > t : k_t' = p}, which moved in the value position t' held before
// step t'; if no such step exists it still holds p.  Following these links
// gives sigma[t] (sigma[0]: the value of position 0 after all steps).  The links
// come from lists of the steps by k (about one step each, ln N for the first
// positions): first[q] is the smallest step of list q, succ[t] the next larger
// step of t's list.
//
// One cluster of 8 blocks of 1024 threads runs a query's phases with a cluster
// barrier between them, one cluster (of 1 to 8 blocks) per query of a batch.  Each phase is a few
// dependent reads of a few thousand threads, so it is the number of phases and
// the price of each step from one to the next that count: as 12 kernels the
// source side took 72 us at 2,018 walks and 139 us at 18,234, now 39 and 102 (of
// which most is the longest walk, a chain of up to 50 dependent reads).
#include <cooperative_groups.h>
#include <stdint.h>

#include <algorithm>

#include "srk_device.cuh"
#include "srk_internal.h"

namespace srk {

namespace cg = cooperative_groups;

constexpr int kSourceBlocks = 8;      // of a cluster (the portable most)
constexpr int kSourceThreads = 1024;

struct SourceShared {
  int32_t P[SRK_MAX_LEN + 2];      // stratum prefix
  int32_t hist[SRK_MAX_LEN + 2];   // this block's pairs by cap, then where they begin
  int32_t cnt[SRK_MAX_LEN + 2];    // pairs with cap >= i
  int32_t R[SRK_MAX_LEN + 2];      // nodes of the longer pairs
};

// Phases of one query by cluster `c` of `blocks`, to sigma (kRows false) or to the cap rows
// and, unless only the `rows` are wanted, the pair records.
template <bool kRows>
__device__ __forceinline__ void source_phases(cg::cluster_group &c, int blocks, bool rows,
                                              SourceShared &S, const GraphView &V, const QueryTab &t,
                                              const Workspace &w, const int32_t *act,
                                              int32_t n_act, int32_t u_begin, int32_t u_end) {
  const int32_t N = t.N_tot, L = t.L;
  const int32_t tid = (int32_t)c.block_rank() * kSourceThreads + (int32_t)threadIdx.x;
  const int32_t nth = blocks * kSourceThreads;
  const Small sm = small_view(w.small);
  int32_t *const head = w.head, *const next = w.next;  // the lists of steps by k
  for (int i = threadIdx.x; i <= L + 1; i += kSourceThreads) {
    S.P[i] = t.P[i];
    S.hist[i] = 0;
  }
  for (int i = tid; i < kSmallBytes / 4; i += nth) w.small[i] = 0;
  __syncthreads();

  // a2: walk r of length stratum(r); step i >= 1 moves to I(x)[k], k the bounded
  // draw below |I(x)| from word (i-1)&1 of the block (((i-1)>>1) << 24 | r, s);
  // it stops early at a node without in-neighbours.  Fisher-Yates draw t = r.
  const int Ls = L > 0 ? L : 1;
  const uint32_t s = (uint32_t)t.s;
  unsigned long long steps = 0;
  {
    const RoundKeys rk = round_keys(t.key0, t.key1);
    auto walks = [&](const auto &G) {
      uint32_t deg_s = 0;
      const int32_t b_s = node_start(G, V.row_ptr, t.s, deg_s);
      for (int32_t r = tid; r < N; r += nth) {
        head[r] = -1;
        w.kdraw[r] = r >= 1 ? fy_draw(rk, s, r) : 0;
        const int eff = source_walk(t.skey, G, s, b_s, deg_s, r, stratum_of(S.P, L, r),
                                    w.spos + (int64_t)r * Ls);
        w.seff[r] = eff;
        steps += (unsigned long long)eff;
      }
    };
    if (V.layout == kNarrow) walks(adj_view<kNarrow>(V));
    else walks(adj_view<kCsr>(V));
  }
  for (int off = 16; off > 0; off >>= 1) steps += __shfl_xor_sync(0xffffffffu, steps, off);
  c.sync();

  // a3: the lists, then the links
  if ((threadIdx.x & 31) == 0 && steps) atomicAdd(sm.ctr + 1, steps);
  for (int32_t r = tid; r < N; r += nth)
    if (r >= 1) next[r] = atomicExch(&head[w.kdraw[r]], r);
  c.sync();
  for (int32_t r = tid; r < N; r += nth) {
    int32_t lo = INT32_MAX;
    for (int32_t x = head[r]; x >= 0; x = next[x]) lo = min(lo, x);
    w.first[r] = lo == INT32_MAX ? -1 : lo;
    if (r >= 1) {
      lo = INT32_MAX;
      for (int32_t x = head[w.kdraw[r]]; x >= 0; x = next[x])
        if (x > r) lo = min(lo, x);
      w.succ[r] = lo == INT32_MAX ? -1 : lo;
    }
  }
  c.sync();

  // sigma[j], and the pair's step cap min(l2, steps of its source walk) (the
  // literal shuffle draws l2 per target) with its rank among the block's
  // pairs of that cap
  int32_t *packed = w.items;
  for (int32_t j = tid; j < N; j += nth) {
    const int32_t p = resolve_sigma(j, w.kdraw, w.first, w.succ, N);
    w.sigma[j] = p;
    if (kRows) {
      const int32_t cap = t.literal ? w.seff[p] : min(stratum_of(S.P, L, j), w.seff[p]);
      packed[j] = cap >= 1 ? cap << 22 | atomicAdd(&S.hist[cap], 1) : 0;
    }
  }
  if (!kRows) return;
  __syncthreads();
  for (int i = threadIdx.x; i <= L; i += kSourceThreads)
    if (i >= 1 && S.hist[i]) S.hist[i] = atomicAdd(&sm.cap_hist[i], S.hist[i]);
  c.sync();

  // cnt[i]: pairs with cap >= i (longest first); R[i]: where the nodes of the
  // pairs of cap i begin or, where only the rows are wanted, row i of the hit table
  for (int i = threadIdx.x; i <= L + 1; i += kSourceThreads)
    S.cnt[i] = i >= 1 && i <= L ? sm.cap_hist[i] : 0;
  __syncthreads();
  if (threadIdx.x == 0) {
    int32_t n = 0, r = 0;
    for (int i = L; i >= 1; --i) {
      const int32_t h = S.cnt[i];
      S.R[i] = r;
      r += i * h;
      n += h;
      S.cnt[i] = n;
    }
    S.cnt[0] = n;
    S.cnt[L + 1] = 0;
    S.R[0] = 0;
    S.R[L + 1] = r;
    if (rows) {
      r = 0;
      for (int i = 1; i <= L + 1; ++i) {
        S.R[i] = r;
        if (i <= L) r += S.cnt[i];
      }
    }
  }
  __syncthreads();
  if (c.block_rank() == 0) {
    for (int i = threadIdx.x; i <= L + 1; i += kSourceThreads) {
      sm.cnt[i] = S.cnt[i];
      sm.R[i] = S.R[i];
      if (i >= 1 && i <= L) sm.cursor[i] = S.cnt[i + 1];
    }
    if (threadIdx.x < 2) {
      // [act_lo, act_hi): the part of the ascending target list in [u_begin, u_end)
      const int32_t v = threadIdx.x == 0 ? u_begin : u_end;
      int32_t lo = 0, hi = n_act;  // first index with act[index] >= v
      if (v == 0) hi = 0;
      if (v == V.n) lo = n_act;
      while (lo < hi) {
        const int32_t mid = lo + (hi - lo) / 2;
        if (act[mid] < v) lo = mid + 1;
        else hi = mid;
      }
      int32_t *bounds = reinterpret_cast<int32_t *>(sm.ctr + 2);
      if (threadIdx.x == 0) {
        bounds[2] = lo;
        bounds[0] = rows ? lo : 0;  // the walk kernel's counter: targets, or units
      } else {
        bounds[1] = lo;
      }
    }
  }
  if (rows) return;

  // the pair records
  int4 *rec = w.rec();
  for (int32_t j = tid; j < N; j += nth) {
    const int32_t pk = packed[j], cap = pk >> 22;
    if (cap < 1) continue;
    const int32_t a = S.cnt[cap + 1] + S.hist[cap] + (pk & ((1 << 22) - 1));
    const int32_t x = w.sigma[j];
    w.pair_w[a] = __double2ull_rn(t.a[stratum_of(S.P, L, x)] * t.a[stratum_of(S.P, L, j)] *
                                  4294967296.0);
    const int32_t off = S.R[cap] + (a - S.cnt[cap + 1]) * cap;
    rec[a] = make_int4(j, cap, off, kNoFilter);
    const int32_t *src = w.spos + (int64_t)x * Ls;
    int32_t last = 0;
    for (int i = 0; i < cap; ++i) {
      last = src[i];
      w.Hc[off + i] = walk_identity(V, last);
    }
    w.pair_j[a] = walk_id(V, last);  // the end node
  }
}

// The end nodes of a query's pairs into the table and the bitmap (cleared
// before), room for every node's list and filter, and the pairs' places there.
__device__ __forceinline__ void end_phases(cg::cluster_group &c, int blocks, const Workspace &w,
                                           const Filters &F) {
  const int32_t tid = (int32_t)c.block_rank() * kSourceThreads + (int32_t)threadIdx.x;
  const int32_t nth = blocks * kSourceThreads;
  const Small sm = small_view(w.small);
  const int32_t n1 = sm.cnt[1], n2 = sm.cnt[2];  // pairs, and those of cap 2 and more
  int4 *rec = w.rec();
  const uint32_t mask = (1u << F.slot_bits) - 1u;
  for (int32_t a = tid; a < n1; a += nth) {
    const uint32_t id = (uint32_t)w.pair_j[a], hash = end_hash(id), bb = hash >> (32 - F.bloom_bits);
    atomicOr(&F.bloom[bb >> 5], 1u << (bb & 31));
    uint32_t sl = hash & mask;
    for (uint32_t probe = 0; probe <= mask; ++probe, sl = (sl + 1u) & mask) {
      const uint32_t prev = atomicCAS(&F.slots[sl].key, 0u, id + 1u);
      if (prev == 0u || prev == id + 1u) break;
    }
    F.slot_of[a] = (int32_t)sl;
    if (a >= n2) F.rank1[a] = atomicAdd(&F.slots[sl].cnt1, 1);
    else F.slots[sl].filt = kWantFilter;
  }
  c.sync();
  if (n1 > 0) {
    const int lane = threadIdx.x & 31;
    for (int32_t base = tid & ~31; base < (1 << F.slot_bits); base += nth) {
      EndSlot &E = F.slots[base + lane];
      if (E.cnt1 > 0) E.off1 = atomicAdd(&F.ctl[1], E.cnt1);
      int32_t at = -1, units = 0;
      if (E.filt == kWantFilter) {
        // 16 bits and more per node of the out-list, so that at most about 6 %
        // of the other nodes pass, up to the largest size (R-MAT 20: 0.7 KB on
        // average; one size of 4 KB for all was slower, a block then stops for
        // its filters every 4 pairs instead of every 11)
        const int32_t d = F.out_deg[E.key - 1u];
        int lg = 5;
        while (lg < kFilterMaxLg && (2 << lg) < d) ++lg;
        units = (1 << lg) / kFilterUnit;
        at = atomicAdd(&F.ctl[0], units);
        if (at > F.max_units - units) at = -1;
        E.filt = at < 0 ? 0 : 1 + (at << 4 | lg);
      }
      for (uint32_t m = __ballot_sync(0xffffffffu, at >= 0); m; m &= m - 1) {
        const int32_t a0 = __shfl_sync(0xffffffffu, at, __ffs(m) - 1),
                      nu = __shfl_sync(0xffffffffu, units, __ffs(m) - 1);
        for (int32_t x = lane; x < nu * kFilterUnit; x += 32)
          F.bits[(int64_t)a0 * kFilterUnit + x] = 0u;
      }
    }
  }
  c.sync();
  for (int32_t a = tid; a < n1; a += nth) {
    const EndSlot &E = F.slots[F.slot_of[a]];
    if (a >= n2) F.list1[E.off1 + F.rank1[a]] = a;
    else rec[a].w = E.filt - 1;
  }
}

// Zeros F's slots, bitmap and counters (16-byte words).
__device__ __forceinline__ void clear_ends(cg::cluster_group &c, int blocks, const Filters &F) {
  const int32_t tid = (int32_t)c.block_rank() * kSourceThreads + (int32_t)threadIdx.x;
  uint4 *p = reinterpret_cast<uint4 *>(F.slots);
  const int64_t n = ((char *)F.ctl + 256 - (char *)F.slots) / 16;
  for (int64_t i = tid; i < n; i += blocks * kSourceThreads) p[i] = make_uint4(0, 0, 0, 0);
}

__global__ void __cluster_dims__(kSourceBlocks, 1, 1) __launch_bounds__(kSourceThreads)
k_source(const __grid_constant__ GraphView V, const __grid_constant__ QueryTab t,
         const __grid_constant__ Workspace w, const __grid_constant__ Filters F, bool rows,
         const int32_t *act, int32_t n_act, int32_t u_begin, int32_t u_end) {
  __shared__ SourceShared S;
  cg::cluster_group c = cg::this_cluster();
  if (F.slots) clear_ends(c, kSourceBlocks, F);
  source_phases<true>(c, kSourceBlocks, rows, S, V, t, w, act, n_act, u_begin, u_end);
  if (F.slots) {
    c.sync();
    end_phases(c, kSourceBlocks, w, F);
  }
}

// The queries of a batch, a cluster each.
template <bool kRows>
__global__ void __launch_bounds__(kSourceThreads)
k_sources(const __grid_constant__ GraphView V, const SourceJob *__restrict__ jobs,
          const int32_t *act, int32_t n_act) {
  __shared__ SourceShared S;
  cg::cluster_group c = cg::this_cluster();
  const int blocks = (int)c.num_blocks();
  const SourceJob &job = jobs[blockIdx.x / blocks];
  source_phases<kRows>(c, blocks, false, S, V, *job.tab, job.w, act, n_act, 0, V.n);
}

// The end nodes of a group of queries, a cluster each.
__global__ void __launch_bounds__(kSourceThreads) k_ends(const WalkJob *__restrict__ jobs) {
  cg::cluster_group c = cg::this_cluster();
  const int blocks = (int)c.num_blocks();
  const Workspace w = jobs[blockIdx.x / blocks].w;
  const Filters F = jobs[blockIdx.x / blocks].F;
  if (!F.slots) return;  // the whole cluster
  clear_ends(c, blocks, F);
  c.sync();
  end_phases(c, blocks, w, F);
}

// ------------------------------------------------------------ host side --

static int launched(const char *what) {
  const cudaError_t e = cudaGetLastError();
  return e == cudaSuccess ? SRK_OK : cuda_fail(e, what);
}

int enqueue_source(const srk_graph *g, const QueryTab &t, const Workspace &w, const Filters &F,
                   bool rows, int32_t u_begin, int32_t u_end, cudaStream_t st) {
  k_source<<<kSourceBlocks, kSourceThreads, 0, st>>>(view_of(g), t, w, F, rows, g->act, g->n_act,
                                                     u_begin, u_end);
  return launched("source walks: launch");
}

// Launches `kernel` with a cluster for each of k queries.  The cluster's size: the
// queries run in rounds over the SMs (a block each), and a round takes about two
// units of time and one for each walk of a thread.  64 queries of 435 walks take 107
// us with clusters of 8 blocks and 30 us with clusters of 2.
template <class... Par, class... Arg>
static cudaError_t launch_clusters(void (*kernel)(Par...), const srk_graph *g, int32_t k, int32_t N,
                                   cudaStream_t st, Arg... arg) {
  const int64_t sms = sm_count(g->device);
  int blocks = 1;
  int64_t least = INT64_MAX;
  for (int b = 1; b <= kSourceBlocks; b *= 2) {
    const int64_t rounds = ((int64_t)k * b + sms - 1) / sms,
                  time = rounds * (2 + (N + b * kSourceThreads - 1) / (b * kSourceThreads));
    if (time <= least) {
      least = time;
      blocks = b;
    }
  }
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(blocks * k));
  cfg.blockDim = dim3(kSourceThreads);
  cfg.stream = st;
  cudaLaunchAttribute attr;
  attr.id = cudaLaunchAttributeClusterDimension;
  attr.val.clusterDim.x = (unsigned)blocks;
  attr.val.clusterDim.y = attr.val.clusterDim.z = 1;
  cfg.attrs = &attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kernel, Par(arg)...);
}

int enqueue_sources(const srk_graph *g, const SourceJob *jobs, int32_t k, int32_t N, bool shared,
                    cudaStream_t st) {
  const cudaError_t e = launch_clusters(shared ? k_sources<false> : k_sources<true>, g, k, N, st,
                                        view_of(g), jobs, (const int32_t *)g->act, g->n_act);
  return e == cudaSuccess ? SRK_OK : cuda_fail(e, "source walks: launch");
}

int enqueue_ends(const srk_graph *g, const WalkJob *jobs, int32_t k, int32_t N, cudaStream_t st) {
  const cudaError_t e = launch_clusters(k_ends, g, k, N, st, jobs);
  return e == cudaSuccess ? SRK_OK : cuda_fail(e, "end nodes: launch");
}

}  // namespace srk
