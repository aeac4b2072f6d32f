// Target walks in lockstep (steps a4-a5 of a query): every target with
// in-neighbours walks its pairs, the first meeting of a pair counts, and the
// scores follow.
//
// A pair j joins the source walk sigma(j), nodes h_1, h_2, ..., with walk j of
// every target, for cap_j steps at most.  A thread holds a few targets and a
// block takes its targets through one pair after the other, so a pair's index,
// nodes, weight and length are the same for all its threads.  Two things follow
// that a warp per target (lanes over pairs, the earlier form) cannot have:
//
//   End filters.  The last step of a pair can only meet when h_cap is an
//   in-neighbour of the node x the walk is at, that is, when x is in the
//   out-list of h_cap.  Each end node has a Bloom filter of its out-list (one
//   hash, 16 bits and more per node), which the block holds in shared memory
//   while it walks the pair; where it says no, the last step is neither drawn
//   nor read.  At R-MAT 20 6.5 % of the walks that reach their last step pass,
//   so of the 1.45 scattered reads a pair costs after its first step 0.92 are
//   left (CPU model of the walk).  The meetings are the same: the filter has no
//   false negatives.  A step counts as taken when the walk gets to take it,
//   whatever its draw, so step counts are the same too.
//   Pairs of cap 1.  Their only step is their last: 40 % of all pairs, which
//   meet at one target in 300.  They are not walked at all.  One pass over the
//   edges (k_edges, which also fills the filters) finds, for every edge from
//   an end node y to a target u, the pairs that end at y after one step, and
//   draws u's step for those only.
//
// What bounds it (GB300): the misses of the scattered list reads, one 32-byte
// sector each, of which a plain random gather gets 3.1e11 per second with the
// graph in L2, then issue slots and the latency of a walk's chain of reads.  At
// R-MAT 20, eps = 0.02 (10,941 pairs, 546,406 targets): 1.17 sectors a pair
// and target and 104 warp instructions per pair and 32 targets (2.0 and 189
// with a warp per target), 2.4e11 sectors per second, 54 % of the issue slots.
// One query 29.0 ms instead of 42.4 ms; R-MAT 16 1.99 ms instead of 2.56 ms;
// 100,003 nodes with uniform lists of 12, eps = 0.03, 1.98 ms instead of 2.95
// ms; R-MAT 22 at eps = 0.05, bound by DRAM (64 bytes fetched per missing
// sector), 41-44 ms instead of 57-62 ms.
//
// Launch shape: 2 blocks of 448 threads per SM, 3 targets a thread (72
// registers).  Measured at R-MAT 20 in an earlier state of the kernel: 1 target
// x 704 threads 44.7 ms, 2 x 512 39.9, 3 x 448 38.2, 4 x 384 38.2, 5 x 320 41:
// several targets share a pair's uniform work, and their chains of dependent
// loads overlap.  Shared memory is kept to 64 KB a block, since the rest of the
// SM's 256 KB holds the lines of reads in flight: 92 KB of it cost nothing
// against 124 KB, 60 KB 10 %, 28 KB half the speed.
#include <stdint.h>
#include <stdlib.h>
#include <string.h>

#include <algorithm>

#include "srk_device.cuh"
#include "srk_internal.h"

namespace srk {

// A query of a group, which a block holds in shared memory: its round keys are
// made as they are needed (kernel parameters have them as constant operands).
struct GroupQuery : LockQuery {};
__device__ __forceinline__ uint32_t round_key(const GroupQuery &Q, int r) {
  return Q.key + (uint32_t)r * kPhiloxW0;
}
template <class QT>
__device__ __forceinline__ uint32_t round_key(const QT &Q, int r) { return Q.rk[r]; }

// -------------------------------------------------- asynchronous copies --
__device__ __forceinline__ uint32_t smem_addr(const void *p) {
  return (uint32_t)__cvta_generic_to_shared(p);
}
__device__ __forceinline__ void mbar_init(uint64_t *bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_addr(bar)), "r"(count)
               : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint64_t *bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_addr(bar)) : "memory");
}
__device__ __forceinline__ void mbar_expect(uint64_t *bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_addr(bar)),
               "r"(bytes)
               : "memory");
}
__device__ __forceinline__ bool mbar_try(uint64_t *bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n.reg .pred p;\nmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
      "selp.u32 %0, 1, 0, p;\n}"
      : "=r"(ok)
      : "r"(smem_addr(bar)), "r"(parity)
      : "memory");
  return ok != 0;
}
// 16-byte aligned addresses, bytes a multiple of 16.
__device__ __forceinline__ void bulk_load(void *dst, const void *src, uint32_t bytes,
                                          uint64_t *bar) {
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
          smem_addr(dst)),
      "l"(src), "r"(bytes), "r"(smem_addr(bar))
      : "memory");
}

// ------------------------------------------------------ the lockstep block --
constexpr int kLockThreads = 448;
constexpr int kLockBlocks = 2;        // per SM
constexpr int kLockTargets = 3;       // per thread
constexpr int kLockWarps = kLockThreads / 32;
constexpr int kStages = 2;            // groups of filters in flight per block,
constexpr int kStageWords = 2048;     //   this many words of filters each (at least the largest)
constexpr int kGroup = 16;            //   of at most this many pairs
constexpr int kListWords = 2048;       // words of targets' own lists held in shared memory
constexpr int kQueue = 128;           // entries of a warp's queue of last steps
constexpr int kHubCache = 512;        // hub records held there (narrow layout),
constexpr int kCodes = 2048;          //   and list starts by degree code
constexpr size_t kLockSmem = 4 * (size_t)kStages * kStageWords + 4 * kListWords +
                             16 * kQueue * kLockWarps + 8 * kHubCache + 4 * kCodes;

// The narrow layout's tables in shared memory.
struct LockTables {
  uint32_t ctab, hub, n_hub;
};

struct LockShared {
  uint64_t full[kStages];   // phase n / kStages: the filters of group n have landed
  uint64_t empty[kStages];  // phase n / kStages: every warp is done with group n
  int32_t pairs[kStages];   // pairs of the stage's group
  int32_t place[kStages][kGroup];  // a pair's filter in the stage: first word, or -1
  uint32_t sums[4];
  uint32_t warp_sum[kLockWarps];
  int32_t unit;
  int32_t broken;  // a wait gave up: filters are read from global memory
};

// Waits, `polls` polls at most, for the phase of parity ph; false when this or
// another wait of the block gave up.
constexpr int32_t kWaitPolls = 1 << 20;
__device__ __forceinline__ bool lock_wait(LockShared &S, uint64_t *bar, uint32_t ph,
                                          int32_t polls) {
  for (int32_t i = 0; i < polls; ++i) {
    if (mbar_try(bar, ph)) return *(volatile int32_t *)&S.broken == 0;
    if (*(volatile int32_t *)&S.broken) return false;
  }
  *(volatile int32_t *)&S.broken = 1;
  return false;
}

__device__ __forceinline__ void mul_wide(uint32_t a, uint32_t b, uint32_t &hi, uint32_t &lo) {
  asm("{\n.reg .u64 p;\nmul.wide.u32 p, %2, %3;\nmov.b64 {%1, %0}, p;\n}"
      : "=r"(hi), "=r"(lo) : "r"(a), "r"(b));
}

// philox2 with the round keys of a query.
template <class QT>
__device__ __forceinline__ void philox2k(const QT &Q, uint32_t c0, uint32_t c1, uint32_t &x0,
                                         uint32_t &x1) {
  x0 = c0;
  x1 = c1;
#pragma unroll
  for (int r = 0; r < 10; ++r) {
    uint32_t hi, lo;
    mul_wide(kPhilox2M, x0, hi, lo);
    x0 = hi ^ x1 ^ round_key(Q, r);
    x1 = lo;
  }
}

// The indices of step i of walk r below d[t] from the words w[t] (step_entry's
// draw; 0 where d[t] is 0).  Lemire's test, which almost no word comes near,
// is one branch for all the thread's targets.
static __device__ __noinline__ uint32_t rare_index(uint32_t w, uint32_t k, int i, uint32_t r,
                                                   uint32_t v, uint32_t d) {
  const uint32_t lo = w * d;
  return lo < d && lo < (0u - d) % d ? step_index_redraw(k, i, r, v, d) : __umulhi(w, d);
}
template <int kT>
__device__ __forceinline__ void lock_index(const uint32_t (&w)[kT], const uint32_t (&d)[kT],
                                           uint32_t k, int i, uint32_t r, const int32_t (&v)[kT],
                                           uint32_t (&idx)[kT]) {
  bool rare = false;
#pragma unroll
  for (int t = 0; t < kT; ++t) {
    uint32_t lo;
    mul_wide(w[t], d[t], idx[t], lo);
    rare |= lo < d[t];
  }
  if (__any_sync(0xffffffffu, rare))
#pragma unroll
    for (int t = 0; t < kT; ++t)
      if (d[t]) idx[t] = rare_index(w[t], k, i, r, (uint32_t)v[t], d[t]);
}

// Loads under a condition, without a branch: v keeps its value where p is false.
__device__ __forceinline__ void load_if(bool p, uint32_t smem, uint32_t &v) {
  asm("{\n.reg .pred q;\nsetp.ne.u32 q, %2, 0;\n@q ld.shared.u32 %0, [%1];\n}"
      : "+r"(v) : "r"(smem), "r"((uint32_t)p) : "memory");
}
__device__ __forceinline__ void load_if(bool p, uint32_t smem, uint2 &v) {
  asm("{\n.reg .pred q;\nsetp.ne.u32 q, %3, 0;\n@q ld.shared.v2.u32 {%0, %1}, [%2];\n}"
      : "+r"(v.x), "+r"(v.y) : "r"(smem), "r"((uint32_t)p) : "memory");
}
__device__ __forceinline__ void load_if(bool p, const uint32_t *g, uint32_t &v) {
  asm("{\n.reg .pred q;\nsetp.ne.u32 q, %2, 0;\n@q ld.global.u32 %0, [%1];\n}"
      : "+r"(v) : "l"(g), "r"((uint32_t)p) : "memory");
}
__device__ __forceinline__ void load_if(bool p, const uint2 *g, uint2 &v) {
  asm("{\n.reg .pred q;\nsetp.ne.u32 q, %3, 0;\n@q ld.global.v2.u32 {%0, %1}, [%2];\n}"
      : "+r"(v.x), "+r"(v.y) : "l"(g), "r"((uint32_t)p) : "memory");
}
__device__ __forceinline__ void load_if(bool p, uint32_t smem, int32_t &v) {
  load_if(p, smem, reinterpret_cast<uint32_t &>(v));
}
__device__ __forceinline__ void load_if(bool p, const int32_t *g, int32_t &v) {
  load_if(p, reinterpret_cast<const uint32_t *>(g), reinterpret_cast<uint32_t &>(v));
}
// The same for a store, and its plain counterpart for a warp's queue.
__device__ __forceinline__ void store_if(bool p, uint32_t smem, uint32_t x, uint32_t y, uint32_t z,
                                         uint32_t w) {
  asm volatile("{\n.reg .pred q;\nsetp.ne.u32 q, %5, 0;\n@q st.shared.v4.u32 [%0], {%1, %2, %3, %4};\n}"
               ::"r"(smem), "r"(x), "r"(y), "r"(z), "r"(w), "r"((uint32_t)p)
               : "memory");
}
__device__ __forceinline__ uint4 load_shared(uint32_t smem) {
  uint4 v;
  asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];"
               : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(smem) : "memory");
  return v;
}
__device__ __forceinline__ const uint32_t *entries(const Adj &G) { return G.adj; }
__device__ __forceinline__ const uint2 *entries(const AdjW &G) { return G.adj; }
__device__ __forceinline__ const int32_t *entries(const AdjC &G) { return G.col; }

// Base and degree of the node x that entry e names, where p holds; degree 0
// elsewhere.
template <class GA, class E>
__device__ __forceinline__ int32_t lock_next(const GA &G, const LockTables &, bool p, E e,
                                             int32_t x, uint32_t &deg) {
  int32_t b = 0;
  deg = 0;
  if (p) b = entry_next(G, e, x, deg);
  return b;
}
__device__ __forceinline__ int32_t lock_next(const Adj &G, const LockTables &T, bool p, uint32_t e,
                                             int32_t x, uint32_t &deg) {
  const uint32_t code = p ? e >> G.pb : 0u;
  uint32_t start = 0;
  load_if(true, T.ctab + 4u * code, start);
  uint2 h = make_uint2(code, start + (uint32_t)x * code);
  const bool hub = code == G.dmax, near = (uint32_t)x < T.n_hub;
  load_if(hub && near, T.hub + 8u * (uint32_t)x, h);
  load_if(hub && !near, G.hub + (uint32_t)x, h);
  deg = h.x;
  return (int32_t)h.y;
}
template <class GA, class E>
__device__ __forceinline__ bool entry_ends(const GA &G, E e, int32_t x) {
  uint32_t d = 0;
  entry_next(G, e, x, d);
  return d == 0;
}
__device__ __forceinline__ bool entry_ends(const Adj &G, uint32_t e, int32_t) {
  return (e >> G.pb) == 0;
}

template <int kT>
struct LockTargets {
  int32_t u[kT], b[kT], at[kT];  // id, list base, list in shared memory (-1: not there,
                                 // -2: no target)
  uint32_t d[kT], st[kT];        // in-degree (0: no target), steps
};

// The first word of an entry (what a queue entry keeps of it; the wide layout
// finds the degree again at the node's head).
__device__ __forceinline__ uint32_t entry_word(uint32_t e) { return e; }
__device__ __forceinline__ uint32_t entry_word(int32_t e) { return (uint32_t)e; }
__device__ __forceinline__ uint32_t entry_word(uint2 e) { return e.x; }
__device__ __forceinline__ uint32_t word_entry(const Adj &, uint32_t w) { return w; }
__device__ __forceinline__ int32_t word_entry(const AdjC &, uint32_t w) { return (int32_t)w; }
__device__ __forceinline__ uint2 word_entry(const AdjW &G, uint32_t w) {
  return make_uint2(w, G.adj[w].y);
}

// Where a pair's filter is: in shared memory (near), or in global.
struct LockFilter {
  uint32_t near;
  const uint32_t *far;
  int lg;
  bool has, landed;
};

// A warp's queue of last steps.  Few walks pass their pair's filter, and
// their last steps would each hold the whole warp for two dependent loads; the
// queue collects them until they fill a warp.  Entry {entry of the node before
// the last step, node to meet, cap << 24 | j, a << 8 | target slot}.
struct LockQueue {
  uint32_t at;  // shared memory
  int32_t n;
  uint32_t below;  // the mask of the lower lanes
};

template <int kT, class GA, class QT>
__device__ __forceinline__ void lock_drain(const GA &G, const LockTables &T, const QT &Q,
                                           LockQueue &B, int take, const int32_t (&u)[kT]) {
  __syncwarp();
  const int lane = threadIdx.x & 31;
  B.n -= take;
  const bool p = lane < take;
  uint4 it = make_uint4(0u, 0u, 1u << 24, 0u);
  if (p) it = load_shared(B.at + 16u * (uint32_t)(B.n + lane));
  int32_t v = 0;
#pragma unroll
  for (int t = 0; t < kT; ++t) {
    const int32_t vt = __shfl_sync(0xffffffffu, u[t], it.w & 31);
    if (((it.w >> 5) & 7) == t) v = vt;
  }
  const uint32_t j = it.z & 0xFFFFFFu;
  const int i = (int)(it.z >> 24);
  uint32_t deg[1] = {0}, x0[1], x1[1], idx[1];
  const int32_t vv[1] = {v};
  int32_t b = 0;
  if (p) {
    const auto e = word_entry(G, it.x);
    b = lock_next(G, T, true, e, entry_pos(G, e), deg[0]);
  }
  philox2k(Q, walk_ctr0(i, j), (uint32_t)v, x0[0], x1[0]);
  if (!(i & 1)) x0[0] = x1[0];
  lock_index(x0, deg, Q.key, i, j, vv, idx);
  if (deg[0]) {
    const auto e = adj_entry(G, b, idx[0]);
    if (entry_pos(G, e) == (int32_t)it.y) {
      atomicAdd(&Q.W[v], Q.w[it.w >> 8]);
      if (Q.counts) atomicAdd(&Q.counts[v], 1u);
    }
  }
  __syncwarp();
}

// One pair (index j, nodes h at steps 1..cap, step 1..32 in the lanes' h32)
// for the thread's targets; kCap = cap, or 0 for any up to 32, or -1 for any.
template <int kCap, int kT, bool kCount, class GA, class E, class QT>
__device__ __forceinline__ void lock_pair(const GA &G, const LockTables &T, const QT &Q,
                                          const LockFilter &F, uint32_t lists, int32_t a, uint32_t j, int cap_,
                                          int32_t h32, const int32_t *__restrict__ h,
                                          LockTargets<kT> &X, LockQueue &B) {
  const int cap = kCap > 0 ? kCap : cap_;
  const int lane = threadIdx.x & 31;
  int32_t b[kT];
  uint32_t deg[kT], x0[kT], x1[kT], idx[kT];
  E e[kT];
#pragma unroll
  for (int t = 0; t < kT; ++t) {
    philox2k(Q, j, (uint32_t)X.u[t], x0[t], x1[t]);
    deg[t] = X.d[t];
  }
  lock_index(x0, deg, Q.key, 1, j, X.u, idx);
#pragma unroll
  for (int t = 0; t < kT; ++t) {
    e[t] = E{};
    load_if(X.at[t] >= 0, lists + (uint32_t)sizeof(E) * ((uint32_t)X.at[t] + idx[t]), e[t]);
    load_if(X.at[t] == -1, entries(G) + ((uint32_t)X.b[t] + idx[t]), e[t]);
  }
#pragma unroll(kCap > 0 ? kCap : 1)
  for (int i = 1;; ++i) {
    // the walks are at the nodes that the entries e of step i name
    int32_t hi = __shfl_sync(0xffffffffu, h32, (i - 1) & 31);
    if (kCap < 0 && i > 32) hi = h[i - 1];
    bool meets = false;
#pragma unroll
    for (int t = 0; t < kT; ++t) {
      meets |= entry_pos(G, e[t]) == hi;  // (or a walk that has ended was there)
      if (kCount && i == cap && deg[t]) X.st[t] += i;
    }
    if (__any_sync(0xffffffffu, meets)) {  // rare: a few times per target and query
#pragma unroll
      for (int t = 0; t < kT; ++t)
        if (deg[t] != 0 && entry_pos(G, e[t]) == hi) {
          atomicAdd(&Q.W[X.u[t]], Q.w[a]);
          if (Q.counts) atomicAdd(&Q.counts[X.u[t]], 1u);
          deg[t] = 0;
          if (kCount && i < cap) X.st[t] += i;
        }
    }
    if (i == cap) break;  // cap 1
    if (i == cap - 1) {   // the last step: into the queue, if the filter lets it
      int32_t he = __shfl_sync(0xffffffffu, h32, i & 31);
      if (kCap < 0 && i >= 32) he = h[i];
      uint32_t word[kT], f[kT];
      if (F.has) {
#pragma unroll
        for (int t = 0; t < kT; ++t) f[t] = filter_bit(entry_pos(G, e[t]), F.lg);
        if (F.landed) {
#pragma unroll
          for (int t = 0; t < kT; ++t) {
            word[t] = 0;
            load_if(true, F.near + 4u * (f[t] >> 5), word[t]);
          }
        } else {
#pragma unroll
          for (int t = 0; t < kT; ++t) word[t] = F.far[f[t] >> 5];
        }
      } else {
#pragma unroll
        for (int t = 0; t < kT; ++t) {
          word[t] = ~0u;
          f[t] = 0;
        }
      }
      const uint32_t len_j = (uint32_t)cap << 24 | j, a_lane = (uint32_t)a << 8 | (uint32_t)lane;
#pragma unroll
      for (int t = 0; t < kT; ++t) {
        bool p = deg[t] != 0;
        if (kCount && p) {
          const bool ends = entry_ends(G, e[t], entry_pos(G, e[t]));
          X.st[t] += ends ? i : cap;
          p = !ends;
        }
        p = p && ((word[t] >> (f[t] & 31)) & 1u);
        const uint32_t m = __ballot_sync(0xffffffffu, p);
        store_if(p, B.at + 16u * (uint32_t)(B.n + __popc(m & B.below)), entry_word(e[t]),
                 (uint32_t)he, len_j, a_lane + 32u * t);
        B.n += __popc(m);
      }
      while (B.n >= 32) lock_drain(G, T, Q, B, 32, X.u);
      break;
    }
    uint32_t any = 0;
#pragma unroll
    for (int t = 0; t < kT; ++t) {
      const bool p = deg[t] != 0;
      b[t] = lock_next(G, T, p, e[t], entry_pos(G, e[t]), deg[t]);
      if (kCount && p && deg[t] == 0) X.st[t] += i;
      any |= deg[t];
    }
    if (!__any_sync(0xffffffffu, any != 0)) break;
    if (!(i & 1)) {
#pragma unroll
      for (int t = 0; t < kT; ++t)
        philox2k(Q, walk_ctr0(i + 1, j), (uint32_t)X.u[t], x0[t], x1[t]);
      lock_index(x0, deg, Q.key, i + 1, j, X.u, idx);
    } else {
      lock_index(x1, deg, Q.key, i + 1, j, X.u, idx);
    }
#pragma unroll
    for (int t = 0; t < kT; ++t)
      load_if(deg[t] != 0, entries(G) + ((uint32_t)b[t] + idx[t]), e[t]);
  }
}

// Pairs first, first + stride, ... (len of them) for the block's targets; seq
// counts the groups of this block.  Warp 0 forms the groups: the next pairs
// whose filters fit a stage.  `staged`: the pairs have filters, and no wait of an
// earlier unit gave up (the same in every thread).  When a wait gives up, the
// block's warps read the filters from global memory instead, one warp after the
// other as each comes to a wait; none frees a stage from then on, so warp 0 forms
// no group into a stage in use, waits for those that it has formed before it
// leaves, and no later unit forms any.
template <int kT, bool kCount, class GA, class E, class QT>
__device__ __forceinline__ void lockstep_walks(const GA &G, const LockTables &T, const QT &Q,
                                               LockShared &S,
                                               uint32_t *ring, uint4 *queues, const E *lists,
                                               int32_t first, int32_t stride, int32_t len,
                                               bool staged, uint32_t &seq, LockTargets<kT> &X) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  LockQueue B{smem_addr(queues + wid * kQueue), 0, lanes_below_mask()};
  int32_t issued = 0;     // warp 0: pairs in the groups formed so far,
  uint32_t formed = seq;  //   and the number of the next group
  auto issue = [&](uint32_t n) {  // warp 0: form group n and fetch its filters
    if (issued >= len) return;
    const uint32_t sg = n % kStages;
    int32_t f = kNoFilter, words = 0;
    const bool in = lane < kGroup && issued + lane < len;
    if (in) f = Q.rec[first + stride * (issued + lane)].w;
    if (f != kNoFilter) words = 1 << filter_lg(f);
    int32_t incl = words;
    for (int o = 1; o < kGroup; o <<= 1) {
      const int32_t y = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += y;
    }
    const uint32_t fits = __ballot_sync(0xffffffffu, in && incl <= kStageWords);
    const int32_t count = __popc(fits);
    const int32_t total = __shfl_sync(0xffffffffu, incl, count - 1);
    const bool mine = lane < count && f != kNoFilter;
    if (lane < count) S.place[sg][lane] = mine ? incl - words : -1;
    if (lane == 0) S.pairs[sg] = count;
    __syncwarp();
    if (lane == 0) mbar_expect(&S.full[sg], 4u * (uint32_t)total);
    __syncwarp();
    if (mine)
      bulk_load(ring + sg * kStageWords + incl - words, Q.bits + filter_place(f),
                4u * (uint32_t)words, &S.full[sg]);
    issued += count;
    formed = n + 1;
  };
  const uint32_t seq0 = seq;
  if (staged && wid == 0)
    for (uint32_t q = 0; q < kStages - 1; ++q) issue(seq0 + q);
  int4 nrec = Q.rec[first];
  int32_t nh = lane < nrec.y ? Q.H[nrec.z + lane] : 0;
  LockFilter F;
  F.landed = staged;
  for (int32_t gk = 0; gk < len; ++seq) {
    const uint32_t sg = seq % kStages;
    int32_t ge = len;
    if (F.landed) {
      if (wid == 0 &&
          __all_sync(0xffffffffu, seq == seq0 || lock_wait(S, &S.empty[(seq - 1) % kStages],
                                                           ((seq - 1) / kStages) & 1u, Q.polls)))
        issue(seq + kStages - 1);
      F.landed = lock_wait(S, &S.full[sg], (seq / kStages) & 1u, Q.polls);
      F.landed = __all_sync(0xffffffffu, F.landed);
      if (F.landed) ge = gk + S.pairs[sg];
    }
    for (int32_t k = gk; k < ge; ++k) {
      const int32_t a = first + stride * k;
      const int4 rec = nrec;
      const int32_t h32 = nh;
      if (k + 1 < len) {
        nrec = Q.rec[a + stride];
        nh = lane < nrec.y ? Q.H[nrec.z + lane] : 0;
      }
      F.has = rec.w != kNoFilter;
      F.lg = filter_lg(rec.w);
      F.near = smem_addr(ring + sg * kStageWords + (F.landed ? S.place[sg][(k - gk) & (kGroup - 1)] : 0));
      F.far = Q.bits + filter_place(rec.w);
#define SRK_PAIR(C)                                                                           \
  lock_pair<C, kT, kCount, GA, E>(G, T, Q, F, smem_addr(lists), a, (uint32_t)rec.x, rec.y, h32, \
                                  Q.H + rec.z, X, B)
      if (rec.y == 2) SRK_PAIR(2);
      else if (rec.y == 3) SRK_PAIR(3);
      else if (rec.y <= 32) SRK_PAIR(0);
      else SRK_PAIR(-1);
#undef SRK_PAIR
    }
    gk = ge;
    if (F.landed) {
      __syncwarp();
      if (lane == 0) mbar_arrive(&S.empty[sg]);
    }
  }
  if (B.n > 0) lock_drain(G, T, Q, B, B.n, X.u);
  if (staged && wid == 0 && !F.landed)  // copies in flight, which nobody waited for
    for (uint32_t q = max(seq0, formed > kStages ? formed - kStages : 0u); q < formed; ++q)
      for (int32_t i = 0; i < kWaitPolls && !mbar_try(&S.full[q % kStages], (q / kStages) & 1u); ++i) {
      }
}

// ------------------------------------------------------- edges, and walks --

// One pass over the edges y -> u (entry k of u's list).  Where y is an end
// node, u joins its filter, and if u is a target, the pairs of cap 1 that end
// at y are decided for u: pair j meets here exactly when its step draws k.
// (Every entry that holds y is its own edge, so repeated in-neighbours count
// once each, as the draw does.)  A bitmap in L1 turns most edges away.  A warp
// takes kEdgeRun consecutive edges and follows their owners along row_ptr, 32
// nodes at a time; a binary search per edge of an end node took 0.37 ms at
// R-MAT 20 (16.1 M edges), this 0.26 ms (R-MAT 16, 0.95 M edges: 0.037, 0.046).
constexpr int kEdgeRun = 1024;

// Meetings of the pairs of cap 1 list1[off + q], q = q0, q0 + dq, ... < cnt, with
// target u, whose entry k of d is the end node.
__device__ __forceinline__ void last_steps(const Filters &F, const int4 *__restrict__ rec,
                                           const unsigned long long *__restrict__ pair_w,
                                           uint32_t key, int32_t u, uint32_t k, uint32_t d,
                                           int32_t off, int32_t cnt, int32_t q0, int32_t dq,
                                           uint32_t &c, unsigned long long &ws) {
  for (int32_t q = q0; q < cnt; q += dq) {
    const int32_t a = F.list1[off + q];
    const uint32_t j = (uint32_t)rec[a].x;
    uint32_t x0, x1;
    philox2(key, walk_ctr0(1, j), (uint32_t)u, x0, x1);
    uint32_t idx = __umulhi(x0, d);
    const uint32_t lo = x0 * d;
    if (lo < d && lo < (0u - d) % d) idx = step_index_redraw(key, 1, j, (uint32_t)u, d);
    if (idx == k) {
      ++c;
      ws += pair_w[a];
    }
  }
}

__device__ __forceinline__ void walk_edges(const Filters &F, const GraphView &V, int64_t m,
                                           const int32_t *__restrict__ cnt,
                                           const int4 *__restrict__ rec,
                                           const unsigned long long *__restrict__ pair_w,
                                           uint32_t key, int32_t s, int32_t u_begin, int32_t u_end,
                                           unsigned long long *__restrict__ W,
                                           uint32_t *__restrict__ counts) {
  if (cnt[1] == 0) return;  // no pair can meet
  const int lane = threadIdx.x & 31;
  const int32_t *__restrict__ row_ptr = V.row_ptr;
  const uint32_t mask = (1u << F.slot_bits) - 1u;
  const int64_t warps = ((int64_t)gridDim.x * blockDim.x) >> 5;
  // short runs when there are few edges, so that all warps have some
  int64_t run = (m + warps - 1) / warps;
  run = run > kEdgeRun ? kEdgeRun : (run + 31) & ~31ll;
  for (int64_t r0 = (((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5) * run; r0 < m;
       r0 += warps * run) {
    int32_t v = -1;  // owners so far are below v + 32 (-1: not looked up yet)
    const int64_t r1 = r0 + run < m ? r0 + run : m;
    for (int64_t e0 = r0; e0 < r1; e0 += 32) {
      const int64_t e = e0 + lane;
      EndSlot S{0u, 0, 0, 0};
      if (e < r1) {
        const uint32_t y = (uint32_t)V.col[e], hash = end_hash(y),
                       bb = hash >> (32 - F.bloom_bits);
        if ((F.bloom[bb >> 5] >> (bb & 31)) & 1u) {
          uint32_t sl = hash & mask;
          for (uint32_t probe = 0; probe <= mask; ++probe, sl = (sl + 1u) & mask) {
            const EndSlot T = F.slots[sl];
            if (T.key == y + 1u) S = T;
            if (T.key == y + 1u || T.key == 0u) break;
          }
        }
      }
      bool open = S.key != 0u;  // owner wanted
      if (!__any_sync(0xffffffffu, open)) continue;
      if (v < 0) {  // the owner of the run's first edge: 32 probes a round
        int32_t lo = 0, hi = V.n;  // row_ptr[lo] <= e0 < row_ptr[hi]
        while (hi - lo > 1) {
          const int64_t step = ((int64_t)hi - lo + 31) / 32;
          const int32_t at = (int32_t)min((int64_t)hi, lo + (lane + 1) * step);
          const uint32_t above = __ballot_sync(0xffffffffu, (int64_t)row_ptr[at] > e0);
          const int f = __ffs(above) - 1;  // the first probe past e0 (row_ptr[hi] is)
          hi = (int32_t)min((int64_t)hi, lo + (f + 1) * step);
          lo += (int32_t)(f * step);
        }
        v = lo;
      }
      int32_t u = 0;
      uint32_t k = 0, d = 1;
      for (;;) {  // the owner is v plus the number of lists that end at or before e
        const int32_t end = row_ptr[min(V.n, v + 1 + lane)];
        int q = 0;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1)
          if ((int64_t)__shfl_sync(0xffffffffu, end, q + o - 1) <= e) q += o;
        const bool in = (int64_t)__shfl_sync(0xffffffffu, end, 31) > e;
        const int32_t b = __shfl_sync(0xffffffffu, end, q > 0 ? q - 1 : 0),
                      f = __shfl_sync(0xffffffffu, end, q);
        if (open && in) {
          u = v + q;
          const int32_t beg = q > 0 ? b : row_ptr[v];
          k = (uint32_t)(e - beg);
          d = (uint32_t)(f - beg);
          open = false;
        }
        if (!__any_sync(0xffffffffu, open)) break;
        v += 32;
      }
      if (S.filt > 0) {
        const uint32_t f = filter_bit(node_identity(V, u), filter_lg(S.filt - 1));
        atomicOr(&F.bits[filter_place(S.filt - 1) + (f >> 5)], 1u << (f & 31));
      }
      const bool todo = S.cnt1 > 0 && u >= u_begin && u < u_end && u != s;
      // a few pairs: each lane decides its edge's; many: the warp's lanes share them
      // (3 queries with L = 1, ER lists of 16 on 100,003 nodes: 0.167 ms when more than
      // one pair is shared, 0.162 from 9 on, 0.229 from 65 on)
      uint32_t c = 0;
      unsigned long long ws = 0;
      if (todo && S.cnt1 <= 8)
        last_steps(F, rec, pair_w, key, u, k, d, S.off1, S.cnt1, 0, 1, c, ws);
      for (uint32_t mm = __ballot_sync(0xffffffffu, todo && S.cnt1 > 8); mm; mm &= mm - 1) {
        const int l = __ffs(mm) - 1;
        uint32_t cl = 0;
        unsigned long long wl = 0;
        last_steps(F, rec, pair_w, key, __shfl_sync(0xffffffffu, u, l),
                   __shfl_sync(0xffffffffu, k, l), __shfl_sync(0xffffffffu, d, l),
                   __shfl_sync(0xffffffffu, S.off1, l), __shfl_sync(0xffffffffu, S.cnt1, l), lane,
                   32, cl, wl);
        for (int o = 16; o > 0; o >>= 1) {
          cl += __shfl_xor_sync(0xffffffffu, cl, o);
          wl += __shfl_xor_sync(0xffffffffu, wl, o);
        }
        if (lane == l) {
          c = cl;
          ws = wl;
        }
      }
      if (c) {
        atomicAdd(&W[u], ws);
        if (counts) atomicAdd(&counts[u], c);
      }
    }
  }
}

__global__ void __launch_bounds__(256)
k_edges(const __grid_constant__ Filters F, const __grid_constant__ GraphView V, int64_t m,
        const int32_t *cnt, const int4 *rec, const unsigned long long *pair_w, uint32_t key,
        int32_t s, int32_t u_begin, int32_t u_end, unsigned long long *W, uint32_t *counts) {
  walk_edges(F, V, m, cnt, rec, pair_w, key, s, u_begin, u_end, W, counts);
}

// For a group of queries (blockIdx.y: the query).  (5 blocks an SM, 48 registers: 62 as
// the compiler takes them leave 3 to 4, and cost 2 to 4 % of a batch on 2,000 nodes.)
__global__ void __launch_bounds__(256, 5)
k_edges_group(const __grid_constant__ GraphView V, int64_t m, const WalkJob *__restrict__ jobs) {
  const WalkJob &J = jobs[blockIdx.y];
  const Filters F = J.F;
  if (F.slots)
    walk_edges(F, V, m, J.Q.cnt, J.Q.rec, J.Q.w, J.Q.key, J.Q.s, 0, V.n, J.Q.W, J.Q.counts);
}

// Into how many strided sets the pairs are cut, so that sets x target blocks
// are units of equal work: up to 16 a block, of at least 128 pairs where there are as
// many, and as near below a whole number of rounds over the grid as a count within
// a quarter of the largest gets; on a graph beyond the L2 up to 1,024 a block, of at
// least 32 pairs (see split_unit).
constexpr int kRounds = 16, kUnitPairs = 128, kFarRounds = 1024, kFarUnitPairs = 32;
__device__ __forceinline__ int32_t lock_chunks(int32_t n_pairs, int32_t n_tb, int32_t grid,
                                               bool far) {
  const int64_t per_block = (int64_t)n_pairs * n_tb / grid;
  const int32_t least = far ? kFarUnitPairs : kUnitPairs;
  const int32_t rounds = per_block < 2 * least
                             ? 1
                             : (int32_t)min(per_block / least, (int64_t)(far ? kFarRounds : kRounds));
  int32_t most = rounds * grid / n_tb;
  if (most > n_pairs) most = n_pairs;
  if (most < 1) most = 1;
  if (rounds > kRounds) return most;  // the last round weighs little
  int32_t best = most;
  float fill = 0.0f;
  for (int32_t c = most, k = 0; c > 0 && c >= most - most / 4 && k < 16; --c, ++k) {
    const float units = (float)(c * n_tb);  // at most rounds x grid, or n_tb: exact
    const float f = units / ((float)grid * ceilf(units / (float)grid));
    if (f > fill) {
      fill = f;
      best = c;
    }
  }
  return best;
}

// Block of targets and strided set of pairs of a unit.  On a graph beyond the L2
// units that follow one another have the same targets, and there are many sets of
// pairs, so that the blocks at work hold few targets between them and those
// targets' lists stay in the L2, where most first steps read them.  On the others the
// targets run first: the narrow layout has them by rank, so the heavy units come
// first.  With the targets first everywhere: wide layout, ER lists of 16, 3 queries,
// 2^20 nodes (143 MB) 54.6 ms, 2^21 165; 48 queries with shared walks, R-MAT 24, 1535.  So,
// with sets of 128 pairs, 44.2 (a warp per target: 44.5), 129 (157) and 1407 (1520).
// Sets of 128, 64 and 32 pairs, one query: R-MAT 22, eps = 0.05, 35.4, 33.9 and 32.8 ms
// (43.8); ER 2^22, eps = 0.1, 29.3, 27.5 and 26.1 (31.3), on the CSR 40.7, 38.9 and 37.8 (39.6).
__device__ __forceinline__ void split_unit(bool far, int32_t unit, int32_t n_tb, int32_t n_chunks,
                                           int32_t &tb, int32_t &first) {
  const int32_t by = far ? n_chunks : n_tb, q = unit / by, r = unit - q * by;
  tb = far ? q : r;
  first = far ? r : q;
}

// The targets act[from .. to) of a block (all but `skip`), at most kT a thread;
// with `stage`, their lists of up to 64 entries go to shared memory while they
// fit.  S.sums is zero on entry; every thread of the block calls.
template <int kT, class GA, class E>
__device__ __forceinline__ void lock_targets(const GA &G, const int32_t *__restrict__ row_ptr,
                                             LockShared &S, E *lists,
                                             const int32_t *__restrict__ act, int32_t from,
                                             int32_t to, int32_t skip, bool stage,
                                             LockTargets<kT> &X) {
  constexpr uint32_t lists_max = kListWords * 4 / (uint32_t)sizeof(E);
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
#pragma unroll
  for (int t = 0; t < kT; ++t) {
    const int32_t i = from + t * kLockThreads + (int32_t)threadIdx.x;
    X.u[t] = i < to ? act[i] : 0;
    X.b[t] = node_start(G, row_ptr, X.u[t], X.d[t]);
    if (i >= to || X.u[t] == skip) X.d[t] = 0;
    X.st[t] = 0;
    X.at[t] = X.d[t] ? -1 : -2;
  }
  if (stage) {
    // lists of at most 64, 32, 16 or 8 entries go to shared memory: the
    // largest bound whose lists fit
    uint32_t sum[4] = {0, 0, 0, 0};
#pragma unroll
    for (int t = 0; t < kT; ++t)
#pragma unroll
      for (int q = 0; q < 4; ++q)
        if (X.d[t] <= (64u >> q)) sum[q] += X.d[t];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      uint32_t v = sum[q];
      for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
      if (lane == 0) atomicAdd(&S.sums[q], v);
    }
    __syncthreads();
    int q = 0;
    while (q < 4 && S.sums[q] > lists_max) ++q;
    // first the lists below that bound, then the longer ones while they fit
    uint32_t base = 0;
    for (int pass = 0; pass < 2; ++pass) {
      auto wanted = [&](uint32_t d) {
        return d <= 64u && (pass == (q < 4 && d <= (64u >> q) ? 0 : 1));
      };
      uint32_t mine = 0;
#pragma unroll
      for (int t = 0; t < kT; ++t)
        if (wanted(X.d[t])) mine += X.d[t];
      uint32_t incl = mine;
      for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += y;
      }
      if (lane == 31) S.warp_sum[wid] = incl;
      __syncthreads();
      uint32_t at = base + incl - mine;
      for (int w = 0; w < kLockWarps; ++w) {
        if (w < wid) at += S.warp_sum[w];
        base += S.warp_sum[w];
      }
#pragma unroll
      for (int t = 0; t < kT; ++t)
        if (X.d[t] && wanted(X.d[t])) {
          if (at + X.d[t] <= lists_max) {
            X.at[t] = (int32_t)at;
            for (uint32_t k = 0; k < X.d[t]; ++k) lists[at + k] = adj_entry(G, X.b[t], k);
          }
          at += X.d[t];
        }
      __syncthreads();
    }
  }
}

// A block's dynamic shared memory, its tables filled and its barriers made (to be
// followed by a __syncthreads); the lists of E begin at the returned ring's end.
template <int kLayout>
__device__ __forceinline__ uint32_t *lock_setup(const GraphView &V, unsigned char *dyn,
                                                LockShared &S, LockTables &tabs, uint4 *&queues) {
  uint32_t *ring = reinterpret_cast<uint32_t *>(dyn);
  queues = reinterpret_cast<uint4 *>(ring + kStages * kStageWords + kListWords);
  uint2 *hub = reinterpret_cast<uint2 *>(queues + kQueue * kLockWarps);
  uint32_t *ctab = reinterpret_cast<uint32_t *>(hub + kHubCache);
  tabs = LockTables{smem_addr(ctab), smem_addr(hub), 0u};
  if (threadIdx.x < kStages) {
    mbar_init(&S.full[threadIdx.x], 1);
    mbar_init(&S.empty[threadIdx.x], kLockWarps);
  }
  if (threadIdx.x == 0) S.broken = 0;
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  if constexpr (kLayout == kNarrow) {
    tabs.n_hub = (uint32_t)min(V.n_hubs, kHubCache);
    for (uint32_t i = threadIdx.x; i < tabs.n_hub; i += kLockThreads) hub[i] = V.hub[i];
    for (uint32_t i = threadIdx.x; i <= V.deg_max; i += kLockThreads) ctab[i] = V.ctab[i];
  }
  return ring;
}

// The steps of a unit's targets, to their totals and the thread's.
template <int kT>
__device__ __forceinline__ void add_steps(const LockTargets<kT> &X, uint32_t *steps,
                                          unsigned long long &total) {
#pragma unroll
  for (int t = 0; t < kT; ++t)
    if (X.st[t]) {
      if (steps) atomicAdd(&steps[X.u[t]], X.st[t]);
      total += X.st[t];
    }
}
// A thread's total of steps, summed over its warp, to *steps_total.
__device__ __forceinline__ void add_total(unsigned long long total,
                                          unsigned long long *steps_total) {
  for (int o = 16; o > 0; o >>= 1) total += __shfl_xor_sync(0xffffffffu, total, o);
  if ((threadIdx.x & 31) == 0 && total) atomicAdd(steps_total, total);
}

// The walks.  A unit of work is a block of targets and a strided set of
// pairs; blocks take units from a counter.  A unit's targets keep their lists
// in shared memory where they fit, for their first steps.  W[u] (in the scores
// until k_finish) and the counts grow by atomics, at the rare meetings.
template <int kLayout, bool kCount, int kT>
__global__ void __launch_bounds__(kLockThreads, kLockBlocks)
k_lockstep(const __grid_constant__ GraphView V, const int32_t *__restrict__ act, int32_t *bounds,
           const __grid_constant__ LockQuery Q) {
  extern __shared__ __align__(128) unsigned char dyn[];
  __shared__ LockShared S;
  const auto G = adj_view<kLayout>(V);
  using E = decltype(adj_entry(G, 0, 0u));
  const int32_t act_lo = bounds[2], act_hi = bounds[1];
  const int32_t n_pairs = Q.cnt[Q.min_cap], n_t = act_hi - act_lo;
  if (n_pairs == 0 || n_t <= 0) return;
  const int32_t T = kLockThreads * kT, n_tb = (n_t + T - 1) / T;
  const int32_t n_chunks = lock_chunks(n_pairs, n_tb, gridDim.x, V.far != 0);
  const int64_t units = (int64_t)n_tb * n_chunks;
  if ((int64_t)blockIdx.x >= units) return;
  LockTables tabs;
  uint4 *queues;
  uint32_t *ring = lock_setup<kLayout>(V, dyn, S, tabs, queues);
  E *lists = reinterpret_cast<E *>(ring + kStages * kStageWords);
  unsigned long long total = 0;
  uint32_t seq = 0;
  for (;;) {
    __syncthreads();
    const bool staged = Q.min_cap == 2 && *(volatile int32_t *)&S.broken == 0;
    if (threadIdx.x == 0) S.unit = atomicAdd(bounds, 1);
    if (threadIdx.x < 4) S.sums[threadIdx.x] = 0;
    __syncthreads();
    if (S.unit >= units) break;
    int32_t tb, first;
    split_unit(V.far, S.unit, n_tb, n_chunks, tb, first);
    const int32_t len = (n_pairs - first + n_chunks - 1) / n_chunks;
    LockTargets<kT> X;
    lock_targets(G, V.row_ptr, S, lists, act, act_lo + tb * T, act_hi, Q.s, len >= 32, X);
    lockstep_walks<kT, kCount>(G, tabs, Q, S, ring, queues, (const E *)lists, first, n_chunks, len,
                               staged, seq, X);
    if (kCount) add_steps(X, Q.steps, total);
  }
  if (kCount) add_total(total, Q.steps_total);
}

// The walks of a group of queries, all targets: the units of all of them that are
// not `alone`, one query's after the other's, from one counter.  Queries that are
// small by themselves fill the GPU together: a batch of 64 of eps = 0.05 on 2,000
// nodes with 8 in-neighbours each took 3.54 ms with launches of their own and 1.34
// ms with a warp per target and query, now 1.05 ms.  A query's unit is a block of
// targets and so many pairs that the group has kGroupRounds units a block; less
// work goes in one round of units of up to kGroupRound pairs.  (A batch of 8
// queries on 900 nodes, eps = 0.1: 0.190 ms with units of 4 pairs and more, 0.219 of
// 16; 8, 16 or 32 rounds differ by less than 2 %.)
constexpr int kGroupRounds = 16, kGroupRound = 64, kGroupPairs = 4;
template <int kLayout, bool kCount, int kT>
__global__ void __launch_bounds__(kLockThreads, kLockBlocks)
k_lockstep_group(const __grid_constant__ GraphView V, const int32_t *__restrict__ act, int32_t n_t,
                 const WalkJob *__restrict__ jobs, int32_t k, int32_t *__restrict__ counter) {
  extern __shared__ __align__(128) unsigned char dyn[];
  __shared__ LockShared S;
  __shared__ GroupQuery Q;
  __shared__ int32_t chunks[kWalkGroup];    // strided sets of pairs by query,
  __shared__ int32_t end[kWalkGroup];       //   and where its units end
  __shared__ int32_t job;
  __shared__ unsigned long long all_pairs;
  static_assert(kWalkGroup <= kLockThreads && kWalkGroup % 32 == 0, "a thread per query");
  const auto G = adj_view<kLayout>(V);
  using E = decltype(adj_entry(G, 0, 0u));
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const int32_t T = kLockThreads * kT, n_tb = (n_t + T - 1) / T;
  int32_t pairs = 0;
  if ((int32_t)threadIdx.x < k && !jobs[threadIdx.x].alone)
    pairs = jobs[threadIdx.x].Q.cnt[jobs[threadIdx.x].Q.min_cap];
  if (threadIdx.x == 0) all_pairs = 0;
  __syncthreads();
  if (pairs > 0) atomicAdd(&all_pairs, (unsigned long long)pairs);
  __syncthreads();
  if (all_pairs == 0 || n_t <= 0) return;
  {
    const unsigned long long per_block = all_pairs * (unsigned)n_tb / gridDim.x;
    const unsigned rounds = V.far ? kFarRounds : kGroupRounds;
    const unsigned long long round = V.far ? kFarUnitPairs : kGroupRound;
    const unsigned long long want = max(per_block / rounds, min(per_block, round));
    const int32_t unit = (int32_t)max(min(want, (unsigned long long)SRK_MAX_WALKS),
                                      (unsigned long long)kGroupPairs);
    const int32_t ch = (pairs + unit - 1) / unit;
    int32_t incl = ch * n_tb;
    for (int o = 1; o < 32; o <<= 1) {
      const int32_t y = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += y;
    }
    if (lane == 31) S.warp_sum[wid] = (uint32_t)incl;
    __syncthreads();
    for (int w = 0; w < wid; ++w) incl += (int32_t)S.warp_sum[w];
    if (threadIdx.x < kWalkGroup) {
      chunks[threadIdx.x] = ch;
      end[threadIdx.x] = incl;
    }
  }
  LockTables tabs;
  uint4 *queues;
  uint32_t *ring = lock_setup<kLayout>(V, dyn, S, tabs, queues);
  E *lists = reinterpret_cast<E *>(ring + kStages * kStageWords);
  uint32_t seq = 0;
  for (;;) {
    __syncthreads();
    const bool whole = *(volatile int32_t *)&S.broken == 0;
    if (threadIdx.x == 0) {
      const int32_t unit = atomicAdd(counter, 1);
      int32_t lo = 0, hi = k;  // the first query whose units end past this one
      while (lo < hi) {
        const int32_t mid = (lo + hi) >> 1;
        if (end[mid] <= unit) lo = mid + 1;
        else hi = mid;
      }
      job = lo;
      S.unit = unit - (lo < k ? end[lo] - chunks[lo] * n_tb : 0);
    }
    if (threadIdx.x < 4) S.sums[threadIdx.x] = 0;
    __syncthreads();
    if (job >= k) break;
    for (int i = threadIdx.x; i < (int)(sizeof(LockQuery) / 8); i += kLockThreads)
      reinterpret_cast<uint64_t *>(&Q)[i] = reinterpret_cast<const uint64_t *>(&jobs[job].Q)[i];
    __syncthreads();
    const int32_t n_chunks = chunks[job];
    int32_t tb, first;
    split_unit(V.far, S.unit, n_tb, n_chunks, tb, first);
    const int32_t n_pairs = Q.cnt[Q.min_cap], len = (n_pairs - first + n_chunks - 1) / n_chunks;
    const bool staged = whole && Q.min_cap == 2;
    LockTargets<kT> X;
    lock_targets(G, V.row_ptr, S, lists, act, tb * T, n_t, Q.s, len >= 32, X);
    uint32_t none = 0;  // (groups are numbered by the units that form some)
    lockstep_walks<kT, kCount>(G, tabs, Q, S, ring, queues, (const E *)lists, first, n_chunks, len,
                               staged, staged ? seq : none, X);
    if (kCount) {
      unsigned long long total = 0;
      add_steps(X, nullptr, total);
      add_total(total, Q.steps_total);
    }
  }
}

// Scores from weight sums.  Most sums are 0, whose bits are the score 0.0
// already; the others of a tile are gathered first, since an FP64 division
// holds a warp for as long with one active lane as with 32 (1.05 M targets: 48
// us with a division in every warp).  row[u] for u in [u0, u1), one tile.
constexpr int kFinishTile = 2048;
__device__ __forceinline__ void finish_tile(double *__restrict__ row, int64_t u0, int64_t u1,
                                            double z, uint16_t *list, int32_t *n_list) {
  if (threadIdx.x == 0) *n_list = 0;
  __syncthreads();
  for (int64_t u = u0 + threadIdx.x; u < u1; u += blockDim.x)
    if (__double_as_longlong(row[u]) != 0) list[atomicAdd(n_list, 1)] = (uint16_t)(u - u0);
  __syncthreads();
  for (int32_t q = threadIdx.x; q < *n_list; q += blockDim.x) {
    const int64_t u = u0 + list[q];
    row[u] = (double)(unsigned long long)__double_as_longlong(row[u]) * 2.3283064365386963e-10 / z;
  }
  __syncthreads();
}

// Scores of a query, and the steps of the pairs that k_edges decided for the
// n_t targets with in-neighbours of the range.
__device__ __forceinline__ void finish_query(const int32_t *__restrict__ row_ptr, int32_t n_t,
                                             const int32_t *__restrict__ cnt, int32_t s,
                                             int32_t u_begin, int32_t u_end, double z,
                                             bool skipped, double *__restrict__ scores,
                                             unsigned long long *__restrict__ wsums,
                                             uint32_t *__restrict__ steps,
                                             unsigned long long *__restrict__ steps_total) {
  __shared__ uint16_t list[kFinishTile];
  __shared__ int32_t n_list;
  // pairs of cap 1 decided per edge: one step each of every target
  const uint32_t one = skipped ? (uint32_t)(cnt[1] - cnt[2]) : 0u;
  for (int64_t u0 = (int64_t)u_begin + (int64_t)blockIdx.x * kFinishTile; u0 < u_end;
       u0 += (int64_t)gridDim.x * kFinishTile) {
    const int64_t u1 = min((int64_t)u_end, u0 + kFinishTile);
    if (wsums || (steps && one))
      for (int64_t u = u0 + threadIdx.x; u < u1; u += blockDim.x) {
        // (the batched path hands in a row that is 1 at s; s has no sum)
        if (wsums) wsums[u] = u == s ? 0ull : (unsigned long long)__double_as_longlong(scores[u]);
        if (steps && one && u != s && row_ptr[u + 1] > row_ptr[u]) steps[u] += one;
      }
    if (cnt[1] > 0) finish_tile(scores, u0, u1, z, list, &n_list);
    __syncthreads();
    if (threadIdx.x == 0 && s >= u0 && s < u1) scores[s] = 1.0;
  }
  if (one && blockIdx.x == 0 && threadIdx.x == 0) {
    int64_t t = n_t;
    if (s >= u_begin && s < u_end && row_ptr[s + 1] > row_ptr[s]) --t;
    atomicAdd(steps_total, (unsigned long long)t * one);
  }
}

__global__ void __launch_bounds__(256)
k_finish(const int32_t *row_ptr, const int32_t *bounds, const int32_t *cnt, int32_t s,
         int32_t u_begin, int32_t u_end, double z, int32_t skipped, double *scores,
         unsigned long long *wsums, uint32_t *steps, unsigned long long *steps_total) {
  finish_query(row_ptr, bounds[1] - bounds[2], cnt, s, u_begin, u_end, z, skipped != 0, scores,
               wsums, steps, steps_total);
}

// For a group of queries (blockIdx.y: the query).
__global__ void __launch_bounds__(256)
k_finish_group(const int32_t *row_ptr, int32_t n, int32_t n_t, const WalkJob *__restrict__ jobs) {
  const WalkJob &J = jobs[blockIdx.y];
  finish_query(row_ptr, n_t, J.Q.cnt, J.Q.s, 0, n, J.z, J.F.slots != nullptr,
               reinterpret_cast<double *>(J.Q.W), nullptr, nullptr, J.Q.steps_total);
}

// ---------------------------------------------------- shared target walks --
// SRK_OPT_SHARED_WALKS: walk j of a target serves pair j of every source of
// the batch, as long as some source's pair can still meet.  In lockstep the
// pending sources, the nodes they wait at and the table of those nodes are the
// same for all targets; a target only keeps the sources that its walk j has
// met.  A node is looked up in the step's table when its bit is set in the
// table's signature: 1024 bits, one L1 line that all the block's warps read,
// so at most 6 % of the walks that meet nobody go to the table (with a 64-bit
// signature in a register, the form before, half of them did).
// A warp per target with lanes over pairs took 10.3 ms for 48 sources on R-MAT
// 18, eps = 0.05; this takes 6.3 ms, with 54 % of the issue slots and 62 % of the
// request cycles to the L2 in use; 2 targets a thread 6.6 ms, 1 8.6 ms.  The
// wide layout, whose lists take twice the room and whose targets come by id,
// wants fewer lists in the L2 between two of their first steps: 48 sources on
// R-MAT 21 and 24, 378 and 33.1 queries/s with 2 targets a thread, 372 and 32.3
// with 3, 357 and 33.1 with 1 (with the targets first; in split_unit's order for
// graphs beyond the L2 2 targets a thread give 435 and 34.2).
constexpr int kSharedTargets = 3;  // per thread, at most
constexpr int shared_targets(int layout) { return layout == kWide ? 2 : kSharedTargets; }

template <int kLayout, bool kCount>
__global__ void __launch_bounds__(kLockThreads, kLockBlocks)
k_lock_shared(const __grid_constant__ GraphView V, const int32_t *__restrict__ act, int32_t n_act,
              const __grid_constant__ SharedWalks Q) {
  constexpr int kT = shared_targets(kLayout);
  extern __shared__ __align__(128) unsigned char dyn[];
  __shared__ LockShared S;
  __shared__ int64_t rowbase[SRK_MAX_LEN + 2];
  __shared__ int32_t src_s[64];
  __shared__ int32_t own_rows;  // some target of the unit is a source
  const auto G = adj_view<kLayout>(V);
  using E = decltype(adj_entry(G, 0, 0u));
  E *lists = reinterpret_cast<E *>(dyn);
  uint2 *hub = reinterpret_cast<uint2 *>(dyn + 4 * kListWords);
  uint32_t *ctab = reinterpret_cast<uint32_t *>(hub + kHubCache);
  unsigned long long *excl = reinterpret_cast<unsigned long long *>(ctab + kCodes);
  LockTables tabs{smem_addr(ctab), smem_addr(hub), 0u};
  const int32_t n_pairs = Q.J - Q.j0;
  if (n_pairs <= 0 || n_act <= 0) return;
  const int32_t T = kLockThreads * kT, n_tb = (n_act + T - 1) / T;
  const int32_t n_chunks = lock_chunks(n_pairs, n_tb, gridDim.x, V.far != 0);
  const int64_t units = (int64_t)n_tb * n_chunks;
  if ((int64_t)blockIdx.x >= units) return;
  const int lane = threadIdx.x & 31;
  for (int i = threadIdx.x; i <= SRK_MAX_LEN + 1; i += kLockThreads)
    rowbase[i] = (i >= 1 && i <= Q.Lmax) ? Q.rowbase[i] : 0;
  for (int i = threadIdx.x; i < 64; i += kLockThreads) src_s[i] = i < Q.k ? Q.src[i].s : -1;
  if constexpr (kLayout == kNarrow) {
    tabs.n_hub = (uint32_t)min(V.n_hubs, kHubCache);
    for (uint32_t i = threadIdx.x; i < tabs.n_hub; i += kLockThreads) hub[i] = V.hub[i];
    for (uint32_t i = threadIdx.x; i <= V.deg_max; i += kLockThreads) ctab[i] = V.ctab[i];
  }
  const uint32_t lists_at = smem_addr(lists), smask = (1u << Q.tbits) - 1u;
  unsigned long long total = 0;
  for (;;) {
    __syncthreads();
    if (threadIdx.x == 0) {
      S.unit = atomicAdd(Q.counter, 1);
      own_rows = 0;
    }
    if (threadIdx.x < 4) S.sums[threadIdx.x] = 0;
    __syncthreads();
    if (S.unit >= units) break;
    int32_t tb, first;
    split_unit(V.far, S.unit, n_tb, n_chunks, tb, first);
    LockTargets<kT> X;
    lock_targets(G, V.row_ptr, S, lists, act, tb * T, n_act, -1, (n_pairs - first) / n_chunks >= 32,
                 X);
#pragma unroll
    for (int t = 0; t < kT; ++t) {
      unsigned long long m = 0ull;
      for (int b = 0; b < Q.k; ++b)
        if (X.d[t] && src_s[b] == X.u[t]) m |= 1ull << b;
      excl[t * kLockThreads + threadIdx.x] = m;
      if (m) own_rows = 1;
    }
    __syncthreads();
    const bool any_own = own_rows != 0;
    uint2 m0 = Q.mask[(int64_t)(Q.j0 + first) * Q.rows];
    for (int32_t q = first; q < n_pairs; q += n_chunks) {
      const int32_t j = Q.j0 + q;
      uint2 m = m0;
      if (q + n_chunks < n_pairs) m0 = Q.mask[(int64_t)(j + n_chunks) * Q.rows];
      if (!(m.x | m.y)) continue;
      const uint2 *mask = Q.mask + (int64_t)j * Q.rows;
      int32_t b[kT];
      uint32_t deg[kT], x0[kT], x1[kT], idx[kT];
      uint2 gone[kT];  // sources met, or whose own row this is
      E e[kT];
#pragma unroll
      for (int t = 0; t < kT; ++t) {
        philox2k(Q, (uint32_t)j, (uint32_t)X.u[t], x0[t], x1[t]);
        gone[t] = make_uint2(0u, 0u);
        deg[t] = X.d[t];
        if (any_own) {
          const unsigned long long g = excl[t * kLockThreads + threadIdx.x];
          gone[t] = make_uint2((uint32_t)g, (uint32_t)(g >> 32));
          if (!((m.x & ~gone[t].x) | (m.y & ~gone[t].y))) deg[t] = 0;
        }
      }
      lock_index(x0, deg, Q.key, 1, (uint32_t)j, X.u, idx);
#pragma unroll
      for (int t = 0; t < kT; ++t) {
        e[t] = E{};
        const bool p = deg[t] != 0;
        load_if(p && X.at[t] >= 0, lists_at + (uint32_t)sizeof(E) * ((uint32_t)X.at[t] + idx[t]),
                e[t]);
        load_if(p && X.at[t] < 0, entries(G) + ((uint32_t)X.b[t] + idx[t]), e[t]);
      }
      for (int i = 1;; ++i) {
        // the walks are at the nodes that the entries e of step i name
        const uint2 mn = mask[i];
        const int64_t table = rowbase[i] + j;
        const uint32_t *sig = Q.sig + table * 32;
        bool cand[kT], any = false;
#pragma unroll
        for (int t = 0; t < kT; ++t) {
          const uint32_t h = sig_bit(entry_pos(G, e[t]));
          uint32_t word = 0;
          load_if(deg[t] != 0, sig + (h >> 5), word);
          cand[t] = (word >> (h & 31)) & 1u;
          any |= cand[t];
          if (kCount && deg[t]) ++X.st[t];
        }
        if (any) {
#pragma unroll
          for (int t = 0; t < kT; ++t) {
            if (!cand[t]) continue;
            const int32_t x = entry_pos(G, e[t]);
            const uint4 *tab = Q.T + (table << Q.tbits);
            uint32_t sl = slot_of(x, Q.tbits);
            for (uint32_t probe = 0; probe <= smask; ++probe, sl = (sl + 1u) & smask) {
              const uint4 c = tab[sl];
              if (c.x == (uint32_t)x + 1u) {
                const uint32_t lo = c.y & m.x & ~gone[t].x, hi = c.z & m.y & ~gone[t].y;
                gone[t].x |= lo;
                gone[t].y |= hi;
                for (unsigned long long w = ((unsigned long long)hi << 32) | lo; w; w &= w - 1) {
                  const SharedSrc &B = Q.src[__ffsll((long long)w) - 1];
                  atomicAdd(&B.W[X.u[t]], B.wj[j]);
                  if (B.counts) atomicAdd(&B.counts[X.u[t]], 1u);
                }
                break;
              }
              if (c.x == 0u) break;
            }
          }
        }
        if (!(mn.x | mn.y)) break;  // no source's pair j reaches step i + 1
        m = mn;
        uint32_t live = 0;
#pragma unroll
        for (int t = 0; t < kT; ++t) {
          const bool p = deg[t] != 0 && ((m.x & ~gone[t].x) | (m.y & ~gone[t].y)) != 0;
          b[t] = lock_next(G, tabs, p, e[t], entry_pos(G, e[t]), deg[t]);
          live |= deg[t];
        }
        if (!__any_sync(0xffffffffu, live != 0)) break;
        if (!(i & 1)) {
#pragma unroll
          for (int t = 0; t < kT; ++t)
            philox2k(Q, walk_ctr0(i + 1, (uint32_t)j), (uint32_t)X.u[t], x0[t], x1[t]);
          lock_index(x0, deg, Q.key, i + 1, (uint32_t)j, X.u, idx);
        } else {
          lock_index(x1, deg, Q.key, i + 1, (uint32_t)j, X.u, idx);
        }
#pragma unroll
        for (int t = 0; t < kT; ++t)
          load_if(deg[t] != 0, entries(G) + ((uint32_t)b[t] + idx[t]), e[t]);
      }
    }
    if (kCount) {
#pragma unroll
      for (int t = 0; t < kT; ++t) total += X.st[t];
    }
  }
  if (kCount) {
    for (int o = 16; o > 0; o >>= 1) total += __shfl_xor_sync(0xffffffffu, total, o);
    if (lane == 0 && total) atomicAdd(Q.steps, total);
  }
}

// The rows' scores from their weight sums (blockIdx.y: the row).
__global__ void __launch_bounds__(256)
k_finish_rows(const SharedSrc *__restrict__ src, int32_t n) {
  __shared__ uint16_t list[kFinishTile];
  __shared__ int32_t n_list;
  const SharedSrc B = src[blockIdx.y];
  double *scores = reinterpret_cast<double *>(B.W);
  for (int64_t u0 = (int64_t)blockIdx.x * kFinishTile; u0 < n;
       u0 += (int64_t)gridDim.x * kFinishTile) {
    const int64_t u1 = min((int64_t)n, u0 + kFinishTile);
    finish_tile(scores, u0, u1, B.z, list, &n_list);
    if (threadIdx.x == 0 && B.s >= u0 && B.s < u1) scores[B.s] = 1.0;
  }
}

// ------------------------------------------------------------ host side --
// Sizes (and, with a base, places) the end nodes and filters of one query in
// at most `avail` bytes; F->slots stays null when the query does without.
// Returns the bytes taken.
static size_t align_up(size_t x) { return (x + 255) & ~(size_t)255; }

WalkWay walk_way(const srk_graph *g, const QueryTab &t, int64_t n_targets, bool batch) {
  const int64_t pairs = t.L >= 1 ? t.N_tot - t.P[1] : 0;
  if (t.literal || pairs == 0 || g->m == 0) return WalkWay::kPlain;
  // Filters cost a pass over the edges and save about a last step in every pair and
  // target.  Where they don't pay, and on some adjacencies that the caches hold less
  // of, a warp per target is the fastest: it reads the target's list from L1 for all
  // its first steps.  The lines, in pairs x targets with in-neighbours an edge, ms
  // with filters, without and with warps (lists of 16, part of the targets):
  //   R-MAT 18 narrow (16 MB)   4.9: 0.26 0.25 0.26;  13: 0.36 0.40 0.40
  //   R-MAT 18 csr (17 MB)      1.1: 0.20 0.15 0.20;  4.9: 0.30 0.30 0.29;  13: 0.44 0.51 0.48
  //   R-MAT 20 narrow (64 MB)   1.2: 0.45 0.27 0.29;  4.9: 0.72 0.68 0.64;  13: 1.15 1.32 1.18
  //   ER 2^20 narrow            2.2: 0.41 0.42 0.41;  7: 0.78 1.06 0.90;  24: 2.09 3.02 2.35
  //   R-MAT 22 narrow (268 MB)  1.1: 1.39 1.11 0.94;  3: 3.08 - 2.32;  12: 5.28 8.00 6.08
  //   ER 2^22 narrow            0.6: - 1.01 0.71;  6.8: 4.95 8.40 5.39;  20: 13.6 23.9 15.8
  //   R-MAT 20 wide (143 MB)    13: 1.58 2.17 1.38;  39: 3.88 6.70 4.19;  78: 7.79 13.8 8.70
  //   ER 2^20 wide              2.2: 0.52 0.66 0.48;  24: 2.61 5.30 2.86;  72: 7.06 14.7 7.79
  //   R-MAT 23 wide (1.1 GB)    3: 7.94 12.6 7.66;  9: 24.2 41.7 26.0
  //   ER 2^23 wide              7: 15.0 30.0 18.4
  //   R-MAT 20 csr (72 MB)      13: 1.56 1.91 1.40;  39: 4.23 5.78 4.17;  78: 8.37 12.3 8.59
  //   R-MAT on 1.7e6 csr (102 MB)  71: 16.8 - 15.7;  ER on 1.5e6 csr (97 MB)  143: 27.8 - 29.0
  //   R-MAT 22 csr (285 MB)     3: 3.71 4.41 2.55;  9: 8.09 11.3 8.16;  18: 16.5 24.1 17.2
  //   ER 2^22 csr               6.8: 6.84 10.8 6.86;  20: 19.2 31.7 20.0
  const int64_t bytes = adj_bytes(g);
  const bool small = bytes <= (48ll << 20), far = bytes > kNearBytes;
  const double targets = (double)n_targets * (double)g->n_act / (double)g->n,
               rate = (double)pairs * targets / (double)g->m;
  // (a small adjacency's line was measured in targets of any kind: 1,000 nodes with
  // lists of 16, L = 2, 126 pairs 53 us without filters, 66 with)
  double least = 6.0;
  if (small) least = 8.0 * (double)g->n_act / (double)g->n;
  else if (batch) least = g->layout == kNarrow && !far ? 6.0 : 1.5;
  else if (g->layout == kNarrow) least = 6.0;
  else if (g->layout == kCsr) least = !far ? 40.0 : bytes <= (200ll << 20) ? 80.0 : 9.0;
  else least = bytes <= (256ll << 20) ? 20.0 : 6.0;
  // with L = 1 the pass over the edges is all there is (R-MAT 20, 4.3: 0.11 ms, 1.15
  // without)
  if (t.L == 1 && !small) least = 0.5;
  // More than 2^20 end nodes would take a table of more than 32 MB.  (So many walks do
  // not: 1.2e6 on R-MAT 16 take 110 ms with filters, 178 without and 168 with a warp per
  // target; 5e6 on 1,000 nodes 28.3, 31.7 and 134 ms.  On fewer targets k_edges, which
  // then has long lists of pairs for a few edges, was not measured with as many.)
  const bool fit = std::min<int64_t>(pairs, g->n) <= (1 << 20) &&
                   (t.N_tot <= (1 << 20) || n_targets >= 1000);
  if (fit && rate >= least) return WalkWay::kFilters;
  // Fewer than 128 pairs are too few rounds for a warp's lanes, and on adjacencies that
  // the caches do hold lockstep without filters is the faster down to few targets.
  if (batch || pairs < 128) return WalkWay::kPlain;
  const double few = g->layout == kNarrow ? (small ? 1e30 : far ? 0.0 : 2.0)
                     : bytes <= (12ll << 20) ? 1e30 : small ? 3.0 : 0.0;
  return rate < few ? WalkWay::kPlain : WalkWay::kWarps;
}

size_t plan_filters(const srk_graph *g, const QueryTab &t, const Workspace &w, WalkWay way,
                    size_t avail, Filters *F, char *base) {
  memset(F, 0, sizeof *F);
  // (arrays of the shuffle, free by then)
  F->list1 = w.items;
  F->slot_of = w.first;
  F->rank1 = w.succ;
  if (way != WalkWay::kFilters) return 0;
  const int64_t pairs = t.N_tot - t.P[1];
  int sb = 5;
  while (((int64_t)1 << sb) < 2 * std::min<int64_t>(pairs, g->n)) ++sb;
  F->slot_bits = sb;
  F->bloom_bits = std::min(20, sb + 3);
  const size_t fixed = align_up((size_t)16 << sb) + align_up((size_t)1 << (F->bloom_bits - 3)) + 256;
  if (avail < fixed) return 0;
  // room for 2 KB per end node of a longer pair; those beyond do without
  const size_t unit = 4 * kFilterUnit;
  const int64_t wanted = std::min<int64_t>(t.L >= 2 ? t.N_tot - t.P[2] : 0, g->n);
  const size_t room = std::min<size_t>(std::min<size_t>(avail - fixed, (size_t)32 << 20),
                                       (size_t)wanted * 2048 + 65536);
  F->max_units = (int32_t)(room / unit);
  F->out_deg = g->out_deg;
  F->slots = reinterpret_cast<EndSlot *>(base);
  F->bloom = reinterpret_cast<uint32_t *>(base + align_up((size_t)16 << sb));
  F->ctl = reinterpret_cast<int32_t *>(base + fixed - 256);
  F->bits = reinterpret_cast<uint32_t *>(base + fixed);
  return fixed + unit * (size_t)F->max_units;
}

size_t filter_bytes(const srk_graph *g, const QueryTab &t, WalkWay way) {
  Filters F;
  Workspace w;
  memset(&w, 0, sizeof w);
  return plan_filters(g, t, w, way, SIZE_MAX, &F, nullptr);
}


static int grid_for(int64_t work, int threads, int device) {
  const int64_t want = (work + threads - 1) / threads;
  const int64_t cap = (int64_t)sm_count(device) * 8;
  return (int)std::max<int64_t>(1, std::min<int64_t>(want, cap));
}

// Lets the lockstep kernels take their shared memory (above the default 48 KB
// a kernel must opt in).  Called at graph load, in the context the queries
// run in and outside any capture.
template <int kLayout>
static cudaError_t allow_lock_t() {
  cudaError_t e = cudaSuccess;
  auto set = [&](const void *f) {
    if (e == cudaSuccess)
      e = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kLockSmem);
  };
  set((const void *)k_lockstep<kLayout, false, 1>);
  set((const void *)k_lockstep<kLayout, true, 1>);
  set((const void *)k_lockstep<kLayout, false, kLockTargets>);
  set((const void *)k_lockstep<kLayout, true, kLockTargets>);
  set((const void *)k_lockstep_group<kLayout, false, 1>);
  set((const void *)k_lockstep_group<kLayout, true, 1>);
  set((const void *)k_lockstep_group<kLayout, false, kLockTargets>);
  set((const void *)k_lockstep_group<kLayout, true, kLockTargets>);
  set((const void *)k_lock_shared<kLayout, false>);
  set((const void *)k_lock_shared<kLayout, true>);
  return e;
}
cudaError_t allow_lockstep(int layout) {
  return layout == kWide ? allow_lock_t<kWide>()
         : layout == kCsr ? allow_lock_t<kCsr>()
                          : allow_lock_t<kNarrow>();
}

template <int kLayout, bool kCount>
static void launch_lockstep(const GraphView &V, const int32_t *act, int32_t *bounds,
                            const LockQuery &Q, int shape, int grid, cudaStream_t st) {
  if (shape == 1)
    k_lockstep<kLayout, kCount, 1><<<grid, kLockThreads, kLockSmem, st>>>(V, act, bounds, Q);
  else
    k_lockstep<kLayout, kCount, kLockTargets><<<grid, kLockThreads, kLockSmem, st>>>(V, act, bounds,
                                                                                     Q);
}

// For a group of queries.
template <int kLayout, bool kCount>
static void launch_group(const GraphView &V, const int32_t *act, int32_t n_act,
                         const WalkJob *jobs, int32_t k, int32_t *counter, int shape, int grid,
                         cudaStream_t st) {
  if (shape == 1)
    k_lockstep_group<kLayout, kCount, 1><<<grid, kLockThreads, kLockSmem, st>>>(V, act, n_act, jobs,
                                                                                k, counter);
  else
    k_lockstep_group<kLayout, kCount, kLockTargets><<<grid, kLockThreads, kLockSmem, st>>>(
        V, act, n_act, jobs, k, counter);
}

// Calls launch<layout, count>(...) for a graph.
#define SRK_BY_LAYOUT(launch, ...)                                       \
  do {                                                                   \
    if (g->layout == kWide) {                                            \
      if (count) launch<kWide, true>(__VA_ARGS__);                       \
      else launch<kWide, false>(__VA_ARGS__);                            \
    } else if (g->layout == kCsr) {                                      \
      if (count) launch<kCsr, true>(__VA_ARGS__);                        \
      else launch<kCsr, false>(__VA_ARGS__);                             \
    } else {                                                             \
      if (count) launch<kNarrow, true>(__VA_ARGS__);                     \
      else launch<kNarrow, false>(__VA_ARGS__);                          \
    }                                                                    \
  } while (0)

// Polls of a wait for filters: 2^20, or the environment variable SRK_WAIT_POLLS.
static int32_t wait_polls() {
  const char *env = getenv("SRK_WAIT_POLLS");
  if (!env || !*env) return kWaitPolls;
  const long v = strtol(env, nullptr, 10);
  return v < 0 || v > kWaitPolls ? kWaitPolls : (int32_t)v;
}

static LockQuery lock_query(const QueryTab &t, const Workspace &w, const Filters &F,
                            const Outputs &o) {
  const Small sm = small_view(w.small);
  LockQuery Q;
  memset(&Q, 0, sizeof Q);
  Q.rec = w.rec();
  Q.w = w.pair_w;
  Q.H = w.Hc;
  Q.bits = F.bits;
  Q.cnt = sm.cnt;
  Q.W = reinterpret_cast<unsigned long long *>(o.scores);
  Q.counts = o.counts;
  Q.steps = o.steps;
  Q.steps_total = sm.ctr;
  Q.key = t.tkey;
  for (int r = 0; r < 10; ++r) Q.rk[r] = t.tkey + (uint32_t)r * kPhiloxW0;
  Q.s = t.s;
  Q.min_cap = F.slots ? 2 : 1;
  Q.polls = wait_polls();
  return Q;
}

// kLockTargets targets a thread (shape 0), or one (1) where there are too few to
// give it several, and on the wide layout far beyond the L2, where fewer of the
// targets' own lists then compete for it.  Wide layout, ms for 3 queries, 3 targets
// a thread and one: 2^20 nodes with lists of 16 (143 MB) 25.1 and 32.7 (R-MAT), 44.2 and
// 53.4 (ER); 2^21 (285 MB) 77.2 and 80.8, 138 and 133; 2^23 153 and 145, 319 and 289.
int walk_shape(const srk_graph *g, int64_t n_targets) {
  const bool far = g->layout == kWide && 8 * ((int64_t)g->n + g->m) > (256ll << 20);
  return n_targets <= kLockThreads || far ? 1 : 0;
}

int enqueue_walks(const srk_graph *g, const QueryTab &t, const Workspace &w, const Filters &F,
                  const Outputs &o, bool count, cudaStream_t st, const cudaEvent_t *timing,
                  int32_t u_begin, int32_t u_end) {
  const int dev = g->device;
  const int64_t nr = (int64_t)u_end - u_begin;
  const GraphView V = view_of(g);
  const Small sm = small_view(w.small);
  int32_t *bounds = reinterpret_cast<int32_t *>(sm.ctr + 2);
  const LockQuery Q = lock_query(t, w, F, o);
  if (F.slots)
    k_edges<<<grid_for(g->m, 256, dev), 256, 0, st>>>(F, V, g->m, sm.cnt, w.rec(), w.pair_w, t.tkey,
                                                      t.s, u_begin, u_end, Q.W, o.counts);
  if (timing) cudaEventRecord(timing[0], st);
  const int grid = sm_count(dev) * kLockBlocks;
  // The targets: by rank where all of them are wanted (the narrow layout ranks
  // the nodes with in-neighbours first), so that a block's lists are of one
  // length: the short ones all fit its shared memory, the heavy units come
  // first.  By id for a part of them.
  const int32_t *act = nr == g->n && g->layout == kNarrow ? g->order : g->act;
  SRK_BY_LAYOUT(launch_lockstep, V, act, bounds, Q, walk_shape(g, nr), grid, st);
  if (timing) cudaEventRecord(timing[1], st);
  if (nr > 0)
    k_finish<<<grid_for(nr, kFinishTile, dev), 256, 0, st>>>(g->row_ptr, bounds, sm.cnt, t.s,
                                                             u_begin, u_end, t.z, F.slots ? 1 : 0, o.scores,
                                                     o.wsums, o.steps, sm.ctr);
  const cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return cuda_fail(e, "kernel launch");
  return SRK_OK;
}

// Queries of more pairs x targets than this fill the GPU by themselves and are walked
// by k_lockstep, whose query is a kernel parameter.  R-MAT 16, 16 queries: of 7e7
// 6.05 ms with launches of their own, 5.39 ms as a group; of 4e8 29.9 and 29.9; with
// those of 2e9 in a batch 70.0 and 73.2.
constexpr double kAlonePairs = 5e8;

WalkJob walk_job(const srk_graph *g, const QueryTab &t, const Workspace &w, const Filters &F,
                 const Outputs &o) {
  WalkJob J;
  memset(&J, 0, sizeof J);
  J.w = w;
  J.F = F;
  J.Q = lock_query(t, w, F, o);
  J.z = t.z;
  const int64_t pairs = t.L >= J.Q.min_cap ? t.N_tot - t.P[J.Q.min_cap] : 0;  // at most
  J.alone = (double)pairs * g->n_act > kAlonePairs ? 1 : 0;
  return J;
}

int enqueue_walk_group(const srk_graph *g, const WalkJob *host, const WalkJob *jobs, int32_t k,
                       int32_t N, int32_t *counter, bool count, cudaStream_t st) {
  const int dev = g->device, sms = sm_count(dev), grid = sms * kLockBlocks;
  const GraphView V = view_of(g);
  bool ends = false, together = false;
  for (int32_t b = 0; b < k; ++b) {
    ends |= host[b].F.slots != nullptr;
    together |= host[b].alone == 0;
  }
  if (ends) {
    const int rc = enqueue_ends(g, jobs, k, N, st);
    if (rc) return rc;
    // (a group's queries share the SMs: longer runs of edges a warp)
    const dim3 by((unsigned)std::min(grid_for(g->m, 256, dev), std::max(8, sms * 16 / k)),
                  (unsigned)k);
    k_edges_group<<<by, 256, 0, st>>>(V, g->m, jobs);
  }
  const int32_t *act = g->layout == kNarrow ? g->order : g->act;  // (see enqueue_walks)
  const int shape = walk_shape(g, g->n_act);
  if (together)
    SRK_BY_LAYOUT(launch_group, V, act, g->n_act, jobs, k, counter, shape, grid, st);
  for (int32_t b = 0; b < k; ++b)
    if (host[b].alone) {
      int32_t *bounds = reinterpret_cast<int32_t *>(small_view(host[b].w.small).ctr + 2);
      SRK_BY_LAYOUT(launch_lockstep, V, act, bounds, host[b].Q, shape, grid, st);
    }
  const dim3 by((unsigned)std::min(grid_for(g->n, kFinishTile, dev), std::max(4, sms * 8 / k)),
                (unsigned)k);
  k_finish_group<<<by, 256, 0, st>>>(g->row_ptr, g->n, g->n_act, jobs);
  const cudaError_t e = cudaGetLastError();
  return e == cudaSuccess ? SRK_OK : cuda_fail(e, "kernel launch");
}

int enqueue_shared_walks(const srk_graph *g, const SharedWalks &Q, cudaStream_t st) {
  const GraphView V = view_of(g);
  const int32_t *act = g->layout == kNarrow ? g->order : g->act;  // (see enqueue_walks)
  const int grid = sm_count(g->device) * kLockBlocks;
  const size_t smem = 4 * (size_t)kListWords + 8 * kHubCache + 4 * kCodes +
                      8 * (size_t)kSharedTargets * kLockThreads;
  static_assert(4 * (size_t)kListWords + 8 * kHubCache + 4 * kCodes +
                        8 * (size_t)kSharedTargets * kLockThreads <= kLockSmem,
                "the opt-in covers both kernels");
#define SRK_SHARED(L)                                                                       \
  do {                                                                                      \
    if (Q.steps) k_lock_shared<L, true><<<grid, kLockThreads, smem, st>>>(V, act, g->n_act, Q); \
    else k_lock_shared<L, false><<<grid, kLockThreads, smem, st>>>(V, act, g->n_act, Q);  \
  } while (0)
  if (g->layout == kWide) SRK_SHARED(kWide);
  else if (g->layout == kCsr) SRK_SHARED(kCsr);
  else SRK_SHARED(kNarrow);
#undef SRK_SHARED
  const dim3 rows((unsigned)std::min<int64_t>((g->n + (int64_t)kFinishTile - 1) / kFinishTile,
                                              (int64_t)sm_count(g->device) * 4),
                  (unsigned)Q.k);
  k_finish_rows<<<rows, 256, 0, st>>>(Q.src, g->n);
  const cudaError_t e = cudaGetLastError();
  return e == cudaSuccess ? SRK_OK : cuda_fail(e, "shared walks: launch");
}

}  // namespace srk
