// srk_multi_source: many single-source queries with uneven walk budgets.
//
// The sources are processed in batches sized by a memory budget.  One launch runs
// the source side (steps a2-a3) of all a batch's sources, a cluster each
// (srk_source.cu).  Their targets are then walked as srk_single_source walks them
// (srk_lockstep.cu), so the results are identical, a group of sources at a time:
// one launch each for the group's end nodes, edges, walks and scores, but that a
// source whose walks fill the GPU by themselves has a walk launch of its own.
// Sources whose walks never leave the source (no pair can meet) find no work
// there: their score rows are prefilled (1 at the source, 0 elsewhere).  A batch's
// launches are captured in a CUDA graph and launched as one.  With shared target
// walks (SRK_OPT_SHARED_WALKS) the batches hold up to 64 sources and the target
// walks run once for all of them (k_lock_shared, srk_lockstep.cu).
#include <stdint.h>
#include <stdlib.h>
#include <string.h>

#include <algorithm>
#include <mutex>
#include <vector>

#include "srk_device.cuh"
#include "srk_internal.h"

namespace srk {

// One source of a batch, as the batched kernels see it (device memory).
struct BatchSrc {
  Workspace w;            // the source's scratch (see plan())
  const QueryTab *tab;    // the source's table (device copy)
  double *scores;         // output row, n entries
  uint32_t *counts;       // output row or null
  unsigned long long *wj;     // shared walks: quantised Lemma 7 weight of pair j
  int32_t s, L, N_tot;
  double z;
};

struct BatchArgs {
  const BatchSrc *src;
  const int64_t *walk_off;  // prefix of N_tot over the batch, k+1 entries
  int32_t k;
  int64_t total_walks;
  GraphView view;
  uint2 *M;       // shared walks: M[j (Lmax + 1) + i - 1] bit b = pair j of batch source b
                  // may still meet at step i (cap_b(j) >= i)
  uint32_t *sig;  // shared walks: 32 words per meeting table, bit sig_bit(node) set for
                  // every node of the table
  uint4 *T;       // shared walks: the meeting tables, one per (step i, pair j) with
                  // j >= Pmin_i (below, no pair of the batch reaches step i) at
                  // T + ((rowbase[i] + j) << tbits): 2^tbits slots {node + 1,
                  // (.y, .z) the sources b with cap_b(j) >= i whose walk
                  // sigma_b(j) is at that node at step i}, empty slots 0,
                  // linear probing from slot_of(node)
  const int64_t *rowbase;  // shared walks: rowbase[i] = tables before step i - Pmin_i
  int32_t tbits;  // shared walks: log2 of the slots per table (>= 2 k)
  int32_t Lmax;   // shared walks: the largest L of the batch
};

__device__ __forceinline__ int find_source(const int64_t *off, int k, int64_t g) {
  int lo = 0, hi = k - 1;  // last i with off[i] <= g
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (off[mid] <= g) lo = mid; else hi = mid - 1;
  }
  return lo;
}

#define SRK_BATCH_LOOP(A, ...)                                                   \
  for (int64_t g_ = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;              \
       g_ < (A).total_walks; g_ += (int64_t)gridDim.x * blockDim.x) {            \
    const int i_ = find_source((A).walk_off, (A).k, g_);                         \
    const BatchSrc &S_ = (A).src[i_];                                            \
    const int32_t r_ = (int32_t)(g_ - (A).walk_off[i_]);                         \
    __VA_ARGS__                                                                  \
  }

// Every output row: 0 (the walks add to the rows), and 1 at the source.
__global__ void kb_prefill(const BatchSrc *__restrict__ src, int32_t k, int32_t n) {
  const int64_t total = (int64_t)k * n;
  for (int64_t g = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; g < total;
       g += (int64_t)gridDim.x * blockDim.x) {
    const int i = (int)(g / n);
    const int32_t u = (int32_t)(g - (int64_t)i * n);
    src[i].scores[u] = (u == src[i].s) ? 1.0 : 0.0;
    if (src[i].counts) src[i].counts[u] = 0;
  }
}

// ------------------------------------------------------------------------
// Shared target walks (SRK_OPT_SHARED_WALKS).  Target walk j of u no longer
// depends on the source, so one walk serves pair j of every source of the
// batch: it goes on while some source's pair j can still meet (it has not met
// and its cap is not reached) and stops at a node without in-neighbours.  For
// source b the pair meets at the first step i <= cap_b(j) where the walk is
// at the node of source b's walk sigma_b(j) at step i, exactly as
// srk_single_source with the same flag decides it.  Those nodes of all the
// batch's sources sit in one small hash table per (step, pair), so a walk
// tests every pending source with one lookup of its own node (one sector,
// rarely two).  Batches hold at most 64 sources (one mask bit each).  The walks
// are k_lock_shared's (srk_lockstep.cu).

// Per source and pair j: the pair's weight, its bit in the step masks, its
// node's bit in the tables' signatures and its bit in the meeting tables of
// steps 1..cap(j) (source walk sigma(j)).  A table holds at most k nodes in
// 2^tbits >= 2k slots, so an insertion always finds its node or a free slot.
__global__ void kb_hitj(const __grid_constant__ BatchArgs A) {
  SRK_BATCH_LOOP(A, {
    const int32_t j = r_;
    const int32_t w = S_.w.sigma[j];
    const int l2 = stratum_of(S_.tab->P, S_.L, j);
    const int32_t cap = min(l2, S_.w.seff[w]);
    const int l1 = stratum_of(S_.tab->P, S_.L, w);
    S_.wj[j] = cap >= 1 ? __double2ull_rn(S_.tab->a[l1] * S_.tab->a[l2] * 4294967296.0) : 0ull;
    const int Ls = S_.L > 0 ? S_.L : 1;
    const int32_t *sp = S_.w.spos + (int64_t)w * Ls;
    const uint32_t bit = 1u << (i_ & 31);  // in word .x (sources 0-31) or .y (32-63)
    const bool high = i_ >= 32;
    const uint32_t smask = (1u << A.tbits) - 1u;
    for (int q = 1; q <= cap; ++q) {
      const int32_t node = walk_identity(A.view, sp[q - 1]);
      uint2 *cell = &A.M[(int64_t)j * (A.Lmax + 1) + q - 1];
      const uint32_t h = sig_bit(node);
      atomicOr(high ? &cell->y : &cell->x, bit);
      atomicOr(&A.sig[(A.rowbase[q] + j) * 32 + (h >> 5)], 1u << (h & 31));
      uint4 *tab = A.T + ((A.rowbase[q] + j) << A.tbits);
      const uint32_t key = (uint32_t)node + 1u;
      uint32_t sl = slot_of(node, A.tbits);
      for (uint32_t probe = 0; probe <= smask; ++probe, sl = (sl + 1u) & smask) {
        const uint32_t prev = atomicCAS(&tab[sl].x, 0u, key);
        if (prev == 0u || prev == key) {
          atomicOr(high ? &tab[sl].z : &tab[sl].y, bit);
          break;
        }
      }
    }
  })
}

static size_t align256(size_t x) { return (x + 255) & ~(size_t)255; }

// The first walk index of source table t whose length is at least i (walks
// are in stratum order): pairs below it cannot reach step i.
static int32_t first_reaching(const QueryTab &t, int i) {
  return i <= t.L ? t.P[i] : t.N_tot;
}

static std::mutex g_stream_mu;
static cudaStream_t g_cap_stream[64] = {};

// One lock per device around a batch's capture and graph launch: the capture
// stream and the handles' cached executables are shared.
static std::mutex g_capture_mu[64];
static std::mutex &capture_mutex(int dev) { return g_capture_mu[dev >= 0 && dev < 64 ? dev : 0]; }

// A library-owned non-blocking stream per device for graph capture (the
// caller's stream may be the legacy default stream, which cannot capture).
static cudaStream_t capture_stream(int dev) {
  std::lock_guard<std::mutex> lk(g_stream_mu);
  if (dev < 0 || dev >= 64) return nullptr;
  if (!g_cap_stream[dev]) {
    cudaStream_t s = nullptr;
    if (cudaStreamCreateWithFlags(&s, cudaStreamNonBlocking) != cudaSuccess) return nullptr;
    g_cap_stream[dev] = s;
  }
  return g_cap_stream[dev];
}

}  // namespace srk

using namespace srk;

namespace srk {

__global__ void k_source_degrees(const int32_t *__restrict__ row_ptr,
                                 int32_t *__restrict__ v, int32_t k) {
  const int32_t i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < k) v[i] = row_ptr[v[i] + 1] - row_ptr[v[i]];
}

int source_in_degrees(const srk_graph *g, const int32_t *sources, int32_t k, cudaStream_t st,
                      std::vector<int32_t> *deg) {
  deg->assign((size_t)k, 0);
  if (k <= 0) return SRK_OK;
  cudaMemPool_t mp = pool(g->device);
  if (!mp) return fail(SRK_ECUDA, "cannot create the device memory pool");
  int32_t *d = nullptr;
  cudaError_t e = cudaMallocFromPoolAsync((void **)&d, sizeof(int32_t) * (size_t)k, mp, st);
  if (e != cudaSuccess) return cuda_fail(e, "source degrees: allocation");
  e = cudaMemcpyAsync(d, sources, sizeof(int32_t) * (size_t)k, cudaMemcpyHostToDevice, st);
  if (e == cudaSuccess) {
    k_source_degrees<<<(k + 255) / 256, 256, 0, st>>>(g->row_ptr, d, k);
    e = cudaGetLastError();
  }
  if (e == cudaSuccess)
    e = cudaMemcpyAsync(deg->data(), d, sizeof(int32_t) * (size_t)k, cudaMemcpyDeviceToHost, st);
  cudaFreeAsync(d, st);
  if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  return e == cudaSuccess ? SRK_OK : cuda_fail(e, "source degrees");
}

}  // namespace srk

extern "C" int srk_multi_source(const srk_graph *g, const int32_t *sources,
                                int32_t k, double c, const double *eps,
                                uint64_t seed, const srk_opts *opt,
                                double *scores, uint32_t *meet_counts,
                                void *cuda_stream) {
  clear_error();
  if (!g) return fail(SRK_EINVAL, "null graph");
  if (k < 0) return fail(SRK_EINVAL, "k = %d is negative", k);
  if (k == 0) return SRK_OK;
  if (!sources || !eps || !scores) return fail(SRK_EINVAL, "null argument");
  if (opt && opt->step_counts)
    return fail(SRK_EINVAL, "step_counts is not supported by srk_multi_source");
  if (opt && (opt->flags & SRK_OPT_LITERAL_SHUFFLE))
    return fail(SRK_EINVAL, "the literal shuffle is not supported by srk_multi_source");
  if (opt && (opt->flags & ~(SRK_OPT_NO_GRAPH | SRK_OPT_WARMUP_RULE | SRK_OPT_SHARED_WALKS)))
    return fail(SRK_EINVAL, "unknown opts.flags 0x%x", opt->flags);
  if (opt && (opt->target_begin != 0 || opt->target_end != 0))
    return fail(SRK_EINVAL, "target ranges are not supported by srk_multi_source");
  const bool use_graph = !(opt && (opt->flags & SRK_OPT_NO_GRAPH));
  const bool shared = opt && (opt->flags & SRK_OPT_SHARED_WALKS);
  const size_t n = (size_t)g->n;
  // a1 for every source (host, FP64)
  std::vector<QueryTab> tabs((size_t)k);
  for (int32_t i = 0; i < k; ++i) {
    int rc = build_table(g->n, sources[i], c, eps[i], seed, opt, &tabs[i]);
    if (rc) return fail(rc, "source %d (index %d): %s", sources[i], i, srk_last_error());
  }
  // batch position -> the caller's row.  With shared target walks the
  // sources are grouped by walk budget (N_tot, then L), so that a batch's
  // sources share as many pairs as possible; a source's results do not
  // depend on its batch, since its target walks do not depend on it.
  std::vector<int32_t> row_of((size_t)k);
  for (int32_t i = 0; i < k; ++i) row_of[(size_t)i] = i;
  DeviceGuard guard(g->device);
  if (shared) {
    // sources without in-neighbours go last: their pairs meet nowhere, so they
    // would hold places in batches that share walks
    std::vector<int32_t> deg;
    const int rcd = source_in_degrees(g, sources, k, (cudaStream_t)cuda_stream, &deg);
    if (rcd) return rcd;
    std::stable_sort(row_of.begin(), row_of.end(), [&](int32_t a, int32_t b) {
      const QueryTab &ta = tabs[(size_t)a], &tb = tabs[(size_t)b];
      const bool za = deg[(size_t)a] == 0, zb = deg[(size_t)b] == 0;
      if (za != zb) return zb;
      return ta.N_tot != tb.N_tot ? ta.N_tot < tb.N_tot : ta.L < tb.L;
    });
    std::vector<QueryTab> sorted((size_t)k);
    for (int32_t p = 0; p < k; ++p) sorted[(size_t)p] = tabs[(size_t)row_of[(size_t)p]];
    tabs.swap(sorted);
  }
  const int dev = g->device;
  const int sms = sm_count(dev);
  cudaStream_t st = (cudaStream_t)cuda_stream;
  const bool d_scores = is_device_ptr(scores);
  const bool d_counts = !meet_counts || is_device_ptr(meet_counts);
  cudaMemPool_t mp = pool(dev);
  if (!mp) return fail(SRK_ECUDA, "cannot create the device memory pool");
  cudaStream_t cs = use_graph ? capture_stream(dev) : st;
  if (use_graph && !cs) return fail(SRK_ECUDA, "cannot create the capture stream");

  // batch shape: as many sources as fit a scratch budget
  size_t free_b = 0, total_b = 0;
  cudaMemGetInfo(&free_b, &total_b);
  size_t budget = std::max<size_t>((size_t)256 << 20,
                                   std::min<size_t>((size_t)8 << 30, free_b / 4));
  if (const char *env = getenv("SRK_BATCH_BYTES")) {  // explicit scratch budget
    const unsigned long long v = strtoull(env, nullptr, 10);
    if (v > 0) budget = (size_t)v;
  }
  srk_stats total;
  memset(&total, 0, sizeof total);
  int32_t i0 = 0;
  int rc = SRK_OK;
  cudaEvent_t ev_in = nullptr, ev_out = nullptr;
  if (use_graph) {
    cudaError_t e = cudaEventCreateWithFlags(&ev_in, cudaEventDisableTiming);
    if (e == cudaSuccess) e = cudaEventCreateWithFlags(&ev_out, cudaEventDisableTiming);
    if (e != cudaSuccess) {
      if (ev_in) cudaEventDestroy(ev_in);
      return cuda_fail(e, "srk_multi_source: creating the graph-launch events");
    }
  }
  while (i0 < k && rc == SRK_OK) {
    // sources [i0, i1) form this batch
    size_t need = 0;
    int32_t i1 = i0;
    std::vector<size_t> ws_off, ends;  // sources' places; bytes of their end filters,
    size_t most = 0;                   //   and the most of them
    int64_t sh_L = 1, sh_N = 0;  // shared walks: the tables' extent so far
    std::vector<int32_t> pmin((size_t)SRK_MAX_LEN + 2, INT32_MAX);
    while (i1 < k && !(shared && i1 - i0 >= 64)) {
      // shared walks: the batch's mask rows and meeting tables with this source
      int64_t L1 = sh_L, N1 = sh_N;
      size_t sb = 0;
      if (shared) {
        const QueryTab &t = tabs[(size_t)i1];
        L1 = std::max<int64_t>(sh_L, std::max(t.L, 1));
        N1 = std::max<int64_t>(sh_N, t.N_tot);
        int tb = 1;
        while ((1 << tb) < 2 * (i1 - i0 + 1)) ++tb;
        size_t tables = 0;
        for (int i = 1; i <= L1; ++i)
          tables += (size_t)(N1 - std::min<int64_t>(pmin[(size_t)i], first_reaching(t, i)));
        sb = 8 * (size_t)(L1 + 1) * (size_t)N1 + 128 * tables + ((16 * tables) << tb);
      }
      Workspace w;
      const QueryTab &t1 = tabs[(size_t)i1];
      const size_t b = align256(plan(t1, &w, nullptr)) +
                       (d_scores ? 0 : align256(8 * n)) + (d_counts ? 0 : align256(4 * n)) +
                       (shared ? align256(8 * (size_t)t1.N_tot) : 0);
      const size_t f = shared ? 0 : align256(filter_bytes(g, t1, walk_way(g, t1, n, true)));
      if (i1 > i0 && need + b + sb + std::max(most, f) > budget) break;
      most = std::max(most, f);
      ends.push_back(f);
      sh_L = L1;
      sh_N = N1;
      if (shared)
        for (int i = 1; i <= SRK_MAX_LEN; ++i)
          pmin[(size_t)i] = std::min(pmin[(size_t)i], first_reaching(tabs[(size_t)i1], i));
      ws_off.push_back(need);
      need += b;
      ++i1;
    }
    const int32_t kb = i1 - i0;
    int Lmax = 0;
    int32_t Jmax = 0, j0 = INT32_MAX;
    for (int32_t b = i0; b < i1; ++b) {
      const QueryTab &t = tabs[(size_t)b];
      Lmax = std::max(Lmax, t.L);
      Jmax = std::max(Jmax, t.N_tot);
      j0 = std::min(j0, t.L >= 1 ? t.P[1] : t.N_tot);  // below, every pair has length 0
    }
    // shared walks: meeting tables of 2^tbits >= 2 kb slots, one per (step i,
    // pair j >= pmin[i]), in rows by step: rowbase[i] + j is the table's index
    int tbits = 1;
    while ((1 << tbits) < 2 * kb) ++tbits;
    std::vector<int64_t> rowbase((size_t)std::max(Lmax, 1) + 1, 0);
    int64_t n_tables = 0;
    for (int i = 1; i <= std::max(Lmax, 1); ++i) {
      const int64_t pm = std::min<int64_t>(pmin[(size_t)i], Jmax);
      rowbase[(size_t)i] = n_tables - pm;
      n_tables += Jmax - pm;
    }
    // shared walks: the step masks (Jmax rows of Lmax + 1), the table rows, the
    // signatures and the tables
    const size_t m_bytes = shared ? 8 * (size_t)(Lmax + 1) * (size_t)Jmax : 0;
    const size_t r_bytes = shared ? sizeof(int64_t) * rowbase.size() : 0;
    const size_t g_bytes = shared ? 128 * (size_t)n_tables : 0;
    const size_t h_bytes = shared ? (16 * (size_t)n_tables) << tbits : 0;
    const size_t c_bytes = shared ? sizeof(SharedSrc) * (size_t)kb : 0;
    size_t head = 0;
    auto part = [&](size_t bytes) {
      const size_t at = head;
      head += align256(bytes);
      return at;
    };
    // the descriptors, which one copy brings to the device, then what it fills itself
    const size_t o_src = part(sizeof(BatchSrc) * (size_t)kb), o_tab = part(sizeof(QueryTab) * (size_t)kb),
                 o_off = part(shared ? sizeof(int64_t) * ((size_t)kb + 1) : 0),
                 o_rowbase = part(r_bytes), o_ssrc = part(c_bytes),
                 o_jobs = part(sizeof(SourceJob) * (size_t)kb),
                 o_walks = part(shared ? 0 : sizeof(WalkJob) * (size_t)kb),
                 o_units = part(shared ? 0 : 4 * (size_t)kb), up_bytes = head;
    const size_t o_ctr = part(256), o_M = part(m_bytes), o_sig = part(g_bytes), o_T = part(h_bytes);
    // End filters: one region, which groups of sources use one after the other,
    // in what the scratch budget leaves.
    size_t room = 0;
    for (size_t f : ends) room += f;
    room = std::min(room, budget > need ? (budget - need) & ~(size_t)255 : 0);
    char *base = nullptr;
    cudaError_t e = cudaMallocFromPoolAsync((void **)&base, head + need + room, mp, st);
    if (e == cudaErrorMemoryAllocation && room > 0) {  // the walks can do without
      cudaGetLastError();
      room = 0;
      e = cudaMallocFromPoolAsync((void **)&base, head + need, mp, st);
    }
    // groups: [groups[q], groups[q + 1]), as many sources as the region holds
    std::vector<int32_t> groups(1, 0);
    size_t held = 0;
    for (int32_t b = 0; b < kb && !shared; ++b) {
      if (b > groups.back() &&
          (b - groups.back() >= kWalkGroup || held + ends[(size_t)b] > room)) {
        groups.push_back(b);
        held = 0;
      }
      held += ends[(size_t)b];
    }
    groups.push_back(kb);
    const int32_t n_groups = (int32_t)groups.size() - 1;
    if (e != cudaSuccess) { rc = cuda_fail(e, "batch workspace allocation"); break; }
    BatchSrc *d_src = (BatchSrc *)(base + o_src);
    QueryTab *d_tab = (QueryTab *)(base + o_tab);
    int64_t *d_off = (int64_t *)(base + o_off), *d_rowbase = (int64_t *)(base + o_rowbase);
    SharedSrc *d_ssrc = (SharedSrc *)(base + o_ssrc);
    SourceJob *d_jobs = (SourceJob *)(base + o_jobs);
    WalkJob *d_walks = (WalkJob *)(base + o_walks);
    int32_t *d_units = (int32_t *)(base + o_units);
    unsigned long long *d_ctr = (unsigned long long *)(base + o_ctr);
    uint2 *d_M = (uint2 *)(base + o_M);
    uint32_t *d_sig = (uint32_t *)(base + o_sig);
    uint4 *d_T = (uint4 *)(base + o_T);
    // shared walks: d_ctr[0] = target counter, d_ctr[1] = steps
    char *ws_base = base + head;
    std::vector<BatchSrc> hsrc((size_t)kb);
    std::vector<int64_t> hoff((size_t)kb + 1);
    hoff[0] = 0;
    for (int32_t b = 0; b < kb; ++b) {
      const QueryTab &t = tabs[(size_t)(i0 + b)];
      BatchSrc &S = hsrc[(size_t)b];
      char *wb = ws_base + ws_off[(size_t)b];
      const size_t core = align256(plan(t, &S.w, wb));
      char *outs = wb + core;
      S.tab = d_tab + b;
      const size_t row = (size_t)row_of[(size_t)(i0 + b)];
      S.scores = d_scores ? scores + row * n : (double *)outs;
      if (!d_scores) outs += align256(8 * n);
      S.counts = !meet_counts ? nullptr
                 : (d_counts ? meet_counts + row * n : (uint32_t *)outs);
      if (meet_counts && !d_counts) outs += align256(4 * n);
      S.wj = nullptr;
      if (shared) {
        S.wj = (unsigned long long *)outs;
        outs += align256(8 * (size_t)t.N_tot);
      }
      S.s = t.s;
      S.L = t.L;
      S.N_tot = t.N_tot;
      S.z = t.z;
      hoff[(size_t)b + 1] = hoff[(size_t)b] + t.N_tot;
    }
    std::vector<SourceJob> jobs;
    for (int32_t b = 0; b < kb; ++b)
      jobs.push_back(SourceJob{hsrc[(size_t)b].w, hsrc[(size_t)b].tab});
    std::vector<WalkJob> walks;
    for (int32_t q = 0; q < n_groups && !shared; ++q) {
      size_t at = 0;
      for (int32_t b = groups[(size_t)q]; b < groups[(size_t)q + 1]; ++b) {
        const BatchSrc &S = hsrc[(size_t)b];
        const QueryTab &t = tabs[(size_t)(i0 + b)];
        Filters F;
        const size_t f = std::min(ends[(size_t)b], room - at);
        plan_filters(g, t, S.w, walk_way(g, t, n, true), f, &F, ws_base + need + at);
        at += f;
        walks.push_back(walk_job(g, t, S.w, F, Outputs{S.scores, S.counts, nullptr, nullptr}));
      }
    }
    std::vector<SharedSrc> ssrc;
    for (int32_t b = 0; shared && b < kb; ++b) {
      const BatchSrc &S = hsrc[(size_t)b];
      ssrc.push_back(SharedSrc{S.wj, reinterpret_cast<unsigned long long *>(S.scores), S.counts,
                               S.z, S.s});
    }
    // tables and source descriptors, and the groups' counters at 0 (synchronous staging
    // of pageable memory; one copy per array took some 10 us more: 8 sources on 1,500
    // nodes, eps = 0.1, 0.207 ms instead of 0.192)
    std::vector<char> up(up_bytes, 0);
    memcpy(up.data() + o_src, hsrc.data(), sizeof(BatchSrc) * (size_t)kb);
    memcpy(up.data() + o_tab, tabs.data() + i0, sizeof(QueryTab) * (size_t)kb);
    memcpy(up.data() + o_jobs, jobs.data(), sizeof(SourceJob) * (size_t)kb);
    if (shared) {
      memcpy(up.data() + o_off, hoff.data(), sizeof(int64_t) * ((size_t)kb + 1));
      memcpy(up.data() + o_rowbase, rowbase.data(), r_bytes);
      memcpy(up.data() + o_ssrc, ssrc.data(), c_bytes);
    } else {
      memcpy(up.data() + o_walks, walks.data(), sizeof(WalkJob) * (size_t)kb);
    }
    if ((e = cudaMemcpyAsync(base, up.data(), up_bytes, cudaMemcpyHostToDevice, st)) !=
        cudaSuccess) {
      rc = cuda_fail(e, "batch descriptors");
      cudaFreeAsync(base, st);
      break;
    }
    BatchArgs A;
    A.src = d_src;
    A.walk_off = d_off;
    A.k = kb;
    A.total_walks = hoff[(size_t)kb];
    A.view = view_of(g);
    A.M = d_M;
    A.sig = d_sig;
    A.T = d_T;
    A.rowbase = d_rowbase;
    A.tbits = tbits;
    A.Lmax = Lmax;
    const int gw = (int)std::max<int64_t>(1, std::min<int64_t>((A.total_walks + 255) / 256,
                                                                (int64_t)sms * 8));
    auto enqueue_source_side = [&](cudaStream_t s2) {
      int r = enqueue_sources(g, d_jobs, kb, Jmax, shared, s2);
      if (shared) {
        cudaMemsetAsync(d_ctr, 0, 256, s2);
        cudaMemsetAsync(d_M, 0, m_bytes, s2);
        cudaMemsetAsync(d_sig, 0, align256(g_bytes) + h_bytes, s2);
        kb_hitj<<<gw, 256, 0, s2>>>(A);
      }
      const int gp = (int)std::min<int64_t>(((int64_t)kb * (int64_t)n + 255) / 256,
                                            (int64_t)sms * 16);
      kb_prefill<<<gp, 256, 0, s2>>>(d_src, kb, (int32_t)n);
      return r;
    };
    const bool count = opt && opt->stats;
    SharedWalks SW;
    memset(&SW, 0, sizeof SW);
    if (shared) {
      SW.mask = d_M;
      SW.sig = d_sig;
      SW.T = d_T;
      SW.rowbase = d_rowbase;
      SW.src = d_ssrc;
      SW.k = kb;
      SW.rows = Lmax + 1;
      SW.tbits = tbits;
      SW.j0 = j0;
      SW.J = Jmax;
      SW.Lmax = Lmax;
      SW.key = walk_key(seed, kSharedWalkKey);
      for (int r = 0; r < 10; ++r) SW.rk[r] = SW.key + (uint32_t)r * kPhiloxW0;
      SW.steps = count ? d_ctr + 1 : nullptr;
      SW.counter = reinterpret_cast<int32_t *>(d_ctr);
    }
    auto enqueue_all = [&](cudaStream_t s2) {
      int r = enqueue_source_side(s2);
      if (r) return r;
      if (shared) return enqueue_shared_walks(g, SW, s2);
      for (int32_t q = 0; q < n_groups && r == SRK_OK; ++q) {
        const int32_t b = groups[(size_t)q];
        r = enqueue_walk_group(g, walks.data() + b, d_walks + b, groups[(size_t)q + 1] - b, Jmax,
                               d_units + q, count, s2);
      }
      return r;
    };
    if (use_graph) {
      // The batch is captured every time (its buffers move), but the graph's
      // executable is kept in the handle and only updated with the new
      // parameters for a batch of as many sources while the launch sequence keeps
      // its shape (same kernels, same order); otherwise it is instantiated anew.
      std::lock_guard<std::mutex> lk(capture_mutex(dev));
      srk_graph *gm = const_cast<srk_graph *>(g);
      cudaGraph_t graph = nullptr;
      e = cudaEventRecord(ev_in, st);
      if (e == cudaSuccess) e = cudaStreamWaitEvent(cs, ev_in, 0);
      if (e == cudaSuccess) e = cudaStreamBeginCapture(cs, cudaStreamCaptureModeThreadLocal);
      if (e == cudaSuccess) {
        rc = enqueue_all(cs);
        e = cudaStreamEndCapture(cs, &graph);
        if (rc && e == cudaSuccess) e = cudaErrorUnknown;
      }
      if (e == cudaSuccess && gm->batch_exec) {
        cudaGraphExecUpdateResultInfo info;
        if (gm->batch_k != kb || cudaGraphExecUpdate(gm->batch_exec, graph, &info) != cudaSuccess) {
          cudaGetLastError();  // a different shape: instantiate below
          cudaGraphExecDestroy(gm->batch_exec);
          gm->batch_exec = nullptr;
        } else {
          ++total.graph_updates;
        }
      }
      if (e == cudaSuccess && !gm->batch_exec) e = cudaGraphInstantiate(&gm->batch_exec, graph, 0);
      gm->batch_k = kb;
      if (e == cudaSuccess) e = cudaGraphLaunch(gm->batch_exec, cs);
      if (e == cudaSuccess) e = cudaEventRecord(ev_out, cs);
      if (e == cudaSuccess) e = cudaStreamWaitEvent(st, ev_out, 0);
      if (e == cudaSuccess) e = cudaStreamSynchronize(cs);
      if (graph) cudaGraphDestroy(graph);
    } else {
      rc = enqueue_all(st);
      e = cudaGetLastError();
    }
    if (e == cudaSuccess) e = cudaGetLastError();
    if (e != cudaSuccess || rc) {
      if (!rc) rc = cuda_fail(e, "batched query launch");
      cudaFreeAsync(base, st);
      break;
    }
    // results of host callers
    for (int32_t b = 0; b < kb && e == cudaSuccess; ++b) {
      const BatchSrc &S = hsrc[(size_t)b];
      if (!d_scores)
        e = cudaMemcpyAsync(scores + (size_t)row_of[(size_t)(i0 + b)] * n, S.scores, 8 * n,
                            cudaMemcpyDeviceToHost, st);
      if (e == cudaSuccess && meet_counts && !d_counts)
        e = cudaMemcpyAsync(meet_counts + (size_t)row_of[(size_t)(i0 + b)] * n, S.counts, 4 * n,
                            cudaMemcpyDeviceToHost, st);
    }
    if (e == cudaSuccess && opt && opt->stats) {
      unsigned long long walked = 0;  // steps of the shared walks
      if (shared)
        e = cudaMemcpyAsync(&walked, d_ctr + 1, sizeof walked, cudaMemcpyDeviceToHost, st);
      for (int32_t b = 0; b < kb && e == cudaSuccess; ++b) {
        unsigned long long sc[2];
        int32_t act = 0;
        const Small sm = small_view(hsrc[(size_t)b].w.small);
        e = cudaMemcpyAsync(sc, sm.ctr, sizeof sc, cudaMemcpyDeviceToHost, st);
        if (e == cudaSuccess)
          e = cudaMemcpyAsync(&act, sm.cnt + 1, sizeof act, cudaMemcpyDeviceToHost, st);
        if (e == cudaSuccess) e = cudaStreamSynchronize(st);
        total.target_steps += sc[0];
        total.source_steps += sc[1];
        total.n_active_pairs += act;
        total.n_walks += tabs[(size_t)(i0 + b)].N_tot;
      }
      if (e == cudaSuccess) e = cudaStreamSynchronize(st);
      total.target_steps += walked;
      total.z = tabs[(size_t)(i1 - 1)].z;
      total.L = tabs[(size_t)(i1 - 1)].L;
    }
    cudaFreeAsync(base, st);
    if (e != cudaSuccess) rc = cuda_fail(e, "batched query results");
    i0 = i1;
  }
  if (ev_in) cudaEventDestroy(ev_in);
  if (ev_out) cudaEventDestroy(ev_out);
  if (rc == SRK_OK && (!d_scores || !d_counts)) {
    cudaError_t e = cudaStreamSynchronize(st);
    if (e != cudaSuccess) rc = cuda_fail(e, "srk_multi_source");
  }
  total.batch_shape = shared ? -1 : walk_shape(g, g->n_act);
  if (rc == SRK_OK && opt && opt->stats) *opt->stats = total;
  return rc;
}
