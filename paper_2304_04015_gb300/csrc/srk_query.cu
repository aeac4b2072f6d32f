// Single- and multi-source queries: the sqrt(c)-walk Monte Carlo estimator of
// arXiv 2304.04015 as kernel phases on one stream.
//
//   a2-a3 enqueue_source (srk_source.cu) the source's walks, their shuffle and
//                        the walk pairs, sorted by step cap (descending)
//   a4-a5 enqueue_walks  (srk_lockstep.cu) the targets' walks
//       k_target_walks   the same by a warp per target, with the literal target
//                        shuffle and where that is faster (walk_way), on a
//                        step-major hit table (k_hit_table): row i holds, for
//                        every pair that can still meet at step i, the source
//                        walk's node at step i
#include <stdint.h>
#include <string.h>

#include <algorithm>

#include "srk_device.cuh"
#include "srk_internal.h"

namespace srk {

// Places every pair with cap >= 1 in its cap group and fills its column of the
// hit table with the source walk's nodes at steps 1..cap.  The pair's Lemma 7
// weight is round(a(l1) a(l2) 2^32) with l1 the source walk's length.
__global__ void __launch_bounds__(256)
k_hit_table(const __grid_constant__ QueryTab tab, GraphView V, const int32_t *__restrict__ sigma,
            const int32_t *__restrict__ seff, const int32_t *__restrict__ spos,
            int32_t *__restrict__ small_base, int32_t *__restrict__ pair_j,
            unsigned long long *__restrict__ pair_w, int32_t *__restrict__ Hc) {
  __shared__ int32_t P[SRK_MAX_LEN + 2];
  __shared__ int32_t R[SRK_MAX_LEN + 2];
  Small sm = small_view(small_base);
  for (int i = threadIdx.x; i <= tab.L + 1; i += blockDim.x) {
    P[i] = tab.P[i];
    R[i] = sm.R[i];
  }
  __syncthreads();
  const int Ls = tab.L > 0 ? tab.L : 1;
  for (int32_t j = blockIdx.x * blockDim.x + threadIdx.x; j < tab.N_tot;
       j += gridDim.x * blockDim.x) {
    const int32_t w = sigma[j];
    const int l2 = stratum_of(P, tab.L, j);
    const int32_t cap = tab.literal ? seff[w] : min(l2, seff[w]);
    if (cap < 1) continue;
    const int l1 = stratum_of(P, tab.L, w);
    const int32_t a = atomicAdd(&sm.cursor[cap], 1);
    pair_j[a] = j;
    // literal mode keeps l1: the weight needs the target walk's length
    pair_w[a] = tab.literal ? (unsigned long long)l1
                            : __double2ull_rn(tab.a[l1] * tab.a[l2] * 4294967296.0);
    const int32_t *src = spos + (int64_t)w * Ls;
    for (int i = 1; i <= cap; ++i) Hc[R[i] + a] = walk_identity(V, src[i - 1]);
  }
}

// -------------------------------------- steps a4-a5 by a warp per target --
// Each warp takes targets u from a global counter.  Its 32 lanes walk the
// target's pairs a = 0, 1, ... of the cap-sorted list; a lane whose walk ends
// takes the next unassigned pair at once (lane refill), so walks that end
// early (cap, meeting, no in-neighbours) do not idle the warp.  (With the literal
// shuffle pairs differ from target to target, so the lockstep form has nothing to
// share.)
// Walks run on the packed adjacency.  Pair a (original index
// j) walks from u: one Philox2x32-10 block, counter (((i-1)>>1) << 24 | j, u)
// under the target walks' key, serves the odd step i (word 0) and the even
// step i+1 (word 1).  A step moves to I(x)[k], k the bounded draw below |I(x)|
// (step_entry); the walk meets when its node equals row i of
// the hit table, ends after cap steps (a >= cnt[i+1]) or at a node without
// in-neighbours.  The first meeting adds 1 to the count and the pair's weight
// to W_u.  The warp then reduces and writes count, W and s~(s,u) = W 2^-32 / z
// (s~(s,s) = 1).
struct TargetArgs {
  GraphView view;
  int32_t s, L;
  uint32_t walk_key;       // walk key of the target walks (the source's or the shared one)
  uint32_t key0, key1;
  double z;
  const int32_t *small_base;
  const int32_t *pair_j;
  const unsigned long long *pair_w;
  const int32_t *Hc;
  double *scores;
  uint32_t *counts;
  unsigned long long *wsums;
  uint32_t *steps_per_target;
  unsigned long long *steps_total;
  int32_t *target_counter;  // next index into act (from act_lo), then act_hi
  const int32_t *act;       // the targets with in-neighbours, ascending
  int32_t u_begin, u_end;   // targets computed: [u_begin, u_end)
  int32_t N_tot;            // the permutation's domain
};

// The stratum prefix and the Lemma 7 weights.
struct LiteralArgs {
  int32_t P[SRK_MAX_LEN + 2];
  double a[SRK_MAX_LEN + 1];
};

// 8 blocks of 256 threads per SM (32 registers): the kernel is bound by the
// rate of scattered L1 misses, and full occupancy keeps the most misses in
// flight.
template <int kLayout, bool kLiteral>
__global__ void __launch_bounds__(256, 8)
k_target_walks(const __grid_constant__ TargetArgs A, const __grid_constant__ LiteralArgs X) {
  __shared__ int2 rc[SRK_MAX_LEN + 3];  // {R[i], cnt[i+1]}, one load per step
  __shared__ int32_t Psh[kLiteral ? SRK_MAX_LEN + 2 : 1];
  {
    const Small sm = small_view(const_cast<int32_t *>(A.small_base));
    for (int i = threadIdx.x; i <= A.L + 2; i += blockDim.x) {
      rc[i] = make_int2((i <= A.L + 1) ? sm.R[i] : 0,
                        (i + 1 <= A.L + 1) ? sm.cnt[i + 1] : 0);  // cnt[L+1] = cnt[L+2] = 0
      if (kLiteral && i <= A.L + 1) Psh[i] = X.P[i];
    }
  }
  __syncthreads();
  const int lane = threadIdx.x & 31;
  const uint32_t lanes_below = (1u << lane) - 1u;
  const auto G = adj_view<kLayout>(A.view);
  PairSet S;
  S.rc = rc;
  S.pair_j = A.pair_j;
  S.pair_w = A.pair_w;
  S.Hc = A.Hc;
  S.n_pairs = rc[0].y;  // cnt[1]
  S.key = A.walk_key;
  FeistelShape fs;
  if constexpr (kLiteral)
    fs = feistel_shape(A.N_tot, ((uint64_t)A.key1 << 32) | A.key0, (uint32_t)A.s);
  unsigned long long warp_steps = 0;
  // the active targets act[counter .. act_hi) (the source side set the counter to
  // the range's first index and act_hi beside it); the outputs of the others
  // were cleared before the launch, and s's score is 1
  if (blockIdx.x == 0 && threadIdx.x == 0 && A.s >= A.u_begin && A.s < A.u_end)
    A.scores[A.s] = 1.0;
  if (S.n_pairs == 0) return;  // no pair can meet: every output is zero
  for (;;) {
    int32_t u = -1;
    if (lane == 0) {
      const int32_t q = atomicAdd(A.target_counter, 1);
      if (q < A.target_counter[1]) u = A.act[q];
    }
    u = __shfl_sync(0xffffffffu, u, 0);
    if (u < 0) break;
    uint32_t c = 0, st = 0;
    unsigned long long W = 0;
    uint32_t deg_u = 0;
    const int32_t b_u = node_start(G, A.view.row_ptr, u, deg_u);
    if (u != A.s && deg_u > 0) {
      if constexpr (kLiteral)
        walk_target_literal(G, S, fs, Psh, A.L, X.a, (uint32_t)u, b_u, deg_u, lanes_below, c, W,
                            st);
      else
        walk_target(G, S, (uint32_t)u, b_u, deg_u, c, W, st);
    }
    for (int off = 16; off > 0; off >>= 1) {
      c += __shfl_xor_sync(0xffffffffu, c, off);
      st += __shfl_xor_sync(0xffffffffu, st, off);
      W += __shfl_xor_sync(0xffffffffu, W, off);
    }
    if (lane == 0) {
      A.scores[u] = (u == A.s) ? 1.0 : (double)W * 2.3283064365386963e-10 / A.z;
      if (A.counts) A.counts[u] = c;
      if (A.wsums) A.wsums[u] = W;
      if (A.steps_per_target) A.steps_per_target[u] = st;
      warp_steps += st;
    }
  }
  if (lane == 0 && warp_steps) atomicAdd(A.steps_total, warp_steps);
}

// ------------------------------------------------------------ host side --

static size_t align_up(size_t x) { return (x + 255) & ~(size_t)255; }

size_t plan(const QueryTab &t, Workspace *w, char *base) {
  const size_t N = (size_t)t.N_tot;
  const size_t Ls = (size_t)(t.L > 0 ? t.L : 1);
  size_t hc = 0;
  for (int l = 1; l <= t.L; ++l) hc += (size_t)l * (size_t)(t.P[l + 1] - t.P[l]);
  if (hc == 0) hc = 1;
  size_t off = 0;
  auto take = [&](size_t bytes) {
    char *p = base ? base + off : nullptr;
    off += align_up(bytes);
    return p;
  };
  w->spos = (int32_t *)take(4 * N * Ls);
  w->seff = (int32_t *)take(4 * N);
  w->kdraw = (int32_t *)take(sizeof(int4) * N);  // the pair records
  w->head = w->kdraw + N;
  w->next = w->kdraw + 2 * N;
  w->items = (int32_t *)take(4 * N);
  w->first = (int32_t *)take(4 * N);
  w->succ = (int32_t *)take(4 * N);
  w->sigma = (int32_t *)take(4 * N);
  w->pair_j = (int32_t *)take(4 * N);
  w->pair_w = (unsigned long long *)take(8 * N);
  w->Hc = (int32_t *)take(4 * hc);
  w->small = (int32_t *)take(kSmallBytes);
  w->bytes = off;
  return off;
}

static int grid_for(int64_t work, int threads, int device) {
  const int64_t want = (work + threads - 1) / threads;
  const int64_t cap = (int64_t)sm_count(device) * 8;
  return (int)std::max<int64_t>(1, std::min<int64_t>(want, cap));
}

static int target_grid(int device) {
  static int blocks_per_sm[64] = {};
  int b = (device >= 0 && device < 64) ? blocks_per_sm[device] : 0;
  if (!b) {
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, k_target_walks<kNarrow, false>, 256, 0) !=
            cudaSuccess || b < 1)
      b = 1;
    if (device >= 0 && device < 64) blocks_per_sm[device] = b;
  }
  return sm_count(device) * b;
}

// Enqueues one query on `st` with device-resident outputs `o`.  Workspace
// `w` (already carved) must hold plan(t) bytes.
int enqueue_query(const srk_graph *g, const QueryTab &t, const Workspace &w,
                  const Outputs &o, char *extra, size_t extra_bytes, bool count, cudaStream_t st,
                  const cudaEvent_t *timing, int32_t u_begin, int32_t u_end) {
  const int dev = g->device;
  cudaError_t e = cudaSuccess;
  Filters F;
  const WalkWay way = walk_way(g, t, (int64_t)u_end - u_begin, false);
  const bool warps = t.literal || way == WalkWay::kWarps;
  plan_filters(g, t, w, way, extra ? extra_bytes : 0, &F, extra);
  const int rc = enqueue_source(g, t, w, F, warps, u_begin, u_end, st);
  if (rc) return rc;
  // targets without in-neighbours have zero outputs (and s, if it is one of
  // them, the score 1): clear the range, then walk only the active targets
  const size_t nr = (size_t)(u_end - u_begin);
  if (nr > 0) {
    e = cudaMemsetAsync(o.scores + u_begin, 0, sizeof(double) * nr, st);
    if (e == cudaSuccess && o.counts)
      e = cudaMemsetAsync(o.counts + u_begin, 0, sizeof(uint32_t) * nr, st);
    if (e == cudaSuccess && o.wsums && warps)
      e = cudaMemsetAsync(o.wsums + u_begin, 0, sizeof(unsigned long long) * nr, st);
    if (e == cudaSuccess && o.steps)
      e = cudaMemsetAsync(o.steps + u_begin, 0, sizeof(uint32_t) * nr, st);
    if (e != cudaSuccess) return cuda_fail(e, "clearing the outputs of the target range");
  }
  if (warps) {
    const GraphView V = view_of(g);
    k_hit_table<<<grid_for(t.N_tot, 256, dev), 256, 0, st>>>(t, V, w.sigma, w.seff, w.spos, w.small, w.pair_j, w.pair_w,
                                    w.Hc);
    TargetArgs A;
    A.view = V;
    A.s = t.s;
    A.walk_key = t.tkey;
    A.L = t.L;
    A.key0 = t.key0;
    A.key1 = t.key1;
    A.z = t.z;
    A.small_base = w.small;
    A.pair_j = w.pair_j;
    A.pair_w = w.pair_w;
    A.Hc = w.Hc;
    A.scores = o.scores;
    A.counts = o.counts;
    A.wsums = o.wsums;
    A.steps_per_target = o.steps;
    A.steps_total = small_view(w.small).ctr;
    A.target_counter = reinterpret_cast<int32_t *>(small_view(w.small).ctr + 2);
    A.act = g->act;
    A.u_begin = u_begin;
    A.u_end = u_end;
    A.N_tot = t.N_tot;
    LiteralArgs X;
    memcpy(X.P, t.P, sizeof X.P);
    memcpy(X.a, t.a, sizeof X.a);
    if (timing) cudaEventRecord(timing[0], st);
    const int tg = target_grid(dev);
    if (g->layout == kWide) {
      if (t.literal) k_target_walks<kWide, true><<<tg, 256, 0, st>>>(A, X);
      else k_target_walks<kWide, false><<<tg, 256, 0, st>>>(A, X);
    } else if (g->layout == kCsr) {
      if (t.literal) k_target_walks<kCsr, true><<<tg, 256, 0, st>>>(A, X);
      else k_target_walks<kCsr, false><<<tg, 256, 0, st>>>(A, X);
    } else {
      if (t.literal) k_target_walks<kNarrow, true><<<tg, 256, 0, st>>>(A, X);
      else k_target_walks<kNarrow, false><<<tg, 256, 0, st>>>(A, X);
    }
    if (timing) cudaEventRecord(timing[1], st);
    e = cudaGetLastError();
    return e == cudaSuccess ? SRK_OK : cuda_fail(e, "kernel launch");
  }
  return enqueue_walks(g, t, w, F, o, count, st, timing, u_begin, u_end);
}

// The target range of a query from its options: [0, n) by default.
int target_range(const srk_graph *g, const srk_opts *opt, int32_t *b, int32_t *e) {
  *b = 0;
  *e = g->n;
  if (opt && (opt->target_begin != 0 || opt->target_end != 0)) {
    if (opt->target_begin < 0 || opt->target_begin > opt->target_end ||
        opt->target_end > g->n)
      return fail(SRK_EINVAL, "target range [%d, %d) outside [0, %d]", opt->target_begin,
                  opt->target_end, g->n);
    *b = opt->target_begin;
    *e = opt->target_end;
  }
  return SRK_OK;
}

// Reads back the counters of the small block into `stats` (synchronous).
int read_stats(const QueryTab &t, const Workspace &w, cudaStream_t st,
               srk_stats *stats, bool accumulate) {
  unsigned long long ctr[2] = {0, 0};
  int32_t active = 0;
  cudaError_t e = cudaMemcpyAsync(ctr, small_view(w.small).ctr, sizeof ctr,
                                  cudaMemcpyDeviceToHost, st);
  if (e == cudaSuccess)
    e = cudaMemcpyAsync(&active, small_view(w.small).cnt + 1, sizeof active,
                        cudaMemcpyDeviceToHost, st);
  if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  if (e != cudaSuccess) return cuda_fail(e, "reading query statistics");
  if (!accumulate) {
    memset(stats, 0, sizeof *stats);
    stats->batch_shape = -1;
  }
  stats->z = t.z;
  stats->L = t.L;
  stats->n_walks = t.N_tot;
  stats->n_active_pairs += active;
  stats->target_steps += ctr[0];
  stats->source_steps += ctr[1];
  return SRK_OK;
}

}  // namespace srk

using namespace srk;

extern "C" int srk_single_source(const srk_graph *g, int32_t s, double c,
                                 double eps, uint64_t seed, const srk_opts *opt,
                                 double *scores, uint32_t *meet_counts,
                                 uint64_t *weight_sums, void *cuda_stream) {
  return single_source(g, s, c, eps, seed, opt, scores, meet_counts, weight_sums, cuda_stream,
                       SIZE_MAX);
}

int srk::single_source(const srk_graph *g, int32_t s, double c, double eps, uint64_t seed,
                       const srk_opts *opt, double *scores, uint32_t *meet_counts,
                       uint64_t *weight_sums, void *cuda_stream, size_t extra_limit) {
  clear_error();
  if (!g) return fail(SRK_EINVAL, "null graph");
  if (!scores) return fail(SRK_EINVAL, "scores is null");
  if (opt && (opt->flags & ~(SRK_OPT_WARMUP_RULE | SRK_OPT_LITERAL_SHUFFLE |
                             SRK_OPT_SHARED_WALKS)))
    return fail(SRK_EINVAL, "unsupported opts.flags 0x%x", opt->flags);
  QueryTab t;
  int rc = build_table(g->n, s, c, eps, seed, opt, &t);
  if (rc) return rc;
  int32_t u_begin = 0, u_end = g->n;
  rc = target_range(g, opt, &u_begin, &u_end);
  if (rc) return rc;
  DeviceGuard guard(g->device);
  cudaStream_t st = (cudaStream_t)cuda_stream;
  const size_t n = (size_t)g->n;
  uint32_t *step_counts = opt ? opt->step_counts : nullptr;
  const bool d_scores = is_device_ptr(scores);
  const bool d_counts = !meet_counts || is_device_ptr(meet_counts);
  const bool d_wsums = !weight_sums || is_device_ptr(weight_sums);
  const bool d_steps = !step_counts || is_device_ptr(step_counts);
  Workspace w;
  size_t ws = plan(t, &w, nullptr);
  const size_t o_scores = ws;
  if (!d_scores) ws += align_up(8 * n);
  const size_t o_counts = ws;
  if (!d_counts) ws += align_up(4 * n);
  const size_t o_wsums = ws;
  if (!d_wsums) ws += align_up(8 * n);
  const size_t o_steps = ws;
  if (!d_steps) ws += align_up(4 * n);
  cudaMemPool_t mp = pool(g->device);
  if (!mp) return fail(SRK_ECUDA, "cannot create the device memory pool");
  const size_t o_extra = ws;
  size_t extra =
      std::min(extra_limit, filter_bytes(g, t, walk_way(g, t, (int64_t)u_end - u_begin, false)));
  char *base = nullptr;
  cudaError_t e = cudaMallocFromPoolAsync((void **)&base, ws + extra, mp, st);
  if (e == cudaErrorMemoryAllocation && extra > 0) {  // the query can do without filters
    cudaGetLastError();
    extra = 0;
    e = cudaMallocFromPoolAsync((void **)&base, ws, mp, st);
  }
  if (e != cudaSuccess) return cuda_fail(e, "workspace allocation");
  plan(t, &w, base);
  Outputs o;
  o.scores = d_scores ? scores : (double *)(base + o_scores);
  o.counts = d_counts ? meet_counts : (uint32_t *)(base + o_counts);
  o.wsums = d_wsums ? (unsigned long long *)weight_sums
                    : (unsigned long long *)(base + o_wsums);
  o.steps = d_steps ? step_counts : (uint32_t *)(base + o_steps);
  rc = enqueue_query(g, t, w, o, base + o_extra, extra, o.steps || (opt && opt->stats), st,
                     opt ? (const cudaEvent_t *)opt->timing_events : nullptr, u_begin, u_end);
  bool host_out = !d_scores || !d_counts || !d_wsums || !d_steps;
  if (!rc) {  // host outputs: copy back the computed range only
    const size_t b = (size_t)u_begin, cnt = (size_t)(u_end - u_begin);
    if (!d_scores)
      e = cudaMemcpyAsync(scores + b, o.scores + b, 8 * cnt, cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess && !d_counts)
      e = cudaMemcpyAsync(meet_counts + b, o.counts + b, 4 * cnt, cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess && !d_wsums)
      e = cudaMemcpyAsync(weight_sums + b, o.wsums + b, 8 * cnt, cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess && !d_steps)
      e = cudaMemcpyAsync(step_counts + b, o.steps + b, 4 * cnt, cudaMemcpyDeviceToHost, st);
    if (e != cudaSuccess) rc = cuda_fail(e, "copying results to the host");
  }
  if (!rc && opt && opt->stats) rc = read_stats(t, w, st, opt->stats, false);
  cudaFreeAsync(base, st);
  if (!rc && host_out) {
    e = cudaStreamSynchronize(st);
    if (e != cudaSuccess) rc = cuda_fail(e, "srk_single_source");
  }
  return rc;
}
