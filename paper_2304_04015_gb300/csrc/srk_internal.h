// Host-side internals shared by the library's translation units.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include <vector>

#include "srk.h"

struct srk_graph {
  int32_t n = 0;
  int64_t m = 0;
  int device = 0;
  const int32_t *row_ptr = nullptr;  // device, n+1
  const int32_t *col = nullptr;      // device, m
  const float *edge_w = nullptr;     // device, m or null
  // Packed adjacency (owned).  Layout 0 (narrow): the lists of m words, by
  // rank; node v's identity inside the walk kernels is its rank npos[v] in
  // the order of build_narrow: in-degree code descending, nodes of one code by
  // how often walks visit them.  The code of degree d is min(d, deg_max); entry
  // k of v's list holds the k-th in-neighbour y as (code(y) << pos_bits) |
  // npos[y].  The d words of a node of degree d < deg_max and rank x begin at
  // ctab[d] + x d (mod 2^32), since the nodes of one degree follow one another
  // in rank and in memory; a hub (degree deg_max or more; they come first)
  // has {degree, first word} in hub[x].  So a walk step learns the next node's
  // degree and list from the entry it reads and a table of deg_max + 1 words.
  // Wide layout (layout = 1, chosen when n + m needs more than 28 bits or
  // forced by SRK_ADJ_WIDE): 2 (n + m) words forming 8-byte entries at
  // positions v + row_ptr[v], adj[pos(v)] = {0, |I(v)|} and entries
  // {pos(y), |I(y)|}, so a step never reads a header.  CSR layout (layout =
  // 2, only when forced by SRK_ADJ_CSR): no packed copy; nodes are their ids
  // and a step reads row_ptr and col.
  uint32_t *adj = nullptr;
  int32_t *npos = nullptr;   // narrow layout (in adj's block): ranks, n,
  int32_t *order = nullptr;  //   the nodes by rank, n,
  uint2 *hub = nullptr;      //   hub records, n_hubs,
  uint32_t *ctab = nullptr;  //   and list starts by degree
  int32_t n_hubs = 0;        // narrow layout: H
  int32_t pos_bits = 1;      // narrow layout: ranks < 2^pos_bits
  uint32_t deg_max = 1;      // narrow layout: largest degree code
  int layout = 0;        // 0 narrow, 1 wide, 2 CSR (no packed adjacency; walks read row_ptr/col)
  // Nodes with at least one in-neighbour, ascending (owned): the only targets
  // whose score can be nonzero.
  int32_t *act = nullptr;
  int32_t n_act = 0;
  int32_t *out_deg = nullptr;  // out-degrees by id, n (in act's block)
  // Executable of the last captured batch (srk_multi_source with a CUDA
  // graph), of batch_k sources, updated in place for the next batch of as many.
  cudaGraphExec_t batch_exec = nullptr;
  int32_t batch_k = 0;
  // Topology of the linearised form (edge owners, a transpose, list size
  // classes), built by the first srk_linear_fwd on the graph.
  struct srk_lin_topo *lin = nullptr;
  int32_t *own_row_ptr = nullptr;    // owned copies (null when borrowed)
  int32_t *own_col = nullptr;
  float *own_w = nullptr;
};

// A graph as the kernels see it (passed by value).
struct GraphView {
  const int32_t *row_ptr;  // CSR offsets
  const int32_t *col;      // in-neighbour lists
  const uint32_t *adj;     // packed adjacency
  const int32_t *npos;     // narrow layout: ranks,
  const int32_t *order;    //   nodes by rank,
  const uint2 *hub;        //   hub records,
  const uint32_t *ctab;    //   list starts by degree
  int32_t pos_bits;
  uint32_t deg_max;
  int32_t n, n_hubs, layout;
  int32_t far;  // the adjacency does not fit the L2
};

namespace srk {

// Bytes of the adjacency that the walks read.
inline int64_t adj_bytes(const srk_graph *g) {
  return g->layout == 1 ? 8 * ((int64_t)g->n + g->m) : 4 * ((int64_t)(g->layout == 2 ? g->n : 0) + g->m);
}
// Adjacencies of more than this do not fit the L2 (129 MB in all, of which the
// walks' other data has a part; between 72 and 143 MB nothing was measured).
constexpr int64_t kNearBytes = 96ll << 20;

inline GraphView view_of(const srk_graph *g) {
  return GraphView{g->row_ptr, g->col,    g->adj,      g->npos,
                   g->order,   g->hub,    g->ctab,     g->pos_bits,
                   g->deg_max, g->n,      g->n_hubs,   g->layout,
                   adj_bytes(g) > kNearBytes ? 1 : 0};
}

// The output function of SplitMix64 (Steele, Lea, Flood, OOPSLA 2014) and
// the 32-bit finalizer "lowbias32" (C. Wellons, 2018); both are bijections.
__host__ __device__ __forceinline__ uint64_t mix64(uint64_t z) {
  z ^= z >> 30;
  z *= 0xBF58476D1CE4E5B9ull;
  z ^= z >> 27;
  z *= 0x94D049BB133111EBull;
  z ^= z >> 31;
  return z;
}
__host__ __device__ __forceinline__ uint32_t h32(uint32_t x) {
  x ^= x >> 16;
  x *= 0x7FEB352Du;
  x ^= x >> 15;
  x *= 0x846CA68Bu;
  x ^= x >> 16;
  return x;
}

// Key word of the shared target walks (SRK_OPT_SHARED_WALKS) in place of a
// source (sources are below 2^31, so it names none).
constexpr uint32_t kSharedWalkKey = 0xFFFFFFFEu;

// The 32-bit Philox2x32-10 key of a query's walks: h32(q ^ low half of
// mix64(seed)), q the source (its source walks, and its target walks by
// default) or kSharedWalkKey (the shared target walks).  Injective in q for a
// given seed, since h32 is a bijection.
__host__ __device__ __forceinline__ uint32_t walk_key(uint64_t seed, uint32_t q) {
  return h32(q ^ (uint32_t)mix64(seed));
}

// Sample-count table of one query (Algorithm 1 lines 3-5, Algorithm 2 line 2,
// Lemma 7).  Passed by value as a kernel parameter (stays below 4 KB).
struct QueryTab {
  int32_t s, n, L, N_tot;
  uint32_t key0, key1;  // the seed's halves (Fisher-Yates draws, literal shuffle)
  uint32_t skey, tkey;  // walk keys of the source walks and of the target walks
  int32_t literal;  // 1: literal target shuffle (SRK_OPT_LITERAL_SHUFFLE)
  int32_t shared;   // 1: shared target walks (SRK_OPT_SHARED_WALKS)
  double z;
  int32_t P[SRK_MAX_LEN + 2];  // stratum prefix: walk r has length l iff P[l] <= r < P[l+1]
  double a[SRK_MAX_LEN + 1];   // rounding weight a(l) = |Z_l| / |Z^_l|
};
static_assert(sizeof(QueryTab) <= 4096, "kernel parameter too large");

// Fills `t`; returns SRK_OK or SRK_EINVAL (message set).
int build_table(int32_t n, int32_t s, double c, double eps, uint64_t seed,
                const srk_opts *opt, QueryTab *t);

// Sets the thread's last-error message (printf-style) and returns `code`.
int fail(int code, const char *fmt, ...);
// Maps a CUDA error to SRK_ECUDA / SRK_ENOMEM with a message.
int cuda_fail(cudaError_t e, const char *what);
void clear_error();

// Library-owned stream-ordered pool of the given device.
cudaMemPool_t pool(int device);
// True when p is device or managed memory visible to the current device.
bool is_device_ptr(const void *p);

// RAII guard that makes `dev` current and restores the previous device.
struct DeviceGuard {
  int prev = -1;
  explicit DeviceGuard(int dev) {
    if (cudaGetDevice(&prev) != cudaSuccess) prev = -1;
    if (prev != dev) cudaSetDevice(dev);
  }
  ~DeviceGuard() {
    int cur = -1;
    if (prev >= 0 && cudaGetDevice(&cur) == cudaSuccess && cur != prev)
      cudaSetDevice(prev);
  }
};

// SM count of the current device (cached per device).
int sm_count(int device);

// Scratch of one query, carved from one device block (srk_query.cu).
struct Workspace {
  // the shuffle's draws, and its lists of steps by draw, are in the room of the pair
  // records, which are made after it
  int32_t *spos, *seff, *kdraw, *head, *next, *items, *first, *succ, *sigma, *pair_j, *Hc, *small;
  unsigned long long *pair_w;
  size_t bytes;
  // the pair records {j, cap, first node in Hc, filter}, longest pairs first
  __host__ __device__ int4 *rec() const { return reinterpret_cast<int4 *>(kdraw); }
};

// Device outputs of one query (null = not wanted, except scores).
struct Outputs {
  double *scores;
  uint32_t *counts;
  unsigned long long *wsums;
  uint32_t *steps;
};

// A slot of the table of end nodes: the node id + 1 (0: empty slot), its
// filter + 1 (0: none; kWantFilter: some pair ends here), and the pairs of cap
// 1 that end here, list1[off1 .. off1 + cnt1).
struct EndSlot {
  uint32_t key;
  int32_t filt;
  int32_t cnt1;
  int32_t off1;
};
constexpr int32_t kWantFilter = -1;
// End nodes and filters of one query (srk_lockstep.cu; null slots: it has none).
struct Filters {
  EndSlot *slots;       // 2^slot_bits of them, linear probing
  uint32_t *bloom;      // 2^bloom_bits bits: ids whose bit is clear are in no slot
  uint32_t *bits;       // the filters, max_units * kFilterUnit words
  int32_t *list1;       // pairs of cap 1, grouped by end node
  int32_t *slot_of;     // per pair: its slot,
  int32_t *rank1;       //   and its place in the slot's list
  int32_t *ctl;         // {units of bits handed out, entries of list1 handed out}
  const int32_t *out_deg;  // out-degrees, by node id
  int slot_bits, bloom_bits;
  int32_t max_units;
};
// How the targets of a query are walked: in lockstep with end filters or without
// (srk_lockstep.cu), or by a warp each (k_target_walks, srk_query.cu).  `batch`: a
// source of a batch, over all targets (never by warps).
enum class WalkWay { kFilters, kPlain, kWarps };
WalkWay walk_way(const srk_graph *g, const QueryTab &t, int64_t n_targets, bool batch);
// The query's end nodes and filters in `avail` bytes at `extra` (0 bytes or a
// null pointer: none), where its way is kFilters; returns the bytes taken.
size_t plan_filters(const srk_graph *g, const QueryTab &t, const Workspace &w, WalkWay way,
                    size_t avail, Filters *F, char *extra);

// The source side of queries (srk_source.cu).  enqueue_source: one query, steps
// a2-a3 to the pair records (with `rows` to the cap rows only) and the end nodes of
// F.  enqueue_sources: of k queries, to the pair records or,
// with `shared`, to sigma.  enqueue_ends: the end nodes of k of them.  N: the most
// walks that one of the k has.
struct SourceJob {
  Workspace w;
  const QueryTab *tab;  // device
};
int enqueue_source(const srk_graph *g, const QueryTab &t, const Workspace &w, const Filters &F,
                   bool rows, int32_t u_begin, int32_t u_end, cudaStream_t st);
int enqueue_sources(const srk_graph *g, const SourceJob *jobs, int32_t k, int32_t N, bool shared,
                    cudaStream_t st);
struct WalkJob;
int enqueue_ends(const srk_graph *g, const WalkJob *jobs, int32_t k, int32_t N, cudaStream_t st);

// Carves `base` (or only sizes the plan when base is null); returns the
// number of bytes one query of table `t` needs.
size_t plan(const QueryTab &t, Workspace *w, char *base);
// Enqueues steps a2-a5 on `st`; `timing` (may be null) gets two events
// recorded around the target-walk kernel; `extra`: scratch for the end filters
// (see filter_bytes); `count`: step totals are wanted.
int enqueue_query(const srk_graph *g, const QueryTab &t, const Workspace &w,
                  const Outputs &o, char *extra, size_t extra_bytes, bool count, cudaStream_t st,
                  const cudaEvent_t *timing, int32_t u_begin, int32_t u_end);
// srk_single_source with at most extra_limit bytes for the end filters.
int single_source(const srk_graph *g, int32_t s, double c, double eps, uint64_t seed,
                  const srk_opts *opt, double *scores, uint32_t *meet_counts,
                  uint64_t *weight_sums, void *cuda_stream, size_t extra_limit);
// Bytes of `extra` scratch a query makes use of (it does
// with less, or none: its end nodes then have fewer filters, or none).
size_t filter_bytes(const srk_graph *g, const QueryTab &t, WalkWay way);
// What the target walks of a query need (srk_lockstep.cu).
struct LockQuery {
  const int4 *rec;              // per pair {j, cap, first node in H, filter}
  const unsigned long long *w;  // per pair: its quantised weight
  const int32_t *H;             // nodes of the pairs' source walks, steps 1..cap
  const uint32_t *bits;         // the filters
  const int32_t *cnt;           // cnt[i]: pairs with cap >= i (longest first)
  unsigned long long *W;        // per target: weight sum
  uint32_t *counts;             // per target: meetings, or null
  uint32_t *steps;              // per target: steps, or null
  unsigned long long *steps_total;
  uint32_t key;                 // walk key of the target walks
  uint32_t rk[10];              //   and its round keys
  int32_t s;
  int32_t min_cap;              // pairs below this cap are not walked here
  int32_t polls;                // of a wait for filters before it gives up
};
// Steps a4-a5 after the source side (the pair records of w and the end nodes
// of F are made, the outputs of the range cleared): srk_lockstep.cu.
int enqueue_walks(const srk_graph *g, const QueryTab &t, const Workspace &w, const Filters &F,
                  const Outputs &o, bool count, cudaStream_t st,
                  const cudaEvent_t *timing, int32_t u_begin, int32_t u_end);
// The same, and the end nodes before it, for a group of queries over all targets
// (at most kWalkGroup, their pair records made and their rows prefilled): `jobs` on
// the device, `host` their copy, N the most walks of one of them, `counter` a device
// word that is zero.
struct WalkJob {
  Workspace w;
  Filters F;
  LockQuery Q;
  double z;
  int32_t alone;  // its targets are walked by a launch of their own
};
constexpr int32_t kWalkGroup = 256;
WalkJob walk_job(const srk_graph *g, const QueryTab &t, const Workspace &w, const Filters &F,
                 const Outputs &o);
int enqueue_walk_group(const srk_graph *g, const WalkJob *host, const WalkJob *jobs, int32_t k,
                       int32_t N, int32_t *counter, bool count, cudaStream_t st);
// Launch shape of the walks of n_targets targets: 0, several a thread, or 1, one.
int walk_shape(const srk_graph *g, int64_t n_targets);
// Shared target walks of up to 64 sources (srk_batch.cu makes the tables).
struct SharedSrc {
  const unsigned long long *wj;  // quantised Lemma 7 weight of pair j
  unsigned long long *W;         // per target: weight sum (in the score row)
  uint32_t *counts;              // per target: meetings, or null
  double z;
  int32_t s;
};
struct SharedWalks {
  const uint2 *mask;       // [j rows + i - 1]: sources whose pair j may meet at step i
  const uint32_t *sig;     // per meeting table: 1024 bits, one for each node of it
  const uint4 *T;          // the meeting tables (BatchArgs in srk_batch.cu)
  const int64_t *rowbase;  // table of (step i, pair j): rowbase[i] + j
  const SharedSrc *src;
  int32_t k, rows, tbits, j0, J, Lmax;
  uint32_t key, rk[10];
  unsigned long long *steps;  // null: not counted
  int32_t *counter;           // units handed out (zero at the start)
};
int enqueue_shared_walks(const srk_graph *g, const SharedWalks &Q, cudaStream_t st);
// The bit of a node in a signature, the first slot in a table of 2^tbits slots.
__host__ __device__ __forceinline__ uint32_t sig_bit(int32_t x) {
  return ((uint32_t)x * 0x9E3779B9u) >> 22;
}
__host__ __device__ __forceinline__ uint32_t slot_of(int32_t x, int tbits) {
  return ((uint32_t)x * 0x85EBCA6Bu) >> (32 - tbits);
}
// Shared-memory opt-in of the walk kernels of a layout, in this context.
cudaError_t allow_lockstep(int layout);
// [*b, *e): the targets a query computes, from its options (SRK_EINVAL when
// the range is malformed).
int target_range(const srk_graph *g, const srk_opts *opt, int32_t *b, int32_t *e);
// Exclusive scan of cnt[0..N) into off[0..N], with scan_scratch(N) bytes of
// scratch (srk_sort.cu).
size_t scan_scratch(int64_t N);
void scan_i32(const int32_t *cnt, int32_t *off, int64_t N, int32_t *tmp, cudaStream_t st);
// Stable sort of m pairs (key, value) by the keys' low `bits` bits, with
// sort_scratch(m) bytes of scratch; returns true when the result is in kB, vB.
size_t sort_scratch(int64_t m);
bool radix_sort(int32_t *kA, int32_t *vA, int32_t *kB, int32_t *vB, int64_t m, int bits,
                int32_t *tmp, cudaStream_t st);

// In-degrees of k sources (ids already checked against n), read from the
// device CSR on stream st (synchronises st).  SRK_OK or an error code.
int source_in_degrees(const srk_graph *g, const int32_t *sources, int32_t k, cudaStream_t st,
                      std::vector<int32_t> *deg);

// Releases the graph's linear topology, if built (srk_linear.cu).
void free_lin_topo(srk_graph *g);

// Copies the query counters into `stats` (synchronises `st`).
int read_stats(const QueryTab &t, const Workspace &w, cudaStream_t st,
               srk_stats *stats, bool accumulate);

}  // namespace srk
