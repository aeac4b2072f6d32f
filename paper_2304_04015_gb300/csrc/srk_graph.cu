// Graph residency, error reporting, memory pools and the sample-count table.
#include <math.h>
#include <stdarg.h>
#include <stdio.h>
#include <string.h>

#include <algorithm>
#include <mutex>
#include <string>
#include <vector>

#include "srk_internal.h"

namespace srk {

static thread_local std::string g_last_error;

int fail(int code, const char *fmt, ...) {
  char buf[512];
  va_list ap;
  va_start(ap, fmt);
  vsnprintf(buf, sizeof buf, fmt, ap);
  va_end(ap);
  g_last_error = buf;
  return code;
}

int cuda_fail(cudaError_t e, const char *what) {
  const int code = (e == cudaErrorMemoryAllocation) ? SRK_ENOMEM : SRK_ECUDA;
  return fail(code, "%s: %s (%s)", what, cudaGetErrorString(e),
              cudaGetErrorName(e));
}

void clear_error() { g_last_error.clear(); }

static std::mutex g_pool_mu;
static cudaMemPool_t g_pools[64] = {};
static int g_sms[64] = {};

cudaMemPool_t pool(int device) {
  if (device < 0 || device >= 64) return nullptr;
  std::lock_guard<std::mutex> lk(g_pool_mu);
  if (!g_pools[device]) {
    cudaMemPoolProps props;
    memset(&props, 0, sizeof props);
    props.allocType = cudaMemAllocationTypePinned;
    props.handleTypes = cudaMemHandleTypeNone;
    props.location.type = cudaMemLocationTypeDevice;
    props.location.id = device;
    cudaMemPool_t p = nullptr;
    if (cudaMemPoolCreate(&p, &props) != cudaSuccess) return nullptr;
    // keep freed blocks cached for the next query
    uint64_t keep = UINT64_MAX;
    cudaMemPoolSetAttribute(p, cudaMemPoolAttrReleaseThreshold, &keep);
    g_pools[device] = p;
  }
  return g_pools[device];
}

int sm_count(int device) {
  if (device < 0 || device >= 64) return 1;
  std::lock_guard<std::mutex> lk(g_pool_mu);
  if (!g_sms[device]) {
    int v = 0;
    if (cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, device) !=
            cudaSuccess || v <= 0)
      v = 1;
    g_sms[device] = v;
  }
  return g_sms[device];
}

bool is_device_ptr(const void *p) {
  if (!p) return false;
  cudaPointerAttributes at;
  if (cudaPointerGetAttributes(&at, p) != cudaSuccess) {
    cudaGetLastError();  // clear the sticky-free error of an unknown pointer
    return false;
  }
  return at.type == cudaMemoryTypeDevice || at.type == cudaMemoryTypeManaged;
}

// Algorithm 1 line 3 (truncation), line 5 (N_i), Algorithm 2 line 2 (z, Z, Z^),
// Lemma 7 (a(l) = |Z_l| / |Z^_l|), Appendix B.5 (p, q).  FP64, evaluated in a
// fixed order (host code is built without floating-point contraction):
//   z   = ln(2 n^q) / (2 lambda^2),  lambda = eps - 3 / n^p
//   L   = floor(p ln n / (-ln sqrt(c)))
//   Z_l = z * (sqrt(c)^l * (1 - sqrt(c))),  N_l = ceil(Z_l),  a(l) = Z_l / N_l
int build_table(int32_t n, int32_t s, double c, double eps, uint64_t seed,
                const srk_opts *opt, QueryTab *t) {
  if (n < 1) return fail(SRK_EINVAL, "graph has no nodes");
  if (s < 0 || s >= n) return fail(SRK_EINVAL, "source %d outside [0, %d)", s, n);
  if (!(c > 0.0 && c < 1.0)) return fail(SRK_EINVAL, "c = %g outside (0, 1)", c);
  double p = 1.0, q = 1.0, z_ovr = 0.0;
  int32_t L_ovr = -1;
  const bool warmup = opt && (opt->flags & SRK_OPT_WARMUP_RULE);
  if (opt) {
    if (opt->p != 0.0) p = opt->p;
    if (opt->q != 0.0) q = opt->q;
    z_ovr = opt->z_override;
    L_ovr = opt->L_override;
  }
  if (!(p >= 1.0) || !(q >= 1.0) || !isfinite(p) || !isfinite(q))
    return fail(SRK_EINVAL, "p = %g and q = %g must be >= 1", p, q);
  if (z_ovr != 0.0 && !(z_ovr > 0.0 && isfinite(z_ovr)))
    return fail(SRK_EINVAL, "z_override = %g must be 0 (none) or positive and finite", z_ovr);
  const double rc = sqrt(c);
  double z;
  if (z_ovr > 0.0) {
    if (!isfinite(z_ovr)) return fail(SRK_EINVAL, "z_override is not finite");
    z = z_ovr;
  } else if (warmup) {  // Section 3: N = ln(2 n^2) / (2 eps^2)
    if (!(eps > 0.0 && eps < 1.0)) return fail(SRK_EINVAL, "eps = %g outside (0, 1)", eps);
    z = log(2.0 * (double)n * (double)n) / (2.0 * eps * eps);
  } else {
    const double thr = 3.0 / pow((double)n, p);
    if (!(eps > thr && eps < 1.0))
      return fail(SRK_EINVAL, "eps = %g must satisfy 3/n^p = %g < eps < 1", eps, thr);
    const double lam = eps - thr;
    z = log(2.0 * pow((double)n, q)) / (2.0 * lam * lam);
  }
  int L;
  if (L_ovr >= 0) {
    L = L_ovr;
  } else if (warmup) {  // Section 3: walks of length >= 3 log_{1/sqrt c}(n/eps) are dropped
    if (!(eps > 0.0 && eps < 1.0)) return fail(SRK_EINVAL, "eps = %g outside (0, 1)", eps);
    const double Lf = floor(3.0 * log((double)n / eps) / (-log(rc)));
    if (!(Lf <= (double)SRK_MAX_LEN))
      return fail(SRK_EINVAL, "truncation length %g exceeds %d", Lf, SRK_MAX_LEN);
    L = (int)Lf;
  } else {
    const double Lf = floor(p * log((double)n) / (-log(rc)));
    if (!(Lf <= (double)SRK_MAX_LEN))
      return fail(SRK_EINVAL, "truncation length %g exceeds %d", Lf, SRK_MAX_LEN);
    L = (int)Lf;
  }
  if (L > SRK_MAX_LEN)
    return fail(SRK_EINVAL, "truncation length %d exceeds %d", L, SRK_MAX_LEN);
  t->s = s;
  t->n = n;
  t->L = L;
  t->key0 = (uint32_t)seed;
  t->key1 = (uint32_t)(seed >> 32);
  t->literal = (opt && (opt->flags & SRK_OPT_LITERAL_SHUFFLE)) ? 1 : 0;
  t->shared = (opt && (opt->flags & SRK_OPT_SHARED_WALKS)) ? 1 : 0;
  t->skey = walk_key(seed, (uint32_t)s);
  t->tkey = t->shared ? walk_key(seed, kSharedWalkKey) : t->skey;
  t->z = z;
  int64_t acc = 0;
  t->P[0] = 0;
  for (int l = 0; l <= L; ++l) {
    const double Zl = z * (pow(rc, (double)l) * (1.0 - rc));
    const double Nl = ceil(Zl);
    if (!(Nl >= 1.0) || Nl > (double)SRK_MAX_WALKS)
      return fail(SRK_EINVAL, "walk count %g for length %d out of range", Nl, l);
    acc += (int64_t)Nl;
    if (acc > SRK_MAX_WALKS)
      return fail(SRK_EINVAL, "N_tot exceeds %d walks", SRK_MAX_WALKS);
    t->a[l] = Zl / Nl;
    t->P[l + 1] = (int32_t)acc;
  }
  t->N_tot = (int32_t)acc;
  // the hit table holds at most sum_l l N_l entries, indexed with int32
  int64_t cells = 0;
  for (int l = 1; l <= L; ++l) cells += (int64_t)l * (t->P[l + 1] - t->P[l]);
  if (cells > INT32_MAX)
    return fail(SRK_EINVAL, "walk budget too large: sum_l l N_l = %lld exceeds 2^31",
                (long long)cells);
  return SRK_OK;
}

// Checks row_ptr[0] = 0, row_ptr[n] = m, row_ptr non-decreasing and
// 0 <= col < n; sets *bad to 1 on any violation.
__global__ void k_validate_csr(const int32_t *__restrict__ row_ptr,
                               const int32_t *__restrict__ col, int32_t n,
                               int64_t m, int *bad) {
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  const int64_t t0 = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (t0 == 0 && (row_ptr[0] != 0 || (int64_t)row_ptr[n] != m)) *bad = 1;
  for (int64_t v = t0; v < n; v += stride)
    if (row_ptr[v + 1] < row_ptr[v]) *bad = 1;
  for (int64_t e = t0; e < m; e += stride) {
    const int32_t x = col[e];
    if (x < 0 || x >= n) *bad = 1;
  }
}

// Packed adjacency with 4-byte entries (layout in srk_internal.h).  A walk
// step reads one entry, which names the next node and, unless that node is a
// hub, its degree too, instead of a row_ptr pair and a col entry.

// Last v with row_ptr[v] <= e: the owner of edge e.
__device__ __forceinline__ int32_t edge_owner(const int32_t *row_ptr, int32_t n, int64_t e) {
  int32_t lo = 0, hi = n - 1;
  while (lo < hi) {
    const int32_t mid = lo + (hi - lo + 1) / 2;
    if ((int64_t)row_ptr[mid] <= e) lo = mid; else hi = mid - 1;
  }
  return lo;
}

// The owner of every edge; a warp writes the lists of 32 nodes one by one.
__global__ void k_owners(const int32_t *__restrict__ row_ptr, int32_t n,
                         int32_t *__restrict__ owner) {
  const int lane = threadIdx.x & 31;
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t v0 = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) & ~31ll; v0 < n;
       v0 += stride) {
    const int64_t v = v0 + lane;
    const int32_t b = v < n ? row_ptr[v] : 0, e = v < n ? row_ptr[v + 1] : 0;
    for (uint32_t todo = __ballot_sync(0xffffffffu, e > b); todo; todo &= todo - 1) {
      const int l = __ffs(todo) - 1;
      const int32_t lb = __shfl_sync(0xffffffffu, b, l), le = __shfl_sync(0xffffffffu, e, l);
      for (int32_t k = lb + lane; k < le; k += 32) owner[k] = (int32_t)(v0 + l);
    }
  }
}

// Expected visits of the walks, used to order the packed adjacency: a walk
// starts at a uniformly drawn node with in-neighbours and moves to a
// uniformly drawn in-neighbour.  In 2^-40 fixed point, p_0 = 2^40 / n_act on
// those nodes and p_{k+1}(y) = sum over the lists I(v) that hold y of
// floor(p_k(v) / |I(v)|); the additions are integer, so their order does not
// change the result.
__global__ void k_visit_init(const int32_t *__restrict__ row_ptr, int32_t n, int32_t n_act,
                             unsigned long long *__restrict__ p) {
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  const unsigned long long unit = (1ull << 40) / (unsigned long long)(n_act > 0 ? n_act : 1);
  for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < n; v += stride)
    p[v] = row_ptr[v + 1] > row_ptr[v] ? unit : 0ull;
}

// p becomes the share that each in-neighbour gets.
__global__ void k_visit_share(const int32_t *__restrict__ row_ptr, int32_t n,
                              unsigned long long *__restrict__ p) {
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < n; v += stride) {
    const int32_t d = row_ptr[v + 1] - row_ptr[v];
    if (d > 1 && p[v]) p[v] /= (unsigned long long)d;
  }
}

__global__ void k_visit_step(const int32_t *__restrict__ owner, const int32_t *__restrict__ col,
                             int64_t m, const unsigned long long *__restrict__ share,
                             unsigned long long *__restrict__ q) {
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < m; e += stride) {
    const unsigned long long s = share[owner[e]];
    if (s) atomicAdd(&q[col[e]], s);
  }
}

// acc += w * p (the visit weights of one step).
__global__ void k_visit_acc(const unsigned long long *__restrict__ p, int32_t n, unsigned int w,
                            unsigned long long *__restrict__ acc) {
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < n; v += stride)
    acc[v] += (unsigned long long)w * p[v];
}

// Sort key of a node in the narrow layout: its degree code, descending, then
// its visits w, descending, by their leading ten bits (exponent and mantissa).
__device__ __forceinline__ uint32_t rank_key(uint32_t code, uint32_t dmax, unsigned long long w) {
  const int e = w ? 64 - __clzll((long long)w) : 0;  // 0..64
  const uint32_t heat = (uint32_t)e << 9 | (e > 10 ? (uint32_t)(w >> (e - 10)) & 511u
                                                   : (uint32_t)(w << (10 - e)) & 511u);
  return (dmax - code) << 16 | (0xFFFFu - heat);
}

__global__ void k_rank_keys(const int32_t *__restrict__ row_ptr, int32_t n, uint32_t dmax,
                            const unsigned long long *__restrict__ vis,
                            int32_t *__restrict__ key, int32_t *__restrict__ id,
                            int32_t *__restrict__ count) {
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  extern __shared__ int32_t hist[];  // nodes by degree code
  for (uint32_t c = threadIdx.x; c <= dmax; c += blockDim.x) hist[c] = 0;
  __syncthreads();
  for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < n; v += stride) {
    const uint32_t d = (uint32_t)(row_ptr[v + 1] - row_ptr[v]), code = d < dmax ? d : dmax;
    key[v] = (int32_t)rank_key(code, dmax, vis[v]);
    id[v] = (int32_t)v;
    atomicAdd(&hist[code], 1);
  }
  __syncthreads();
  for (uint32_t c = threadIdx.x; c <= dmax; c += blockDim.x)
    if (hist[c]) atomicAdd(&count[c], hist[c]);
}

// The visits, keys and order of a small graph (at most kRankNodes nodes, one block):
// what the kernels above and the radix sort do for a large one in 27 launches, which
// on 1,000 nodes made up a third of the load.  p, q: scratch of n words each.
constexpr int32_t kRankNodes = 4096, kRankEdges = 65536;
__global__ void __launch_bounds__(1024)
k_rank_small(const int32_t *__restrict__ row_ptr, const int32_t *__restrict__ col, int32_t n,
             int32_t m, int32_t n_act, uint32_t dmax, const int32_t *__restrict__ owner,
             unsigned long long *p, unsigned long long *q, int32_t *__restrict__ order,
             int32_t *__restrict__ count) {
  constexpr int kPer = kRankNodes / 1024;
  __shared__ unsigned long long s[kRankNodes];  // key << 32 | id
  const int t = threadIdx.x;
  unsigned long long acc[kPer];
  uint32_t deg[kPer];
  const unsigned long long unit = (1ull << 40) / (unsigned long long)(n_act > 0 ? n_act : 1);
#pragma unroll
  for (int k = 0; k < kPer; ++k) {
    const int32_t v = t + 1024 * k;
    acc[k] = 0;
    deg[k] = v < n ? (uint32_t)(row_ptr[v + 1] - row_ptr[v]) : 0u;
    if (v < n) p[v] = deg[k] ? unit : 0ull;
  }
  for (uint32_t c = t; c <= dmax; c += 1024) count[c] = 0;
#pragma unroll 1
  for (int step = 0; step < 3; ++step) {
#pragma unroll
    for (int k = 0; k < kPer; ++k) {
      const int32_t v = t + 1024 * k;
      if (v < n) {
        if (deg[k] > 1) p[v] /= (unsigned long long)deg[k];
        q[v] = 0ull;
      }
    }
    __syncthreads();
    for (int32_t e = t; e < m; e += 1024) {
      const unsigned long long share = p[owner[e]];
      if (share) atomicAdd(&q[col[e]], share);
    }
    __syncthreads();
    const unsigned long long w = step == 0 ? 25ull : step == 1 ? 15ull : 9ull;
#pragma unroll
    for (int k = 0; k < kPer; ++k) {
      const int32_t v = t + 1024 * k;
      if (v < n) acc[k] += w * q[v];
    }
    unsigned long long *const x = p;
    p = q;
    q = x;
  }
  int32_t size = 2;  // of the sort
  while (size < n) size <<= 1;
#pragma unroll
  for (int k = 0; k < kPer; ++k) {
    const int32_t v = t + 1024 * k;
    if (v < n) {
      const uint32_t code = deg[k] < dmax ? deg[k] : dmax;
      s[v] = (unsigned long long)rank_key(code, dmax, acc[k]) << 32 | (uint32_t)v;
      atomicAdd(&count[code], 1);
    } else if (v < size) {
      s[v] = ~0ull;
    }
  }
  for (int32_t run = 2; run <= size; run <<= 1)
    for (int32_t d = run >> 1; d > 0; d >>= 1) {
      __syncthreads();
      for (int32_t i = t; i < size / 2; i += 1024) {
        const int32_t a = 2 * i - (i & (d - 1)), b = a + d;  // bit d of a is clear
        const unsigned long long x = s[a], y = s[b];
        if ((x > y) == ((a & run) == 0)) {
          s[a] = y;
          s[b] = x;
        }
      }
    }
  __syncthreads();
  for (int32_t i = t; i < n; i += 1024) order[i] = (int32_t)(uint32_t)s[i];
}

// npos of the ranked nodes; the hubs' degrees by rank.
__global__ void k_ranks(const int32_t *__restrict__ row_ptr, int32_t n, int32_t H,
                        const int32_t *__restrict__ order, int32_t *__restrict__ npos,
                        int32_t *__restrict__ hub_deg) {
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t x = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; x < n; x += stride) {
    const int32_t v = order[x];
    npos[v] = (int32_t)x;
    if (x < H) hub_deg[x] = row_ptr[v + 1] - row_ptr[v];
  }
}

__global__ void k_hubs(int32_t H, const int32_t *__restrict__ deg, const int32_t *__restrict__ off,
                       uint2 *__restrict__ hub) {
  for (int32_t x = blockIdx.x * blockDim.x + threadIdx.x; x < H; x += gridDim.x * blockDim.x)
    hub[x] = make_uint2((uint32_t)deg[x], (uint32_t)off[x]);
}

// Edge e of list v lands at first(v) + (e - row_ptr[v]).
__global__ void k_narrow_lists(GraphView V, const int32_t *__restrict__ owner, int64_t m,
                               uint32_t *__restrict__ adj) {
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < m; e += stride) {
    const int32_t v = owner[e];
    const uint32_t dv = (uint32_t)(V.row_ptr[v + 1] - V.row_ptr[v]), x = (uint32_t)V.npos[v];
    const uint32_t first = dv < V.deg_max ? V.ctab[dv] + x * dv : V.hub[x].y;
    const int32_t y = V.col[e];
    const uint32_t dy = (uint32_t)(V.row_ptr[y + 1] - V.row_ptr[y]);
    const uint32_t code = dy < V.deg_max ? dy : V.deg_max;
    adj[first + (uint32_t)(e - V.row_ptr[v])] = (code << V.pos_bits) | (uint32_t)V.npos[y];
  }
}

// The wide layout (srk_internal.h): adj2[pos(v)] = {0, |I(v)|} and entry e
// of list v = {pos(y), |I(y)|} for y = col[e], at the same positions.
__global__ void k_build_adjw_heads(const int32_t *__restrict__ row_ptr, int32_t n,
                                   uint2 *__restrict__ adj2) {
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < n; v += stride)
    adj2[v + row_ptr[v]] = make_uint2(0u, (uint32_t)(row_ptr[v + 1] - row_ptr[v]));
}

__global__ void k_build_adjw_lists(const int32_t *__restrict__ row_ptr,
                                   const int32_t *__restrict__ col, int32_t n, int64_t m,
                                   uint2 *__restrict__ adj2) {
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < m; e += stride) {
    const int32_t lo = edge_owner(row_ptr, n, e);
    const int32_t y = col[e];
    adj2[(int64_t)lo + 1 + e] =
        make_uint2((uint32_t)(y + row_ptr[y]), (uint32_t)(row_ptr[y + 1] - row_ptr[y]));
  }
}

__global__ void k_out_degrees(const int32_t *__restrict__ col, int64_t m,
                              int32_t *__restrict__ deg) {
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < m;
       e += (int64_t)gridDim.x * blockDim.x)
    atomicAdd(&deg[col[e]], 1);
}

__global__ void k_active_flags(const int32_t *__restrict__ row_ptr, int32_t n,
                               int32_t *__restrict__ flag) {
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < n; v += stride)
    flag[v] = row_ptr[v + 1] > row_ptr[v] ? 1 : 0;
}

__global__ void k_active_scatter(const int32_t *__restrict__ flag,
                                 const int32_t *__restrict__ off, int32_t n,
                                 int32_t *__restrict__ act) {
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < n; v += stride)
    if (flag[v]) act[off[v]] = (int32_t)v;
}

}  // namespace srk

using namespace srk;

extern "C" const char *srk_last_error(void) { return g_last_error.c_str(); }

extern "C" int srk_pool_stats(int32_t device, uint64_t *reserved, uint64_t *used,
                              uint64_t *used_high, int reset_high) {
  clear_error();
  int count = 0;
  cudaError_t e = cudaGetDeviceCount(&count);
  if (e != cudaSuccess) return cuda_fail(e, "srk_pool_stats: device count");
  if (device < 0 || device >= count || device >= 64)
    return fail(SRK_EINVAL, "device %d outside [0, %d)", device, count);
  DeviceGuard guard(device);
  cudaMemPool_t p = pool(device);
  if (!p) return fail(SRK_ECUDA, "srk_pool_stats: cannot create the memory pool");
  uint64_t r = 0, u = 0, h = 0;  // the attributes are 64-bit values
  e = cudaMemPoolGetAttribute(p, cudaMemPoolAttrReservedMemCurrent, &r);
  if (e == cudaSuccess) e = cudaMemPoolGetAttribute(p, cudaMemPoolAttrUsedMemCurrent, &u);
  if (e == cudaSuccess) e = cudaMemPoolGetAttribute(p, cudaMemPoolAttrUsedMemHigh, &h);
  if (e == cudaSuccess && reset_high) {
    uint64_t zero = 0;  // resets the high-water mark to the current use
    e = cudaMemPoolSetAttribute(p, cudaMemPoolAttrUsedMemHigh, &zero);
  }
  if (e != cudaSuccess) return cuda_fail(e, "srk_pool_stats");
  if (reserved) *reserved = r;
  if (used) *used = u;
  if (used_high) *used_high = h;
  return SRK_OK;
}

extern "C" int srk_graph_layout(const srk_graph *g, int32_t *layout) {
  if (!g || !layout) return fail(SRK_EINVAL, "null argument");
  *layout = g->layout == 1 ? SRK_ADJ_WIDE : g->layout == 2 ? SRK_ADJ_CSR : SRK_ADJ_NARROW;
  return SRK_OK;
}

extern "C" int srk_graph_info(const srk_graph *g, int32_t *n, int64_t *m) {
  if (!g) return fail(SRK_EINVAL, "null graph");
  if (n) *n = g->n;
  if (m) *m = g->m;
  return SRK_OK;
}

extern "C" int srk_graph_free(srk_graph *g) {
  if (!g) return SRK_OK;
  int rc = SRK_OK;
  {
    DeviceGuard guard(g->device);
    cudaError_t e = cudaDeviceSynchronize();
    if (e != cudaSuccess) rc = cuda_fail(e, "srk_graph_free: synchronize");
    if (g->own_row_ptr) cudaFree(g->own_row_ptr);
    if (g->own_col) cudaFree(g->own_col);
    if (g->own_w) cudaFree(g->own_w);
    if (g->adj) cudaFree(g->adj);
    if (g->act) cudaFree(g->act);
    if (g->batch_exec) cudaGraphExecDestroy(g->batch_exec);
    free_lin_topo(g);
  }
  delete g;
  return rc;
}

// Smallest b with 2^b >= x (x >= 1), at most 31.
static int bits_for(int64_t x) {
  int b = 1;
  while (b < 31 && ((int64_t)1 << b) < x) ++b;
  return b;
}

// Degree codes of the narrow layout have at most this many bits: a table of
// list starts that the walk kernels hold in shared memory (8 KB).
constexpr int kCodeBits = 11;

// Builds the 4-byte-entry adjacency of g (sets adj, npos, hub, ctab, n_hubs,
// pos_bits, deg_max).  Nodes are ranked by degree code, descending, so that
// a list's place follows from its node's rank and degree, and within a code by
// expected visits, descending, so that the lists read most lie together; ties
// by id.  Expected visits (k_visit_*): 25 p_1 + 15 p_2 + 9 p_3, the landing
// mass of the first three steps weighted by survival at c = 0.6 (the layout
// does not depend on a query's c).  The layout is a function of the graph alone
// and is made on the device: R-MAT 20 loads in 1.8 ms and R-MAT 22 in 5.0 ms,
// where an order sorted on the host took 61 and 282 ms.
static int build_narrow(srk_graph *g, int dev) {
  const int32_t n = g->n;
  const int64_t m = g->m;
  // the documented bound of this layout (n + m + n_act past 2^30 edges and nodes)
  if ((int64_t)n + m > (1 << 30) && (int64_t)n + m + g->n_act > INT32_MAX)
    return fail(SRK_EINVAL, "graph too large for 4-byte adjacency entries (n + m + hubs = %lld)",
                (long long)n + (long long)m + (long long)g->n_act);
  const int pb = bits_for(n);
  const uint32_t dmax = (1u << std::min(32 - pb, kCodeBits)) - 1u;
  auto up = [](size_t b) { return (b + 255) & ~(size_t)255; };
  const size_t nb = up(sizeof(int32_t) * ((size_t)n + 1)), n8 = up(8 * (size_t)n);
  const size_t mb = up(sizeof(int32_t) * (size_t)(m > 0 ? m : 1));
  const size_t sort_b = up(sort_scratch(n)), count_b = up(sizeof(int32_t) * ((size_t)dmax + 1));
  char *tmp = nullptr;
  cudaError_t e = cudaMalloc(&tmp, 3 * n8 + 4 * nb + mb + sort_b + count_b);
  if (e != cudaSuccess) return cuda_fail(e, "srk_graph_load: ranking scratch");
  unsigned long long *p = (unsigned long long *)tmp, *q = (unsigned long long *)(tmp + n8),
                     *acc = (unsigned long long *)(tmp + 2 * n8);
  char *at = tmp + 3 * n8;
  int32_t *kA = (int32_t *)at, *vA = (int32_t *)(at + nb), *kB = (int32_t *)(at + 2 * nb),
          *vB = (int32_t *)(at + 3 * nb);
  at += 4 * nb;
  int32_t *owner = (int32_t *)at, *sort_tmp = (int32_t *)(at + mb),
          *count = (int32_t *)(at + mb + sort_b);
  const int bn = sm_count(dev) * 4, bm = sm_count(dev) * 8;
  if (m > 0) k_owners<<<bm, 256>>>(g->row_ptr, n, owner);
  const int32_t *order = vA;
  if (n <= kRankNodes && m <= kRankEdges) {
    k_rank_small<<<1, 1024>>>(g->row_ptr, g->col, n, (int32_t)m, g->n_act, dmax, owner, p, q, vA,
                              count);
  } else {
    cudaMemsetAsync(acc, 0, 8 * (size_t)n, 0);
    cudaMemsetAsync(count, 0, sizeof(int32_t) * ((size_t)dmax + 1), 0);
    k_visit_init<<<bn, 256>>>(g->row_ptr, n, g->n_act, p);
    const unsigned int w[3] = {25u, 15u, 9u};
    for (int k = 0; k < 3; ++k) {
      cudaMemsetAsync(q, 0, 8 * (size_t)n, 0);
      k_visit_share<<<bn, 256>>>(g->row_ptr, n, p);
      if (m > 0) k_visit_step<<<bm, 256>>>(owner, g->col, m, p, q);
      k_visit_acc<<<bn, 256>>>(q, n, w[k], acc);
      std::swap(p, q);
    }
    k_rank_keys<<<bn, 256, sizeof(int32_t) * ((size_t)dmax + 1)>>>(g->row_ptr, n, dmax, acc, kA,
                                                                   vA, count);
    if (radix_sort(kA, vA, kB, vB, n, 16 + std::min(32 - pb, kCodeBits), sort_tmp, 0)) order = vB;
  }
  // list starts by degree, from the number of nodes of each code
  std::vector<int32_t> cnt((size_t)dmax + 1);
  e = cudaMemcpy(cnt.data(), count, sizeof(int32_t) * cnt.size(), cudaMemcpyDeviceToHost);
  const int32_t H = e == cudaSuccess ? cnt[dmax] : 0;
  int64_t rest = m;  // entries of the hubs' lists
  for (uint32_t d = 1; d < dmax; ++d) rest -= (int64_t)d * cnt[d];
  std::vector<uint32_t> ctab((size_t)dmax + 1, 0u);
  uint32_t first = (uint32_t)rest, rank = (uint32_t)H;
  for (uint32_t d = dmax - 1; d >= 1 && d < dmax; --d) {
    ctab[d] = first - rank * d;
    first += d * (uint32_t)cnt[d];
    rank += (uint32_t)cnt[d];
  }
  // one block: the lists, ranks, nodes by rank, hub records and list starts
  const size_t adj_b = up(sizeof(uint32_t) * (size_t)(m > 0 ? m : 1)),
               hub_b = up(sizeof(uint2) * (size_t)(H > 0 ? H : 1));
  if (e == cudaSuccess)
    e = cudaMalloc(&g->adj, adj_b + 2 * nb + hub_b + sizeof(uint32_t) * ctab.size());
  if (e == cudaSuccess) {
    char *p8 = (char *)g->adj + adj_b;
    g->npos = (int32_t *)p8;
    g->order = (int32_t *)(p8 + nb);
    g->hub = (uint2 *)(p8 + 2 * nb);
    g->ctab = (uint32_t *)(p8 + 2 * nb + hub_b);
    e = cudaMemcpyAsync(g->order, order, sizeof(int32_t) * (size_t)n, cudaMemcpyDeviceToDevice, 0);
  }
  if (e == cudaSuccess)
    e = cudaMemcpy(g->ctab, ctab.data(), sizeof(uint32_t) * ctab.size(), cudaMemcpyHostToDevice);
  if (e == cudaSuccess) {
    g->pos_bits = pb;
    g->deg_max = dmax;
    g->n_hubs = H;
    int32_t *hub_deg = (int32_t *)p, *hub_off = (int32_t *)q;  // n words of 8 bytes each
    k_ranks<<<bn, 256>>>(g->row_ptr, n, H, order, g->npos, hub_deg);
    if (H > 0) {
      scan_i32(hub_deg, hub_off, H, sort_tmp, 0);
      k_hubs<<<bn, 256>>>(H, hub_deg, hub_off, g->hub);
    }
    if (m > 0) k_narrow_lists<<<bm, 256>>>(view_of(g), owner, m, g->adj);
    e = cudaGetLastError();
    if (e == cudaSuccess) e = cudaDeviceSynchronize();
  }
  cudaFree(tmp);
  if (e != cudaSuccess) return cuda_fail(e, "srk_graph_load: building the packed adjacency");
  return SRK_OK;
}

extern "C" int srk_graph_load(const int32_t *row_ptr, const int32_t *col,
                              int32_t n, int64_t m, int flags,
                              const float *edge_w, srk_graph **out) {
  clear_error();
  if (!out) return fail(SRK_EINVAL, "out is null");
  *out = nullptr;
  if (n < 1) return fail(SRK_EINVAL, "n = %d must be >= 1", n);
  if (m < 0 || m > INT32_MAX) return fail(SRK_EINVAL, "m = %lld outside [0, 2^31)", (long long)m);
  if ((int64_t)n + m > INT32_MAX)
    return fail(SRK_EINVAL, "n + m = %lld must stay below 2^31", (long long)n + (long long)m);
  if (!row_ptr || (m > 0 && !col)) return fail(SRK_EINVAL, "null CSR array");
  if (flags & ~(SRK_DEVICE_PTRS | SRK_VALIDATE | SRK_ADJ_NARROW | SRK_ADJ_WIDE | SRK_ADJ_CSR))
    return fail(SRK_EINVAL, "unknown flags 0x%x", flags);
  {
    const int layouts = !!(flags & SRK_ADJ_NARROW) + !!(flags & SRK_ADJ_WIDE) +
                        !!(flags & SRK_ADJ_CSR);
    if (layouts > 1)
      return fail(SRK_EINVAL, "SRK_ADJ_NARROW, SRK_ADJ_WIDE and SRK_ADJ_CSR exclude each other");
  }
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return cuda_fail(e, "srk_graph_load: no CUDA device");
  srk_graph *g = new srk_graph;
  g->n = n;
  g->m = m;
  g->device = dev;
  if (flags & SRK_DEVICE_PTRS) {
    if (!is_device_ptr(row_ptr) || (m > 0 && !is_device_ptr(col)) ||
        (edge_w && m > 0 && !is_device_ptr(edge_w))) {
      delete g;
      return fail(SRK_EINVAL, "SRK_DEVICE_PTRS given but an array is not device memory");
    }
    g->row_ptr = row_ptr;
    g->col = col;
    g->edge_w = edge_w;
  } else {
    const size_t rb = sizeof(int32_t) * ((size_t)n + 1);
    const size_t cb = sizeof(int32_t) * (size_t)(m > 0 ? m : 1);
    if ((e = cudaMalloc(&g->own_row_ptr, rb)) != cudaSuccess ||
        (e = cudaMalloc(&g->own_col, cb)) != cudaSuccess ||
        (edge_w && (e = cudaMalloc(&g->own_w, sizeof(float) * (size_t)(m > 0 ? m : 1))) !=
                       cudaSuccess)) {
      int rc = cuda_fail(e, "srk_graph_load: device allocation");
      srk_graph_free(g);
      return rc;
    }
    if ((e = cudaMemcpy(g->own_row_ptr, row_ptr, rb, cudaMemcpyDefault)) != cudaSuccess ||
        (m > 0 && (e = cudaMemcpy(g->own_col, col, sizeof(int32_t) * (size_t)m,
                                  cudaMemcpyDefault)) != cudaSuccess) ||
        (edge_w && m > 0 && (e = cudaMemcpy(g->own_w, edge_w, sizeof(float) * (size_t)m,
                                            cudaMemcpyDefault)) != cudaSuccess)) {
      int rc = cuda_fail(e, "srk_graph_load: copy to device");
      srk_graph_free(g);
      return rc;
    }
    g->row_ptr = g->own_row_ptr;
    g->col = g->own_col;
    g->edge_w = g->own_w;
  }
  {
    // Always validate: the walk kernels index with these values.  In the same
    // go, the ascending list of the nodes with in-neighbours and the
    // out-degrees (sizes of the queries' filters): few allocations and waits,
    // since those are what a small graph's load consists of.
    const size_t words = ((size_t)n + 64) & ~(size_t)63;  // at least n + 1
    int32_t *flag = nullptr;
    if ((e = cudaMalloc(&flag, sizeof(int32_t) * (2 * words + 64) + scan_scratch(n))) !=
        cudaSuccess) {
      int rc = cuda_fail(e, "srk_graph_load: active-node list");
      srk_graph_free(g);
      return rc;
    }
    int32_t *off = flag + words, *bad = off + n + 1, *scan_tmp = off + words + 64;
    const int blocks = sm_count(dev) * 4;
    cudaMemsetAsync(bad, 0, sizeof(int), 0);
    k_validate_csr<<<blocks, 256>>>(g->row_ptr, g->col, n, m, bad);
    k_active_flags<<<blocks, 256>>>(g->row_ptr, n, flag);
    scan_i32(flag, off, n, scan_tmp, 0);
    int32_t got[2] = {0, 0};  // nodes with in-neighbours, malformed
    e = cudaGetLastError();
    if (e == cudaSuccess) e = cudaMemcpy(got, off + n, sizeof got, cudaMemcpyDeviceToHost);
    const size_t act_words = ((size_t)got[0] + 64) & ~(size_t)63;
    if (e == cudaSuccess && !got[1] &&
        (e = cudaMalloc(&g->act, sizeof(int32_t) * (act_words + (size_t)n))) == cudaSuccess) {
      g->n_act = got[0];
      g->out_deg = g->act + act_words;
      cudaMemsetAsync(g->out_deg, 0, sizeof(int32_t) * (size_t)n, 0);
      k_active_scatter<<<blocks, 256>>>(flag, off, n, g->act);
      if (m > 0) k_out_degrees<<<2 * blocks, 256>>>(g->col, m, g->out_deg);
      e = cudaGetLastError();
    }
    cudaFree(flag);
    if (e != cudaSuccess) {
      int rc = cuda_fail(e, "srk_graph_load: validation and target list");
      srk_graph_free(g);
      return rc;
    }
    if (got[1]) {
      srk_graph_free(g);
      return fail(SRK_EINVAL, "malformed CSR: row_ptr must start at 0, end at m and "
                              "not decrease; col entries must lie in [0, n)");
    }
  }
  {
    const int pb = bits_for((int64_t)n + m);  // positions < n + m (wide layout)
    // Layout by size: 4-byte entries while n + m needs 28 bits at most (degree
    // codes of 9 bits at R-MAT 23), 8-byte entries beyond, which carry the full
    // degree.  Forced at R-MAT 24 and 25 (codes of 8 and 7 bits), 4-byte entries
    // give 4.93 and 2.30 queries/s at eps = 0.05 against 4.59 and 2.12 (the
    // latter with 3 targets a thread): half the bytes weigh more than the
    // hubs' records.  The default stays where
    // callers find it documented.  The CSR layout is only taken when asked for.
    g->layout = (flags & SRK_ADJ_WIDE)     ? 1
                : (flags & SRK_ADJ_CSR)    ? 2
                : (flags & SRK_ADJ_NARROW) ? 0
                : pb <= 28                 ? 0
                                           : 1;
    int rc = SRK_OK;
    if (g->layout == 0) {
      rc = build_narrow(g, dev);
    } else if ((e = cudaMalloc(&g->adj, sizeof(uint32_t) *
                                            (g->layout == 2 ? 1 : 2 * ((size_t)n + (size_t)m)))) !=
               cudaSuccess) {
      rc = cuda_fail(e, "srk_graph_load: packed adjacency");
    } else if (g->layout == 1) {
      uint2 *adj2 = reinterpret_cast<uint2 *>(g->adj);
      k_build_adjw_heads<<<sm_count(dev) * 4, 256>>>(g->row_ptr, n, adj2);
      if (m > 0) k_build_adjw_lists<<<sm_count(dev) * 8, 256>>>(g->row_ptr, g->col, n, m, adj2);
      e = cudaGetLastError();
      if (e == cudaSuccess) e = cudaDeviceSynchronize();
      if (e != cudaSuccess) rc = cuda_fail(e, "srk_graph_load: building the packed adjacency");
    }  // CSR: the walks read row_ptr and col directly
    if (rc != SRK_OK) {
      srk_graph_free(g);
      return rc;
    }
  }
  if ((e = allow_lockstep(g->layout)) != cudaSuccess) {
    int rc = cuda_fail(e, "srk_graph_load: shared memory of the walk kernels");
    srk_graph_free(g);
    return rc;
  }
  if ((e = cudaDeviceSynchronize()) != cudaSuccess) {
    int rc = cuda_fail(e, "srk_graph_load");
    srk_graph_free(g);
    return rc;
  }
  *out = g;
  return SRK_OK;
}
