// Scans and sorts of the graph builders: an exclusive scan of any length and a
// stable LSD radix sort of 32-bit keys with values.
#include <stdint.h>

#include "srk_internal.h"

namespace srk {

// Radix sort: 8-bit digits, tiles of 256 threads x 16 keys.
constexpr int kSortBlock = 256, kSortItems = 16, kSortTile = kSortBlock * kSortItems;
// Scan: tiles of 1024 threads x 4 entries.
constexpr int kScanTile = 4096;

// Radix sort pass, step 1: digit histogram of each tile, stored digit-major
// (hist[d * tiles + tile]) so that its exclusive scan gives each
// (digit, tile) its first output position.
__global__ void __launch_bounds__(kSortBlock)
k_sort_hist(const int32_t *__restrict__ keys, int64_t m, int shift, int32_t tiles,
            int32_t *__restrict__ hist) {
  __shared__ int32_t cnt[256];
  cnt[threadIdx.x] = 0;
  __syncthreads();
  const int64_t base = (int64_t)blockIdx.x * kSortTile;
  for (int r = 0; r < kSortItems; ++r) {
    const int64_t i = base + (int64_t)r * kSortBlock + threadIdx.x;
    if (i < m) atomicAdd(&cnt[(keys[i] >> shift) & 255], 1);
  }
  __syncthreads();
  hist[(int64_t)threadIdx.x * tiles + blockIdx.x] = cnt[threadIdx.x];
}

// Radix sort pass, step 2: stable scatter.  Round r of a tile covers 256
// consecutive keys; a key goes to its (digit, tile) offset plus the number of
// keys of its digit in earlier rounds, earlier warps and lower lanes.
__global__ void __launch_bounds__(kSortBlock)
k_sort_scatter(const int32_t *__restrict__ keys, const int32_t *__restrict__ vals, int64_t m,
               int shift, int32_t tiles, const int32_t *__restrict__ off,
               int32_t *__restrict__ keys_out, int32_t *__restrict__ vals_out) {
  constexpr int kWarps = kSortBlock / 32;
  __shared__ int32_t base[256];
  __shared__ int32_t wcnt[kWarps][256];
  const int t = threadIdx.x, lane = t & 31, w = t >> 5;
  base[t] = off[(int64_t)t * tiles + blockIdx.x];
  for (int i = 0; i < kWarps; ++i) wcnt[i][t] = 0;
  __syncthreads();
  const int64_t tile0 = (int64_t)blockIdx.x * kSortTile;
  for (int r = 0; r < kSortItems; ++r) {
    // the last tile's rounds past the end: most of them on a small graph
    if (tile0 + (int64_t)r * kSortBlock >= m) break;
    const int64_t i = tile0 + (int64_t)r * kSortBlock + t;
    const bool valid = i < m;
    int32_t key = 0, val = 0, d = 256;  // 256: no key in this slot
    if (valid) {
      key = keys[i];
      val = vals[i];
      d = (key >> shift) & 255;
    }
    const unsigned peers = __match_any_sync(0xffffffffu, d);
    const int rank = __popc(peers & ((1u << lane) - 1u));
    if (valid && rank == 0) wcnt[w][d] = __popc(peers);
    __syncthreads();
    int32_t run = 0;  // thread t: digit t's counts over the warps, made exclusive
    for (int k = 0; k < kWarps; ++k) {
      const int32_t c = wcnt[k][t];
      wcnt[k][t] = run;
      run += c;
    }
    __syncthreads();
    if (valid) {
      const int64_t pos = (int64_t)base[d] + wcnt[w][d] + rank;
      keys_out[pos] = key;
      vals_out[pos] = val;
    }
    __syncthreads();
    base[t] += run;
    for (int k = 0; k < kWarps; ++k) wcnt[k][t] = 0;
    __syncthreads();
  }
}

// Exclusive scan of cnt[0..N) into off[0..N], one block of 1024 threads.
static __global__ void __launch_bounds__(1024)
k_scan(const int32_t *__restrict__ cnt, int32_t *__restrict__ off, int32_t N) {
  __shared__ int32_t warp_sum[32];
  __shared__ int32_t carry;
  if (threadIdx.x == 0) carry = 0;
  __syncthreads();
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  for (int64_t base = 0; base < N; base += 4096) {
    const int64_t i0 = base + 4 * (int64_t)threadIdx.x;
    int32_t v[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) v[k] = (i0 + k < N) ? cnt[i0 + k] : 0;
    const int32_t local = v[0] + v[1] + v[2] + v[3];
    int32_t incl = local;
    for (int o = 1; o < 32; o <<= 1) {
      const int32_t y = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += y;
    }
    if (lane == 31) warp_sum[wid] = incl;
    __syncthreads();
    if (wid == 0) {
      int32_t ws = warp_sum[lane];
      for (int o = 1; o < 32; o <<= 1) {
        const int32_t y = __shfl_up_sync(0xffffffffu, ws, o);
        if (lane >= o) ws += y;
      }
      warp_sum[lane] = ws;  // inclusive over warps
    }
    __syncthreads();
    int32_t run = carry + (wid ? warp_sum[wid - 1] : 0) + incl - local;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      if (i0 + k < N) off[i0 + k] = run;
      run += v[k];
    }
    __syncthreads();
    if (threadIdx.x == 1023) carry = run;
    __syncthreads();
  }
  if (threadIdx.x == 0) off[N] = carry;
}

// Sums of the scan's tiles.
__global__ void __launch_bounds__(1024)
k_scan_sums(const int32_t *__restrict__ cnt, int64_t N, int32_t *__restrict__ sums) {
  __shared__ int32_t ws[32];
  const int64_t i0 = (int64_t)blockIdx.x * kScanTile + threadIdx.x;
  int32_t v = 0;
#pragma unroll
  for (int k = 0; k < 4; ++k) v += (i0 + k * 1024 < N) ? cnt[i0 + k * 1024] : 0;
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  if ((threadIdx.x & 31) == 0) ws[threadIdx.x >> 5] = v;
  __syncthreads();
  if (threadIdx.x < 32) {
    v = ws[threadIdx.x];
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if (threadIdx.x == 0) sums[blockIdx.x] = v;
  }
}

// The tiles' entries, from the scanned sums of the tiles (base).
__global__ void __launch_bounds__(1024)
k_scan_tiles(const int32_t *__restrict__ cnt, int64_t N, const int32_t *__restrict__ base,
             int32_t *__restrict__ off) {
  __shared__ int32_t ws[32];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const int64_t i0 = (int64_t)blockIdx.x * kScanTile + 4 * (int64_t)threadIdx.x;
  int32_t v[4];
#pragma unroll
  for (int k = 0; k < 4; ++k) v[k] = (i0 + k < N) ? cnt[i0 + k] : 0;
  const int32_t local = v[0] + v[1] + v[2] + v[3];
  int32_t incl = local;
  for (int o = 1; o < 32; o <<= 1) {
    const int32_t y = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += y;
  }
  if (lane == 31) ws[wid] = incl;
  __syncthreads();
  if (wid == 0) {
    int32_t s = ws[lane];
    for (int o = 1; o < 32; o <<= 1) {
      const int32_t y = __shfl_up_sync(0xffffffffu, s, o);
      if (lane >= o) s += y;
    }
    ws[lane] = s;  // inclusive over warps
  }
  __syncthreads();
  int32_t run = base[blockIdx.x] + (wid ? ws[wid - 1] : 0) + incl - local;
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    if (i0 + k < N) off[i0 + k] = run;
    run += v[k];
    if (i0 + k == N - 1) off[N] = run;
  }
}

size_t scan_scratch(int64_t N) {
  return 2 * sizeof(int32_t) * (size_t)((N + kScanTile - 1) / kScanTile + 1);
}

// One block scans up to a few tiles itself (two launches more cost about as
// much as eight of its rounds); beyond, all SMs scan tiles: 1 M entries in
// 0.011 ms.
void scan_i32(const int32_t *cnt, int32_t *off, int64_t N, int32_t *tmp, cudaStream_t st) {
  const int64_t tiles = (N + kScanTile - 1) / kScanTile;
  if (tiles <= 8) {
    k_scan<<<1, 1024, 0, st>>>(cnt, off, (int32_t)N);
    return;
  }
  int32_t *sums = tmp, *base = tmp + tiles;
  k_scan_sums<<<(unsigned)tiles, 1024, 0, st>>>(cnt, N, sums);
  k_scan<<<1, 1024, 0, st>>>(sums, base, (int32_t)tiles);
  k_scan_tiles<<<(unsigned)tiles, 1024, 0, st>>>(cnt, N, base, off);
}

size_t sort_scratch(int64_t m) {
  const size_t tiles = (size_t)((m + kSortTile - 1) / kSortTile), H = 256 * (tiles ? tiles : 1);
  return sizeof(int32_t) * (2 * H + 1) + 256 + scan_scratch((int64_t)H);
}

bool radix_sort(int32_t *kA, int32_t *vA, int32_t *kB, int32_t *vB, int64_t m, int bits,
                int32_t *tmp, cudaStream_t st) {
  if (m <= 0) return false;
  const int32_t tiles = (int32_t)((m + kSortTile - 1) / kSortTile);
  const int64_t H = (int64_t)256 * tiles;
  int32_t *hist = tmp, *hoff = tmp + H, *scan = hoff + H + 1;
  bool swapped = false;
  for (int shift = 0; shift < bits; shift += 8) {
    k_sort_hist<<<tiles, kSortBlock, 0, st>>>(kA, m, shift, tiles, hist);
    scan_i32(hist, hoff, H, scan, st);
    k_sort_scatter<<<tiles, kSortBlock, 0, st>>>(kA, vA, m, shift, tiles, hoff, kB, vB);
    int32_t *tk = kA, *tv = vA;
    kA = kB;
    vA = vB;
    kB = tk;
    vB = tv;
    swapped = !swapped;
  }
  return swapped;
}

}  // namespace srk
