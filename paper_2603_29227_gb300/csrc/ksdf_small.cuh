// ksdf_small.cuh -- grouping of a small batch of queries by one CTA (included by ksdf_query.cu and ksdf_backward.cu).
//
// For a few queries the grouping passes are all launch latency: binning, hashing, five scans, scatters and tile lists
// take 17 launches before phase A and 8 before phase B, about 0.23 ms.  Up to kSmallQ queries fit one CTA's shared
// memory, which sorts them by group, numbers the groups and cuts the tiles in a single launch.
#pragma once
#include "ksdf_internal.cuh"

namespace ksdf {
namespace {

// two keys per thread of a 1,024-thread CTA, 33 KB of shared memory.  Measured, grouping before phase A: 37 queries 177 ->
// 14 us, 512 queries 181 -> 21 us; regrouping by winner 59 -> 11 and 15 us.
constexpr int kSmallQ = 2048;
constexpr int kSmallThreads = kSmallQ / 2;

struct SmallSort {
  uint64_t key[kSmallQ];   // group key; kEmptyKey: not grouped (sorts last)
  int idx[kSmallQ];        // item
  int start[kSmallQ + 1];  // first position of each group, then the number of grouped items
  int sw[32];
  int base[3], cnt[3];
};

// exclusive scan of one int per thread over the CTA; *total gets the sum
__device__ __forceinline__ int small_exscan(int v, int* sw, int* total) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  int x = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int y = __shfl_up_sync(0xffffffffu, x, o);
    if (lane >= o) x += y;
  }
  if (lane == 31) sw[warp] = x;
  __syncthreads();
  if (warp == 0) {
    int w = sw[lane];
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int y = __shfl_up_sync(0xffffffffu, w, o);
      if (lane >= o) w += y;
    }
    sw[lane] = w;
  }
  __syncthreads();
  const int r = (warp ? sw[warp - 1] : 0) + x - v;
  *total = sw[31];
  __syncthreads();
  return r;
}

// Sorts the items 0 .. n - 1 by (key, item) and finds the groups: returns their number, with start[] filled and gid[]
// the groups of this thread's positions 2 tid and 2 tid + 1 (-1: not grouped).
__device__ __forceinline__ int small_group(SmallSort& s, int n, int gid[2]) {
  const int tid = threadIdx.x;
  int P = 2;
  while (P < n) P <<= 1;
  for (int i = n + tid; i < P; i += kSmallThreads) {
    s.key[i] = kEmptyKey;
    s.idx[i] = i;
  }
  __syncthreads();
  for (int k = 2; k <= P; k <<= 1)
    for (int j = k >> 1; j > 0; j >>= 1) {
      if (tid < P / 2) {
        const int a = 2 * tid - (tid & (j - 1)), b = a + j;  // the tid-th pair of this stride
        const uint64_t ka = s.key[a], kb = s.key[b];
        const int ia = s.idx[a], ib = s.idx[b];
        const bool gt = ka > kb || (ka == kb && ia > ib);
        if (gt == ((a & k) == 0)) {
          s.key[a] = kb;
          s.key[b] = ka;
          s.idx[a] = ib;
          s.idx[b] = ia;
        }
      }
      __syncthreads();
    }
  bool head[2], live[2];
#pragma unroll
  for (int u = 0; u < 2; ++u) {
    const int i = 2 * tid + u;
    live[u] = i < n && s.key[i] != kEmptyKey;
    head[u] = live[u] && (i == 0 || s.key[i] != s.key[i - 1]);
  }
  int ng, nl;
  const int before = small_exscan((int)head[0] + (int)head[1], s.sw, &ng);
  small_exscan((int)live[0] + (int)live[1], s.sw, &nl);
  gid[0] = before + (int)head[0] - 1;
  gid[1] = gid[0] + (int)head[1];
#pragma unroll
  for (int u = 0; u < 2; ++u) {
    if (head[u]) s.start[gid[u]] = 2 * tid + u;
    if (!live[u]) gid[u] = -1;
  }
  if (tid == 0) s.start[ng] = nl;
  __syncthreads();
  return ng;
}

// tiles of at most T items of every group, in group order: each thread takes the groups 2 tid, 2 tid + 1; fn(g, first
// tile, number of tiles); returns the number of tiles
template <class F>
__device__ __forceinline__ int small_tiles(SmallSort& s, int ng, int T, F&& fn) {
  int nt[2] = {0, 0};
#pragma unroll
  for (int u = 0; u < 2; ++u) {
    const int g = 2 * threadIdx.x + u;
    if (g < ng) nt[u] = (s.start[g + 1] - s.start[g] + T - 1) / T;
  }
  int total;
  const int t0 = small_exscan(nt[0] + nt[1], s.sw, &total);
  if (nt[0]) fn(2 * (int)threadIdx.x, t0, nt[0]);
  if (nt[1]) fn(2 * (int)threadIdx.x + 1, t0 + nt[0], nt[1]);
  return total;
}

}  // namespace
}  // namespace ksdf
