// ksdf_sort.cu -- device-wide exclusive scan and stable LSD radix sort used by the fit and the query
// grouping.  Written for one GPU; every launch is stream ordered and allocation free once `tmp` is large
// enough.
#include "ksdf_internal.cuh"

#include <algorithm>

namespace ksdf {

namespace {

constexpr int kScanThreads = 256;
constexpr int kScanItems = 8;
constexpr int kScanTile = kScanThreads * kScanItems;

// exclusive scan of one value per thread over a 256-thread block; returns the block total in *total
__device__ inline int64_t block_exscan(int64_t v, int64_t* smem_warp, int64_t* total) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  int64_t x = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    int64_t y = __shfl_up_sync(0xffffffffu, x, o);
    if (lane >= o) x += y;
  }
  if (lane == 31) smem_warp[warp] = x;
  __syncthreads();
  if (warp == 0) {
    int64_t w = lane < (kScanThreads / 32) ? smem_warp[lane] : 0;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      int64_t y = __shfl_up_sync(0xffffffffu, w, o);
      if (lane >= o) w += y;
    }
    if (lane < (kScanThreads / 32)) smem_warp[lane] = w;  // inclusive warp prefix
  }
  __syncthreads();
  int64_t warp_base = warp ? smem_warp[warp - 1] : 0;
  *total = smem_warp[kScanThreads / 32 - 1];
  __syncthreads();
  return warp_base + x - v;
}

// n_dev (may be NULL): the scan covers min(n, *n_dev) elements, a count known only on the device
__device__ __forceinline__ int64_t scan_len(int64_t n, const int64_t* n_dev) {
  return n_dev ? (*n_dev < n ? *n_dev : n) : n;
}

// Several arrays are scanned by the same launches, one per blockIdx.y (the query's groupings scan two and four at a time:
// at most sizes each launch is latency only).
struct ScanJobs {
  ScanJob j[kMaxScanJobs];
};

__global__ void k_scan_reduce(ScanJobs jobs) {
  __shared__ int64_t sw[kScanThreads / 32];
  const ScanJob& job = jobs.j[blockIdx.y];
  const int64_t* in = job.in;
  const int64_t n = scan_len(job.n, job.n_dev);
  if ((int64_t)blockIdx.x * kScanTile >= n) return;  // the whole block is past the end (uniform)
  int64_t base = (int64_t)blockIdx.x * kScanTile + (int64_t)threadIdx.x * kScanItems;
  int64_t s = 0;
#pragma unroll
  for (int i = 0; i < kScanItems; ++i)
    if (base + i < n) s += in[base + i];
  int64_t tot;
  block_exscan(s, sw, &tot);
  if (threadIdx.x == 0) job.sums[blockIdx.x] = tot;
}

__global__ void k_scan_sums(ScanJobs jobs) {
  __shared__ int64_t sw[kScanThreads / 32];
  const ScanJob& job = jobs.j[blockIdx.y];
  int64_t* sums = job.sums;
  const int64_t nb = (scan_len(job.n, job.n_dev) + kScanTile - 1) / kScanTile;
  int64_t carry = 0;
  for (int64_t c0 = 0; c0 < nb; c0 += kScanThreads) {
    int64_t i = c0 + threadIdx.x;
    int64_t v = i < nb ? sums[i] : 0;
    int64_t tot;
    int64_t ex = block_exscan(v, sw, &tot);
    if (i < nb) sums[i] = carry + ex;
    carry += tot;
  }
  if (threadIdx.x == 0 && job.total) *job.total = carry;
}

__global__ void k_scan_apply(ScanJobs jobs) {
  __shared__ int64_t sw[kScanThreads / 32];
  const ScanJob& job = jobs.j[blockIdx.y];
  const int64_t* in = job.in;
  int64_t* out = job.out;
  const int64_t n = scan_len(job.n, job.n_dev);
  if ((int64_t)blockIdx.x * kScanTile >= n) return;  // the whole block is past the end (uniform)
  int64_t base = (int64_t)blockIdx.x * kScanTile + (int64_t)threadIdx.x * kScanItems;
  int64_t v[kScanItems];
  int64_t s = 0;
#pragma unroll
  for (int i = 0; i < kScanItems; ++i) {
    v[i] = base + i < n ? in[base + i] : 0;
    s += v[i];
  }
  int64_t tot;
  int64_t ex = block_exscan(s, sw, &tot) + job.sums[blockIdx.x];
#pragma unroll
  for (int i = 0; i < kScanItems; ++i) {
    if (base + i < n) out[base + i] = ex;
    ex += v[i];
  }
}

// small arrays: the whole exclusive scan in one 1024-thread block (one launch instead of three).  Each warp owns a
// contiguous run and walks it 32 elements at a time (coalesced), once for its sum and once, from its base, to write:
// with a run per thread instead, the loads of a warp fall on 32 sectors each (the grouping of a million queries, with
// its scan of 65,536 buckets, went from 0.32 to 0.23 ms).
constexpr int kScanSingleThreads = 1024;
constexpr int kScanSingleItems = 64;

__global__ void __launch_bounds__(kScanSingleThreads) k_scan_single(ScanJobs jobs) {
  constexpr unsigned FULL = 0xffffffffu;
  __shared__ int64_t sw[kScanSingleThreads / 32];
  const ScanJob& job = jobs.j[blockIdx.y];
  const int64_t* in = job.in;
  int64_t* out = job.out;
  const int64_t n = scan_len(job.n, job.n_dev);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int64_t per = 32 * ((n + kScanSingleThreads - 1) / kScanSingleThreads);  // elements of a warp
  const int64_t b = warp * per, e = b + per < n ? b + per : n;
  int64_t s = 0;
#pragma unroll 8
  for (int64_t i = b + lane; i < e; i += 32) s += in[i];
#pragma unroll
  for (int o = 16; o; o >>= 1) s += __shfl_xor_sync(FULL, s, o);
  if (lane == 0) sw[warp] = s;
  __syncthreads();
  if (warp == 0) {
    int64_t w = sw[lane];
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int64_t y = __shfl_up_sync(FULL, w, o);
      if (lane >= o) w += y;
    }
    sw[lane] = w;  // inclusive prefix over the warps
    if (lane == 31 && job.total) *job.total = w;
  }
  __syncthreads();
  int64_t run = warp ? sw[warp - 1] : 0;
  for (int64_t i0 = b; i0 < e; i0 += 128) {  // four loads in flight
    int64_t v[4], x[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int64_t i = i0 + 32 * u + lane;
      x[u] = v[u] = i < e ? in[i] : 0;
    }
#pragma unroll
    for (int o = 1; o < 32; o <<= 1)
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int64_t y = __shfl_up_sync(FULL, x[u], o);
        if (lane >= o) x[u] += y;
      }
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int64_t i = i0 + 32 * u + lane;
      if (i < e) out[i] = run + x[u] - v[u];
      run += __shfl_sync(FULL, x[u], 31);
    }
  }
}

// ---- radix sort ----
constexpr int kRsThreads = 256;
constexpr int kRsWarps = kRsThreads / 32;
constexpr int kRsChunks = 8;  // chunks of 256 elements per tile
constexpr int kRsTile = kRsThreads * kRsChunks;

__global__ void k_rs_hist(const uint64_t* keys, int64_t n, int shift, int64_t* hist, int nblocks) {
  __shared__ int h[256];
  h[threadIdx.x] = 0;
  __syncthreads();
  int64_t base = (int64_t)blockIdx.x * kRsTile;
#pragma unroll
  for (int c = 0; c < kRsChunks; ++c) {
    int64_t i = base + c * kRsThreads + threadIdx.x;
    if (i < n) atomicAdd(&h[(keys[i] >> shift) & 0xFF], 1);
  }
  __syncthreads();
  hist[(int64_t)threadIdx.x * nblocks + blockIdx.x] = h[threadIdx.x];
}

// stable scatter: elements of a chunk are ranked by (warp, lane) order; chunks in order; blocks in order
__global__ void k_rs_scatter(const uint64_t* keys, const uint32_t* vals, uint64_t* okeys, uint32_t* ovals, int64_t n,
                             int shift, const int64_t* offs, int nblocks) {
  __shared__ int64_t running[256];
  __shared__ int64_t wcnt[kRsWarps][256];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  running[threadIdx.x] = offs[(int64_t)threadIdx.x * nblocks + blockIdx.x];
  int64_t base = (int64_t)blockIdx.x * kRsTile;
  const unsigned lt_mask = (1u << lane) - 1u;
  for (int c = 0; c < kRsChunks; ++c) {
#pragma unroll
    for (int w = 0; w < kRsWarps; ++w) wcnt[w][threadIdx.x] = 0;
    __syncthreads();
    int64_t i = base + c * kRsThreads + threadIdx.x;
    bool valid = i < n;
    uint64_t k = valid ? keys[i] : 0;
    uint32_t v = valid ? vals[i] : 0;
    int d = valid ? (int)((k >> shift) & 0xFF) : 256;  // 256: no element
    unsigned m = __match_any_sync(0xffffffffu, d);
    int rank = __popc(m & lt_mask);
    if (valid && rank == 0) wcnt[warp][d] = __popc(m);
    __syncthreads();
    {
      int64_t r = running[threadIdx.x];
#pragma unroll
      for (int w = 0; w < kRsWarps; ++w) {
        int64_t t = wcnt[w][threadIdx.x];
        wcnt[w][threadIdx.x] = r;
        r += t;
      }
      running[threadIdx.x] = r;
    }
    __syncthreads();
    if (valid) {
      int64_t pos = wcnt[warp][d] + rank;
      okeys[pos] = k;
      ovals[pos] = v;
    }
    __syncthreads();
  }
}

}  // namespace

// the launches of a scan whose jobs have their sums
static void scan_launch(const ScanJobs& js, int nj, int64_t n, cudaStream_t st) {
  const unsigned y = (unsigned)nj;
  if (n <= (int64_t)kScanSingleThreads * kScanSingleItems) {
    launch(k_scan_single, dim3(1, y), kScanSingleThreads, 0, st, js);
    return;
  }
  const unsigned nb = (unsigned)((n + kScanTile - 1) / kScanTile);
  launch(k_scan_reduce, dim3(nb, y), kScanThreads, 0, st, js);
  launch(k_scan_sums, dim3(1, y), kScanThreads, 0, st, js);
  launch(k_scan_apply, dim3(nb, y), kScanThreads, 0, st, js);
}

cudaError_t scan_i64(const ScanJob* jobs, int nj, DevBuf& tmp, cudaStream_t st) {
  ScanJobs js{};
  int64_t n = 0, sums = 0;
  int k = 0;
  for (int i = 0; i < nj; ++i) {
    if (jobs[i].n > 0) {
      js.j[k++] = jobs[i];
      n = std::max(n, jobs[i].n);
      sums += scan_sums_len(jobs[i].n);
    } else if (jobs[i].total) {
      cudaError_t e = cudaMemsetAsync(jobs[i].total, 0, sizeof(int64_t), st);
      if (e != cudaSuccess) return e;
    }
  }
  if (k == 0) return cudaSuccess;
  if (n > (int64_t)kScanSingleThreads * kScanSingleItems) {
    cudaError_t e = ensure(tmp, sizeof(int64_t) * (size_t)sums);
    if (e != cudaSuccess) return e;
    int64_t* p = ptr<int64_t>(tmp);
    for (int i = 0; i < k; ++i) {
      js.j[i].sums = p;
      p += scan_sums_len(js.j[i].n);
    }
  }
  scan_launch(js, k, n, st);
  return cudaGetLastError();
}

cudaError_t scan_i64(const int64_t* in, int64_t* out, int64_t n, int64_t* total, DevBuf& tmp, cudaStream_t st,
                     const int64_t* n_dev) {
  const ScanJob job{in, out, n, total, n_dev, nullptr};
  return scan_i64(&job, 1, tmp, st);
}

cudaError_t radix_sort_u64(uint64_t* keys, uint32_t* vals, int64_t n, int bits, DevBuf& tmp, cudaStream_t st) {
  if (n <= 1 || bits <= 0) return cudaSuccess;
  const int passes = (bits + 7) / 8;
  const int nblocks = (int)((n + kRsTile - 1) / kRsTile);
  const int64_t nh = 256LL * nblocks;
  const int64_t nb_scan = (nh + kScanTile - 1) / kScanTile;
  size_t need = sizeof(uint64_t) * n + sizeof(uint32_t) * n + sizeof(int64_t) * (size_t)(nh + nb_scan + 2) + 64;
  cudaError_t e = ensure(tmp, need);
  if (e != cudaSuccess) return e;
  char* b = static_cast<char*>(tmp.p);
  uint64_t* k2 = reinterpret_cast<uint64_t*>(b);
  b += sizeof(uint64_t) * n;
  uint32_t* v2 = reinterpret_cast<uint32_t*>(b);
  b += sizeof(uint32_t) * n;
  b = reinterpret_cast<char*>((reinterpret_cast<uintptr_t>(b) + 15) & ~uintptr_t(15));
  int64_t* hist = reinterpret_cast<int64_t*>(b);
  int64_t* sums = hist + nh;
  uint64_t *ki = keys, *ko = k2;
  uint32_t *vi = vals, *vo = v2;
  for (int p = 0; p < passes; ++p) {
    int shift = 8 * p;
    launch(k_rs_hist, nblocks, kRsThreads, 0, st, ki, n, shift, hist, nblocks);
    ScanJobs js{};
    js.j[0] = ScanJob{hist, hist, nh, nullptr, nullptr, sums};
    scan_launch(js, 1, nh, st);
    launch(k_rs_scatter, nblocks, kRsThreads, 0, st, ki, vi, ko, vo, n, shift, hist, nblocks);
    uint64_t* tk = ki; ki = ko; ko = tk;
    uint32_t* tv = vi; vi = vo; vo = tv;
  }
  if (ki != keys) {
    e = cudaMemcpyAsync(keys, ki, sizeof(uint64_t) * n, cudaMemcpyDeviceToDevice, st);
    if (e != cudaSuccess) return e;
    e = cudaMemcpyAsync(vals, vi, sizeof(uint32_t) * n, cudaMemcpyDeviceToDevice, st);
    if (e != cudaSuccess) return e;
  }
  return cudaGetLastError();
}

}  // namespace ksdf
