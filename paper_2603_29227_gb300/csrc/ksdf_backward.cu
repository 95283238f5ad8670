// ksdf_backward.cu -- adjoint of the Kernel-SDF query with respect to the query points and the sample
// positions (differentiation path; the paper states the SDF is differentiable, Sec. IV-B).
//
// With d held constant (u does not depend on the scaling of App. D), for a query q whose min-fusion
// winner is cell g with training set {x_i, alpha_i}:
//   u^2 = -log f'/lambda + d^2,  f' = sum_i alpha_i k'_i,  k'_i = exp(-lambda (|x - x_i|^2 - d^2))
//   dL/df'  = -s dsdf / (2 lambda u f')                                   (sdf = s u)
//   x_bar  += dL/df' grad_x f' = dL/df' (-2 lambda G),  G = sum_i alpha_i k'_i (x - x_i)
//   X_bar_i += dL/df' 2 lambda alpha_i k'_i (x - x_i),   alpha_bar_i += dL/df' k'_i
// For the gradient output s G/|G| with cotangent gb: v = s (I - g g^T) gb / |G|, and
//   x_bar += sum_i alpha_i k'_i (v - 2 lambda r_i (r_i . v)),  X_bar_i -= the i-th term,
//   alpha_bar_i += k'_i (r_i . v).
// Through alpha = A^{-1} 1 (A = K + Sigma = L L^T): b = A^{-1} alpha_bar (FP32 L^{-1} products with one
// FP64 refinement step against L), X_bar_i += sum_j 2 lambda K_ij (b_i alpha_j + b_j alpha_i)(x_i - x_j).
// Kernel 1 recomputes k' per (query, winner) tile and accumulates alpha_bar / X_bar per sample; kernel 2 runs
// once per touched cell.
#include "ksdf_internal.cuh"
#include "ksdf_small.cuh"

#include <algorithm>

namespace ksdf {

namespace {

constexpr int kTW = 128;  // queries per backward tile
constexpr float kLog2e = 1.4426950408889634f;

__device__ inline float ex2(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
__device__ __forceinline__ float sqrt_approx(float x) {
  float y;
  asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

__global__ void k_bw_count(const int32_t* winner, int64_t Q, int64_t G, int32_t* rank, int64_t* cnt, float* d_xq,
                           int dim, uint32_t* st) {
  const int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  int w = q < Q ? winner[q] : -1;
  if (w >= G) {
    atomicOr(st, ST_CAPACITY);
    w = -1;
  }
  const int r = warp_rank(cnt, w < 0 ? -1 : w);
  if (q >= Q) return;
  rank[q] = w < 0 ? -1 : r;
  if (w < 0)
    for (int j = 0; j < dim; ++j) d_xq[q * dim + j] = 0.f;
}

__global__ void k_bw_scatter(const int32_t* winner, const int32_t* rank, int64_t Q, int64_t G, const int64_t* off,
                             int32_t* sorted) {
  int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (q >= Q) return;
  int w = winner[q];
  if (w >= 0 && w < G && rank[q] >= 0) sorted[off[w] + rank[q]] = (int32_t)q;
}

__global__ void k_bw_tiles(const int64_t* cnt, const int64_t* off, const int64_t* toff, int64_t G, int4* tiles) {
  int64_t g = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (g >= G) return;
  int64_t c = cnt[g];
  for (int64_t t = 0; t * kTW < c; ++t)
    tiles[toff[g] + t] = make_int4((int)g, (int)(off[g] + t * kTW), (int)(c - t * kTW < kTW ? c - t * kTW : kTW), 0);
}

__global__ void k_ntiles_w(const int64_t* cnt, int64_t n, int64_t* nt) {
  int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) nt[i] = (cnt[i] + kTW - 1) / kTW;
}

// the same for a small batch in one CTA (ksdf_small.cuh); cnt holds zeros on entry
__global__ void __launch_bounds__(kSmallThreads) k_bw_group_small(const int32_t* winner, int Q, int64_t G, int64_t* cnt,
                                                                  float* d_xq, int dim, int32_t* sorted, int4* tiles,
                                                                  int64_t* tot, uint32_t* st) {
  __shared__ SmallSort s;
  for (int q = threadIdx.x; q < Q; q += kSmallThreads) {
    int w = winner[q];
    if (w >= G) {
      atomicOr(st, ST_CAPACITY);
      w = -1;
    }
    if (w < 0)
      for (int j = 0; j < dim; ++j) d_xq[(int64_t)q * dim + j] = 0.f;
    s.key[q] = w < 0 ? kEmptyKey : (uint64_t)w;
    s.idx[q] = q;
  }
  int gid[2];
  const int ng = small_group(s, Q, gid);
#pragma unroll
  for (int u = 0; u < 2; ++u) {
    const int i = 2 * threadIdx.x + u;
    if (i < Q) sorted[i] = s.idx[i];
  }
  const int nt = small_tiles(s, ng, kTW, [&](int g, int t0, int n) {
    const int b = s.start[g], c = s.start[g + 1] - b;
    const int w = (int)s.key[b];
    cnt[w] = c;
    for (int t = 0; t < n; ++t) tiles[t0 + t] = make_int4(w, b + t * kTW, min(c - t * kTW, kTW), 0);
  });
  if (threadIdx.x < 4) tot[threadIdx.x] = threadIdx.x == 0 ? nt : 0;
}

struct BwArgs {
  const int4* tiles;
  const int64_t* n_tiles;
  int* counter;
  const int32_t* sorted;
  const int64_t* ts_off;
  const int32_t* cell_n;
  const uint64_t* cell_key;
  const float4* mf4;
  const int32_t* mgid;
  const float4* mnrm;
  int has_normals;
  const int8_t* sign;
  const float* d_sdf;
  const float* d_grad;
  float* d_xq;
  float* d_x;
  double* abar;  // per member
};

// Per (winner, tile of up to kTW queries), two passes.
//  Pass 1, a thread per query: the forward recomputation around the nearest sample x_n -- with p = x - x_n and
//  delta_i = x_n - x_i (so r_i = x - x_i = p + delta_i) and the exponent relative to x_n (excess_sq):
//    f' = sum_i alpha_i k'_i (compensated),  D = sum_i alpha_i k'_i delta_i,  M = sum_i alpha_i k'_i delta_i delta_i^T,
//  hence G = sum_i alpha_i k'_i r_i = f' p + D and, for any v, H v = sum_i alpha_i k'_i r_i (r_i . v) =
//  f' (p.v) p + (p.v) D + p (D.v) + M v.  (Sums of r_i r_i^T would hold d^2 p p^T-sized entries whose product
//  with v -- orthogonal to the gradient -- cancels; the offsets delta_i are small.)  Then the cotangent scalars
//  fb = dL/df', v (from d grad) and
//    x_bar = -2 lambda (fb G + H v) + f' v
//  (the sum over samples of alpha_i k'_i (v - 2 lambda r_i (r_i . v)) folded into f' and H v), written out; the
//  query's fb, v, x_n and 2 p go to shared memory.
//  Pass 2, a thread per sample (and per group of queries when the cell is small): over the tile's queries,
//    alpha_bar_i += k'_i c,   X_bar_i += alpha_i k'_i (2 lambda c r_i - v),   c = fb + r_i . v,
//  accumulated in registers, then added once per sample to the global accumulators.
// A query whose f' <= 0 (the distance fallback) has fb = 0 and its term on the nearest sample added directly.
// With the Matern 3/2 kernel (u = -log f'/lambda + d, k'_i = (1 + lambda r_i) w_i, w_i = e^{-lambda (r_i - d)},
// grad k'_i = -lambda^2 w_i r_i): fb = -s d_sdf / (lambda f'), G = sum_i alpha_i w_i r_i, the gradient output's
// Jacobian sum_i alpha_i w_i (I - (lambda / |r_i|) r_i r_i^T), so that
//   x_bar = -lambda^2 fb G + f_w v - lambda H' v  (f_w = sum alpha_i w_i, H' = sum (alpha_i w_i / |r_i|) r_i r_i^T),
//   alpha_bar_i += fb k'_i + w_i (r_i . v),  X_bar_i += alpha_i w_i ((lambda^2 fb + lambda (r_i . v) / |r_i|) r_i - v).
//
// FP32 bound.  HASV, a cotangent of the gradient, is a template parameter: without one H v = 0, so pass 1 leaves M out and
// pass 2 the terms in v (46 of 61 operations per query and sample are left).  Pass 2 takes two queries per packed
// instruction.  Pass 1 does not: f' in two partial sums differs from the sequential sum in its last bits, which 1 / u
// magnifies without bound near the surface.  Measured without a gradient cotangent: 16,777,216 queries on cells of mean N 81,
// 4.07 -> 2.84 ms.
constexpr int kTQ = 128;  // backward tile: queries (pass 1) and threads
constexpr int kPair = 64;  // pairs of queries of a tile

// shared memory: the cell's samples [n_max]; the tile's queries as pairs (both queries' x, both queries' y): x y | z fb | wx wy | wz nx | ny nz (w = 2 (x - x_n)), then v0 v1 | v2 m where HASV or MATERN; [kTQ] group partial sums
__host__ __device__ constexpr int bq_rows(bool ext) { return ext ? 7 : 5; }
__host__ __device__ inline size_t bq_smem_bytes(int n_max, bool ext) {
  return sizeof(float4) * (size_t)(n_max + bq_rows(ext) * kPair + kTQ);
}

template <bool MATERN, bool HASV>
__global__ void __launch_bounds__(kTQ) k_bw_query(BwArgs a, const float* xq, Params p) {
  typedef unsigned long long u64;
  extern __shared__ __align__(16) float4 s_x[];
  __shared__ int s_tile;
  __shared__ float s_bh[3], s_bl[3];
  float4* s_q = s_x + p.n_max;
  float4* RED = s_q + bq_rows(HASV || MATERN) * kPair;
  const int tid = threadIdx.x;
  const float lam = (float)p.lambda;
  const float c1 = lam * kLog2e;
  const float tl = 2.f * lam;
  const u64 NC1 = f2pack(-c1, -c1), LAM = f2pack(lam, lam), ONE = f2pack(1.f, 1.f);
  const int64_t ntiles = *a.n_tiles;
  for (;;) {
    if (tid == 0) s_tile = atomicAdd(a.counter, 1);
    __syncthreads();
    const int t = s_tile;
    if (t >= ntiles) break;
    const int4 tile = a.tiles[t];
    const int g = tile.x;
    const int n = a.cell_n[g];
    const int64_t m0 = a.ts_off[g];
    for (int i = tid; i < n; i += kTQ) s_x[i] = __ldg(a.mf4 + m0 + i);
    if (tid == 0) {
      int cc[3];
      unpack_key(a.cell_key[g], cc[0], cc[1], cc[2]);
      for (int j = 0; j < 3; ++j) base_split(p.o[j], cc[j], p.h, s_bh[j], s_bl[j]);
    }
    __syncthreads();
    // ---- pass 1: a thread per query ----
    const int nq = tile.z;
    if (tid < nq) {
      const int q = a.sorted[tile.y + tid];
      float ql[3] = {0.f, 0.f, 0.f};
      for (int j = 0; j < p.dim; ++j) ql[j] = local32(xq[(int64_t)q * p.dim + j], s_bh[j], s_bl[j]);
      float m = INFINITY;
      int nn = 0;
      for (int i = 0; i < n; ++i) {
        const float4 v = s_x[i];
        const float dx = ql[0] - v.x, dy = ql[1] - v.y, dz = ql[2] - v.z;
        const float r2 = fmaf(dx, dx, fmaf(dy, dy, dz * dz));
        if (r2 < m) {
          m = r2;
          nn = i;
        }
      }
      const float4 xn = s_x[nn];
      const float px = ql[0] - xn.x, py = ql[1] - xn.y, pz = ql[2] - xn.z;
      const float wx = 2.f * px, wy = 2.f * py, wz = 2.f * pz;
      const float zmin = sqrtf(m);
      // f' (compensated); the gradient weights' sums fw, D (G = fw p + D); the Jacobian weights' sums fc, Dc, M
      // (RBF: the same weights; Matern: alpha_i w_i / |r_i|)
      float f = 0.f, comp = 0.f, fw = 0.f, D0 = 0.f, D1 = 0.f, D2 = 0.f;
      float fc = 0.f, C0 = 0.f, C1 = 0.f, C2 = 0.f;
      float M00 = 0.f, M01 = 0.f, M02 = 0.f, M11 = 0.f, M12 = 0.f, M22 = 0.f;
      for (int i = 0; i < n; ++i) {
        const float4 v = s_x[i];
        const float ax = v.x - xn.x, ay = v.y - xn.y, az = v.z - xn.z;  // -delta_i
        const float e = fmaf(ax, ax - wx, fmaf(ay, ay - wy, az * (az - wz)));
        float ak, aw, ac;
        if (MATERN) {
          const float r2 = m + e, z = r2 > 0.f ? r2 * rsqrtf(r2) : 0.f;
          const float den = z + zmin;
          const float y = den > 0.f ? fmaxf(e, 0.f) * __frcp_rn(den) : 0.f;
          aw = v.w * ex2(-c1 * y);
          ak = aw * fmaf(lam, z, 1.f);
          ac = HASV && z > 0.f ? aw * __frcp_rn(z) : 0.f;
        } else {
          ak = v.w * ex2(-c1 * e);
          aw = ak;
          ac = ak;
        }
        const float y = ak - comp;
        const float tt = f + y;
        comp = (tt - f) - y;
        f = tt;
        fw += aw;
        D0 -= aw * ax;
        D1 -= aw * ay;
        D2 -= aw * az;
        if (HASV) {
          const float bx = ac * ax, by = ac * ay, bz = ac * az;
          if (MATERN) {
            fc += ac;
            C0 -= bx;
            C1 -= by;
            C2 -= bz;
          }
          M00 = fmaf(bx, ax, M00);
          M01 = fmaf(bx, ay, M01);
          M02 = fmaf(bx, az, M02);
          M11 = fmaf(by, ay, M11);
          M12 = fmaf(by, az, M12);
          M22 = fmaf(bz, az, M22);
        }
      }
      f -= comp;
      if (!MATERN) {
        fw = f;  // the compensated sum
        fc = f;
        C0 = D0;
        C1 = D1;
        C2 = D2;
      }
      const float G0 = fmaf(fw, px, D0), G1 = fmaf(fw, py, D1), G2 = fmaf(fw, pz, D2);
      float s = 1.f;
      if (a.sign) {
        s = a.sign[q] < 0 ? -1.f : 1.f;
      } else if (p.sign_mode == 1 && a.has_normals) {
        const float4 nv = a.mnrm[m0 + nn];
        s = (nv.x * (ql[0] - xn.x) + nv.y * (ql[1] - xn.y) + nv.z * (ql[2] - xn.z)) >= 0.f ? 1.f : -1.f;
      }
      const float ub = s * a.d_sdf[q];
      float fb = 0.f;
      const bool fallback = !(f > 0.f);
      if (!fallback) {
        if (MATERN) {
          fb = fmaf(-logf(f), 1.f / lam, zmin) > 0.f ? -ub / (lam * f) : 0.f;
        } else {
          const float u2 = fmaf(-logf(f), 1.f / lam, m);
          fb = u2 > 0.f ? -ub / (2.f * lam * sqrtf(u2) * f) : 0.f;
        }
      }
      float v0 = 0.f, v1 = 0.f, v2 = 0.f;
      if (HASV) {
        const float gn = sqrtf(G0 * G0 + G1 * G1 + G2 * G2);
        if (gn > 0.f) {
          const float g0 = G0 / gn, g1 = G1 / gn, g2 = G2 / gn;
          const float b0 = a.d_grad[(int64_t)q * p.dim + 0], b1 = a.d_grad[(int64_t)q * p.dim + 1];
          const float b2 = p.dim == 3 ? a.d_grad[(int64_t)q * p.dim + 2] : 0.f;
          const float dot = g0 * b0 + g1 * b1 + g2 * b2;
          const float sc = s / gn;
          v0 = sc * (b0 - g0 * dot);
          v1 = sc * (b1 - g1 * dot);
          v2 = sc * (b2 - g2 * dot);
        }
      }
      // x_bar = -cg fb G + fw v - beta H v with H v = fc (p.v) p + (p.v) C + p (C.v) + M v; RBF cg = beta = 2 lambda,
      // Matern cg = lambda^2, beta = lambda (the 1/|r_i| is inside the weights of fc, C, M)
      const float cg = MATERN ? lam * lam : tl, beta = MATERN ? lam : tl;
      float xb0 = -cg * fb * G0, xb1 = -cg * fb * G1, xb2 = -cg * fb * G2;
      if (HASV) {
        const float pv = fmaf(px, v0, fmaf(py, v1, pz * v2)), cv = fmaf(C0, v0, fmaf(C1, v1, C2 * v2));
        const float fpv = fc * pv;
        const float hv0 = fmaf(fpv, px, fmaf(pv, C0, fmaf(px, cv, fmaf(M00, v0, fmaf(M01, v1, M02 * v2)))));
        const float hv1 = fmaf(fpv, py, fmaf(pv, C1, fmaf(py, cv, fmaf(M01, v0, fmaf(M11, v1, M12 * v2)))));
        const float hv2 = fmaf(fpv, pz, fmaf(pv, C2, fmaf(pz, cv, fmaf(M02, v0, fmaf(M12, v1, M22 * v2)))));
        xb0 = fmaf(-cg * fb, G0, fmaf(-beta, hv0, fw * v0));
        xb1 = fmaf(-cg * fb, G1, fmaf(-beta, hv1, fw * v1));
        xb2 = fmaf(-cg * fb, G2, fmaf(-beta, hv2, fw * v2));
      }
      if (fallback && m > 0.f) {
        // u = distance to the nearest sample: its own derivative, on the query and on that sample
        const float d = sqrtf(m);
        const float e0 = ub * (ql[0] - xn.x) / d, e1 = ub * (ql[1] - xn.y) / d, e2 = ub * (ql[2] - xn.z) / d;
        xb0 += e0;
        xb1 += e1;
        xb2 += e2;
        const int gid = a.mgid[m0 + nn];
        atomicAdd(&a.d_x[(int64_t)gid * p.dim + 0], -e0);
        atomicAdd(&a.d_x[(int64_t)gid * p.dim + 1], -e1);
        if (p.dim == 3) atomicAdd(&a.d_x[(int64_t)gid * p.dim + 2], -e2);
      }
      a.d_xq[(int64_t)q * p.dim + 0] = xb0;
      a.d_xq[(int64_t)q * p.dim + 1] = xb1;
      if (p.dim == 3) a.d_xq[(int64_t)q * p.dim + 2] = xb2;
      float* e = reinterpret_cast<float*>(s_q + (tid >> 1)) + (tid & 1);
      const float rec[10] = {ql[0], ql[1], ql[2], fb, wx, wy, wz, xn.x, xn.y, xn.z};
      // an odd last pair's second query repeats the first with cotangents of zero
      const bool twin = tid == nq - 1 && !(tid & 1);
#pragma unroll
      for (int k = 0; k < 10; ++k) {
        e[(k >> 1) * 4 * kPair + (k & 1) * 2] = rec[k];
        if (twin) e[(k >> 1) * 4 * kPair + (k & 1) * 2 + 1] = k == 3 ? 0.f : rec[k];
      }
      if (HASV || MATERN) {
        const float ext[4] = {v0, v1, v2, m};
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          e[(5 + (k >> 1)) * 4 * kPair + (k & 1) * 2] = ext[k];
          if (twin) e[(5 + (k >> 1)) * 4 * kPair + (k & 1) * 2 + 1] = k < 3 ? 0.f : m;
        }
      }
    }
    __syncthreads();
    // ---- pass 2: a thread per (sample, group of query pairs) ----
    const int nrep = n < kTQ ? kTQ / n : 1;  // query groups when the cell is small
    const int grp = tid / (n < kTQ ? n : kTQ);
    const int np = (nq + 1) >> 1;
    for (int i0 = 0; i0 < n; i0 += kTQ) {
      const int i = i0 + (n < kTQ ? tid - grp * n : tid);
      const bool act = grp < nrep && i < n;
      float ab = 0.f, X0 = 0.f, X1 = 0.f, X2 = 0.f;
      if (act) {
        const float4 xi = s_x[i];
        const u64 IX = f2pack(xi.x, xi.x), IY = f2pack(xi.y, xi.y), IZ = f2pack(xi.z, xi.z);
        const u64 TL = f2pack(tl, tl), L2 = f2pack(lam * lam, lam * lam);
        u64 AB = 0ull, Y0 = 0ull, Y1 = 0ull, Y2 = 0ull;  // X = (the factors that the queries share) Y
#pragma unroll 2
        for (int qq = grp; qq < np; qq += nrep) {
          const float4 s0 = s_q[qq], s1 = s_q[kPair + qq], s2 = s_q[2 * kPair + qq], s3 = s_q[3 * kPair + qq];
          const float4 s4 = s_q[4 * kPair + qq];
          const u64 r0 = f2sub(f2pack(s0.x, s0.y), IX), r1 = f2sub(f2pack(s0.z, s0.w), IY);
          const u64 r2 = f2sub(f2pack(s1.x, s1.y), IZ), FB = f2pack(s1.z, s1.w);
          const u64 ax = f2sub(IX, f2pack(s3.z, s3.w)), ay = f2sub(IY, f2pack(s4.x, s4.y));
          const u64 az = f2sub(IZ, f2pack(s4.z, s4.w));
          const u64 e = f2fma(ax, f2sub(ax, f2pack(s2.x, s2.y)),
                              f2fma(ay, f2sub(ay, f2pack(s2.z, s2.w)), f2mul(az, f2sub(az, f2pack(s3.x, s3.y)))));
          float4 s5 = {}, s6 = {};
          u64 rv = 0ull;
          if (HASV || MATERN) s6 = s_q[6 * kPair + qq];
          if (HASV) {
            s5 = s_q[5 * kPair + qq];
            rv = f2fma(r0, f2pack(s5.x, s5.y), f2fma(r1, f2pack(s5.z, s5.w), f2mul(r2, f2pack(s6.x, s6.y))));
          }
          u64 kw, t2;  // the weight w_i (RBF: k'_i) and the factor of r_i beside it
          if (MATERN) {
            const float2 es = f2unpack(e);
            const float ra = s6.z + es.x, rb = s6.w + es.y, ma = sqrtf(s6.z), mb = sqrtf(s6.w);
            const float za = ra > 0.f ? ra * rsqrtf(ra) : 0.f, zb = rb > 0.f ? rb * rsqrtf(rb) : 0.f;
            const float da = za + ma, db = zb + mb;
            const float ya = da > 0.f ? fmaxf(es.x, 0.f) * __frcp_rn(da) : 0.f;
            const float yb = db > 0.f ? fmaxf(es.y, 0.f) * __frcp_rn(db) : 0.f;
            const float2 ey = f2unpack(f2mul(NC1, f2pack(ya, yb)));
            kw = f2pack(ex2(ey.x), ex2(ey.y));
            const u64 c = f2mul(FB, f2fma(f2pack(za, zb), LAM, ONE));
            AB = f2fma(HASV ? f2add(c, rv) : c, kw, AB);
            t2 = f2mul(L2, FB);
            if (HASV) {
              const u64 iz = f2pack(za > 0.f ? __frcp_rn(za) : 0.f, zb > 0.f ? __frcp_rn(zb) : 0.f);
              t2 = f2fma(f2mul(LAM, rv), iz, t2);
            }
          } else {
            const float2 ee = f2unpack(f2mul(NC1, e));
            kw = f2pack(ex2(ee.x), ex2(ee.y));
            const u64 c = HASV ? f2add(rv, FB) : FB;
            AB = f2fma(kw, c, AB);
            t2 = HASV ? f2mul(TL, c) : c;  // (without v the factor 2 lambda waits for the end)
          }
          if (HASV) {
            const u64 nk = kw ^ 0x8000000080000000ull;
            const u64 kt = f2mul(kw, t2);
            Y0 = f2fma(kt, r0, f2fma(nk, f2pack(s5.x, s5.y), Y0));
            Y1 = f2fma(kt, r1, f2fma(nk, f2pack(s5.z, s5.w), Y1));
            Y2 = f2fma(kt, r2, f2fma(nk, f2pack(s6.x, s6.y), Y2));
          } else {
            const u64 kt = f2mul(kw, t2);
            Y0 = f2fma(kt, r0, Y0);
            Y1 = f2fma(kt, r1, Y1);
            Y2 = f2fma(kt, r2, Y2);
          }
        }
        const float2 a2 = f2unpack(AB), y0 = f2unpack(Y0), y1 = f2unpack(Y1), y2 = f2unpack(Y2);
        const float sc = HASV || MATERN ? xi.w : xi.w * tl;
        ab = a2.x + a2.y;
        X0 = sc * (y0.x + y0.y);
        X1 = sc * (y1.x + y1.y);
        X2 = sc * (y2.x + y2.y);
      }
      if (nrep > 1) {  // combine the query groups of each sample
        RED[tid] = make_float4(ab, X0, X1, X2);
        __syncthreads();
        if (grp == 0 && act)
          for (int r = 1; r < nrep; ++r) {
            const float4 o = RED[r * n + tid];
            ab += o.x;
            X0 += o.y;
            X1 += o.z;
            X2 += o.w;
          }
      }
      if (grp == 0 && act) {
        atomicAdd(&a.abar[m0 + i], (double)ab);
        const int gid = a.mgid[m0 + i];
        atomicAdd(&a.d_x[(int64_t)gid * p.dim + 0], X0);
        atomicAdd(&a.d_x[(int64_t)gid * p.dim + 1], X1);
        if (p.dim == 3) atomicAdd(&a.d_x[(int64_t)gid * p.dim + 2], X2);
      }
    }
    __syncthreads();
  }
}

// Per touched cell: b = A^{-1} alpha_bar.  b0 = L^{-T} L^{-1} alpha_bar with the FP32 L^{-1}; one step of
// iterative refinement against the FP64 factor, r = alpha_bar - L (L^T b0) (the only FP64 work, N^2
// FMAs), b = b0 + L^{-T} L^{-1} r; then the alpha-path X_bar terms in FP32.
//
// Every step is a chain of dependent loads and FMAs per thread.  With many cells touched the SM hides it behind other
// cells: 64 threads a cell and little shared memory, the factors read through the caches (cells above kBwSplitN apart,
// so that the others are not charged their shared memory).  A small batch (kSmallQ) touches a few dozen cells and
// waits for the slowest: 128 threads a cell, both factors copied to shared memory first with all loads in flight, up
// to kBwSmemN samples (copying in the large batches too took 8.9 instead of 3.9 ms for 61,000 cells: four to seven
// cells per SM in place of 32), and 256 threads above.  The terms through alpha take two samples per packed instruction.
// Measured: 61,000 cells 3.85 -> 2.80 ms, 512 queries' cells 151 -> 58 us.  Bound by load latency, the FP64 pipe at 36%.
constexpr int kBwSplitN = 128;
constexpr int kBwSmemN = 160;
// shared memory: [n] alpha_bar, [n] t, [n] b0 (double) | [n] rhs, [n] y, [n] b, then the samples' x, y, z, alpha
// (floats), n rounded up to 4 | staged: L^{-1} | L (double)
__host__ __device__ inline size_t bw_vec_bytes(int n) { return (size_t)52 * ((n + 3) & ~3); }
__host__ __device__ inline size_t bw_smem_bytes(int n, bool staged) {
  return bw_vec_bytes(n) + (staged ? 4 * (size_t)linv_blocked_size(n) + 8 * (size_t)tri_sz(n) : 0);
}

// the cells with queries in two lists of G ints, those of at most `bound` samples and the larger ones; cnt their lengths
__global__ void k_bw_cells(const int64_t* qcnt, const int32_t* cell_n, int64_t G, int bound, int32_t* list, int* cnt) {
  const int64_t g = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const int lane = threadIdx.x & 31;
  const bool hit = g < G && qcnt[g] != 0;
  const int cl = hit ? (cell_n[g] <= bound ? 0 : 1) : -1;
#pragma unroll
  for (int c = 0; c < 2; ++c) {
    const unsigned m = __ballot_sync(0xffffffffu, cl == c);
    if (m == 0) continue;
    int base = 0;
    if (lane == 0) base = atomicAdd(&cnt[c], __popc(m));
    base = __shfl_sync(0xffffffffu, base, 0);
    if (cl == c) list[c * G + base + __popc(m & ((1u << lane) - 1u))] = (int32_t)g;
  }
}

template <int NT>
__device__ __forceinline__ void linv_solve32(const float* Lb, int n, const float* rhs, float* y, float* out, bool add) {
  // y = L^{-1} rhs (rows over threads; 8 consecutive rows share a 32-byte sector per column)
  for (int j = threadIdx.x; j < n; j += NT) {
    const float* row = Lb + linv_block_off(j >> 3) + (j & 7);
    float a0 = 0.f, a1 = 0.f, a2 = 0.f, a3 = 0.f;  // four independent chains
    int i = 0;
#pragma unroll 2
    for (; i + 3 <= j; i += 4) {
      a0 = fmaf(row[i * 8], rhs[i], a0);
      a1 = fmaf(row[(i + 1) * 8], rhs[i + 1], a1);
      a2 = fmaf(row[(i + 2) * 8], rhs[i + 2], a2);
      a3 = fmaf(row[(i + 3) * 8], rhs[i + 3], a3);
    }
    for (; i <= j; ++i) a0 = fmaf(row[i * 8], rhs[i], a0);
    y[j] = (a0 + a1) + (a2 + a3);
  }
  __syncthreads();
  // out (+)= L^{-T} y (columns over threads; the 8 rows of a block at one column are contiguous)
  const int nb = (n + 7) >> 3;
  for (int i = threadIdx.x; i < n; i += NT) {
    float acc = 0.f;
#pragma unroll 2
    for (int R = i >> 3; R < nb; ++R) {
      const float4* v = reinterpret_cast<const float4*>(Lb + linv_block_off(R) + i * 8);
      const float4 l0 = v[0], l1 = v[1];
      const float* yy = y + 8 * R;
      const int rmax = min(8, n - 8 * R);
      const float lr[8] = {l0.x, l0.y, l0.z, l0.w, l1.x, l1.y, l1.z, l1.w};
#pragma unroll
      for (int r = 0; r < 8; ++r)
        if (r < rmax) acc = fmaf(lr[r], yy[r], acc);
    }
    out[i] = add ? out[i] + acc : acc;
  }
  __syncthreads();
}

struct BwCellArgs {
  const int32_t* list;  // the class's cells
  const int* count;
  const int64_t* ts_off;
  const int32_t* cell_n;
  const int64_t* chol_off;
  const double* chol64;
  const int64_t* linv_off;
  const float* linv32;
  const float4* mf4;
  const int32_t* mgid;
  const double* abar;
  float* d_x;
};

template <bool MATERN, bool SM, int NT>
__global__ void __launch_bounds__(NT) k_bw_cell(BwCellArgs a, Params p) {
  extern __shared__ __align__(16) unsigned char bwsm[];
  const int tid = threadIdx.x;
  const int count = *a.count;
  for (int e = blockIdx.x; e < count; e += gridDim.x) {
    const int g = a.list[e];
    const int n = a.cell_n[g], n4 = (n + 3) & ~3;
    const int64_t m0 = a.ts_off[g];
    double* sa = reinterpret_cast<double*>(bwsm);
    double* st = sa + n4;
    double* sbd = st + n4;
    float* srhs = reinterpret_cast<float*>(sbd + n4);
    float* sy = srhs + n4;
    float* sb = sy + n4;
    float* sx = sb + n4;  // x, y, z, alpha, n4 each
    const float* Lb = a.linv32 + a.linv_off[g];
    const double* L = a.chol64 + a.chol_off[g];
    if (SM) {
      float4* sl = reinterpret_cast<float4*>(bwsm + bw_vec_bytes(n));
      const int nl = (int)(linv_blocked_size(n) >> 2), T = (int)tri_sz(n);
      double* sd = reinterpret_cast<double*>(sl + nl);
      const float4* src = reinterpret_cast<const float4*>(Lb);
#pragma unroll 8
      for (int i = tid; i < nl; i += NT) sl[i] = src[i];
#pragma unroll 8
      for (int i = tid; i < T; i += NT) sd[i] = L[i];
      Lb = reinterpret_cast<const float*>(sl);
      L = sd;
    }
    for (int i = tid; i < n4; i += NT) {
      const float4 v = i < n ? a.mf4[m0 + i] : make_float4(0.f, 0.f, 0.f, 0.f);  // (padding: zero weight)
      sx[i] = v.x;
      sx[n4 + i] = v.y;
      sx[2 * n4 + i] = v.z;
      sx[3 * n4 + i] = v.w;
      if (i >= n) sb[i] = 0.f;
    }
    for (int i = tid; i < n; i += NT) {
      sa[i] = a.abar[m0 + i];
      srhs[i] = (float)sa[i];
    }
    __syncthreads();
    linv_solve32<NT>(Lb, n, srhs, sy, sb, false);  // b0
    for (int i = tid; i < n; i += NT) sbd[i] = (double)sb[i];  // converted once, not per FMA
    __syncthreads();
    // t = L^T b0: rows in lockstep, threads over columns k (coalesced row reads)
    for (int k0 = 0; k0 < n; k0 += NT) {
      const int k = k0 + tid;
      double c0 = 0.0, c1 = 0.0, c2 = 0.0, c3 = 0.0;  // four independent chains (DFMA latency ~64 cycles)
      // a warp walks rows from its first lane's column so that a row's loads coalesce; entries above the
      // diagonal (k > i) are not loaded and count as zero
      int i = k0 + (tid & ~31);
      if (k < n) {
        for (; i + 3 < n; i += 4) {
          c0 = fma(k <= i ? L[tri_sz(i) + k] : 0.0, sbd[i], c0);
          c1 = fma(k <= i + 1 ? L[tri_sz(i + 1) + k] : 0.0, sbd[i + 1], c1);
          c2 = fma(k <= i + 2 ? L[tri_sz(i + 2) + k] : 0.0, sbd[i + 2], c2);
          c3 = fma(k <= i + 3 ? L[tri_sz(i + 3) + k] : 0.0, sbd[i + 3], c3);
        }
        for (; i < n; ++i) c0 = fma(k <= i ? L[tri_sz(i) + k] : 0.0, sbd[i], c0);
        st[k] = (c0 + c1) + (c2 + c3);
      }
    }
    __syncthreads();
    // r = alpha_bar - L t (rows over threads)
    for (int i = tid; i < n; i += NT) {
      const double* Li = L + tri_sz(i);
      double c0 = sa[i], c1 = 0.0, c2 = 0.0, c3 = 0.0;
      int k = 0;
      for (; k + 3 <= i; k += 4) {
        c0 = fma(-Li[k], st[k], c0);
        c1 = fma(-Li[k + 1], st[k + 1], c1);
        c2 = fma(-Li[k + 2], st[k + 2], c2);
        c3 = fma(-Li[k + 3], st[k + 3], c3);
      }
      for (; k <= i; ++k) c0 = fma(-Li[k], st[k], c0);
      srhs[i] = (float)((c0 + c1) + (c2 + c3));
    }
    __syncthreads();
    linv_solve32<NT>(Lb, n, srhs, sy, sb, true);  // b = b0 + L^{-T} L^{-1} r
    const float c1 = (float)p.lambda * kLog2e;
    const float tl = 2.f * (float)p.lambda, cm = (float)(p.lambda * p.lambda);
    for (int i = tid; i < n; i += NT) {
      // two samples j per packed instruction (j == i adds zero: its offset is zero)
      const float bi = sb[i], ai = sx[3 * n4 + i];
      const unsigned long long XI = f2pack(sx[i], sx[i]), YI = f2pack(sx[n4 + i], sx[n4 + i]);
      const unsigned long long ZI = f2pack(sx[2 * n4 + i], sx[2 * n4 + i]);
      const unsigned long long BI = f2pack(bi, bi), AI = f2pack(ai, ai), NC1 = f2pack(-c1, -c1);
      const float cg = MATERN ? cm : tl;
      const unsigned long long CG = f2pack(cg, cg);
      unsigned long long S0 = 0ull, S1 = 0ull, S2 = 0ull;
      auto pair = [&](int e, int j) { return *reinterpret_cast<const unsigned long long*>(sx + e * n4 + j); };
#pragma unroll 2
      for (int j = 0; j < n4; j += 2) {
        const unsigned long long dx = f2sub(XI, pair(0, j)), dy = f2sub(YI, pair(1, j)), dz = f2sub(ZI, pair(2, j));
        const float2 r2 = f2unpack(f2fma(dx, dx, f2fma(dy, dy, f2mul(dz, dz))));
        // grad_{x_i} A_ij = -cg w_ij (x_i - x_j): RBF cg w = 2 lambda K_ij, Matern lambda^2 e^{-lambda r_ij}
        const float2 ev = f2unpack(f2mul(NC1, MATERN ? f2pack(sqrt_approx(r2.x), sqrt_approx(r2.y)) : f2pack(r2.x, r2.y)));
        const unsigned long long cw = f2mul(CG, f2pack(ex2(ev.x), ex2(ev.y)));
        const unsigned long long bj = *reinterpret_cast<const unsigned long long*>(sb + j);
        const unsigned long long cf = f2mul(cw, f2fma(BI, pair(3, j), f2mul(bj, AI)));
        S0 = f2fma(cf, dx, S0);
        S1 = f2fma(cf, dy, S1);
        S2 = f2fma(cf, dz, S2);
      }
      const float2 s0 = f2unpack(S0), s1 = f2unpack(S1), s2 = f2unpack(S2);
      const float X0 = s0.x + s0.y, X1 = s1.x + s1.y, X2 = s2.x + s2.y;
      const int gid = a.mgid[m0 + i];
      atomicAdd(&a.d_x[(int64_t)gid * p.dim + 0], X0);
      atomicAdd(&a.d_x[(int64_t)gid * p.dim + 1], X1);
      if (p.dim == 3) atomicAdd(&a.d_x[(int64_t)gid * p.dim + 2], X2);
    }
    __syncthreads();
  }
}

}  // namespace

ksdf_status run_backward(ksdf_ctx* c, const float* xq, int64_t Q, const int8_t* sign, const int32_t* winner,
                         const float* d_sdf, const float* d_grad, float* d_xq, float* d_x) {
  cudaStream_t st = c->stream;
  const Params& p = c->p;
  Model& m = c->m;
  const int64_t G = m.G;
  uint32_t* stw = ptr<uint32_t>(c->status_word);
  KSDF_CUDA(c, ensure(c->ws[WS_QRANK], sizeof(int32_t) * Q));
  KSDF_CUDA(c, ensure(c->ws[WS_QWSORT], sizeof(int32_t) * Q));
  KSDF_CUDA(c, ensure(c->ws[WS_CELLQ], sizeof(int64_t) * (4 * G + 8)));
  const int64_t max_tiles = Q / kTW + G + 1;
  KSDF_CUDA(c, ensure(c->ws[WS_TILE], sizeof(int4) * max_tiles));
  KSDF_CUDA(c, ensure(c->ws[WS_BW], sizeof(double) * (m.M + 1)));
  int32_t* rank = ptr<int32_t>(c->ws[WS_QRANK]);
  int32_t* sorted = ptr<int32_t>(c->ws[WS_QWSORT]);
  int64_t* cb = ptr<int64_t>(c->ws[WS_CELLQ]);
  int64_t *cnt = cb, *off = cb + G, *nt = cb + 2 * G, *toff = cb + 3 * G, *tot = cb + 4 * G;
  int* counter = reinterpret_cast<int*>(tot + 2);
  int4* tiles = ptr<int4>(c->ws[WS_TILE]);
  double* abar = ptr<double>(c->ws[WS_BW]);
  cudaEvent_t e_b = prof_begin(c), e0 = prof_begin(c);
  KSDF_CUDA(c, cudaMemsetAsync(cnt, 0, sizeof(int64_t) * G, st));
  KSDF_CUDA(c, cudaMemsetAsync(tot, 0, sizeof(int64_t) * 6, st));
  KSDF_CUDA(c, cudaMemsetAsync(abar, 0, sizeof(double) * (m.M + 1), st));
  if (Q <= kSmallQ) {
    launch(k_bw_group_small, 1, kSmallThreads, 0, st, winner, (int)Q, G, cnt, d_xq, p.dim, sorted, tiles, tot, stw);
  } else {
    launch(k_bw_count, ceil_div(Q, 256), 256, 0, st, winner, Q, G, rank, cnt, d_xq, p.dim, stw);
    launch(k_ntiles_w, ceil_div(G, 256), 256, 0, st, cnt, G, nt);
    const ScanJob jobs[2] = {{cnt, off, G, nullptr, nullptr, nullptr}, {nt, toff, G, &tot[0], nullptr, nullptr}};
    KSDF_CUDA(c, scan_i64(jobs, 2, c->ws[WS_SCAN], st));
    launch(k_bw_scatter, ceil_div(Q, 256), 256, 0, st, winner, rank, Q, G, off, sorted);
    launch(k_bw_tiles, ceil_div(G, 256), 256, 0, st, cnt, off, toff, G, tiles);
  }
  prof_end(c, e0, "backward.group");
  BwArgs a;
  a.tiles = tiles;
  a.n_tiles = &tot[0];
  a.counter = counter;
  a.sorted = sorted;
  a.ts_off = ptr<int64_t>(m.ts_off);
  a.cell_n = ptr<int32_t>(m.n);
  a.cell_key = ptr<uint64_t>(m.key);
  a.mf4 = ptr<float4>(m.mf4);
  a.mgid = ptr<int32_t>(m.mgid);
  a.mnrm = m.has_normals ? ptr<float4>(m.mnrm) : nullptr;
  a.has_normals = m.has_normals ? 1 : 0;
  a.sign = sign;
  a.d_sdf = d_sdf;
  a.d_grad = d_grad;
  a.d_xq = d_xq;
  a.d_x = d_x;
  a.abar = abar;
  const bool matern = p.kernel == KSDF_KERNEL_MATERN32;
  const size_t smem = bq_smem_bytes(p.n_max, matern || d_grad);
  auto kq = matern ? (d_grad ? k_bw_query<true, true> : k_bw_query<true, false>)
                   : (d_grad ? k_bw_query<false, true> : k_bw_query<false, false>);
  KSDF_CUDA(c, cudaFuncSetAttribute(kq, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
  int occ = 0;
  KSDF_CUDA(c, cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, kq, kTQ, smem));
  e0 = prof_begin(c);
  launch(kq, std::max(1, occ) * c->num_sms, kTQ, smem, st, a, xq, p);
  prof_end(c, e0, "backward.query");
  e0 = prof_begin(c);
  // two size classes, the larger cells beside the others on an auxiliary stream; their lists take the place of the tile
  // counts and offsets, which are done with
  const bool small = Q <= kSmallQ;
  int32_t* list = reinterpret_cast<int32_t*>(nt);
  int* ccnt = reinterpret_cast<int*>(tot + 4);
  const int maxn = std::max(m.max_n, 1), bound = std::min(maxn, small ? kBwSmemN : kBwSplitN);
  launch(k_bw_cells, ceil_div(G, 256), 256, 0, st, cnt, ptr<int32_t>(m.n), G, bound, list, ccnt);
  const bool two = maxn > bound;
  if (two) KSDF_CUDA(c, fork_streams(c, 1));
  for (int part = two ? 1 : 0; part >= 0; --part) {
    const bool sm = small && part == 0;
    const size_t smem2 = bw_smem_bytes(part == 0 ? bound : maxn, sm);
    const int threads = !small ? 64 : sm ? 128 : 256;
    auto kc = !small ? (matern ? k_bw_cell<true, false, 64> : k_bw_cell<false, false, 64>)
              : sm   ? (matern ? k_bw_cell<true, true, 128> : k_bw_cell<false, true, 128>)
                     : (matern ? k_bw_cell<true, false, 256> : k_bw_cell<false, false, 256>);
    KSDF_CUDA(c, cudaFuncSetAttribute(kc, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem2));
    int occ2 = 0;
    KSDF_CUDA(c, cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ2, kc, threads, smem2));
    BwCellArgs ca;
    ca.list = list + part * G;
    ca.count = ccnt + part;
    ca.ts_off = ptr<int64_t>(m.ts_off);
    ca.cell_n = ptr<int32_t>(m.n);
    ca.chol_off = ptr<int64_t>(m.chol_off);
    ca.chol64 = ptr<double>(m.chol64);
    ca.linv_off = ptr<int64_t>(m.linv_off);
    ca.linv32 = ptr<float>(m.linv32);
    ca.mf4 = ptr<float4>(m.mf4);
    ca.mgid = ptr<int32_t>(m.mgid);
    ca.abar = abar;
    ca.d_x = d_x;
    const int64_t grid2 = std::min<int64_t>(std::min<int64_t>(G, Q), (int64_t)std::max(1, occ2) * c->num_sms);
    launch(kc, (unsigned)grid2, threads, smem2, part == 0 ? st : c->aux[0], ca, p);
  }
  if (two) KSDF_CUDA(c, join_streams(c, 1));
  KSDF_CUDA(c, cudaGetLastError());
  prof_end(c, e0, "backward.cell");
  prof_end(c, e_b, "backward");
  return KSDF_OK;
}

}  // namespace ksdf
