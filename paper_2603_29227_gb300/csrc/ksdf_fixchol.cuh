// ksdf_fixchol.cuh -- the Cholesky factorisation and the forward solve of the fit in 64-bit fixed point on the integer
// pipe, and the backward solve (included by ksdf_fit.cu).
//
// Why: an SM of this part retires 2.0 FP64 FMA lanes per cycle but 32 lanes of 32 x 32 + 64 -> 64-bit integer
// multiply-add (measured: 0.63 and 10.0 T/s at 2070 MHz), and a GP's kernel matrix is the friendliest input fixed point can have: A = K + diag(s^2)
// has a diagonal in [1, 1.25] and every entry of A, of its Schur complements and of L bounded by sqrt(1.25).  An FMA
// on 57 fractional bits takes three integer multiply-adds, so the pipe's bound is five times the FP64 pipe's, and the
// absolute rounding (2^-58 per entry of L, 2^-60 per sum) is below binary64's on these numbers: against extended precision
// alpha's largest relative error is 0.76 to 1.02 of the binary64 factorisation's (geometric means over 24 to 119 cells of
// each of six maps; one of them above 1), L's root mean square error 0.92 to 0.99 (both carry the kernel entries'
// rounding).
// Measured (with the L^-1 kernels that run beside it): 81,700 cells of mean N 80, 29.3 -> 19.0 ms; 865 cells of mean N
// 473, 48.6 -> 12.4 ms; a stream frame with a tenth of its cells at N = 256, 34.4 -> 8.3 ms.  What bounds it now: in the
// largest class the multiply-adds (their pipe is 55% busy) and the two barriers around the panel's 8 x 8 block; in the teams
// below the barriers; in the one-warp class the latency of the block's serial columns, at 7 to 8 warps per SM.
//
// Numbers.  "Q57 pair": v = h 2^27 + l with |l| <= 2^26 (two int32), value v 2^-57: L, y.  "Q60": int64, value 2^-60:
// A, sums.  The product of two pairs is h h' 2^54 + (h l' + l h') 2^27 + l l' in units of 2^-114, i.e. h h' in Q60
// plus (h l' + l h') >> 27; l l' < 2^-62 is dropped.  Sums of h h' are bounded by the Cauchy-Schwarz inequality
// (sum_k L_ik L_jk <= sqrt(A_ii A_jj)), so they fit an int64 for every N; the cross terms are folded every 16 columns
// (each below 2^57.2, 32 of them plus the panel's own 14 below 2^63).
//
// Eligibility (k_order_keys): every sigma_i^2 in [2^-20, 0.25].  Then lambda_min(A) >= 2^-20, so the factorisation
// cannot fail (in binary64 neither: N^2 2^-53 is far below 2^-20) and every pivot is at least 2^-20.  Other cells
// take the binary64 factorisation (k_fit).  y = L^-1 1 is formed along with L, held times 2^-2: |y_i| is the standard
// score of a label 1 given the earlier samples', hardly ever above 1 (a kernel without negative values).  While every
// |y_i| is below 1, sums of L_ik y_k 2^-2 are below sqrt(1.25 N) / 4 < 2^3 and fit; a cell where one reaches 1 gets its
// y from the binary64 solve of k_alpha, which also solves L^T alpha = y.
#pragma once
#include "ksdf_internal.cuh"

namespace ksdf {
namespace {

constexpr float kFxMinVar = 0x1p-20f, kFxMaxVar = 0.25f;
constexpr int kFxYs = 2;  // y is held times 2^-kFxYs

// Storage of the pairs: panels of 8 columns; panel p holds rows 8p .. N8 - 1 (N8 = N rounded up to 8), column-major
// with a column stride of N8 - 8p + 2 pairs: a warp's 32 consecutive rows of a column are conflict-free, the 8 rows
// of a later panel are 64 contiguous bytes on a 16-byte boundary (read as broadcasts), and the stride's +2 spreads
// the rows' walk along k (output) over the banks.
__host__ __device__ inline int fx_n8(int n) { return (n + 7) & ~7; }
__host__ __device__ inline int fx_panel_off(int n8, int p) { return 8 * p * (n8 + 2) - 32 * p * (p - 1); }
__host__ __device__ inline int64_t fx_elems(int n) { return fx_panel_off(fx_n8(n), fx_n8(n) / 8); }
// shared memory of a team: the pairs, or (when they live in a global slot) the staged rows of a panel; then the
// partial sums of the warps that share a group's columns
__host__ __device__ inline size_t fx_team_red_off(int np, bool smem_mat) {
  return (8 * (size_t)(smem_mat ? fx_elems(np + 1) : 8 * fx_n8(np + 1)) + 15) & ~(size_t)15;
}
__host__ __device__ inline size_t fx_team_smem(int np, bool smem_mat, int warps) {
  return fx_team_red_off(np, smem_mat) + (warps >= 7 ? (size_t)warps * 8 * 32 * (8 + 4) : 0);
}

__device__ __forceinline__ long long fx_mad(int a, int b, long long c) {
  // (a product and a sum in one asm statement: with mad.wide.s32 in it the factorisation of 81,700 cells of mean N 80 took
  // 17.5 instead of 17.0 ms, with C++ arithmetic 18.6; of 865 cells of mean N 473 13.9 and 14.8 instead of 13.8)
  long long r;
  asm("{.reg .s64 t; mul.wide.s32 t, %1, %2; add.s64 %0, t, %3;}" : "=l"(r) : "r"(a), "r"(b), "l"(c));
  return r;
}
__device__ __forceinline__ long long fx_mul(int a, int b) {
  long long r;
  asm("mul.wide.s32 %0, %1, %2;" : "=l"(r) : "r"(a), "r"(b));
  return r;
}
__device__ __forceinline__ long long fx_join(int2 p) { return ((long long)p.x << 27) + p.y; }

// v 2^(x - 57) as binary64, round to nearest (ties up in magnitude)
__device__ __forceinline__ double fx_to_double(long long v, int x) {
  if (v == 0) return 0.0;
  const unsigned long long u = v < 0 ? (unsigned long long)(-v) : (unsigned long long)v;
  const int z = __clzll((long long)u);
  const unsigned long long m = u << z;
  const unsigned long long mant = (m >> 11) + ((m >> 10) & 1ull);
  const unsigned long long b = ((unsigned long long)(63 - z - 57 + x + 1022) << 52) + mant;  // the carry moves on
  return __longlong_as_double((long long)(b | ((unsigned long long)v & (1ull << 63))));
}
// binary64 in [0, 2) -> Q60, truncated below 2^-60
__device__ __forceinline__ long long fx_from_double(double d) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(d);
  const int e = (int)(b >> 52) - 1023;
  if (e < -61) return 0;
  const unsigned long long m = (b & 0xFFFFFFFFFFFFFull) | (1ull << 52);
  const int s = e + 8;
  return (long long)(s >= 0 ? m << s : m >> (-s));
}

// 1 / sqrt(d) of a pivot d (Q60, 2^-20 <= d <= 1.25): D 2^-60 2^s2 with D in [2^59, 2^60].  An FP32 seed Y 2^-24 of
// the normalised d' = d 2^(2 s2) in [1, 4), e = 1 - d' y0^2 exactly in integers (units of 2^-64), and the
// second-order correction y0 (1 + e/2 + 3 e^2/8): |e| < 2^-21, so the next term is below 2^-64.
__device__ __forceinline__ int2 fx_rsqrt(long long d, int& s2) {
  const int s = (__clzll(d) - 2) & ~1;
  s2 = s >> 1;
  const unsigned long long dn = (unsigned long long)d << s;
  float y0;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y0) : "f"((float)(int)(dn >> 31) * 0x1p-29f));
  const unsigned Y = __float2uint_rn(y0 * 0x1p24f);
  const unsigned long long Y2 = (unsigned long long)Y * Y;
  const unsigned long long plo = dn * Y2, phi = __umul64hi(dn, Y2);
  const long long E = -(long long)((phi << 20) | (plo >> 44));
  const int e1 = (int)(E >> 16);
  const long long e2 = fx_mul(e1, e1) >> 32;
  const long long w = (E >> 1) + ((3 * e2) >> 3);
  const long long y = ((long long)Y << 36) + (fx_mul((int)Y, (int)(w >> 32)) << 4) +
                      (long long)(((unsigned long long)Y * (unsigned)w) >> 28);
  return make_int2((int)(y >> 31), (int)y & 0x7fffffff);
}

// t / L_jj (t in Q60) as a Q57 pair: (t 2^s2) (D 2^-60), |t| 2^s2 < 2^61.2; both factors split at 2^31, so the
// product is th Dh 2^62 + (th Dl + tl Dh) 2^31 (Q120), i.e. Q58 after dropping 62 bits, rounded to Q57
__device__ __forceinline__ int2 fx_scale(long long t, int2 D, int s2) {
  const long long tn = t << s2;
  const int th = (int)(tn >> 31), tl = (int)tn & 0x7fffffff;
  const long long q = fx_mad(th, D.x, fx_mad(tl, D.x, fx_mul(th, D.y)) >> 31);
  const int h = (int)((q + (1ll << 27)) >> 28);
  return make_int2(h, ((int)q - (int)((unsigned)h << 28) + 1) >> 1);
}

struct FixArgs {
  const uint32_t* order;  // this launch takes order[first .. first + count)
  int64_t first, count;
  int* counter;
  const int32_t* n32;
  const int64_t* ts_off;
  const int64_t* chol_off;
  D4* md4;         // .w receives y (NaN in the first member's when k_alpha has to form it)
  double* chol64;  // holds A in Q60 (int64) on entry (k_kmat), L in binary64 on return
  int2* gscr;      // per-CTA global slot (largest class)
  int64_t gstride;
  int np;
};

// L as packed binary64 rows: thread t of nt takes the entries t, t + nt, ... (consecutive threads, consecutive entries)
__device__ __forceinline__ void fx_write_l(const int2* Ls, int n8, int N, int t, int nt, double* Lg) {
  const int T = (int)tri_sz(N);
  int i = t < T ? tri_row(t) : 0;
  int k = t - (int)tri_sz(i);
  for (int e = t; e < T; e += nt) {
    const int k0 = k & ~7;
    Lg[e] = fx_to_double(fx_join(Ls[fx_panel_off(n8, k >> 3) + (k - k0) * (n8 - k0 + 2) + (i - k0)]), 0);
    k += nt;
    while (k > i) {
      k -= i + 1;
      ++i;
    }
  }
}

// whether an entry of row N (t = its sum in Q60, v the entry) left the range |y_i| < 1, i.e. 2^-kFxYs
__device__ __forceinline__ bool fx_y_out(long long t, int s2, int2 v) {
  return (t >> (60 - s2)) != (t >> 63) || abs(v.x) >= 1 << (30 - kFxYs);
}

// One panel of a cell owned by one warp: a lane holds NS rows kb + lane + 32 s of the rows kb .. N (row N is the
// right-hand side, ones times 2^-kFxYs, which becomes y).  The gather reads the panel rows' pairs once for all NS
// rows; the pivots and the panel's multipliers go through shuffles, and all rows take the eight columns together.
// Returns whether a y_i reached 1.
template <int NS>
__device__ __forceinline__ bool fx_panel(int2* Ls, const long long* A, int N, int n8, int kb) {
  constexpr unsigned FULL = 0xffffffffu;
  const int lane = threadIdx.x & 31;
  const int p = kb >> 3, nc = min(8, N - kb);
  long long HH[NS][8], MI[NS][8], T[NS][8];
#pragma unroll
  for (int s = 0; s < NS; ++s) {
    const int i = kb + lane + 32 * s;
    const long long* Ai = A + tri_sz(min(i, N - 1)) + kb;
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      T[s][j] = i >= N ? 1ll << (60 - kFxYs) : (j < nc && kb + j <= i ? Ai[j] : 0ll);
      HH[s][j] = 0;
      MI[s][j] = 0;
    }
  }
  const int2* own = Ls + kb + lane;  // row kb + lane of the columns, one after another (panel q starts at row 8 q)
  const int last = n8 - 1 - kb - lane;
  for (int q = 0; q < p; ++q) {
    const int cq = n8 - 8 * q + 2;
#pragma unroll 2
    for (int c = 0; c < 8; ++c) {
      int2 o[NS];
#pragma unroll
      for (int s = 0; s < NS; ++s) o[s] = own[min(32 * s, last)];
      const int4* p4 = reinterpret_cast<const int4*>(own - lane);
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int4 v = p4[u];
#pragma unroll
        for (int s = 0; s < NS; ++s) {
          HH[s][2 * u] = fx_mad(o[s].x, v.x, HH[s][2 * u]);
          HH[s][2 * u + 1] = fx_mad(o[s].x, v.z, HH[s][2 * u + 1]);
          MI[s][2 * u] = fx_mad(o[s].x, v.y, MI[s][2 * u]);
          MI[s][2 * u + 1] = fx_mad(o[s].x, v.w, MI[s][2 * u + 1]);
          MI[s][2 * u] = fx_mad(o[s].y, v.x, MI[s][2 * u]);
          MI[s][2 * u + 1] = fx_mad(o[s].y, v.z, MI[s][2 * u + 1]);
        }
      }
      own += cq;
    }
    own -= 8;  // the next panel's columns start 8 rows further down
    if (q & 1) {
#pragma unroll
      for (int s = 0; s < NS; ++s)
#pragma unroll
        for (int j = 0; j < 8; ++j) {
          HH[s][j] += MI[s][j] >> 27;
          MI[s][j] &= (1 << 27) - 1;
        }
    }
  }
  const int cs = n8 - kb + 2;
  int2* Lp = Ls + fx_panel_off(n8, p) + lane;
  bool bad = false;
#pragma unroll
  for (int j = 0; j < 8; ++j) {
    if (j < nc) {
      long long t[NS];
#pragma unroll
      for (int s = 0; s < NS; ++s) t[s] = T[s][j] - (HH[s][j] + (MI[s][j] >> 27));
      int s2;
      const int2 D = fx_rsqrt(__shfl_sync(FULL, t[0], j), s2);
      int2 v[NS];
#pragma unroll
      for (int s = 0; s < NS; ++s) {
        v[s] = fx_scale(t[s], D, s2);
        if (kb + lane + 32 * s < n8 && (s > 0 || lane >= j)) Lp[j * cs + 32 * s] = v[s];
        if (s == NS - 1) bad |= kb + lane + 32 * s == N && fx_y_out(t[s], s2, v[s]);
      }
#pragma unroll
      for (int k = j + 1; k < 8; ++k) {
        const int bh = __shfl_sync(FULL, v[0].x, k), bl = __shfl_sync(FULL, v[0].y, k);
#pragma unroll
        for (int s = 0; s < NS; ++s) {
          HH[s][k] = fx_mad(v[s].x, bh, HH[s][k]);
          MI[s][k] = fx_mad(v[s].x, bl, MI[s][k]);
          MI[s][k] = fx_mad(v[s].y, bh, MI[s][k]);
        }
      }
    }
  }
  return bad;
}

// The fixed-point factorisation of cells of N <= 95 samples, one warp per cell (persistent): left-looking in panels
// of 8 columns, up to three rows per lane.  Shared memory holds few cells per SM (seven of N = 80), so a warp's
// instruction-level parallelism has to fill the pipes: several rows per lane give independent chains, share the
// panel rows' loads and need no barrier.
constexpr int kFxOneN = 95;
__global__ void __launch_bounds__(32, 8) k_fit_fx1(FixArgs a) {
  extern __shared__ __align__(16) unsigned char fxsm[];
  int2* Ls = reinterpret_cast<int2*>(fxsm);
  const int lane = threadIdx.x & 31;
  for (;;) {
    int w = 0;
    if (lane == 0) w = atomicAdd(a.counter, 1);
    w = __shfl_sync(0xffffffffu, w, 0);
    if (w >= a.count) break;
    const int g = (int)a.order[a.first + w];
    const int N = a.n32[g], n8 = fx_n8(N + 1);
    const int64_t m0 = a.ts_off[g];
    double* Ag = a.chol64 + a.chol_off[g];
    const long long* A = reinterpret_cast<const long long*>(Ag);
    bool bad = false;
    for (int kb = 0; kb < N; kb += 8) {
      const int rows = N + 1 - kb;
      if (rows > 64) bad |= fx_panel<3>(Ls, A, N, n8, kb);
      else if (rows > 32) bad |= fx_panel<2>(Ls, A, N, n8, kb);
      else bad |= fx_panel<1>(Ls, A, N, n8, kb);
      __syncwarp();
    }
    bad = __any_sync(0xffffffffu, bad);
    for (int i = lane; i < N; i += 32) {
      const int k0 = i & ~7;
      const double y = fx_to_double(fx_join(Ls[fx_panel_off(n8, i >> 3) + (i - k0) * (n8 - k0 + 2) + (N - k0)]), kFxYs);
      a.md4[m0 + i].w = i == 0 && bad ? (double)NAN : y;
    }
    fx_write_l(Ls, n8, N, lane, 32, Ag);
    __syncwarp();
  }
}

// Larger cells, one per iteration of a persistent team of W warps (one per 32 rows; the first panel of a cell with
// 32 W + 1 rows, row N included, has one group more).  Per panel: the sums over the finished columns are formed by
// groups of 32 rows, a lane per row; when the remaining rows leave warps free, nsp warps share a group's columns
// (teams of 7 and more, which have an SM nearly to themselves).  Warp 0's group holds the panel's own rows and factors
// the 8 x 8 block; the others solve against it.  GM: the pairs live in a global slot (L2) and the panel
// rows, which every lane reads, are staged in shared memory.
// A share of the columns is handed over as its whole part and the 27 bits of its cross terms below it, so that the sum over
// the shares is exact and is cut to Q60 once: the factor does not depend on the team (with every share cut on its own, 4 to
// 15% of the entries differed in their last bit between teams of 5, 7 and 8).  Handing both over left the times as they
// were (fit and query of 150,000 densely scanned samples, cells of mean N 473: 24.2 and 24.1 ms).
template <int W, bool GM>
__global__ void __launch_bounds__(32 * W, W == 7 ? 1 : 16 / W) k_fit_fx(FixArgs a) {
  constexpr bool SPLIT = W >= 7;
  extern __shared__ __align__(16) unsigned char fxsm[];
  __shared__ int s_cell, s_bad;
  __shared__ int2 s_d[8];
  __shared__ int s_e[8];
  constexpr unsigned FULL = 0xffffffffu;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  int2* Ls = GM ? a.gscr + (int64_t)blockIdx.x * a.gstride : reinterpret_cast<int2*>(fxsm);
  long long* red = reinterpret_cast<long long*>(fxsm + fx_team_red_off(a.np, !GM));  // [W][8][32]: the shares' whole parts
  int* redl = reinterpret_cast<int*>(red + W * 8 * 32);                              // [W][8][32]: the bits below them
  int2* stage = reinterpret_cast<int2*>(fxsm);  // GM: [column][8] the panel's rows
  for (;;) {
    if (tid == 0) {
      const int w = atomicAdd(a.counter, 1);
      s_cell = w < a.count ? (int)a.order[a.first + w] : -1;
      s_bad = 0;
    }
    __syncthreads();
    const int g = s_cell;
    if (g < 0) break;
    const int N = a.n32[g], n8 = fx_n8(N + 1);
    const int64_t m0 = a.ts_off[g];
    double* Ag = a.chol64 + a.chol_off[g];
    bool bad = false;
    for (int kb = 0; kb < N; kb += 8) {
      const int p = kb >> 3, nc = min(8, N - kb);
      const int groups = (N + 1 - kb + 31) >> 5;
      int nsp = 1;
      while (SPLIT && groups * nsp * 2 <= W) nsp *= 2;
      const int part = SPLIT ? warp / groups : 0, gi = warp - part * groups;
      const bool act = SPLIT ? part < nsp : warp < groups;
      const int i = kb + 32 * gi + lane, ic = min(i, n8 - 1);
      const int cs = n8 - kb + 2;
      int2* Lp = Ls + fx_panel_off(n8, p);
      long long HH[8], MI[8], T[8];
      if (act && part == 0) {
        const long long* Ai = reinterpret_cast<const long long*>(Ag) + tri_sz(min(i, N - 1)) + kb;
#pragma unroll
        for (int j = 0; j < 8; ++j)
          T[j] = i >= N ? 1ll << (60 - kFxYs) : (j < nc && kb + j <= i ? Ai[j] : 0ll);
      }
      if (GM) {
        for (int e = tid; e < 4 * kb; e += 32 * W) {
          const int k = e >> 2, k0 = k & ~7;
          reinterpret_cast<int4*>(stage)[e] = reinterpret_cast<const int4*>(
              Ls + fx_panel_off(n8, k >> 3) + (k - k0) * (n8 - k0 + 2) + (kb - k0))[e & 3];
        }
        __syncthreads();
      }
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        HH[j] = 0;
        MI[j] = 0;
      }
      if (act) {
        const int q0 = SPLIT ? part * p / nsp : 0, q1 = SPLIT ? (part + 1) * p / nsp : p;
        auto load = [&](int q, int2* o) {  // the lane's row of panel q's columns
          const int cq = n8 - 8 * q + 2;
          const int2* own = Ls + fx_panel_off(n8, q) + (ic - 8 * q);
#pragma unroll
          for (int c = 0; c < 8; ++c) o[c] = own[c * cq];
        };
        auto column = [&](int2 o, const int2* pan) {
          const int4* p4 = reinterpret_cast<const int4*>(pan);
#pragma unroll
          for (int u = 0; u < 4; ++u) {
            const int4 v = p4[u];
            HH[2 * u] = fx_mad(o.x, v.x, HH[2 * u]);
            HH[2 * u + 1] = fx_mad(o.x, v.z, HH[2 * u + 1]);
            MI[2 * u] = fx_mad(o.x, v.y, MI[2 * u]);
            MI[2 * u + 1] = fx_mad(o.x, v.w, MI[2 * u + 1]);
            MI[2 * u] = fx_mad(o.y, v.x, MI[2 * u]);
            MI[2 * u + 1] = fx_mad(o.y, v.z, MI[2 * u + 1]);
          }
        };
        int2 o[GM ? 8 : 1];
        if (GM && q0 < q1) load(q0, o);
        for (int q = q0; q < q1; ++q) {
          if (GM) {
            int2 on[8];
            if (q + 1 < q1) load(q + 1, on);  // ahead: the slot is in L2
#pragma unroll
            for (int c = 0; c < 8; ++c) column(o[c], stage + 64 * q + 8 * c);
#pragma unroll
            for (int c = 0; c < 8; ++c) o[c] = on[c];
          } else {
            const int cq = n8 - 8 * q + 2;
            const int2* pan = Ls + fx_panel_off(n8, q) + (kb - 8 * q);
#pragma unroll 2
            for (int c = 0; c < 8; ++c) column(pan[c * cq + (ic - kb)], pan + c * cq);
          }
          if (q & 1) {
#pragma unroll
            for (int j = 0; j < 8; ++j) {
              HH[j] += MI[j] >> 27;
              MI[j] &= (1 << 27) - 1;
            }
          }
        }
        if (SPLIT && part > 0)
#pragma unroll
          for (int j = 0; j < 8; ++j) {
            red[(warp * 8 + j) * 32 + lane] = HH[j] + (MI[j] >> 27);
            redl[(warp * 8 + j) * 32 + lane] = (int)MI[j] & ((1 << 27) - 1);
          }
      }
      if (SPLIT && nsp > 1) {
        __syncthreads();
        if (act && part == 0)
          for (int q = 1; q < nsp; ++q)
#pragma unroll
            for (int j = 0; j < 8; ++j) {
              HH[j] += red[((q * groups + gi) * 8 + j) * 32 + lane];
              MI[j] += redl[((q * groups + gi) * 8 + j) * 32 + lane];
            }
      }
      if (warp == 0) {
#pragma unroll
        for (int j = 0; j < 8; ++j) {
          if (j < nc) {
            const long long t = T[j] - (HH[j] + (MI[j] >> 27));
            int s2;
            const int2 D = fx_rsqrt(__shfl_sync(FULL, t, j), s2);
            if (lane == 0) {
              s_d[j] = D;
              s_e[j] = s2;
            }
            const int2 v = fx_scale(t, D, s2);
            if (lane >= j && i < n8) Lp[j * cs + lane] = v;
            if (GM && lane < 8) stage[8 * (kb + j) + lane] = v;
            bad |= i == N && fx_y_out(t, s2, v);
#pragma unroll
            for (int k = j + 1; k < 8; ++k) {
              const int bh = __shfl_sync(FULL, v.x, k), bl = __shfl_sync(FULL, v.y, k);
              HH[k] = fx_mad(v.x, bh, HH[k]);
              MI[k] = fx_mad(v.x, bl, MI[k]);
              MI[k] = fx_mad(v.y, bh, MI[k]);
            }
          }
        }
      }
      __syncthreads();
      for (int gg = warp; gg < groups; gg += W) {  // (then the panel is full: 8 columns)
        if (gg == 0) continue;
        const int r = kb + 32 * gg + lane;
        if (gg >= W) {  // kb == 0: nothing to subtract
          const long long* Ai = reinterpret_cast<const long long*>(Ag) + tri_sz(min(r, N - 1));
#pragma unroll
          for (int j = 0; j < 8; ++j) {
            T[j] = r >= N ? 1ll << (60 - kFxYs) : Ai[j];
            HH[j] = 0;
            MI[j] = 0;
          }
        }
#pragma unroll
        for (int j = 0; j < 8; ++j) {
          const long long t = T[j] - (HH[j] + (MI[j] >> 27));
          const int s2 = s_e[j];
          const int2 v = fx_scale(t, s_d[j], s2);
          if (r < n8) Lp[j * cs + (r - kb)] = v;
          bad |= r == N && fx_y_out(t, s2, v);
#pragma unroll
          for (int k = j + 1; k < 8; ++k) {
            const int2 b = GM ? stage[8 * (kb + j) + k] : Lp[j * cs + k];
            HH[k] = fx_mad(v.x, b.x, HH[k]);
            MI[k] = fx_mad(v.x, b.y, MI[k]);
            MI[k] = fx_mad(v.y, b.x, MI[k]);
          }
        }
      }
      __syncthreads();
    }
    if (bad) s_bad = 1;
    __syncthreads();
    for (int i = tid; i < N; i += 32 * W) {
      const int k0 = i & ~7;
      const double y = fx_to_double(fx_join(Ls[fx_panel_off(n8, i >> 3) + (i - k0) * (n8 - k0 + 2) + (N - k0)]), kFxYs);
      a.md4[m0 + i].w = i == 0 && s_bad ? (double)NAN : y;
    }
    fx_write_l(Ls, n8, N, tid, 32 * W, Ag);
    __syncthreads();
  }
}

struct AlphaArgs {
  const uint32_t* order;  // cells order[first .. first + count)
  int64_t first, count;
  const int32_t* n32;
  const int64_t* ts_off;
  const int64_t* chol_off;
  D4* md4;
  float4* mf4;
  const double* chol64;
};

// alpha = L^-T y in binary64, a warp per cell of N <= 32 NR samples: lane l holds the unknowns l, l + 32, ... in
// registers and the rows of L stream by from the last (contiguous, independent of the chain, so loaded ahead).  A
// kernel of its own: this chain of N dependent steps would idle the factorisation's CTAs, of which shared memory
// allows few, while here every SM holds dozens of them.  A cell whose y the factorisation could not hold (NaN) gets
// it here first, by dot products.
constexpr int kAlphaWarps = 4;
template <int NR>
__global__ void __launch_bounds__(32 * kAlphaWarps) k_alpha(AlphaArgs a) {
  constexpr unsigned FULL = 0xffffffffu;
  const int lane = threadIdx.x & 31;
  const int64_t w = (int64_t)blockIdx.x * kAlphaWarps + (threadIdx.x >> 5);
  if (w >= a.count) return;
  const int g = (int)a.order[a.first + w];
  const int N = a.n32[g];
  const int64_t m0 = a.ts_off[g];
  const double* L = a.chol64 + a.chol_off[g];
  double r[NR], d[NR];
#pragma unroll
  for (int j = 0; j < NR; ++j) {
    const int i = lane + 32 * j;
    r[j] = i < N ? a.md4[m0 + i].w : 0.0;
    d[j] = i < N ? 1.0 / L[tri_sz(i) + i] : 0.0;
  }
  if (__any_sync(FULL, r[0] != r[0])) {
    for (int k = 0; k < N; ++k) {
      const double* Lk = L + tri_sz(k);
      double s = 0.0;
#pragma unroll
      for (int j = 0; j < NR; ++j)
        if (lane + 32 * j < k) s = fma(Lk[lane + 32 * j], r[j], s);
#pragma unroll
      for (int o = 16; o; o >>= 1) s += __shfl_xor_sync(FULL, s, o);
#pragma unroll
      for (int j = 0; j < NR; ++j)
        if (lane + 32 * j == k) r[j] = (1.0 - s) * d[j];
    }
  }
#pragma unroll
  for (int j = NR - 1; j >= 0; --j) {
    const int mt = min(32, N - 32 * j);  // unknowns of this block (<= 0: none)
#pragma unroll(NR > 4 ? 2 : 4)
    for (int m = mt - 1; m >= 0; --m) {
      const double* Lk = L + tri_sz(32 * j + m);
      double l[NR];
#pragma unroll
      for (int q = 0; q < NR; ++q) l[q] = q < j || (q == j && lane < m) ? Lk[lane + 32 * q] : 0.0;
      const double ak = __shfl_sync(FULL, r[j] * d[j], m);
#pragma unroll
      for (int q = 0; q < NR; ++q)
        if (q <= j) r[q] = q == j && lane == m ? ak : fma(-l[q], ak, r[q]);
    }
  }
#pragma unroll
  for (int j = 0; j < NR; ++j) {
    const int i = lane + 32 * j;
    if (i < N) {
      a.md4[m0 + i].w = r[j];
      a.mf4[m0 + i].w = d2f_bits(r[j]);
    }
  }
}

}  // namespace
}  // namespace ksdf
