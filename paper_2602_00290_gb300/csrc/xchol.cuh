// Cholesky factor of an exact integer Gram matrix in 128-bit fixed point: R with R^T R = G, for the
// triangular factor of the merged core's columns (xgram.cuh).
//
// G comes as 192-bit integers.  Column c is scaled by 2^-s_c so that every diagonal entry lies in
// (1/4, 1], and the entries, Schur complements and rows of R (all at most 1 in magnitude) are held as
// signed 128-bit integers of unit 2^-125.  Absolute round-off stays near n 2^-125, so a column's
// remainder after the earlier columns is resolved down to about 2^-57 of its norm; a pivot below
// n 2^-118 is dead (the column is a combination of the earlier ones to that accuracy).  The pivot of a
// step is the remaining column of largest norm, so the rows of R come graded, which a one-sided Jacobi
// on R^T needs fewer sweeps for, and the factor ends where nothing is left.  128-bit integers rather than double-double: this part's FP64 pipe runs at 1/64 of
// the integer rate, and a double-double update (20 FP64 operations) would take 4 ms at 160 columns.
//
// Right-looking, one cluster: CTA r holds the columns i = r mod C (all rows), the pivot's row is
// exchanged through distributed shared memory, one cluster barrier per step.  Every CTA keeps all
// diagonals (r_p is known to all of them), so pivots and reciprocal square roots need no exchange; the
// next pivot's row is updated and sent first, the rest of the update and the next reciprocal square
// root run between the barrier's arrival and its wait.
#pragma once
#include "common.cuh"
#include "instr.cuh"

namespace ttk {

typedef unsigned __int128 u128;
typedef __int128 i128;

constexpr int kXcThreads = 512;
constexpr int kXcMaxN = 256;
constexpr int kXcMaxCluster = 8;

// floor(a b / 2^128) up to 2 units
__device__ __forceinline__ u128 mulhi128(u128 a, u128 b) {
  const unsigned long long a1 = (unsigned long long)(a >> 64), a0 = (unsigned long long)a;
  const unsigned long long b1 = (unsigned long long)(b >> 64), b0 = (unsigned long long)b;
  return (u128)a1 * b1 + __umul64hi(a1, b0) + __umul64hi(a0, b1);
}
// product of two magnitudes of unit 2^-125 (each at most 2^126)
__device__ __forceinline__ u128 mulq125(u128 a, u128 b) { return mulhi128(a << 2, b << 1); }
__device__ __forceinline__ u128 mag128(i128 x) { return x < 0 ? (u128)(-x) : (u128)x; }
__device__ __forceinline__ int clz128(u128 x) {
  const unsigned long long h = (unsigned long long)(x >> 64);
  return h ? __clzll((long long)h) : 64 + __clzll((long long)(unsigned long long)x);
}

// 1 / sqrt(v) in (1, 2], unit 2^-126, for v in [1/4, 1) of unit 2^-128: Newton steps y (3 - v y^2) / 2
// from the FP32 reciprocal square root, two in 64 bits (2^-22, 2^-43, 2^-56) and one in 128 (2^-111).
__device__ __forceinline__ u128 rsqrt128(u128 v) {
  const unsigned long long v64 = (unsigned long long)(v >> 64);  // unit 2^-64
  const float vf = (float)(unsigned)(v64 >> 32) * 2.3283064365386963e-10f;
  unsigned long long y = (unsigned long long)(rsqrtf(vf) * 1073741824.0f) << 32;  // unit 2^-62
#pragma unroll
  for (int it = 0; it < 2; ++it) {
    const unsigned long long t = __umul64hi(y, y);            // 2^-60
    const unsigned long long w = __umul64hi(t, v64);          // 2^-60
    y = __umul64hi(y, (3ull << 60) - w) << 3;                 // 2^-58 -> halved, 2^-62
  }
  const u128 y1 = (u128)y << 64;                              // 2^-126
  const u128 t = mulhi128(y1, y1);                            // 2^-124
  const u128 w = mulhi128(t, v);                              // 2^-124
  return mulhi128(y1, ((u128)3 << 124) - w) << 3;             // 2^-122 -> halved, 2^-126
}

__device__ __forceinline__ double to_double125(u128 m) {  // m 2^-125
  return __ull2double_rn((unsigned long long)(m >> 64)) * 4.3368086899420177e-19 +       // 2^-61
         __ull2double_rn((unsigned long long)m) * 2.3509887016445750e-38;                // 2^-125
}

__device__ __forceinline__ unsigned xc_cluster_rank() {
  unsigned r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ unsigned xc_cluster_size() {
  unsigned r;
  asm volatile("mov.u32 %0, %%cluster_nctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ void xc_arrive() { asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory"); }
__device__ __forceinline__ void xc_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }
// store a 128-bit value at the same shared-memory address of CTA `rank` of the cluster
__device__ __forceinline__ void xc_store_remote(i128* local, unsigned rank, i128 v) {
  unsigned a = (unsigned)__cvta_generic_to_shared(local), r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(rank));
  asm volatile("st.shared::cluster.v2.u64 [%0], {%1, %2};" ::"r"(r), "l"((unsigned long long)v),
               "l"((unsigned long long)((u128)v >> 64))
               : "memory");
}

// columns of a matrix of n per CTA of a cluster of C
__host__ __device__ inline int xc_cols(int n, int C) { return (n + C - 1) / C; }
inline size_t xchol_smem_bytes(int n, int C) { return sizeof(i128) * ((size_t)xc_cols(n, C) * n + 5 * (size_t)n); }
inline int xchol_cluster(int n) { return n <= 24 ? 1 : n <= 48 ? 2 : n <= 96 ? 4 : 8; }

// Shift right (left for negative sh) a 192-bit two's complement integer to 128 bits.
__device__ __forceinline__ i128 shift192(unsigned long long w0, unsigned long long w1, unsigned long long w2, int sh) {
  if (sh <= 0) return (i128)((((u128)w1 << 64) | w0) << (sh < -127 ? 127 : -sh));
  const i128 hi = ((i128)(long long)w2 << 64) | w1;  // words 2, 1
  if (sh >= 64) return sh >= 191 ? (hi < 0 ? (i128)-1 : (i128)0) : hi >> (sh - 64);
  return (i128)(((u128)hi << (64 - sh)) | (w0 >> sh));
}

// Pivot key of a remaining diagonal d (unit 2^-125) of a column with binary exponent `ex` of its squared
// scale: exponent, leading bits, position (so that equal keys resolve the same way in every CTA).
__device__ __forceinline__ unsigned xc_key(u128 d, int ex, int pos) {
  const int lz = clz128(d);
  int e = ex - lz + 2048;
  e = min(max(e, 1), 4095);
  const unsigned m = (unsigned)((d << lz) >> 116) & 0xfffu;  // leading bits
  return ((unsigned)e << 20) | (m << 8) | (unsigned)(255 - pos);
}

// gint: word planes of the upper triangle of G (row-major, n x n).  Rows k of R (n x n row-major, pivot
// order; zero beyond the rank) get r_kc 2^(s_c) coef_c 2^(U_c), U_c the unit exponent of column c's fixed
// point and coef_c its coefficient in the sum (nullable).
static __global__ void __launch_bounds__(kXcThreads) k_xg_chol(int n, const unsigned long long* __restrict__ gint,
                                                               const int* __restrict__ unit,
                                                               const double* __restrict__ coef,
                                                               double* __restrict__ R) {
  extern __shared__ __align__(16) unsigned char xc_smem[];
  __shared__ int act[kXcMaxN], sc[kXcMaxN], ex[kXcMaxN], order[kXcMaxN], piv[kXcMaxN], perm[2][kXcMaxN];
  __shared__ int wcount[kXcThreads / 32], na_s;
  __shared__ unsigned wkey[2][kXcMaxN / 32];
  const int C = (int)xc_cluster_size(), rank = (int)xc_cluster_rank();
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int ncl = xc_cols(n, C);
  const size_t plane = (size_t)n * n;
  i128* S = reinterpret_cast<i128*>(xc_smem);  // [ncl][n]: column lc C + rank; row of a finished pivot: r
  i128* rowbuf = S + (size_t)ncl * n;          // [2][n]: the exchanged row
  i128* rs = rowbuf + 2 * n;                   // [2][n]: its scaled form, a row of R
  i128* dg = rs + 2 * n;                       // [n]: remaining diagonals
  // columns with a nonzero diagonal, in order, and their scales
  {
    bool on = false;
    int scale = 0;
    if (tid < n) {
      const size_t o = (size_t)tid * n + tid;
      const unsigned long long w0 = gint[o], w1 = gint[plane + o], w2 = gint[2 * plane + o];
      const int len = w2 ? 192 - __clzll((long long)w2) : w1 ? 128 - __clzll((long long)w1) : 64 - __clzll((long long)w0);
      on = (w0 | w1 | w2) != 0ull;
      scale = (len + 1) >> 1;
    }
    const unsigned m = __ballot_sync(0xffffffffu, on);
    if (lane == 0) wcount[warp] = __popc(m);
    __syncthreads();
    int before = 0;
    for (int w = 0; w < warp; ++w) before += wcount[w];
    if (on) {
      const int i = before + __popc(m & ((1u << lane) - 1u));
      act[i] = tid;
      sc[i] = scale;
      int e = 0;
      if (coef) e = (int)((__double_as_longlong(coef[tid]) >> 52) & 0x7ff) - 1023;
      ex[i] = 2 * (scale + unit[tid] + e);
      perm[0][i] = i;
      order[i] = n;
    }
    if (tid == kXcThreads - 1) na_s = before + __popc(m);
    __syncthreads();
  }
  const int na = na_s;
  for (int lc = warp; lc < ncl; lc += kXcThreads / 32) {
    const int i = lc * C + rank;
    if (i >= na) continue;
    for (int p = lane; p < na; p += 32) {
      const int u = p < i ? p : i, v = p < i ? i : p;
      const size_t o = (size_t)act[u] * n + act[v];
      S[(size_t)lc * n + p] = shift192(gint[o], gint[plane + o], gint[2 * plane + o], sc[p] + sc[i] - 125);
    }
  }
  const i128 thr = (i128)n << 7;  // n 2^-118
  // key exponents relative to the largest column
  int exmax = -(1 << 30);
  for (int i = lane; i < na; i += 32) exmax = max(exmax, ex[i]);
  exmax = __reduce_max_sync(0xffffffffu, exmax);
  if (tid < kXcMaxN) {
    unsigned key = 0;
    if (tid < na) {
      const size_t o = (size_t)act[tid] * n + act[tid];
      const i128 d = shift192(gint[o], gint[plane + o], gint[2 * plane + o], 2 * sc[tid] - 125);
      dg[tid] = d;
      key = d > thr ? xc_key((u128)d, ex[tid] - exmax, tid) : 0u;
    }
    key = __reduce_max_sync(0xffffffffu, key);
    if (lane == 0) wkey[0][warp] = key;
  }
  __syncthreads();
  auto best = [&](const unsigned* w) {
    unsigned k = 0;
#pragma unroll
    for (int i = 0; i < kXcMaxN / 32; ++i) k = max(k, w[i]);
    return k;
  };
  unsigned key = best(wkey[0]);
  int rnk = 0;
  int pos = 255 - (int)(key & 255u);
  int pv = key ? perm[0][pos] : 0;
  if (key) {
    const int lc = tid / C, dst = tid - (tid / C) * C, i = lc * C + rank;
    if (lc < ncl && i < na) xc_store_remote(rowbuf + i, (unsigned)dst, S[(size_t)lc * n + pv]);
    xc_arrive();
  }
  while (key) {
    const int k = rnk, buf = k & 1;
    const i128* row = rowbuf + buf * n;
    i128* r = rs + buf * n;
    const int* pm = perm[buf];
    int* pn = perm[buf ^ 1];
    // the pivot's reciprocal square root, while its row travels
    u128 y = 0;
    int t = 0;
    if (tid < na - k) {
      const u128 v = (u128)dg[pv] << 3;
      t = clz128(v) >> 1;
      y = rsqrt128(v << (2 * t));
    }
    xc_wait();
    if (tid < kXcMaxN) {
      unsigned kk = 0;
      if (tid < na - k) {
        const int p = pm[k + tid];
        const i128 x = row[p];
        const u128 mag = mulhi128((mag128(x) << t) << 2, y);
        const i128 rp = x < 0 ? -(i128)mag : (i128)mag;
        r[p] = rp;
        if (p % C == rank) S[(size_t)(p / C) * n + pv] = rp;
        // the pivot moves to position k, what was there to the pivot's place
        if (p == pv) {
          pn[k] = pv;
          order[pv] = k;
          piv[k] = pv;
        } else {
          const int np = k + tid == k ? pos : k + tid;
          pn[np] = p;
          const i128 d = dg[p] - (i128)mulq125(mag, mag);
          dg[p] = d;
          kk = d > thr ? xc_key((u128)d, ex[p] - exmax, np) : 0u;
        }
      }
      kk = __reduce_max_sync(0xffffffffu, kk);
      if (lane == 0) wkey[buf ^ 1][warp] = kk;
    }
    __syncthreads();
    key = best(wkey[buf ^ 1]);
    ++rnk;
    if (!key) break;
    pos = 255 - (int)(key & 255u);
    const int pnext = pn[pos];
    {
      // the next pivot's row first, to every CTA
      const int lc = tid / C, dst = tid - (tid / C) * C, i = lc * C + rank;
      if (lc < ncl && i < na && order[i] == n) {
        const i128 a = r[pnext], b = r[i];
        const u128 m = mulq125(mag128(a), mag128(b));
        const i128 v = S[(size_t)lc * n + pnext] - (((a < 0) != (b < 0)) ? -(i128)m : (i128)m);
        xc_store_remote(rowbuf + (buf ^ 1) * n + i, (unsigned)dst, v);
      }
      xc_arrive();
    }
    // the remaining rows of the own columns
    for (int l = warp; l < ncl; l += kXcThreads / 32) {
      const int i = l * C + rank;
      if (i >= na || order[i] != n) continue;
      const i128 b = r[i];
      const u128 bm = mag128(b);
      i128* col = S + (size_t)l * n;
      for (int q = k + 1 + lane; q < na; q += 32) {
        const int p = pn[q];
        if (p == pnext) continue;
        const i128 a = r[p];
        const u128 m = mulq125(mag128(a), bm);
        col[p] -= ((a < 0) != (b < 0)) ? -(i128)m : (i128)m;
      }
    }
    pv = pnext;
  }
  // rows of R, own columns (and the CTA's share of the columns that are zero)
  __syncthreads();
  for (int idx = tid; idx < n * xc_cols(n, C); idx += kXcThreads) {
    const int k = idx / xc_cols(n, C), lc = idx - k * xc_cols(n, C), i = lc * C + rank;
    if (i < na) {
      const int c = act[i];
      double d = 0.0;
      if (k < rnk && order[i] >= k) {
        const i128 x = S[(size_t)lc * n + piv[k]];
        d = ldexp(to_double125(mag128(x)), sc[i] + unit[c]) * (coef ? coef[c] : 1.0);
        if (x < 0) d = -d;
      }
      R[(size_t)k * n + c] = d;
    }
  }
  // inactive columns
  if (rank == 0)
    for (int idx = tid; idx < n * n; idx += kXcThreads) {
      const int c = idx % n;
      const size_t o = (size_t)c * n + c;
      if ((gint[o] | gint[plane + o] | gint[2 * plane + o]) == 0ull) R[idx] = 0.0;
    }
}

// R (n x n) from gint on stream s: one cluster.
inline tt_status launch_xg_chol(cudaStream_t s, int n, const unsigned long long* gint, const int* unit,
                                const double* coef, double* R) {
  if (n > kXcMaxN) return TT_ERR_UNSUPPORTED;
  const int C = xchol_cluster(n);
  const size_t smem = xchol_smem_bytes(n, C);
  if (const tt_status a = smem_optin(k_xg_chol, smem); a != TT_OK) return a;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(C);
  cfg.blockDim = dim3(kXcThreads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute at{};
  at.id = cudaLaunchAttributeClusterDimension;
  at.val.clusterDim.x = C;
  at.val.clusterDim.y = 1;
  at.val.clusterDim.z = 1;
  cfg.attrs = &at;
  cfg.numAttrs = 1;
  if (cudaLaunchKernelEx(&cfg, k_xg_chol, n, gint, unit, coef, R) != cudaSuccess) return TT_ERR_CUDA;
  count_launch();
  return TT_OK;
}

}  // namespace ttk
