// Cholesky factor of an exact integer Gram matrix in 128-bit fixed point: R with R^T R = G, for the
// triangular factor of the merged core's columns (xgram.cuh).
//
// G comes as 192-bit integers.  Column c is scaled by 2^-s_c so that every diagonal entry lies in
// (1/4, 1], and the entries, Schur complements and rows of R (all at most 1 in magnitude) are held as
// signed integers: FP64 passes 128 bits of unit 2^-125, FP32 passes 64 bits of unit 2^-61.  Absolute
// round-off stays near n 2^-125 (n 2^-60), so a column's remainder after the earlier columns is resolved
// down to about 2^-57 (2^-27) of its norm, as a Householder QR in FP64 (FP32) resolves it; a pivot below
// n 2^-118 (n 2^-56) is dead (the column is a combination of the earlier ones to that accuracy).  The pivot of a
// step is the remaining column of largest norm, so the rows of R come graded, which a one-sided Jacobi
// on R^T needs fewer sweeps for, and the factor ends where nothing is left.  128-bit integers rather than double-double: this part's FP64 pipe runs at 1/64 of
// the integer rate, and a double-double update (20 FP64 operations) would take 4 ms at 160 columns.
//
// Right-looking, one cluster: CTA r holds the columns i = r mod C (all rows), the pivot's row is
// exchanged through distributed shared memory, one cluster barrier per step (and one before the first
// exchange: a peer's shared memory may be written only once that CTA runs).  Every CTA keeps all
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

// 1 / sqrt(v) in (1, 2], unit 2^-62, for v in [1/4, 1) of unit 2^-64: two Newton steps y + y (1 - v y^2) / 2
// from the FP32 reciprocal square root (2^-22, 2^-43, 2^-59).
__device__ __forceinline__ unsigned long long rsqrt64(unsigned long long v) {
  const float vf = (float)(unsigned)(v >> 32) * 2.3283064365386963e-10f;
  unsigned long long y = (unsigned long long)(rsqrtf(vf) * 1073741824.0f) << 32;
#pragma unroll
  for (int it = 0; it < 2; ++it) {
    const unsigned long long w = __umul64hi(__umul64hi(y, y), v);  // v y^2, unit 2^-60
    const long long e = (long long)((1ull << 60) - w);
    const unsigned long long m = (unsigned long long)(e < 0 ? -e : e);
    const unsigned long long c = __umul64hi(y, m << 3);            // y |e| 2^3, unit 2^-58: halved, 2^-62 is itself
    y = e < 0 ? y - c : y + c;
  }
  return y;
}

// The integer type of a pass: WD 64-bit words, unit 2^-F.
template <int WD>
struct XcWord;
template <>
struct XcWord<1> {
  using S = long long;
  using U = unsigned long long;
  static constexpr int F = 61, kThr = 5;  // dead pivots: n 2^(kThr - F)
  __device__ static __forceinline__ U mulhi(U a, U b) { return __umul64hi(a, b); }
  __device__ static __forceinline__ int clz(U x) { return __clzll((long long)x); }
  __device__ static __forceinline__ U rsqrt(U v) { return rsqrt64(v); }
  __device__ static __forceinline__ double to_double(U m) { return __ull2double_rn(m) * 4.3368086899420177e-19; }
};
template <>
struct XcWord<2> {
  using S = i128;
  using U = u128;
  static constexpr int F = 125, kThr = 7;
  __device__ static __forceinline__ U mulhi(U a, U b) { return mulhi128(a, b); }
  __device__ static __forceinline__ int clz(U x) {
    const unsigned long long h = (unsigned long long)(x >> 64);
    return h ? __clzll((long long)h) : 64 + __clzll((long long)(unsigned long long)x);
  }
  // a third Newton step in 128 bits (2^-118); unit 2^-126
  __device__ static __forceinline__ U rsqrt(U v) {
    const u128 y = (u128)rsqrt64((unsigned long long)(v >> 64)) << 64;
    const u128 w = mulhi128(mulhi128(y, y), v);  // unit 2^-124
    const i128 e = (i128)(((u128)1 << 124) - w);
    const u128 c = mulhi128(y, (e < 0 ? (u128)(-e) : (u128)e) << 3);
    return e < 0 ? y - c : y + c;
  }
  __device__ static __forceinline__ double to_double(U m) {
    return __ull2double_rn((unsigned long long)(m >> 64)) * 4.3368086899420177e-19 +
           __ull2double_rn((unsigned long long)m) * 2.3509887016445750e-38;
  }
};

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
// store a value at the same shared-memory address of CTA `rank` of the cluster
__device__ __forceinline__ unsigned xc_map(const void* local, unsigned rank) {
  const unsigned a = (unsigned)__cvta_generic_to_shared(local);
  unsigned r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(rank));
  return r;
}
__device__ __forceinline__ void xc_store_remote(i128* local, unsigned rank, i128 v) {
  asm volatile("st.shared::cluster.v2.u64 [%0], {%1, %2};" ::"r"(xc_map(local, rank)), "l"((unsigned long long)v),
               "l"((unsigned long long)((u128)v >> 64))
               : "memory");
}
__device__ __forceinline__ void xc_store_remote(long long* local, unsigned rank, long long v) {
  asm volatile("st.shared::cluster.u64 [%0], %1;" ::"r"(xc_map(local, rank)), "l"(v) : "memory");
}

// columns of a matrix of n per CTA of a cluster of C (at most 32)
__host__ __device__ inline int xc_cols(int n, int C) { return (n + C - 1) / C; }
inline size_t xchol_smem_bytes(int n, int C, int word) { return (size_t)word * ((size_t)xc_cols(n, C) * n + 5 * (size_t)n); }
inline int xchol_cluster(int n) { return n <= 32 ? 1 : n <= 64 ? 2 : n <= 96 ? 4 : 8; }

// Shift right (left for negative sh) a 192-bit two's complement integer to 128 bits.
__device__ __forceinline__ i128 shift192(unsigned long long w0, unsigned long long w1, unsigned long long w2, int sh) {
  if (sh <= 0) return (i128)((((u128)w1 << 64) | w0) << (sh < -127 ? 127 : -sh));
  const i128 hi = ((i128)(long long)w2 << 64) | w1;  // words 2, 1
  if (sh >= 64) return sh >= 191 ? (hi < 0 ? (i128)-1 : (i128)0) : hi >> (sh - 64);
  return (i128)(((u128)hi << (64 - sh)) | (w0 >> sh));
}

// Pivot key of a remaining diagonal d of a column whose squared scale has the binary exponent `ex`:
// exponent, leading bits, position (so that equal keys resolve the same way in every CTA).
template <int WD>
__device__ __forceinline__ unsigned xc_key(typename XcWord<WD>::U d, int ex, int pos) {
  const int lz = XcWord<WD>::clz(d);
  const int e = min(max(ex - lz + 2048, 1), 4095);
  const unsigned m = (unsigned)((d << lz) >> (64 * WD - 12)) & 0xfffu;
  return ((unsigned)e << 20) | (m << 8) | (unsigned)(255 - pos);
}

// gint: word planes of the upper triangle of G (row-major, n x n).  Rows k of R (n x n row-major, pivot
// order; zero beyond the rank) get r_kc 2^(s_c) coef_c 2^(U_c), U_c the unit exponent of column c's fixed
// point and coef_c its coefficient in the sum (nullable).
template <int WD>
__global__ void __launch_bounds__(kXcThreads) k_xg_chol(int n, const unsigned long long* __restrict__ gint,
                                                        const int* __restrict__ unit, const double* __restrict__ coef,
                                                        double* __restrict__ R) {
  using Wd = XcWord<WD>;
  using SI = typename Wd::S;
  using UI = typename Wd::U;
  extern __shared__ __align__(16) unsigned char xc_smem[];
  __shared__ int act[kXcMaxN], sc[kXcMaxN], ex[kXcMaxN], order[kXcMaxN], piv[kXcMaxN], perm[2][kXcMaxN];
  __shared__ int wcount[kXcThreads / 32], na_s;
  __shared__ __align__(16) unsigned wkey[2][kXcMaxN / 32];
  const int C = (int)xc_cluster_size(), rank = (int)xc_cluster_rank();
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  if (C > 1) xc_arrive();  // this CTA runs (waited for before the first exchange)
  const int ncl = xc_cols(n, C);
  const size_t plane = (size_t)n * n;
  SI* S = reinterpret_cast<SI*>(xc_smem);  // [ncl][n]: column lc C + rank; row of a finished pivot: r
  SI* rowbuf = S + (size_t)ncl * n;        // [2][n]: the exchanged row
  SI* rs = rowbuf + 2 * n;                 // [2][n]: its scaled form, a row of R
  SI* dg = rs + 2 * n;                     // [n]: remaining diagonals
  auto mag = [](SI x) -> UI { return x < 0 ? (UI)(-x) : (UI)x; };
  // x - (a b) for entries of rows of R
  auto sub_prod = [&](SI x, SI a, SI b) -> SI {
    const UI m = Wd::mulhi(mag(a) << 2, mag(b) << 1);
    const SI neg = (a ^ b) >> (64 * WD - 1);  // -1 where the product is negative
    return x - (((SI)m ^ neg) - neg);
  };
  auto arrive = [&]() {
    if (C > 1) xc_arrive();
  };
  auto wait = [&]() {
    if (C > 1) xc_wait();
    else __syncthreads();
  };
  auto send = [&](SI* local, int dst, SI v) {
    if (C > 1) xc_store_remote(local, (unsigned)dst, v);
    else *local = v;
  };
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
      S[(size_t)lc * n + p] = (SI)shift192(gint[o], gint[plane + o], gint[2 * plane + o], sc[p] + sc[i] - Wd::F);
    }
  }
  const SI thr = (SI)n << Wd::kThr;
  // key exponents relative to the largest column
  int exmax = -(1 << 30);
  for (int i = lane; i < na; i += 32) exmax = max(exmax, ex[i]);
  exmax = __reduce_max_sync(0xffffffffu, exmax);
  if (tid < kXcMaxN) {
    unsigned key = 0;
    if (tid < na) {
      const size_t o = (size_t)act[tid] * n + act[tid];
      const SI d = (SI)shift192(gint[o], gint[plane + o], gint[2 * plane + o], 2 * sc[tid] - Wd::F);
      dg[tid] = d;
      key = d > thr ? xc_key<WD>((UI)d, ex[tid] - exmax, tid) : 0u;
    }
    key = __reduce_max_sync(0xffffffffu, key);
    if (lane == 0) wkey[0][warp] = key;
  }
  __syncthreads();
  auto best = [&](const unsigned* w) {
    const uint4 a = *reinterpret_cast<const uint4*>(w), b = *reinterpret_cast<const uint4*>(w + 4);
    return max(max(max(a.x, a.y), max(a.z, a.w)), max(max(b.x, b.y), max(b.z, b.w)));
  };
  unsigned key = best(wkey[0]);
  int rnk = 0;
  int pos = 255 - (int)(key & 255u);
  int pv = key ? perm[0][pos] : 0;
  // threads of the row exchange: one per (own column, destination)
  const int xl = tid / C, xd = tid - (tid / C) * C, xi = xl * C + rank;
  const bool xon = xl < ncl && xi < na;
  if (C > 1) xc_wait();  // every CTA of the cluster runs
  if (key) {
    if (xon) send(rowbuf + xi, xd, S[(size_t)xl * n + pv]);
    arrive();
  }
  while (key) {
    const int k = rnk, buf = k & 1;
    const SI* row = rowbuf + buf * n;
    SI* r = rs + buf * n;
    const int* pm = perm[buf];
    int* pn = perm[buf ^ 1];
    // the pivot's reciprocal square root, while its row travels
    UI y = 0;
    int t = 0;
    if (tid < na - k) {
      const UI v = (UI)dg[pv] << 3;
      t = Wd::clz(v) >> 1;
      y = Wd::rsqrt(v << (2 * t));
    }
    wait();
    if (tid < kXcMaxN) {
      unsigned kk = 0;
      if (tid < na - k) {
        const int p = pm[k + tid];
        const SI x = row[p];
        const UI m = Wd::mulhi((mag(x) << t) << 2, y);
        const SI rp = x < 0 ? -(SI)m : (SI)m;
        r[p] = rp;
        if (p % C == rank) S[(size_t)(p / C) * n + pv] = rp;
        // the pivot moves to position k, what was there to the pivot's place
        if (p == pv) {
          pn[k] = pv;
          piv[k] = pv;
        } else {
          const int np = k + tid == k ? pos : k + tid;
          pn[np] = p;
          const SI d = dg[p] - (SI)Wd::mulhi(m << 2, m << 1);
          dg[p] = d;
          kk = d > thr ? xc_key<WD>((UI)d, ex[p] - exmax, np) : 0u;
        }
      }
      kk = __reduce_max_sync(0xffffffffu, kk);
      if (lane == 0) wkey[buf ^ 1][warp] = kk;
    }
    __syncthreads();
    key = best(wkey[buf ^ 1]);
    ++rnk;
    // (a slow thread still in the previous step's update never reads order[] of this pivot as finished)
    if (tid == 0) order[pv] = k;
    if (!key) break;
    pos = 255 - (int)(key & 255u);
    const int pnext = pn[pos];
    // the next pivot's row first, to every CTA
    if (xon && xi != pv && order[xi] == n) send(rowbuf + (buf ^ 1) * n + xi, xd, sub_prod(S[(size_t)xl * n + pnext], r[pnext], r[xi]));
    arrive();
    // the remaining rows of the own unfinished columns: 16 warps over the columns, several to a column
    // where few are left
    {
      const int i = lane * C + rank;
      const bool on = lane < ncl && i < na && i != pv && order[i] == n;
      const unsigned mask = __ballot_sync(0xffffffffu, on);
      const int m = __popc(mask), mine = __popc(mask & ((1u << lane) - 1u));
      const int wsh = m > 8 ? 0 : m > 4 ? 1 : m > 2 ? 2 : m > 1 ? 3 : 4;  // log2 warps per column
      const int sub = warp & ((1 << wsh) - 1);
      for (int j = warp >> wsh; j < m; j += 16 >> wsh) {
        const int l = __ffs(__ballot_sync(0xffffffffu, on && mine == j)) - 1;
        const SI b = r[l * C + rank];
        SI* col = S + (size_t)l * n;
        for (int q = k + 1 + lane + 32 * sub; q < na; q += 32 << wsh) {
          const int p = pn[q];
          if (p != pnext) col[p] = sub_prod(col[p], r[p], b);
        }
      }
    }
    pv = pnext;
  }
  // rows of R in the own columns, zeros in the columns without entries
  __syncthreads();
  for (int idx = tid; idx < n * ncl; idx += kXcThreads) {
    const int k = idx / ncl, lc = idx - k * ncl, i = lc * C + rank;
    if (i < na) {
      const int c = act[i];
      double d = 0.0;
      if (k < rnk && order[i] >= k) {
        const SI x = S[(size_t)lc * n + piv[k]];
        d = ldexp(Wd::to_double(mag(x)), sc[i] + unit[c]) * (coef ? coef[c] : 1.0);
        if (x < 0) d = -d;
      }
      R[(size_t)k * n + c] = d;
    }
  }
  if (rank == 0 && na < n)
    for (int idx = tid; idx < n * n; idx += kXcThreads) {
      const int c = idx % n;
      const size_t o = (size_t)c * n + c;
      if ((gint[o] | gint[plane + o] | gint[2 * plane + o]) == 0ull) R[idx] = 0.0;
    }
}

// R (n x n) from gint on stream s: one cluster.
template <int WD>
inline tt_status launch_xg_chol(cudaStream_t s, int n, const unsigned long long* gint, const int* unit,
                                const double* coef, double* R) {
  if (n > kXcMaxN) return TT_ERR_UNSUPPORTED;
  const int C = xchol_cluster(n);
  const size_t smem = xchol_smem_bytes(n, C, 8 * WD);
  if (const tt_status a = smem_optin(k_xg_chol<WD>, smem); a != TT_OK) return a;
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
  if (cudaLaunchKernelEx(&cfg, k_xg_chol<WD>, n, gint, unit, coef, R) != cudaSuccess) return TT_ERR_CUDA;
  count_launch();
  return TT_OK;
}

}  // namespace ttk
