// One-sided Jacobi SVD of a small triangular (or square) factor in one cluster: the columns of R^T (the
// rows of R, n <= 256) are spread over the CTAs' shared memory, two blocks of b columns per CTA, and
// the blocks go round the cluster through distributed shared memory (round-robin tournament of the 2 C
// blocks).  Between two moves a CTA rotates all b x b cross pairs of its two blocks (and once per sweep
// the pairs inside each block), one warp per pair, with CTA barriers only: a sweep of n columns takes
// 2 C - 1 cluster exchanges and about n short rounds.
//
// Why: the one-CTA FP32 form is bound by shared-memory traffic (every round reads and writes all
// columns: 1.4 us a round at 160 columns), and the grid-wide FP64 form (one pair per CTA, a barrier
// through global memory per round) by its barrier, 5.3 us a round.  Here a round moves 1/C of the
// columns per SM and waits on a CTA barrier.  FP64: the pipe runs at 1/64 of the FP32 rate, so the pair
// dot is the only reduction (norms follow the rotations and are renewed before every block pair), and
// the rotation's angle is formed in FP32 (the rotation itself is orthogonal to FP64 round-off; an angle
// accurate to 2^-22 only costs a sweep's final factor).
#pragma once
#include "common.cuh"
#include "instr.cuh"
#include "xchol.cuh"

namespace ttk {

constexpr int kJcMaxN = 256;
constexpr int kJcMaxB = 16;  // columns of a block (a warp per pair)

// Cluster size, up to the eight CTAs that every cluster launch may have: blocks of at most 16 columns, small enough
// that an inner round is one or two pairs per sub-partition.  FP64 takes more SMs for its slow pipe up to 64 columns.
template <typename T>
inline int jc_cluster(int n) {
  if (sizeof(T) == 8) return n <= 8 ? 1 : n <= 16 ? 2 : n <= 40 ? 4 : 8;
  return n <= 32 ? 1 : n <= 64 ? 4 : 8;
}
__host__ __device__ inline int jc_ld(int n) { return (n + 31) & ~31; }
__host__ __device__ inline int jc_b(int n, int C) { return (n + 2 * C - 1) / (2 * C); }
template <typename T>
inline size_t jc_smem_bytes(int n, int C) {
  const int b = jc_b(n, C);
  return sizeof(T) * ((size_t)4 * b * jc_ld(n) + 2 * b) + sizeof(int) * 4 * (size_t)b + 64;
}

__device__ __forceinline__ unsigned jc_map(const void* p, unsigned rank) {
  const unsigned a = (unsigned)__cvta_generic_to_shared(p);
  unsigned r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(rank));
  return r;
}

// tan of the rotation that makes a pair with squared norms a, b and product g orthogonal (columns scaled
// to norms <= 1), in FP32; 0 when the pair is orthogonal to the working accuracy or below round-off.
__device__ __forceinline__ float jc_tan(float d, float g) {  // d = b - a
  const float zeta = __fdividef(d, 2.f * g);
  const float az = fabsf(zeta);
  if (!(az < 1e18f)) return __fdividef(g, d);  // 1 / (2 zeta)
  const float s = fmaf(zeta, zeta, 1.f);
  return copysignf(__fdividef(1.f, az + s * rsqrtf(s)), zeta);
}
__device__ __forceinline__ void jc_cs(float t, float& c, float& s) {
  c = rsqrtf(fmaf(t, t, 1.f));
  s = c * t;
}
__device__ __forceinline__ void jc_cs(double t, double& c, double& s) {
  const double x = fma(t, t, 1.0);
  double y = (double)rsqrtf((float)x);  // two Newton steps: 2^-22, 2^-43, below 2^-53
  const double h = 0.5 * x;
  y = y * fma(-h * y, y, 1.5);
  y = y * fma(-h * y, y, 1.5);
  c = y;
  s = y * t;
}
template <typename T>
__device__ __forceinline__ T jc_warp_sum(T v) {
#pragma unroll
  for (int o = 16; o; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

template <typename T>
struct JcTol {
  T rel2, floor;
};

// One pair: rotates x (registers) against y, norms na, nb updated; returns whether it rotated.
template <typename T, int E>
__device__ __forceinline__ bool jc_pair(T (&x)[E], T (&y)[E], T& na, T& nb, const JcTol<T>& tol) {
  T g = T(0);
#pragma unroll
  for (int e = 0; e < E; ++e) g = fma(x[e], y[e], g);
  g = jc_warp_sum(g);
  if (!(fabs(g) > tol.floor && g * g > tol.rel2 * na * nb)) return false;
  const T t = (T)jc_tan((float)(nb - na), (float)g);
  T c, s;
  jc_cs(t, c, s);
#pragma unroll
  for (int e = 0; e < E; ++e) {
    const T u = x[e], v = y[e];
    x[e] = fma(c, u, -s * v);
    y[e] = fma(s, u, c * v);
  }
  na = fma(-t, g, na);
  nb = fma(t, g, nb);
  return true;
}

// R: n x n row-major FP64.  U[i][c] (row-major n x n): the normalised columns, raw[c] their norms, perm[r]
// the column of rank r by decreasing raw (ties by index).  Rows of R below drop ||R||_F stay out (zero
// columns of U).  maxsweep: cap on the sweeps; at the cap with rotations left TT_ERR_TIMEOUT is latched
// (FP64).  Every wait for the other CTAs is bounded (ctrl->spin_limit, else 2^24 tries; ctrl->barrier_extra
// arrivals that never come are a test setting) and latches TT_ERR_TIMEOUT when it runs out.
template <typename T, int E>
__global__ void __launch_bounds__(512) k_jacobi_cl(int n, const double* __restrict__ R, double* __restrict__ U,
                                                   double* __restrict__ raw, int* __restrict__ perm, int maxsweep,
                                                   float drop, DevCtrl* ctrl) {
  extern __shared__ __align__(16) unsigned char jc_smem[];
  __shared__ uint64_t bar;
  __shared__ float rn2[kJcMaxN];
  __shared__ int kept[kJcMaxN], nk_s, rotflag, wmax[16];
  __shared__ int cflag[2][16];
  __shared__ float wsum[16];
  const int C = (int)xc_cluster_size(), rank = (int)xc_cluster_rank();
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, nw = blockDim.x >> 5;
  const int ld = jc_ld(n), bm = jc_b(n, C);
  T* data = reinterpret_cast<T*>(jc_smem);                    // [2 buffers][2 blocks][bm][ld]
  T* norm = data + (size_t)4 * bm * ld;                       // [2 blocks][bm]
  int* ids = reinterpret_cast<int*>(norm + 2 * bm);           // [2 buffers][2 blocks][bm]
  const int extra = ctrl ? ctrl->barrier_extra : 0;
  const long long limit = (ctrl && ctrl->spin_limit > 0) ? ctrl->spin_limit : (1LL << 24);
  if (tid == 0) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"((unsigned)__cvta_generic_to_shared(&bar)), "r"(C + extra)
                 : "memory");
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  // largest binary exponent of R, then FP32 row norms of R 2^-e
  int em = 0;
  for (int i = tid; i < n * n; i += blockDim.x) em = max(em, (int)((__double_as_longlong(R[i]) >> 52) & 0x7ff));
  em = __reduce_max_sync(0xffffffffu, em);
  if (lane == 0) wmax[warp] = em;
  __syncthreads();
  for (int w = 0; w < nw; ++w) em = max(em, wmax[w]);
  const int es = min(max(em - 1022, -1000), 1000);
  const double scale = __longlong_as_double((long long)(1023 - es) << 52), unscale = __longlong_as_double((long long)(1023 + es) << 52);
  float fl = 0.f;
  for (int c = warp; c < n; c += nw) {
    float s2 = 0.f;
    for (int i = lane; i < n; i += 32) {
      const float v = (float)(R[(size_t)c * n + i] * scale);
      s2 = fmaf(v, v, s2);
    }
    s2 = jc_warp_sum(s2);
    if (lane == 0) rn2[c] = s2;
    fl += s2;
  }
  if (lane == 0) wsum[warp] = fl;
  __syncthreads();
  float fro2 = 0.f;
  for (int w = 0; w < nw; ++w) fro2 += wsum[w];
  if (warp == 0) {  // rows kept, in order
    const float thr = fro2 * drop * drop;
    int m = 0;
    for (int c0 = 0; c0 < n; c0 += 32) {
      const bool on = c0 + lane < n && rn2[c0 + lane] > thr;
      const unsigned mask = __ballot_sync(0xffffffffu, on);
      if (on) kept[m + __popc(mask & ((1u << lane) - 1u))] = c0 + lane;
      m += __popc(mask);
    }
    if (lane == 0) nk_s = m;
  }
  __syncthreads();
  const int nk = nk_s;
  const int b = nk > 0 ? jc_b(nk, C) : 0;
  // kept row s to block s mod 2C, place s / 2C: block 2 rank above, 2 rank + 1 below
  for (int q = warp; q < 2 * b; q += nw) {
    const int blk = q / b, i = q - blk * b, s = i * 2 * C + 2 * rank + blk;
    T* col = data + (size_t)(blk * bm + i) * ld;
    const bool on = s < nk;
    const double* row = R + (size_t)(on ? kept[s] : 0) * n;
    for (int k = lane; k < ld; k += 32) col[k] = (on && k < n) ? (T)(row[k] * scale) : T(0);
    if (lane == 0) ids[blk * bm + i] = on ? s : -1;
  }
  JcTol<T> tol;
  {
    // round-off of a pair's dot: FP32 sums 8 terms a lane and 5 levels of lanes
    const T rel = sizeof(T) == 4 ? fmaxf(4.f, sqrtf((float)n)) * T(1.1920929e-7f) : T(2.0 * n * 2.220446049250313e-16);
    tol.rel2 = rel * rel;
    tol.floor = (sizeof(T) == 4 ? T(1e-14) : T(1e-32)) * (T)fro2;
  }
  if (ctrl && sizeof(T) == 8 && ctrl->jac_sweep_cap > 0 && ctrl->jac_sweep_cap < maxsweep) maxsweep = ctrl->jac_sweep_cap;
  // every CTA's barrier is initialised, and every CTA runs, before any remote access
  xc_arrive();
  xc_wait();
  int cur = 0, sweeps = 0, phase = 0;
  bool lost = false;
  auto load = [&](const T* col, T(&v)[E]) {
#pragma unroll
    for (int e = 0; e < E; ++e) v[e] = (lane + 32 * e < ld) ? col[lane + 32 * e] : T(0);
  };
  auto store = [&](T* col, const T(&v)[E]) {
#pragma unroll
    for (int e = 0; e < E; ++e)
      if (lane + 32 * e < ld) col[lane + 32 * e] = v[e];
  };
  // arrivals of every CTA, then a bounded wait for all of them
  auto cluster_step = [&]() -> bool {
    asm volatile("fence.acq_rel.cluster;" ::: "memory");
    __syncthreads();
    if (tid < C) {
      const unsigned a = jc_map(&bar, (unsigned)tid);
      asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(a) : "memory");
    }
    bool ok = false;
    for (long long i = 0; i < limit && !ok; ++i) {
      unsigned p;
      asm volatile(
          "{\n.reg .pred p;\nmbarrier.test_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\nselp.u32 %0, 1, 0, "
          "p;\n}\n"
          : "=r"(p)
          : "r"((unsigned)__cvta_generic_to_shared(&bar)), "r"((unsigned)(phase & 1))
          : "memory");
      ok = p != 0;
    }
    ++phase;
    return __syncthreads_and(ok) != 0;
  };
  for (int sweep = 0; sweep < maxsweep && nk > 1 && !lost; ++sweep) {
    sweeps = sweep + 1;
    if (tid == 0) rotflag = 0;
    bool rotated = false;
    for (int br = 0; br < 2 * C - 1 && !lost; ++br) {
      T* X = data + (size_t)cur * 2 * bm * ld;
      T* Y = X + (size_t)bm * ld;
      const int* idx = ids + cur * 2 * bm;
      const int* idy = idx + bm;
      __syncthreads();
      if (br == 0) {
        // squared norms of all columns, then the pairs inside each block
        for (int q = warp; q < 2 * b; q += nw) {
          const int blk = q / b, i = q - blk * b;
          T v[E];
          load(X + (size_t)(blk * bm + i) * ld, v);
          T a = T(0);
#pragma unroll
          for (int e = 0; e < E; ++e) a = fma(v[e], v[e], a);
          a = jc_warp_sum(a);
          if (lane == 0) norm[blk * bm + i] = a;
        }
        __syncthreads();
        const int bb = b + (b & 1), hp = bb / 2;
        for (int rd = 0; rd < bb - 1; ++rd) {
          for (int w = warp; w < 2 * hp; w += nw) {
            const int blk = w / hp, pr = w - blk * hp;
            int p, q;
            if (pr == 0) {
              p = rd;
              q = bb - 1;
            } else {
              p = rd + pr;
              if (p >= bb - 1) p -= bb - 1;
              q = rd - pr;
              if (q < 0) q += bb - 1;
            }
            if (p > q) {
              const int u = p;
              p = q;
              q = u;
            }
            if (q < b && idx[blk * bm + p] >= 0 && idx[blk * bm + q] >= 0) {
              T* cp = X + (size_t)(blk * bm + p) * ld;
              T* cq = X + (size_t)(blk * bm + q) * ld;
              T x[E], y[E];
              load(cp, x);
              load(cq, y);
              T na = norm[blk * bm + p], nb = norm[blk * bm + q];
              if (jc_pair<T, E>(x, y, na, nb, tol)) {
                store(cp, x);
                store(cq, y);
                rotated = true;
                if (lane == 0) {
                  norm[blk * bm + p] = na;
                  norm[blk * bm + q] = nb;
                }
              }
            }
          }
          __syncthreads();
        }
      }
      // cross pairs: warp w keeps column w of X in registers, the columns of Y pass by
      {
        const bool mine = warp < b && idx[warp] >= 0;
        T x[E];
        T na = T(0);
        if (mine) {
          load(X + (size_t)warp * ld, x);
#pragma unroll
          for (int e = 0; e < E; ++e) na = fma(x[e], x[e], na);
          na = jc_warp_sum(na);
        }
        if (warp < b) {
          T v[E];
          load(Y + (size_t)warp * ld, v);
          T a = T(0);
#pragma unroll
          for (int e = 0; e < E; ++e) a = fma(v[e], v[e], a);
          a = jc_warp_sum(a);
          if (lane == 0) norm[bm + warp] = a;
        }
        __syncthreads();
        for (int rd = 0; rd < b; ++rd) {
          if (mine) {
            int q = warp + rd;
            if (q >= b) q -= b;
            if (idy[q] >= 0) {
              T* cq = Y + (size_t)q * ld;
              T y[E];
              load(cq, y);
              T nb = norm[bm + q];
              if (jc_pair<T, E>(x, y, na, nb, tol)) {
                store(cq, y);
                rotated = true;
                if (lane == 0) norm[bm + q] = nb;
              }
            }
          }
          __syncthreads();
        }
        if (mine) store(X + (size_t)warp * ld, x);
      }
      if (rotated && lane == 0) rotflag = 1;
      __syncthreads();
      if (br == 2 * C - 2 && tid < C) {  // the sweep's flag to every CTA
        const unsigned a = jc_map(&cflag[sweep & 1][rank], (unsigned)tid);
        asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(a), "r"(rotflag) : "memory");
      }
      if (C > 1) {
        // the blocks move: above to the right (the last one below itself), below to the left, block 0 stays
        T* N = data + (size_t)(cur ^ 1) * 2 * bm * ld;
        int* nid = ids + (cur ^ 1) * 2 * bm;
#pragma unroll
        for (int blk = 0; blk < 2; ++blk) {
          int dst, slot;
          if (blk == 0) {
            dst = rank == 0 ? 0 : rank < C - 1 ? rank + 1 : C - 1;
            slot = (rank == C - 1) ? 1 : 0;
          } else {
            dst = rank == 0 ? 1 : rank - 1;
            slot = rank == 0 ? 0 : 1;
          }
          const uint4* from = reinterpret_cast<const uint4*>(X + (size_t)blk * bm * ld);
          const unsigned to = jc_map(N + (size_t)slot * bm * ld, (unsigned)dst);
          const int nv = (int)((size_t)b * ld * sizeof(T) / 16);
          for (int i = tid; i < nv; i += blockDim.x) {
            const uint4 v = from[i];
            asm volatile("st.shared::cluster.v4.u32 [%0], {%1, %2, %3, %4};" ::"r"(to + 16u * i), "r"(v.x), "r"(v.y),
                         "r"(v.z), "r"(v.w)
                         : "memory");
          }
          const unsigned tid_to = jc_map(nid + slot * bm, (unsigned)dst);
          if (tid < b)
            asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(tid_to + 4u * tid), "r"(idx[blk * bm + tid]) : "memory");
        }
      }
      if (!cluster_step()) {
        lost = true;
        break;
      }
      if (C > 1) cur ^= 1;
    }
    if (lost) break;
    int any = 0;
    for (int c = 0; c < C; ++c) any |= cflag[sweep & 1][c];
    if (!any) break;
    if (sizeof(T) == 8 && sweep == maxsweep - 1 && rank == 0 && tid == 0 && ctrl) latch(&ctrl->status, TT_ERR_TIMEOUT);
  }
  if (lost && tid == 0 && ctrl) latch(&ctrl->status, TT_ERR_TIMEOUT);
  if (ctrl && tid == 0 && rank == 0) {
    atomicMax(&ctrl->jac_sweeps_max, sweeps);
    atomicAdd(&ctrl->jac_calls, 1);
    atomicAdd(&ctrl->jac_sweeps_sum, sweeps);
  }
  __syncthreads();
  // normalised columns (FP64 norms of the stored columns)
  for (int q = warp; q < 2 * b; q += nw) {
    const int blk = q / b, i = q - blk * b;
    const int c = ids[cur * 2 * bm + blk * bm + i];
    if (c < 0) continue;
    const T* col = data + ((size_t)cur * 2 * bm + blk * bm + i) * ld;
    double s2 = 0.0;
    for (int k = lane; k < n; k += 32) s2 += (double)col[k] * (double)col[k];
    s2 = jc_warp_sum(s2);
    const double inv = (s2 > 0.0) ? 1.0 / sqrt(s2) : 0.0;
    for (int k = lane; k < n; k += 32) U[(size_t)k * n + c] = (double)col[k] * inv;
    if (lane == 0) raw[c] = sqrt(s2) * unscale;
  }
  for (int c = nk + rank; c < n; c += C) {
    for (int k = tid; k < n; k += blockDim.x) U[(size_t)k * n + c] = 0.0;
    if (tid == 0) raw[c] = 0.0;
  }
  // the order of all columns, in the first CTA (its peers' stores are visible after the barrier)
  __threadfence();
  xc_arrive();
  xc_wait();
  if (rank == 0 && perm) {
    double* key = reinterpret_cast<double*>(jc_smem);
    for (int c = tid; c < n; c += blockDim.x) key[c] = rank_key(__ldcg(raw + c));
    __syncthreads();
    for (int c = tid; c < n; c += blockDim.x) {
      const double v = key[c];
      int rk = 0;
      for (int q = 0; q < n; ++q) {
        const double w = key[q];
        rk += (w > v) || (w == v && q < c);
      }
      perm[rk] = c;
    }
  }
}

template <typename T, int E>
inline tt_status launch_jacobi_cl_e(cudaStream_t s, int n, const double* R, double* U, double* raw, int* perm, float drop,
                                    DevCtrl* ctrl) {
  auto kern = k_jacobi_cl<T, E>;
  const int C = jc_cluster<T>(n);
  size_t smem = jc_smem_bytes<T>(n, C);
  if (smem < sizeof(double) * (size_t)n) smem = sizeof(double) * (size_t)n;
  if (const tt_status a = smem_optin(kern, smem); a != TT_OK) return a;
  int nwarp = jc_b(n, C);
  nwarp += nwarp & 1;
  if (nwarp < 4) nwarp = 4;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(C);
  cfg.blockDim = dim3(32 * nwarp);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute at{};
  at.id = cudaLaunchAttributeClusterDimension;
  at.val.clusterDim.x = C;
  at.val.clusterDim.y = 1;
  at.val.clusterDim.z = 1;
  cfg.attrs = &at;
  cfg.numAttrs = 1;
  if (cudaLaunchKernelEx(&cfg, kern, n, R, U, raw, perm, 40, drop, ctrl) != cudaSuccess) return TT_ERR_CUDA;
  count_launch();
  return TT_OK;
}
// U, raw and perm of the n x n factor R (see k_jacobi_cl) on stream s.
template <typename T>
tt_status launch_jacobi_cl(cudaStream_t s, int n, const double* R, double* U, double* raw, int* perm, DevCtrl* ctrl) {
  // rows below drop ||R||_F together change R by less than sqrt(n) drop ||R||_F: below the rounding of R
  const float drop = sizeof(T) == 4 ? 9.31322574615478515625e-10f : 8.6736173798840355e-19f;  // 2^-30, 2^-60
  if (n > kJcMaxN) return TT_ERR_UNSUPPORTED;
  if (n <= 32) return launch_jacobi_cl_e<T, 1>(s, n, R, U, raw, perm, drop, ctrl);
  if (n <= 64) return launch_jacobi_cl_e<T, 2>(s, n, R, U, raw, perm, drop, ctrl);
  if (n <= 160) return launch_jacobi_cl_e<T, 5>(s, n, R, U, raw, perm, drop, ctrl);
  return launch_jacobi_cl_e<T, 8>(s, n, R, U, raw, perm, drop, ctrl);
}

}  // namespace ttk
