// TT primitives: materialised transport sum, axpy by rank concatenation, inner product.
#include "bigpass.cuh"
#include "small.cuh"
#include "step.cuh"
#include "xgram.cuh"

namespace ttk {
namespace {

// lam (a + b + c) rounded to FP32 with the sum and the product in pairs of FP32 numbers (two-sums, an FMA for the
// product's low part; about 2^-47), since FP64 arithmetic (1/64 of the FP32 rate) took longer than the memory.
// lh + ll = lam.  Where the low parts may leave the normal numbers: FP64.
__device__ __noinline__ float tr_scaled64(double lam, float a, float b, float c) {
  return (float)(lam * (((double)a + (double)b) + (double)c));
}
__device__ __forceinline__ float tr_scaled(double lam, float lh, float ll, float a, float b, float c) {
  const float s = a + b, bb = s - a, e1 = (a - (s - bb)) + (b - bb);
  const float t = s + c, cb = t - s, e2 = (s - (t - cb)) + (c - cb);
  const float e = e1 + e2, h = t + e, hb = h - t, l = (t - (h - hb)) + (e - hb);
  const float p = h * lh;
  if (fabsf(p) > 1e-25f && fabsf(p) < 1e30f && fabsf(h) > 1e-25f && fabsf(h) < 1e30f)
    return p + (fmaf(h, lh, -p) + fmaf(h, ll, l * lh));
  if (h == 0.0f) return p;
  return tr_scaled64(lam, a, b, c);  // (inlined, its FP64 instructions were executed under a predicate)
}
__device__ __forceinline__ double tr_scaled(double lam, float, float, double a, double b, double c) {
  return lam * ((a + b) + c);
}

// Merged core of the materialised transport sum in compact layout: columns t*r + q
// (t = 0 state, t = 1..nterm operator images) and the nbc inflow columns after them.  A thread keeps
// one column (its operator is looked up once), a CTA takes 64 rows at a time (their neighbour flags are
// formed once, by 64 threads), four rows of a thread in flight.  1,048,576 x 81 FP32: 0.37 ms (340 MB written); with a
// thread per entry, which divides for its row, column and neighbours in 64 bits and scales in FP64: 1.47 ms.
// Below 32,768 rows (FP64: 64 a CTA) a CTA takes fewer rows, so that all of them have some: 7,488 x 180 FP32 37 -> 29 us,
// 16,384 x 180 FP64 62 -> 48.  A thread per entry (k_transport_entry) stays where it is faster, thread per entry / columns:
//   FP32, up to 5 x 2^16 entries: 576 x 100 19 / 25 us, 2,048 x 100 20 / 26, 7,488 x 40 20 / 22, 7,488 x 72 26 / 22
//   FP64 central differences, up to 2^20: 576 x 180 24 / 46, 7,488 x 72 21 / 29, 16,384 x 72 32 / 30, 55,296 x 27 39 / 35
//   FP64 upwind, up to 6 x 2^20 or where the columns leave a fifth of a CTA idle: 55,296 x 15 25 / 27, 131,072 x 40 78 /
//     83, 442,368 x 15 102 / 100, 442,368 x 40 258 / 240; 100 columns: 131,072 173 / 193, 1,048,576 1,316 / 1,373
constexpr int kTrRows = 64;
// SrcStencil::row_flags in 32 bits where the rows allow it (64-bit division runs on the FP64 pipe).
template <typename S>
__device__ __forceinline__ unsigned tr_flags(const SrcStencil<S>& src, long k, long N) {
  if (N >= (1L << 31)) return src.row_flags(k);
  unsigned f = 0u;
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    const unsigned idx = ((unsigned)k / (unsigned)src.stride[a]) % (unsigned)src.ext[a];
    f |= (idx > 0u ? 1u : 0u) << (2 * a);
    f |= (idx + 1u < (unsigned)src.ext[a] ? 1u : 0u) << (2 * a + 1);
  }
  return f | (((unsigned)k % (unsigned)src.G) << 8);
}
template <typename S>
__global__ void __launch_bounds__(256) k_transport_entry(long N, SrcStencil<S> src, const int* __restrict__ rank_in,
                                                         S* __restrict__ Zo, int ldo, int nbc,
                                                         const int* __restrict__ rank_in2, int rcapo2, int,
                                                         int* status) {
  const int r = rank_in[1];
  const int R = (src.nterm + 1) * r + nbc;
  bool over = R > ldo;
  if (rank_in2) over = over || ((src.nterm + 1) * (*rank_in2) + nbc > rcapo2);
  if (over) {
    if (blockIdx.x == 0 && threadIdx.x == 0) latch(status, TT_ERR_CAPACITY);
    return;
  }
  src.rcap = r > 0 ? r : 1;
  const long tot = N * (long)ldo;
  for (long idx = blockIdx.x * (long)blockDim.x + threadIdx.x; idx < tot; idx += (long)gridDim.x * blockDim.x) {
    const long k = idx / ldo;
    const int c = (int)(idx - k * ldo);
    S v = S(0);
    if (c < R && r > 0) {
      const auto cc = src.col(c);
      if (sizeof(S) == 8 || (cc.kind != 1 && cc.kind < 4)) {
        v = (S)src.load(cc, k);
      } else {  // as k_transport_Z forms it
        const double lam = cc.kind == 4 ? -0.5 * cc.lam : cc.kind == 5 ? 0.5 * cc.lam : -cc.lam;
        const float lh = fabs(lam) > 1e-25 ? (float)lam : 0.0f, ll = (float)(lam - (double)lh);
        const unsigned f = tr_flags(src, k, N) >> (2 * cc.ax);
        const S* z = src.Z + k * src.ldz + cc.q;
        const long st = cc.s * src.ldz;
        const bool both = cc.kind >= 4;
        const S zl = (both || cc.w > 0) && (f & 1u) ? z[-st] : S(0), zh = (both || cc.w <= 0) && (f & 2u) ? z[st] : S(0);
        const S x = !both && cc.w > 0 ? z[0] : zh;
        const S y = cc.kind == 5 ? S(-2) * z[0] : !both && cc.w <= 0 ? -z[0] : -zl;
        v = tr_scaled(lam, lh, ll, x, y, cc.kind == 5 ? zl : S(0));
      }
    }
    Zo[idx] = v;
  }
}
template <typename S, int ROWS>
__global__ void __launch_bounds__(256) k_transport_Z(long N, SrcStencil<S> src, const int* __restrict__ rank_in,
                                                     S* __restrict__ Zo, int ldo, int nbc,
                                                     const int* __restrict__ rank_in2, int rcapo2, int nrow,
                                                     int* status) {
  __shared__ unsigned fl[kTrRows];
  const int rows = ROWS ? ROWS : nrow;
  const int r = rank_in[1];
  const int R = (src.nterm + 1) * r + nbc;
  bool over = R > ldo;
  if (rank_in2) over = over || ((src.nterm + 1) * (*rank_in2) + nbc > rcapo2);
  if (over) {
    if (blockIdx.x == 0 && threadIdx.x == 0) latch(status, TT_ERR_CAPACITY);
    return;
  }
  src.rcap = r > 0 ? r : 1;
  const int tid = threadIdx.x;
  // ldo <= 256: 256 / ldo rows side by side; wider: column chunks of 256
  const int cw = ldo < 256 ? ldo : 256, rpb = 256 / cw, sub = tid / cw;
  for (int c0 = 0; c0 < ldo; c0 += 256) {
    const int c = c0 + tid - sub * cw;
    const bool mine = sub < rpb && c < ldo;
    typename SrcStencil<S>::Col cc{3, 0, 0, 0, 0, 0.0, 0.0f, 0};
    if (mine && c < R && r > 0) cc = src.col(c);
    // coefficient of the (second) difference
    const double lam = cc.kind == 4 ? -0.5 * cc.lam : cc.kind == 5 ? 0.5 * cc.lam : -cc.lam;
    // (a coefficient whose parts would be subnormal: zero, which sends every entry to FP64)
    const float lh = fabs(lam) > 1e-25 ? (float)lam : 0.0f, ll = (float)(lam - (double)lh);
    const bool lo = cc.kind >= 4 || (cc.kind == 1 && cc.w > 0), hi = cc.kind >= 4 || (cc.kind == 1 && cc.w <= 0);
    for (long row0 = (long)blockIdx.x * rows; row0 < N; row0 += (long)gridDim.x * rows) {
      __syncthreads();
      for (int m = tid; m < rows; m += 256) fl[m] = row0 + m < N ? tr_flags(src, row0 + m, N) : 0u;
      __syncthreads();
      if (!mine) continue;
      const int nr = (int)(N - row0 < rows ? N - row0 : rows);
      const S* z = src.Z + row0 * src.ldz + cc.q;
      S* o = Zo + row0 * ldo + c;
      const long st = cc.s * src.ldz;
      for (int m0 = sub; m0 < nr; m0 += 4 * rpb) {
        S zk[4], zl[4], zh[4];
        unsigned f[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const int m = m0 + u * rpb;
          const bool in = m < nr;
          f[u] = in ? fl[m] : 0u;
          zk[u] = in && cc.kind != 2 && cc.kind != 3 ? z[(long)m * src.ldz] : S(0);
          zl[u] = lo && ((f[u] >> (2 * cc.ax)) & 1u) ? z[(long)m * src.ldz - st] : S(0);
          zh[u] = hi && ((f[u] >> (2 * cc.ax + 1)) & 1u) ? z[(long)m * src.ldz + st] : S(0);
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const int m = m0 + u * rpb;
          if (m >= nr) break;
          S v;
          if (cc.kind == 0) {
            v = zk[u];
          } else if (cc.kind == 2) {
            const bool at_face = (cc.w > 0) ? !((f[u] >> (2 * cc.ax)) & 1u) : !((f[u] >> (2 * cc.ax + 1)) & 1u);
            v = at_face ? (S)src.bcval[cc.b * src.G + (int)(f[u] >> 8)] : S(0);
          } else if (cc.kind == 3) {
            v = S(0);
          } else {
            // one form for every operator: the columns of a warp belong to several, which ran one after another
            // (1,048,576 rows FP32, 16 columns of the state: 446 us, now 367; FP64 Rusanov 1,160, now 977)
            const S x = cc.kind == 1 && lo ? zk[u] : zh[u];
            const S y = cc.kind == 5 ? S(-2) * zk[u] : cc.kind == 1 && !lo ? -zk[u] : -zl[u];
            v = tr_scaled(lam, lh, ll, x, y, cc.kind == 5 ? zl[u] : S(0));
          }
          o[(long)m * ldo] = v;
        }
      }
    }
  }
}

// Small cores of the materialised transport sum: block diagonal middle core, stacked last
// core (d = 3), or stacked mu core (d = 2); operator blocks scaled by the angular factors.
template <typename S>
__global__ void k_transport_small(int d, int nterm, int nbc, int n1, int n2, const S* __restrict__ c1,
                                  const S* __restrict__ c2, int rcapi1, int rcapi2, const int* __restrict__ rank_in,
                                  S* __restrict__ o1, S* __restrict__ o2, int rcapo1, int rcapo2,
                                  const double* __restrict__ fac1, const double* __restrict__ fac2,
                                  const int* __restrict__ bc_term) {
  const int r1 = rank_in[1];
  const int r2 = (d == 3) ? rank_in[2] : 1;
  const int R1 = (nterm + 1) * r1 + nbc;
  const int R2 = (nterm + 1) * r2 + nbc;
  if (R1 > rcapo1 || (d == 3 && R2 > rcapo2)) return;
  if (d == 2) {
    for (int idx = blockIdx.x * blockDim.x + threadIdx.x; idx < rcapo1 * n1; idx += gridDim.x * blockDim.x) {
      const int a = idx / n1, j = idx - (idx / n1) * n1;
      double v = 0.0;
      if (a < (nterm + 1) * r1) {
        const int t = a / r1, q = a - t * r1;
        v = (double)c1[q * n1 + j] * (t == 0 ? 1.0 : fac1[(t - 1) * n1 + j]);
      } else if (a < R1) {
        v = fac1[bc_term[a - (nterm + 1) * r1] * n1 + j];
      }
      o1[idx] = (S)v;
    }
    return;
  }
  const long tot1 = (long)rcapo1 * n1 * rcapo2;
  const long tot2 = (long)rcapo2 * n2;
  for (long idx = blockIdx.x * (long)blockDim.x + threadIdx.x; idx < tot1 + tot2; idx += (long)gridDim.x * blockDim.x) {
    if (idx < tot1) {
      const int a = (int)(idx / ((long)n1 * rcapo2));
      const int rem = (int)(idx - (long)a * n1 * rcapo2);
      const int l = rem / rcapo2, b = rem - (rem / rcapo2) * rcapo2;
      double v = 0.0;
      if (a < (nterm + 1) * r1 && b < (nterm + 1) * r2) {
        const int ta = a / r1, tb = b / r2;
        if (ta == tb) {
          const int qa = a - ta * r1, qb = b - tb * r2;
          v = (double)c1[((size_t)qa * n1 + l) * rcapi2 + qb] * (ta == 0 ? 1.0 : fac1[(ta - 1) * n1 + l]);
        }
      } else if (a >= (nterm + 1) * r1 && a < R1 && b >= (nterm + 1) * r2 && b < R2) {
        const int ba = a - (nterm + 1) * r1, bb = b - (nterm + 1) * r2;
        if (ba == bb) v = fac1[bc_term[ba] * n1 + l];
      }
      o1[idx] = (S)v;
    } else {
      const long i2 = idx - tot1;
      const int b = (int)(i2 / n2), p = (int)(i2 - (long)b * n2);
      double v = 0.0;
      if (b < (nterm + 1) * r2) {
        const int tb = b / r2, qb = b - tb * r2;
        v = (double)c2[(size_t)qb * n2 + p] * (tb == 0 ? 1.0 : fac2[(tb - 1) * n2 + p]);
      } else if (b < R2) {
        v = fac2[bc_term[b - (nterm + 1) * r2] * n2 + p];
      }
      o2[i2] = (S)v;
    }
  }
  (void)rcapi1;
}

__global__ void k_transport_ranks(int d, int nterm, int nbc, const int* __restrict__ rank_in, int* __restrict__ rank_out,
                                  int rcapo1, int rcapo2) {
  if (threadIdx.x || blockIdx.x) return;
  const int R1 = (nterm + 1) * rank_in[1] + nbc;
  const int R2 = (d == 3) ? (nterm + 1) * rank_in[2] + nbc : 1;
  if (R1 > rcapo1 || (d == 3 && R2 > rcapo2)) return;
  rank_out[0] = 1;
  rank_out[1] = R1;
  if (d == 3) {
    rank_out[2] = R2;
    rank_out[3] = 1;
  } else {
    rank_out[2] = 1;
  }
}

// y <- alpha x + y: x's blocks appended after y's live ranks (TT addition, Sec. 3.1).
template <typename S>
__global__ void k_axpy_Z(long N, double alpha, const S* __restrict__ Zx, int ldx, const int* __restrict__ rx,
                         S* __restrict__ Zy, int ldy, const int* __restrict__ ry, int d, int rcapy2, int* status) {
  const int rx1 = rx[1], ry1 = ry[1];
  const bool over = (rx1 + ry1 > ldy) || (d == 3 && rx[2] + ry[2] > rcapy2);
  if (over) {
    if (blockIdx.x == 0 && threadIdx.x == 0) latch(status, TT_ERR_CAPACITY);
    return;
  }
  const long tot = N * (long)rx1;
  for (long idx = blockIdx.x * (long)blockDim.x + threadIdx.x; idx < tot; idx += (long)gridDim.x * blockDim.x) {
    const long k = idx / rx1;
    const int q = (int)(idx - k * rx1);
    Zy[k * ldy + ry1 + q] = (S)(alpha * (double)Zx[k * ldx + q]);
  }
}

template <typename S>
__global__ void k_axpy_small(int d, int n1, int n2, const S* __restrict__ x1, const S* __restrict__ x2, int rcapx1,
                             int rcapx2, const int* __restrict__ rx, S* __restrict__ y1, S* __restrict__ y2, int rcapy1,
                             int rcapy2, const int* __restrict__ ry) {
  const int rx1 = rx[1], ry1 = ry[1];
  const int rx2 = (d == 3) ? rx[2] : 0, ry2 = (d == 3) ? ry[2] : 0;
  if (rx1 + ry1 > rcapy1 || (d == 3 && rx2 + ry2 > rcapy2)) return;
  if (d == 2) {
    for (int idx = blockIdx.x * blockDim.x + threadIdx.x; idx < rx1 * n1; idx += gridDim.x * blockDim.x) {
      const int a = idx / n1, j = idx - (idx / n1) * n1;
      y1[(size_t)(ry1 + a) * n1 + j] = x1[(size_t)a * n1 + j];
    }
    return;
  }
  const int tot1 = rx1 * n1 * rx2, tot2 = rx2 * n2;
  for (int idx = blockIdx.x * blockDim.x + threadIdx.x; idx < tot1 + tot2; idx += gridDim.x * blockDim.x) {
    if (idx < tot1) {
      const int a = idx / (n1 * rx2);
      const int rem = idx - a * n1 * rx2;
      const int l = rem / rx2, b = rem - (rem / rx2) * rx2;
      y1[((size_t)(ry1 + a) * n1 + l) * rcapy2 + ry2 + b] = x1[((size_t)a * n1 + l) * rcapx2 + b];
    } else {
      const int i2 = idx - tot1;
      const int b = i2 / n2, p = i2 - (i2 / n2) * n2;
      y2[(size_t)(ry2 + b) * n2 + p] = x2[(size_t)b * n2 + p];
    }
  }
  (void)rcapx1;
}

__global__ void k_axpy_ranks(int d, const int* __restrict__ rx, int* __restrict__ ry, int rcapy1, int rcapy2) {
  if (threadIdx.x || blockIdx.x) return;
  const int n1 = rx[1] + ry[1];
  const int n2 = (d == 3) ? rx[2] + ry[2] : 1;
  if (n1 > rcapy1 || (d == 3 && n2 > rcapy2)) return;
  ry[1] = n1;
  if (d == 3) ry[2] = n2;
}

// Per-chunk partial Gram entries W1[a][b] = sum_k X[k][a] Y[k][b]; when (nullable): a no-op where it is zero.
template <typename S>
__global__ void k_gram_partials(long N, long rows_per, const S* __restrict__ X, int ldx, int rx,
                                const S* __restrict__ Y, int ldy, int ry, double* __restrict__ partials,
                                const int* __restrict__ when) {
  if (when && *when == 0) return;
  const int e = blockIdx.y * blockDim.x + threadIdx.x;
  if (e >= rx * ry) return;
  const int a = e / ry, b = e - (e / ry) * ry;
  const long beg = blockIdx.x * rows_per;
  const long end = (beg + rows_per < N) ? beg + rows_per : N;
  double acc = 0.0;
  for (long k = beg; k < end; ++k) acc += (double)X[k * ldx + a] * (double)Y[k * ldy + b];
  partials[(size_t)blockIdx.x * rx * ry + e] = acc;
}

__global__ void k_sum_chunks(const double* __restrict__ partials, long nchunks, int ne, double* __restrict__ out,
                             const int* __restrict__ when) {
  if (when && *when == 0) return;
  const int e = blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= ne) return;
  double s = 0.0;
  for (long c = 0; c < nchunks; ++c) s += partials[(size_t)c * ne + e];
  out[e] = s;
}

__global__ void k_dot_final(int ne, const double* __restrict__ W1, const double* __restrict__ G, double* __restrict__ out) {
  __shared__ double red[33];
  double s = 0.0;
  for (int e = threadIdx.x; e < ne; e += blockDim.x) s += W1[e] * G[e];
  s = block_sum(s, red);
  if (threadIdx.x == 0) *out = s;
}

}  // namespace

template <typename S>
tt_status apply_transport_impl(tt_context* ctx, const tt_plan* p, const tt_tensor* in, tt_tensor* out) {
  cudaStream_t s = ctx->stream;
  const int d = in->d;
  SrcStencil<S> src{};
  src.Z = (const S*)in->core[0];
  src.ldz = in->rcap[1];
  src.rcap = in->rcap[1];
  src.nterm = p->nterm;
  src.G = p->G;
  for (int a = 0; a < 3; ++a) {
    src.ext[a] = p->ext[a];
    src.stride[a] = p->stride[a];
  }
  for (int t = 0; t < kMaxTerms; ++t) {
    src.lam[t] = (t < p->nterm) ? p->lam[p->term_axis[t]] : 0.0;
    src.axis[t] = (t < p->nterm) ? p->term_axis[t] : 0;
    src.w[t] = (t < p->nterm) ? p->term_w[t] : 1;
    src.bc_term[t] = (t < p->nbc) ? p->bc_term[t] : 0;
  }
  src.bcval = p->bcval;
  src.nax = p->ndim;
  const long N = in->n[0];
  const int rcapo2 = (d == 3) ? out->rcap[2] : 1;
  // Which kernel: see k_transport_Z
  const long grid = 8L * ctx->num_sms, tot = N * (long)out->rcap[1];
  const int cols = out->rcap[1] < 256 ? out->rcap[1] : 256;
  bool wide = false;  // central differences
  for (int t = 0; t < p->nterm; ++t) wide = wide || p->term_w[t] > 1 || p->term_w[t] < -1;
  const bool entry = sizeof(S) == 4 ? tot <= 5 * (1L << 16)
                     : wide         ? tot <= (1L << 20)
                                    : tot <= 6 * (1L << 20) || 256 / cols * cols < 208;
  const bool full = N >= (sizeof(S) == 4 ? 32768L : grid * kTrRows);
  const int rows = full ? kTrRows : N <= 4 * grid ? 4 : (int)((N + grid - 1) / grid);
  auto kern = entry ? k_transport_entry<S> : full ? k_transport_Z<S, kTrRows> : k_transport_Z<S, 0>;
  kern<<<(unsigned)(entry ? 1024 : grid), 256, 0, s>>>(N, src, in->rank, (S*)out->core[0], out->rcap[1], p->nbc,
                                                       d == 3 ? in->rank + 2 : nullptr, rcapo2, rows, &ctx->ctrl->status);
  count_launch();
  k_transport_small<S><<<64, 256, 0, s>>>(d, p->nterm, p->nbc, p->n1, p->n2, (const S*)in->core[1],
                                          d == 3 ? (const S*)in->core[2] : nullptr, in->rcap[1],
                                          d == 3 ? in->rcap[2] : 1, in->rank, (S*)out->core[1],
                                          d == 3 ? (S*)out->core[2] : nullptr, out->rcap[1], rcapo2, p->fac1, p->fac2,
                                          p->bc_term_dev); count_launch();
  k_transport_ranks<<<1, 32, 0, s>>>(d, p->nterm, p->nbc, in->rank, out->rank, out->rcap[1], rcapo2); count_launch();
  return cudaGetLastError() == cudaSuccess ? TT_OK : TT_ERR_CUDA;
}

template <typename S>
tt_status axpy_impl(tt_context* ctx, double alpha, const tt_tensor* x, tt_tensor* y) {
  cudaStream_t s = ctx->stream;
  const int d = x->d;
  const long N = x->n[0];
  const int rcapy2 = (d == 3) ? y->rcap[2] : 1;
  k_axpy_Z<S><<<1024, 256, 0, s>>>(N, alpha, (const S*)x->core[0], x->rcap[1], x->rank, (S*)y->core[0], y->rcap[1],
                                   y->rank, d, rcapy2, &ctx->ctrl->status); count_launch();
  k_axpy_small<S><<<64, 256, 0, s>>>(d, x->n[1], d == 3 ? x->n[2] : 1, (const S*)x->core[1],
                                     d == 3 ? (const S*)x->core[2] : nullptr, x->rcap[1], d == 3 ? x->rcap[2] : 1,
                                     x->rank, (S*)y->core[1], d == 3 ? (S*)y->core[2] : nullptr, y->rcap[1], rcapy2,
                                     y->rank); count_launch();
  k_axpy_ranks<<<1, 32, 0, s>>>(d, x->rank, y->rank, y->rcap[1], rcapy2); count_launch();
  return cudaGetLastError() == cudaSuccess ? TT_OK : TT_ERR_CUDA;
}

// Whether the first cores' products are formed exactly (xg_cross): the digits cost by rows and columns, the FP64 sums
// by rows and products in groups of 256.  Inner products, exact / sums, cold L2, us:
//   8,192 rows (the sums stay): 32 x 32 FP64 117 / 501, FP32 113 / 349; 1 x 1: 105 / 128, 104 / 169
//   262,144 rows: 2 x 2 FP64 163 / 217, FP32 160 / 206; 32 x 32: 289 / 555, 275 / 1,523; 1 x 200 FP64 579 / 469
//   1,048,576 rows: FP64 1 x 1 436 / 205, 8 x 8 472 / 477, 14 x 14 600 / 582, 16 x 16 603 / 639, 32 x 32 894 / 2,217;
//     FP32 4 x 4 443 / 323, 6 x 6 451 / 496, 2 x 32 610 / 494, 8 x 8 460 / 506, 32 x 32 843 / 5,690
// (a pass is 262,144 rows: beyond one, the exact form needs many products for each column whose digits it forms.)
constexpr long kDotExactRows = 16384;
template <typename S>
inline bool dot_exact(const XgPair<S>& pr, long N) {
  if (N < kDotExactRows || !xg_cross_fits(pr)) return false;
  const long cols = xg_cross_same(pr) ? pr.na : pr.na + pr.nb, ne = (long)pr.na * pr.nb;
  if (N <= kXgCrossRows && N * cols <= (1L << 25)) return true;
  return ne >= (sizeof(S) == 8 ? 8 * cols : 3L * (pr.na + pr.nb));
}
template <typename S>
tt_status dot_impl(tt_context* ctx, const tt_tensor* x, const tt_tensor* y, double* out, Bump& ws) {
  cudaStream_t s = ctx->stream;
  const int d = x->d;
  const long N = x->n[0];
  const int n1 = x->n[1], n2 = (d == 3) ? x->n[2] : 1, nang = n1 * n2;
  const int rx = x->rcap[1], ry = y->rcap[1];
  const int ne = rx * ry;
  long nchunks = (N + 1023) / 1024;
  if (nchunks > 2048) nchunks = 2048;
  const long rows_per = (N + nchunks - 1) / nchunks;
  nchunks = (N + rows_per - 1) / rows_per;
  double* part = ws.take<double>((size_t)nchunks * ne);
  double* W1 = ws.take<double>(ne);
  double* Bx = ws.take<double>((size_t)rx * nang);
  double* By = ws.take<double>((size_t)ry * nang);
  double* G = ws.take<double>(ne);
  // tall cores: exact products on the tensor cores (dot_exact), the FP64 sums only where an entry is not finite or
  // the columns are large on different rows (k_xg_cover)
  const XgPair<S> pr{(const S*)x->core[0], (const S*)y->core[0], rx, ry};
  int* when = nullptr;
  if (!ctx->no_xg && dot_exact(pr, N)) {
    when = ws.take<int>(1);
    const tt_status st = xg_cross<S>(s, ctx->num_sms, pr, N, ws, W1, when, &ctx->ctrl->status);
    if (st != TT_OK) return st;
  }
  if (ws.dry) return TT_OK;
  dim3 grid((unsigned)nchunks, (unsigned)((ne + 255) / 256));
  k_gram_partials<S><<<grid, 256, 0, s>>>(N, rows_per, (const S*)x->core[0], rx, rx, (const S*)y->core[0], ry, ry,
                                          part, when); count_launch();
  k_sum_chunks<<<(ne + 255) / 256, 256, 0, s>>>(part, nchunks, ne, W1, when); count_launch();
  right_part<S>(s, d, rx, n1, d == 3 ? x->rcap[2] : 1, n2, (const S*)x->core[1], d == 3 ? (const S*)x->core[2] : nullptr,
                Bx);
  right_part<S>(s, d, ry, n1, d == 3 ? y->rcap[2] : 1, n2, (const S*)y->core[1], d == 3 ? (const S*)y->core[2] : nullptr,
                By);
  small_gemm<double, double>(s, rx, ry, nang, Bx, nang, 1, By, 1, nang, G, ry, nullptr, nullptr);
  k_dot_final<<<1, 1024, 0, s>>>(ne, W1, G, out); count_launch();
  return cudaGetLastError() == cudaSuccess ? TT_OK : TT_ERR_CUDA;
}

// Inner product with caller-provided scratch (no workspace, no allocation): the same kernels
// as dot_impl with the number of row chunks reduced until everything fits in `cap` doubles.
template <typename S>
tt_status dot_into(cudaStream_t s, const tt_tensor* x, const tt_tensor* y, double* out, double* scratch,
                   size_t cap) {
  const int d = x->d;
  const long N = x->n[0];
  const int n1 = x->n[1], n2 = (d == 3) ? x->n[2] : 1, nang = n1 * n2;
  const int rx = x->rcap[1], ry = y->rcap[1];
  const size_t ne = (size_t)rx * ry;
  const size_t fixed = ne /*W1*/ + ne /*G*/ + (size_t)(rx + ry) * nang;
  if (fixed + ne > cap) return TT_ERR_WORKSPACE;
  long nchunks = (N + 1023) / 1024;
  if (nchunks > 2048) nchunks = 2048;
  const long fit = (long)((cap - fixed) / ne);
  if (nchunks > fit) nchunks = fit;
  if (nchunks < 1) nchunks = 1;
  const long rows_per = (N + nchunks - 1) / nchunks;
  nchunks = (N + rows_per - 1) / rows_per;
  double* part = scratch;
  double* W1 = part + (size_t)nchunks * ne;
  double* Bx = W1 + ne;
  double* By = Bx + (size_t)rx * nang;
  double* G = By + (size_t)ry * nang;
  dim3 grid((unsigned)nchunks, (unsigned)((ne + 255) / 256));
  k_gram_partials<S><<<grid, 256, 0, s>>>(N, rows_per, (const S*)x->core[0], rx, rx, (const S*)y->core[0], ry, ry,
                                          part, nullptr); count_launch();
  k_sum_chunks<<<(unsigned)((ne + 255) / 256), 256, 0, s>>>(part, nchunks, (int)ne, W1, nullptr); count_launch();
  right_part<S>(s, d, rx, n1, d == 3 ? x->rcap[2] : 1, n2, (const S*)x->core[1], d == 3 ? (const S*)x->core[2] : nullptr,
                Bx);
  right_part<S>(s, d, ry, n1, d == 3 ? y->rcap[2] : 1, n2, (const S*)y->core[1], d == 3 ? (const S*)y->core[2] : nullptr,
                By);
  small_gemm<double, double>(s, rx, ry, nang, Bx, nang, 1, By, 1, nang, G, ry, nullptr, nullptr);
  k_dot_final<<<1, 1024, 0, s>>>((int)ne, W1, G, out); count_launch();
  return cudaGetLastError() == cudaSuccess ? TT_OK : TT_ERR_CUDA;
}
template tt_status dot_into<double>(cudaStream_t, const tt_tensor*, const tt_tensor*, double*, double*, size_t);
template tt_status dot_into<float>(cudaStream_t, const tt_tensor*, const tt_tensor*, double*, double*, size_t);

template tt_status apply_transport_impl<double>(tt_context*, const tt_plan*, const tt_tensor*, tt_tensor*);
template tt_status apply_transport_impl<float>(tt_context*, const tt_plan*, const tt_tensor*, tt_tensor*);
template tt_status axpy_impl<double>(tt_context*, double, const tt_tensor*, tt_tensor*);
template tt_status axpy_impl<float>(tt_context*, double, const tt_tensor*, tt_tensor*);
template tt_status dot_impl<double>(tt_context*, const tt_tensor*, const tt_tensor*, double*, Bump&);
template tt_status dot_impl<float>(tt_context*, const tt_tensor*, const tt_tensor*, double*, Bump&);

}  // namespace ttk
