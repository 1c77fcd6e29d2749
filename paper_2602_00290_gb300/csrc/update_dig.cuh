// Update pass Z_new = Z_sum W from digits on the tensor cores: rows and weights as fixed-point integers in
// balanced base 256 (xgram.cuh), FP32 passes with 4 digits, FP64 passes with 8.
//
// The columns x_c of a row are the centre row, its differences with the neighbours (exact subtractions, as in
// k_update_blk) and the inflow columns.  With a power of two per column (2^a_c, its size: in the
// triangular factor, or its largest entry) and one per row (2^r), v_c = round(x_c 2^-(r + a_c) ..) keeps 2^-30 (FP32)
// or 2^-62 (FP64) of the row's largest scaled entry: rows and columns of any grading keep more bits than
// the arithmetic that the pass stands for.  The weights w_cn 2^a_c get a power of two per output column.  Then
//   sum_c v_c w_cn = sum_o 256^(2 NS - 2 - o) A_o,   A_o = sum_{i + j = o} sum_c d_j e_i
// for digits d_j of v and e_i of w, and the A_o are integers below 2^24 in the FP32 accumulators of
// tcgen05.mma.kind::f16, exact except in the lowest orders of wide FP64 passes (where a lost bit is 2^-60 of the
// result).  Orders from NS (FP32: NS + 1 where the accumulators fit) on are dropped: 2^-28 (2^-36) and 2^-59
// of the largest product; the read-back rounds once.  For digit j of the rows the operand B is [e_0 | .. | e_(NS-1-j)], a prefix
// of one resident tile, and its products land in the orders j, j + 1, ..: one MMA does all of them.
//
// Eight or twelve warps form the digits (a row and 16 columns each) in a ring of K steps, one thread issues the
// MMAs, eight warps read one of two accumulator sets back (half a row per thread) and run the epilogue.
//
// Why: the FP64 pass ran on the FP64 FMA pipe, 1/64 of the FP32 rate; the FP32 passes between block barriers (FMAs
// at wide ranks, split TF32).  Measured for both updates of a step, scales included: FP64, 1,048,576 rows x
// 160 columns x 32 outputs 12.6 -> 1.6 ms; FP32 storage 1.06 -> 0.72 ms; 3,538,944 x 242 x 48, FP32 11.5 -> 3.4
// ms; FP64 storage in an FP32 pass, 131,072 rows x 32: 0.63 -> 0.17 ms.  Bound by the integer work of the digits (FP32: about
// half of the issue slots; the tensor cores are busy 15 % of the time), not by memory.
#pragma once
#include "update_blk.cuh"
#include "xgram.cuh"

namespace ttk {

constexpr int kUdEpi = 8;                        // epilogue warps: two per 32 rows, half of the columns each
// Digit-forming warps: three K steps at a time, FP64 passes two (their rows take twice the registers).
__host__ __device__ constexpr int ud_prod(int ns) { return ns == 4 ? 12 : 8; }
__host__ __device__ constexpr int ud_threads(int ns) { return 32 * (kUdEpi + ud_prod(ns) + 1); }
constexpr int kUdMaxSlots = 8;
constexpr int kUdMaxUnits = 64;                  // K steps of 16 columns
// Passes of fewer rows stay with the other kernels (eight tiles leave most SMs idle there).  Both updates of a plane
// step, all launches, digits against before: 1,024 rows, rank 32: FP64 78 / 123 us, FP32 60 / 82 us; rank 8: 59 / 75,
// 46 / 65 us; rank 2: 56 / 64, 47 / 67 us; 4,096 rows, rank 32: 69 / 114, 50 / 83 us; 65,536 rows, rank 32:
// 151 / 883, 82 / 166 us; 589,824 rows, rank 48, FP32: 596 / 1,783 us.
constexpr long kUdMinRows = 1024;
// Where the caller asked for 3xTF32 (k_update_tc, FP32 storage): 4,096 rows, rank 32: 50 / 94 us; 131,072 rows:
// 118 / 218 us.  Below, the split-TF32 kernel that the precision names keeps the first update (1,024 rows, rank 32:
// 60 / 92 us), for the arithmetic asked for, not for speed.
constexpr long kUdMinRowsTc = 4096;
constexpr int kUdDead = 1 << 20;                 // column scale that makes every digit zero
constexpr int kUdMinExp = -8000;                 // row scale of a zero row
// Rows of FP32 storage in an FP32 pass whose scales (row + column) reach below kUdPowMin, where the power of two of an
// entry leaves FP32 (rows below about 1e-29): their entries are multiplied by 2^kUdRaise first, and the row's scale
// is stored as much larger.  Not where the columns' sizes differ by 2^kUdWide or more: the raised entries could
// leave FP32 at the other end, and rows end at kUdPowMin.
constexpr int kUdRaised = 1 << 22, kUdRaise = 28, kUdPowMin = -98, kUdWide = 180;

// Scales of a pass and where its weights' digits go (workspace).
struct UdBufs {
  int* cexp = nullptr;        // [ncap] size of each column (launch_ud_scales, launch_ud_scales_cols)
  unsigned long long* slots = nullptr;  // [columns] largest entries (launch_ud_scales_cols)
  short* rho = nullptr;       // [nrows] exponent of a storage row (stencil passes)
  int* rinfo = nullptr;       // [nrows] scale of a row of the pass (16 bits), neighbour flags from bit 16, kUdRaised
  unsigned char* w = nullptr; // digits of the weights, exponents
};

__host__ __device__ inline int ud_kp(int kcap) { return (kcap + 15) & ~15; }  // the MMA's N: multiples of 16
// Orders kept.
__host__ __device__ inline int ud_orders(int ns, int kp) { return ns == 4 && 5 * kp <= 256 ? 5 : ns; }

// K steps.  Stencil sums: pairs of 8 centre columns; then 8 lower and 8 upper differences of one axis;
// then the inflow columns.  Explicit rows: 16 columns each.
template <typename S>
__host__ __device__ inline int ud_units(const SrcStencil<S>& s, const LivePattern& lp) {
  const int ng = (s.rcap + 7) / 8;
  return (ng + 1) / 2 + s.nax * ng + (lp.nextra ? 1 : 0);
}
template <typename S>
__host__ __device__ inline int ud_units(const SrcRows<S>&, const LivePattern& lp) { return (lp.ncap() + 15) / 16; }

// Column of K step u, half h, place e: block (0 centre, 1 + 2 axis lower, 2 + 2 axis upper, 8 inflow, -1
// none) and column of it.
struct UdCol {
  int b, q;
};
template <typename S>
__device__ __forceinline__ UdCol ud_col(const SrcStencil<S>& s, const LivePattern& lp, int u, int h, int e) {
  const int ng = (s.rcap + 7) / 8, np = (ng + 1) / 2;
  UdCol c{-1, 0};
  if (u < np) {
    c.q = 16 * u + 8 * h + e;
    if (c.q < s.rcap) c.b = 0;
  } else if (u < np + s.nax * ng) {
    const int ax = (u - np) / ng;
    c.q = 8 * (u - np - ax * ng) + e;
    if (c.q < s.rcap) c.b = 1 + 2 * ax + h;
  } else if (h == 0 && e < lp.nextra) {
    c.b = 8;
    c.q = e;
  }
  return c;
}
template <typename S>
__device__ __forceinline__ UdCol ud_col(const SrcRows<S>&, const LivePattern& lp, int u, int h, int e) {
  UdCol c{-1, 16 * u + 8 * h + e};
  if (c.q < lp.ncap()) c.b = 0;
  return c;
}
// Its column of the pass that gives the scale, or -1 for a dead one.
template <typename S>
__device__ __forceinline__ int ud_scale_col(const SrcStencil<S>& s, const LivePattern& lp, UdCol c, int r) {
  if (c.b < 0) return -1;
  if (c.b == 8) {
    const int k = (s.nterm + 1) * s.rcap + c.q;
    return lp.live(k, r) ? k : -1;
  }
  return c.q < r ? c.q : -1;
}
template <typename S>
__device__ __forceinline__ int ud_scale_col(const SrcRows<S>&, const LivePattern& lp, UdCol c, int r) {
  return c.b == 0 && lp.live(c.q, r) ? c.q : -1;
}
// Weight of the column for output n (live columns).
template <typename S>
__device__ __forceinline__ double ud_weight(const SrcRows<S>&, UdCol c, int n, const double* W, int kcap) {
  return W[(size_t)c.q * kcap + n];
}
template <typename S>
__device__ __forceinline__ double ud_weight(const SrcStencil<S>& s, UdCol c, int n, const double* W, int kcap) {
  if (c.b == 0) return W[(size_t)c.q * kcap + n];
  if (c.b == 8) return W[(size_t)((s.nterm + 1) * s.rcap + c.q) * kcap + n];
  double sum = 0.0;
  for (int t = 1; t <= s.nterm; ++t) {
    const int ax = s.axis[t - 1];
    if (c.b != 1 + 2 * ax && c.b != 2 + 2 * ax) continue;
    double cL, cH;
    blk_coefs(s, t, cL, cH);
    const double cf = (c.b == 1 + 2 * ax) ? cL : cH;
    if (cf != 0.0) sum += cf * W[(size_t)(t * s.rcap + c.q) * kcap + n];
  }
  return sum;
}

// Exponent of every column's largest entry in the triangular factor (one block per column).
__global__ void __launch_bounds__(128) k_ud_colexp(const double* __restrict__ RZ, int n, int* __restrict__ cexp) {
  __shared__ int m;
  const int c = blockIdx.x;
  if (threadIdx.x == 0) m = 0;
  __syncthreads();
  int e = 0;
  for (int i = threadIdx.x; i < n; i += blockDim.x)
    e = max(e, (int)((__double_as_longlong(RZ[(size_t)i * n + c]) >> 52) & 0x7ff));
  e = __reduce_max_sync(0xffffffffu, e);
  if ((threadIdx.x & 31) == 0) atomicMax(&m, e);
  __syncthreads();
  if (threadIdx.x == 0) cexp[c] = m ? m - 1023 : 0;
}

// Exponent of every storage column's largest entry (slots, k_xg_colmax) and, behind the operators' columns, of the
// inflow columns'; the operators' own columns have no digits of their own.
static __global__ void __launch_bounds__(256) k_ud_slotexp(int ncol, int extra0, int nextra,
                                                    const unsigned long long* __restrict__ slots,
                                                    int* __restrict__ cexp) {
  for (int c = threadIdx.x; c < ncol + nextra; c += blockDim.x) {
    const int e = (int)((slots[c] >> 52) & 0x7ff);
    cexp[c < ncol ? c : extra0 + c - ncol] = e ? e - 1023 : 0;
  }
}

__device__ __forceinline__ int ud_exp(double x) { return (int)((__double_as_longlong(x) >> 52) & 0x7ff) - 1023; }
__device__ __forceinline__ int ud_exp(float x) { return max((int)((__float_as_uint(x) >> 23) & 0xff), 1) - 127; }
// Row information of scale m and neighbour flags f; raise: an FP32 pass over FP32 storage, amin, amax: the smallest and
// largest column.
__device__ __forceinline__ int ud_rinfo(int m, unsigned f, bool raise, int amin, int amax) {
  const bool up = raise && amax - amin < kUdWide && m + amin < kUdPowMin && m > kUdMinExp + 1;
  return (int)((f << 16) | (up ? (unsigned)kUdRaised : 0u) | ((unsigned)(up ? m + kUdRaise : m) & 0xffffu));
}
__device__ __forceinline__ int ud_row_scale(int inf) {
  return (int)(short)(inf & 0xffff) - ((inf & kUdRaised) ? kUdRaise : 0);
}
__device__ __forceinline__ float ud_row_raise(int inf) {
  return __int_as_float(0x3f800000 + ((inf & kUdRaised) ? kUdRaise << 23 : 0));
}

// Smallest and largest of the live columns (kUdDead, 0 where there are none); a full warp.
__device__ __forceinline__ void ud_col_range(const int* cexp, int ncol, const LivePattern& lp, int r, int& amin,
                                             int& amax) {
  amin = kUdDead;
  amax = -kUdDead;
  for (int c = threadIdx.x & 31; c < ncol; c += 32)
    if (lp.live(c, r)) {
      amin = min(amin, cexp[c]);
      amax = max(amax, cexp[c]);
    }
  amin = __reduce_min_sync(0xffffffffu, amin);
  amax = __reduce_max_sync(0xffffffffu, amax);
}

// rho of the rows of a storage matrix: largest exponent of an entry against its column's; eight lanes take
// a row (rows of 33 columns waste little), a warp 16 rows at a time.
template <typename S, typename O>
__global__ void __launch_bounds__(256) k_ud_rows(const S* __restrict__ A, long ld, LivePattern lp, int ncol, long nrows,
                                                 const int* __restrict__ cexp, O* __restrict__ out, bool raise) {
  const int lane = threadIdx.x & 31, l8 = lane & 7, g = lane >> 3;
  const long warp = ((long)blockIdx.x * blockDim.x + threadIdx.x) >> 5, nw = ((long)gridDim.x * blockDim.x) >> 5;
  const int r = lp.r_ptr ? *lp.r_ptr : lp.rcap;
  int amin, amax;
  ud_col_range(cexp, ncol, lp, r, amin, amax);
  // rows at the end of the storage's numbers against their columns share one scale
  const int low = amin == kUdDead ? kUdMinExp
                                  : (sizeof(S) == 8 ? -950 : amax - amin < kUdWide ? -126 : kUdPowMin) - amin;
  for (long k0 = 16 * warp; k0 < nrows; k0 += 16 * nw) {
    int m[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) m[u] = low;
#pragma unroll 2
    for (int c = l8; c < ncol; c += 8) {
      if (!lp.live(c, r)) continue;
      const int ce = cexp[c];
      S x[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) x[u] = k0 + 4 * u + g < nrows ? A[(k0 + 4 * u + g) * ld + c] : S(0);
#pragma unroll
      for (int u = 0; u < 4; ++u) m[u] = x[u] != S(0) ? max(m[u], ud_exp(x[u]) - ce) : m[u];
    }
#pragma unroll
    for (int u = 0; u < 4; ++u) {
#pragma unroll
      for (int o = 1; o < 8; o <<= 1) m[u] = max(m[u], __shfl_xor_sync(0xffffffffu, m[u], o));
    }
    const int v = l8 == 0 ? m[0] : l8 == 1 ? m[1] : l8 == 2 ? m[2] : m[3];
    const long k = k0 + 4 * l8 + g;
    if (l8 < 4 && k < nrows) out[k] = sizeof(O) == 2 ? (O)v : (O)ud_rinfo(v, 0u, raise, amin, amax);
  }
}

// Scale of a row of the stencil pass, from its own row and its neighbours' (a difference is at most twice
// the larger one), the inflow columns, and the neighbour flags.
template <typename S>
__global__ void __launch_bounds__(256) k_ud_info(const __grid_constant__ SrcStencil<S> src, LivePattern lp, long nrows,
                                                 const int* __restrict__ cexp, const short* __restrict__ rho,
                                                 int* __restrict__ rinfo, bool raise) {
  const long k = (long)blockIdx.x * blockDim.x + threadIdx.x;
  int amin, amax;
  ud_col_range(cexp, src.rcap, LivePattern{lp.r_ptr, lp.rcap, 1, 0}, lp.r_ptr ? *lp.r_ptr : lp.rcap, amin, amax);
  if (k >= nrows) return;
  int m = rho[k];
  unsigned f = 0u;
  for (int a = 0; a < src.nax; ++a) {
    const unsigned idx = ((unsigned)k / (unsigned)src.stride[a]) % (unsigned)src.ext[a];
    if (idx > 0u) {
      f |= 1u << (2 * a);
      m = max(m, (int)rho[k - src.stride[a]]);
    }
    if (idx + 1u < (unsigned)src.ext[a]) {
      f |= 2u << (2 * a);
      m = max(m, (int)rho[k + src.stride[a]]);
    }
  }
  ++m;
  for (int e = 0; e < lp.nextra; ++e) {
    const int tt = src.bc_term[e], ax = src.axis[tt];
    const bool at_face = src.w[tt] > 0 ? !((f >> (2 * ax)) & 1u) : !((f >> (2 * ax + 1)) & 1u);
    const double v = at_face ? src.bcval[e * src.G + (int)((unsigned)k % (unsigned)src.G)] : 0.0;
    if (v != 0.0) m = max(m, ud_exp(v) - cexp[(src.nterm + 1) * src.rcap + e]);
  }
  rinfo[k] = ud_rinfo(m, f, raise, amin, amax);
}

// Digits of the weights, one block per output column n, in the layout of the B operand (K-major core
// matrices): K step u, K eight h, row i kp + n (digit i).  wexp[n]: exponent of the column's
// largest scaled weight.
template <int NS, class Src>
__global__ void __launch_bounds__(256) k_ud_weights(const __grid_constant__ Src src, LivePattern lp,
                                                    const double* __restrict__ W, int kcap, int kp,
                                                    const int* __restrict__ cexp, unsigned short* __restrict__ B,
                                                    int* __restrict__ wexp, int* __restrict__ aexp,
                                                    int* __restrict__ status) {
  __shared__ double wv[16 * kUdMaxUnits];
  __shared__ int em_s;
  const int n = blockIdx.x, tid = threadIdx.x;
  const int r = lp.r_ptr ? *lp.r_ptr : lp.rcap;
  const int K = 16 * ud_units(src, lp);
  if (tid == 0) em_s = 0;
  __syncthreads();
  int em = 0;
  for (int k = tid; k < K; k += blockDim.x) {
    const UdCol c = ud_col(src, lp, k >> 4, (k >> 3) & 1, k & 7);
    const int sc = ud_scale_col(src, lp, c, r);
    double v = 0.0;
    if (sc >= 0 && n < kcap) {
      v = ud_weight(src, c, n, W, kcap);
      if (v != 0.0) v = ldexp(v, cexp[sc]);
      em = max(em, (int)((__double_as_longlong(v) >> 52) & 0x7ff));
    }
    wv[k] = v;
    if (n == 0) aexp[k] = sc >= 0 ? cexp[sc] : kUdDead;
  }
  atomicMax(&em_s, em);
  __syncthreads();
  em = em_s;
  if (tid == 0) wexp[n] = em - 1023;
  if (tid == 0 && em == 0x7ff) latch(status, TT_ERR_NONFINITE);
  const int nr8 = NS * kp / 8;
  for (int k = tid; k < K; k += blockDim.x) {
    unsigned dig[NS];
    xg_digits2<NS>(xg_fix(wv[k], em + 62 - (8 * NS - 2)), 0ll, dig);
#pragma unroll
    for (int i = 0; i < NS; ++i) {
      const int row = i * kp + n;
      B[(((size_t)(k >> 3) * nr8 + (row >> 3)) * 128 + (row & 7) * 16) / 2 + (k & 7)] = (unsigned short)(dig[i] & 0xffffu);
    }
  }
}

// x 2^(8 NS - 3 - scale) as an integer below 2^(8 NS - 2), scale: row scale + column scale.  FP64 entries on the
// integer units, truncated (the FP64 pipe is narrow; the scales keep zero's exponent out of range); `top`
// collects the largest exponent field.
template <int NS>
__device__ __forceinline__ auto ud_fix(double x, int scale, int& top) {
  using V = typename std::conditional<NS == 4, int, long long>::type;
  const unsigned long long b = (unsigned long long)__double_as_longlong(x);
  const unsigned hi = (unsigned)(b >> 32);
  const int e = (int)((hi >> 20) & 0x7ffu);
  top = max(top, e);
  const int sh = scale + 1024 - e;  // at least 1
  const V sg = (V)((int)hi >> 31);
  if constexpr (NS == 4) {
    const unsigned m = __funnelshift_l((unsigned)b, (hi & 0xfffffu) | 0x100000u, 10);  // 31 bits
    return ((V)(m >> min(max(sh, 1), 31)) ^ sg) - sg;
  } else {
    const unsigned long long m = ((b & 0xfffffffffffffull) | 0x10000000000000ull) << 10;  // 63 bits
    return ((V)(m >> min(max(sh, 1), 63)) ^ sg) - sg;
  }
}
// FP32 entries of an FP64 pass: exact.
template <int NS>
__device__ __forceinline__ long long ud_fix(float x, int scale, int& top) {
  const unsigned b = __float_as_uint(x);
  const int e = (int)((b >> 23) & 0xff);
  top = max(top, e);
  const unsigned long long m = (unsigned long long)((b & 0x7fffffu) | (e ? 0x800000u : 0u)) << 39;
  const long long sg = (long long)((int)b >> 31);
  return ((long long)(m >> min(max(scale + 128 - max(e, 1), 1), 63)) ^ sg) - sg;
}
// FP32 entries of an FP32 pass: a power of two (zero for dead columns) and a conversion, rounded to nearest.
__device__ __forceinline__ float ud_pow(int scale) { return __int_as_float(max(156 - scale, 0) << 23); }

// Four balanced digits of two biased 32-bit words (see xg_digits2).
__device__ __forceinline__ void ud_digits4(unsigned a, unsigned b, unsigned (&dig)[4]) {
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    const unsigned k = (unsigned)(3 - j);
    unsigned x = (__byte_perm(a, b, k | (4u + k) << 8) & 0x00ff00ffu) | 0x64006400u;
    asm("sub.rn.f16x2 %0, %0, %1;" : "+r"(x) : "r"(0x64806480u));  // - 1152
    dig[j] = x;
  }
}

// Rows and columns of a digit-forming thread: 32 rows of a warp in four groups of eight, four lanes per row, two
// neighbouring columns each.  A load of the warp covers whole 32-byte sectors (a lane with eight columns of a
// row to itself fetched every sector twice), a store whole core matrices.
template <typename S>
struct alignas(2 * sizeof(S)) UdPair {
  S a, b;
};
template <typename S>
__device__ __forceinline__ void ud_load2(const S* p, bool vec, int left, UdPair<S>& x) {
  if (vec) {
    x = *reinterpret_cast<const UdPair<S>*>(p);
  } else {
    x.a = left > 0 ? p[0] : S(0);
    x.b = left > 1 ? p[1] : S(0);
  }
}

// Digits of two fixed-point columns of a row to the stage (digit j at 2 j + h K eights), four at a time.
template <int NS, typename V>
__device__ __forceinline__ void ud_store2(V v0, V v1, unsigned char* at) {
#pragma unroll
  for (int w = 0; w < NS / 4; ++w) {
    unsigned a, b, dig[4];
    if constexpr (NS == 4) {
      a = (unsigned)v0 + 0x80808080u;
      b = (unsigned)v1 + 0x80808080u;
    } else {
      const unsigned long long p = (unsigned long long)v0 + 0x8080808080808080ull;
      const unsigned long long q = (unsigned long long)v1 + 0x8080808080808080ull;
      a = w ? (unsigned)p : (unsigned)(p >> 32);
      b = w ? (unsigned)q : (unsigned)(q >> 32);
    }
    ud_digits4(a, b, dig);
#pragma unroll
    for (int j = 0; j < 4; ++j) *reinterpret_cast<unsigned*>(at + (size_t)(4 * w + j) * 4096) = dig[j];
  }
}
// Fixed point of two columns; `bad` on an Inf or NaN in a live one.
template <int NS, typename S, typename V>
__device__ __forceinline__ void ud_fix2(const UdPair<S>& x, int2 a, int r, V& v0, V& v1, bool& bad) {
  int top = 0;
  v0 = ud_fix<NS>(x.a, r + a.x, top);
  v1 = ud_fix<NS>(x.b, r + a.y, top);
  if (top == (sizeof(S) == 4 ? 255 : 2047))
    bad = bad || (!isfinite(x.a) && a.x != kUdDead) || (!isfinite(x.b) && a.y != kUdDead);
}
__device__ __forceinline__ void ud_fix2f(float x0, float x1, float up, float f0, float f1, int& v0, int& v1, bool& bad) {
  v0 = __float2int_rn((x0 * up) * f0);
  v1 = __float2int_rn((x1 * up) * f1);
  const float t = fmaf(x1, 0.0f, x0 * 0.0f);
  if (t != 0.0f) bad = bad || (!isfinite(x0) && f0 != 0.0f) || (!isfinite(x1) && f1 != 0.0f);
}

// What a K step needs from memory: 16 columns of four rows, or 8 columns of the rows and their neighbours.
template <typename S>
struct UdRaw {
  UdPair<S> x[4], y[4], c[4];
};
// k[g] < 0: a row past the end; c2: the thread's first column of eight; f[g]: neighbour flags.
template <typename S>
__device__ __forceinline__ void ud_load(const SrcStencil<S>& s, const LivePattern& lp, int u, long k0, long nrows,
                                        const int (&inf)[4], int c2, bool vec, UdRaw<S>& w) {
  const int ng = (s.rcap + 7) / 8, np = (ng + 1) / 2;
  const UdPair<S> zero{S(0), S(0)};
  if (u < np) {
    const int q = 16 * u + c2;
#pragma unroll
    for (int g = 0; g < 4; ++g) {
      w.x[g] = w.y[g] = zero;
      if (k0 + 8 * g >= nrows) continue;
      const S* row = s.Z + (k0 + 8 * g) * s.ldz;
      ud_load2(row + q, vec, s.rcap - q, w.x[g]);
      if (16 * u + 8 < s.rcap) ud_load2(row + q + 8, vec, s.rcap - q - 8, w.y[g]);
    }
  } else if (u < np + s.nax * ng) {
    const int ax = (u - np) / ng, q = 8 * (u - np - ax * ng) + c2;
    const long st = s.stride[ax] * s.ldz;
#pragma unroll
    for (int g = 0; g < 4; ++g) {
      w.x[g] = w.y[g] = w.c[g] = zero;
      if (k0 + 8 * g >= nrows) continue;
      const S* row = s.Z + (k0 + 8 * g) * s.ldz;
      const unsigned f = (unsigned)inf[g] >> (16 + 2 * ax);
      ud_load2(row + q, vec, s.rcap - q, w.c[g]);
      if (f & 1u) ud_load2(row - st + q, vec, s.rcap - q, w.x[g]);
      if (f & 2u) ud_load2(row + st + q, vec, s.rcap - q, w.y[g]);
    }
  }
}
template <typename S>
__device__ __forceinline__ void ud_load(const SrcRows<S>& s, const LivePattern& lp, int u, long k0, long nrows,
                                        const int (&)[4], int c2, bool vec, UdRaw<S>& w) {
  const int nc = lp.ncap(), q = 16 * u + c2;
  const UdPair<S> zero{S(0), S(0)};
#pragma unroll
  for (int g = 0; g < 4; ++g) {
    w.x[g] = w.y[g] = zero;
    if (k0 + 8 * g >= nrows) continue;
    const S* row = s.A + (k0 + 8 * g) * s.ld + q;
    ud_load2(row, vec && q + 2 <= nc, nc - q, w.x[g]);
    ud_load2(row + 8, vec && q + 10 <= nc, nc - q - 8, w.y[g]);
  }
}
// Its digits.  The differences C - L and H - C are formed in the row's fixed point: the same unit as their
// digits have.  at: the stage at the thread's first row and columns (groups of rows 128 bytes apart).
template <int NS, typename S>
__device__ __forceinline__ void ud_digits(const SrcStencil<S>& s, const LivePattern& lp, int u, long k0, long nrows,
                                          const int (&inf)[4], int c2, const UdRaw<S>& w, const int* a,
                                          unsigned char* at, bool& bad) {
  using V = typename std::conditional<NS == 4, int, long long>::type;
  const int ng = (s.rcap + 7) / 8, np = (ng + 1) / 2;
  const int2 a0 = *reinterpret_cast<const int2*>(a + c2), a1 = *reinterpret_cast<const int2*>(a + 8 + c2);
  if constexpr (NS == 4 && sizeof(S) == 4) {
    if (u < np + s.nax * ng) {
#pragma unroll
      for (int g = 0; g < 4; ++g) {
        const int r = (int)(short)(inf[g] & 0xffff);
        UdPair<S> x = w.x[g], y = w.y[g];
        if (u >= np) {  // differences, then scaled: both exact but for the difference's own rounding
          const UdPair<S> c = w.c[g];
          x = UdPair<S>{c.a - x.a, c.b - x.b};
          y = UdPair<S>{y.a - c.a, y.b - c.b};
        }
        const int2 ay = u < np ? a1 : a0;
        const float up = ud_row_raise(inf[g]);
        int v0, v1;
        ud_fix2f(x.a, x.b, up, ud_pow(r + a0.x), ud_pow(r + a0.y), v0, v1, bad);
        ud_store2<NS>(v0, v1, at + 128 * g);
        ud_fix2f(y.a, y.b, up, ud_pow(r + ay.x), ud_pow(r + ay.y), v0, v1, bad);
        ud_store2<NS>(v0, v1, at + 2048 + 128 * g);
      }
      return;
    }
  }
  if (u < np) {
#pragma unroll
    for (int g = 0; g < 4; ++g) {
      const int r = (int)(short)(inf[g] & 0xffff);
      V v0, v1;
      ud_fix2<NS>(w.x[g], a0, r, v0, v1, bad);
      ud_store2<NS>(v0, v1, at + 128 * g);
      ud_fix2<NS>(w.y[g], a1, r, v0, v1, bad);
      ud_store2<NS>(v0, v1, at + 2048 + 128 * g);
    }
  } else if (u < np + s.nax * ng) {
#pragma unroll
    for (int g = 0; g < 4; ++g) {
      const int r = (int)(short)(inf[g] & 0xffff);
      V v0, v1, c0, c1;
      ud_fix2<NS>(w.c[g], a0, r, c0, c1, bad);
      ud_fix2<NS>(w.x[g], a0, r, v0, v1, bad);
      ud_store2<NS>(c0 - v0, c1 - v1, at + 128 * g);
      ud_fix2<NS>(w.y[g], a0, r, v0, v1, bad);
      ud_store2<NS>(v0 - c0, v1 - c1, at + 2048 + 128 * g);
    }
  } else {
    for (int g = 0; g < 4; ++g) {
      const int r = ud_row_scale(inf[g]);
      const unsigned f = (unsigned)inf[g] >> 16;
      UdPair<double> x{0.0, 0.0};
      for (int e = c2; e < c2 + 2 && e < lp.nextra; ++e) {
        const int tt = s.bc_term[e], ax = s.axis[tt];
        const bool at_face = s.w[tt] > 0 ? !((f >> (2 * ax)) & 1u) : !((f >> (2 * ax + 1)) & 1u);
        if (at_face && k0 + 8 * g < nrows) (e == c2 ? x.a : x.b) = s.bcval[e * s.G + (int)((unsigned)(k0 + 8 * g) % (unsigned)s.G)];
      }
      V v0, v1;
      ud_fix2<NS>(x, a0, r, v0, v1, bad);
      // (a small face value's scale may leave zero's exponent in range)
      ud_store2<NS>(x.a != 0.0 ? v0 : (V)0, x.b != 0.0 ? v1 : (V)0, at + 128 * g);
      ud_store2<NS>((V)0, (V)0, at + 2048 + 128 * g);
    }
  }
}
template <int NS, typename S>
__device__ __forceinline__ void ud_digits(const SrcRows<S>&, const LivePattern&, int, long, long, const int (&inf)[4],
                                          int c2, const UdRaw<S>& w, const int* a, unsigned char* at, bool& bad) {
  const int2 a0 = *reinterpret_cast<const int2*>(a + c2), a1 = *reinterpret_cast<const int2*>(a + 8 + c2);
#pragma unroll
  for (int g = 0; g < 4; ++g) {
    const int r = (int)(short)(inf[g] & 0xffff);
    typename std::conditional<NS == 4, int, long long>::type v0, v1;
    if constexpr (NS == 4 && sizeof(S) == 4) {
      const float up = ud_row_raise(inf[g]);
      ud_fix2f(w.x[g].a, w.x[g].b, up, ud_pow(r + a0.x), ud_pow(r + a0.y), v0, v1, bad);
      ud_store2<NS>(v0, v1, at + 128 * g);
      ud_fix2f(w.y[g].a, w.y[g].b, up, ud_pow(r + a1.x), ud_pow(r + a1.y), v0, v1, bad);
    } else {
      ud_fix2<NS>(w.x[g], a0, r, v0, v1, bad);
      ud_store2<NS>(v0, v1, at + 128 * g);
      ud_fix2<NS>(w.y[g], a1, r, v0, v1, bad);
    }
    ud_store2<NS>(v0, v1, at + 2048 + 128 * g);
  }
}
template <typename S>
inline bool ud_vec(const SrcStencil<S>& s) {
  return s.rcap % 8 == 0 && ((size_t)s.ldz * sizeof(S)) % 16 == 0 && (size_t)s.Z % 16 == 0;
}
template <typename S>
inline bool ud_vec(const SrcRows<S>& s) { return ((size_t)s.ld * sizeof(S)) % 16 == 0 && (size_t)s.A % 16 == 0; }

// (hi 2^32 + lo) 2^e, rounded once (FP64, on the integer units: the FP64 pipe is narrow).
__device__ __forceinline__ double ud_make(long long hi, unsigned lo, int e) {
  const bool neg = hi < 0;
  if (neg) {
    lo = 0u - lo;
    hi = ~hi + (lo == 0u ? 1 : 0);
  }
  const unsigned long long a = (unsigned long long)hi, b = (unsigned long long)lo << 32;
  int lz;
  unsigned long long nm;  // the leading 64 bits
  if (a != 0ull) {
    lz = __clzll((long long)a);
    nm = lz ? (a << lz) | (b >> (64 - lz)) : a;
  } else {
    if (lo == 0u) return 0.0;
    lz = 64 + __clz((int)lo);
    nm = b << (lz - 64);
  }
  const int f = 1023 + 95 - lz + e;
  if (f < 2 || f > 2044) {
    const double v = ldexp(__ull2double_rn(nm), f - 1086);
    return neg ? -v : v;
  }
  const unsigned long long m = (nm >> 11) + ((nm >> 10) & 1ull);
  const unsigned long long r = ((unsigned long long)(f - 1) << 52) + m;
  return __longlong_as_double((long long)(r | (neg ? 0x8000000000000000ull : 0ull)));
}

template <int Q>
__device__ __forceinline__ void ud_tmem_ld(uint32_t taddr, uint32_t (&v)[Q]) {
  if constexpr (Q == 8) tc::tmem_ld8(taddr, v);
  else tc::tmem_ld4(taddr, v);
}

inline size_t ud_b_bytes(int nunit, int ns, int kp) { return (size_t)nunit * 32 * ns * kp; }
template <typename T>
__host__ __device__ inline size_t ud_misc_bytes(int nunit, int kp) {
  // column scales, weights' exponents, per-row scale and half dots, vJ, output tile
  return sizeof(int) * (size_t)(16 * nunit + kp) + 256 * sizeof(T) + sizeof(T) * ((size_t)kp + 128 * (size_t)(kp + 1)) + 16;
}
template <typename T>
inline int ud_slots(int nunit, int kp) {
  constexpr int NS = sizeof(T) == 4 ? 4 : 8;
  const size_t fixed = ud_b_bytes(nunit, NS, kp) + ud_misc_bytes<T>(nunit, kp);
  if (fixed >= 225 * 1024) return 0;
  const int n = (int)((225 * 1024 - fixed) / (NS * 4096));
  return n < kUdMaxSlots ? n : kUdMaxSlots;
}

namespace tc {
// Barrier `id` of two warps; the AND form gives both the same answer.
__device__ __forceinline__ void pair_sync(int id) { asm volatile("barrier.cta.sync %0, 64;\n" ::"r"(id) : "memory"); }
__device__ __forceinline__ bool pair_and(int id, bool x) {
  uint32_t out;
  asm volatile(
      "{\n.reg .pred p, q;\nsetp.ne.u32 p, %1, 0;\nbarrier.cta.red.and.pred q, %2, 64, p;\nselp.u32 %0, 1, 0, q;\n}\n"
      : "=r"(out)
      : "r"((uint32_t)x), "r"(id)
      : "memory");
  return out != 0;
}
__device__ __forceinline__ bool wait_warp(uint64_t* bar, uint32_t parity) {
  return __all_sync(0xffffffffu, mbar_wait(bar, parity)) != 0;
}
}  // namespace tc

template <int NS, class Src, class Epi>
__global__ void __launch_bounds__(ud_threads(NS), 1)
    k_update_dig(const __grid_constant__ Src src, const __grid_constant__ LivePattern lp, long nrows,
                 const int* __restrict__ rinfo, const unsigned short* __restrict__ B, const int* __restrict__ wexp,
                 const int* __restrict__ aexp, int kcap, int nslot, bool vec, const __grid_constant__ Epi epi,
                 double* __restrict__ partials, int* __restrict__ status) {
  using T = typename std::conditional<NS == 4, float, double>::type;
  using S = typename XgElem<Src>::type;
  using SO = typename std::remove_pointer<decltype(epi.out)>::type;
  extern __shared__ __align__(1024) unsigned char ud_smem[];
  __shared__ uint64_t full[kUdMaxSlots], empty[kUdMaxSlots], dfull[2], dempty[2], bbar;
  __shared__ uint32_t tbase;
  constexpr int kUdProd = ud_prod(NS), kUdThreads = ud_threads(NS);
  constexpr uint32_t kStage = NS * 4096u;  // a K step: 128 rows x 16 columns x NS digits x 2 bytes
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int kp = ud_kp(kcap), no = ud_orders(NS, kp);
  const int nunit = ud_units(src, lp);
  unsigned char* ring = ud_smem;
  unsigned char* Bs = ring + (size_t)nslot * kStage;
  const uint32_t bstep = 32u * NS * (uint32_t)kp, bbytes = bstep * (uint32_t)nunit;
  int* as = reinterpret_cast<int*>(Bs + bbytes);         // [16 nunit]
  int* we = as + 16 * nunit;                             // [kp]
  T* scs = reinterpret_cast<T*>(we + kp);                // [128]
  T* jps = scs + 128;                                    // [128]
  T* vJs = jps + 128;                                    // [kp]
  T* Os = vJs + kp;                                      // [128][kp + 1]
  constexpr uint32_t kCols = 512;
  if (warp == kUdEpi + kUdProd) {
    tc::tmem_alloc(&tbase, kCols);
    tc::tmem_relinquish();
  }
  if (tid == 0) {
    for (int i = 0; i < nslot; ++i) {
      tc::mbar_init(&full[i], 4);
      tc::mbar_init(&empty[i], 1);
    }
    for (int i = 0; i < 2; ++i) {
      tc::mbar_init(&dfull[i], 1);
      tc::mbar_init(&dempty[i], kUdEpi);
    }
    tc::mbar_init(&bbar, 1);
  }
  const double* vJ = epi_vj(epi);
  for (int j = tid; j < kp; j += kUdThreads) {
    we[j] = wexp[j];
    vJs[j] = (vJ && j < kcap) ? (T)vJ[j] : T(0);
  }
  for (int j = tid; j < 16 * nunit; j += kUdThreads) as[j] = aexp[j];
  tc::fence_before_sync();
  __syncthreads();
  tc::fence_after_sync();
  const uint32_t tmem = tbase;
  const long ntiles = (nrows + 127) / 128;
  double e0t = 0.0, e1t = 0.0;
  bool lost = false, bad = false;

  if (warp < kUdEpi) {
    // ---- epilogue: warps q and q + 4 have the rows 32 q .. of every tile, half of the columns each
    const int q = warp & 3, h = warp >> 2;
    T* O = Os + (size_t)(32 * q) * (kp + 1);
    const int nh = ((kp / 8 + 1) / 2) * 8, nlo = h ? nh : 0, nhi = h ? kp : nh;
    long it = 0;
    for (long tile = blockIdx.x; tile < ntiles; tile += gridDim.x, ++it) {
      const int buf = (int)(it & 1);
      const long k0 = tile * 128 + 32 * q, k = k0 + lane;
      const int r = k < nrows ? ud_row_scale(rinfo[k]) : kUdMinExp;
      // the two warps of a quarter leave together
      if (!tc::pair_and(1 + q, tc::mbar_wait(&dfull[buf], (uint32_t)((it >> 1) & 1)))) {
        lost = true;
        break;
      }
      tc::fence_after_sync();
      const uint32_t ta = tmem + ((uint32_t)(32 * q) << 16) + (uint32_t)(buf * 256);
      T js[4] = {T(0), T(0), T(0), T(0)};
      constexpr int Q = NS == 4 ? 8 : 4;  // columns at a time
      for (int n0 = nlo; n0 < nhi; n0 += Q) {
        uint32_t v[NS == 4 ? 5 : NS][Q];
#pragma unroll
        for (int o = 0; o < NS; ++o) ud_tmem_ld<Q>(ta + (uint32_t)(o * kp + n0), v[o]);
        if constexpr (NS == 4) {
          if (no > NS) ud_tmem_ld<Q>(ta + (uint32_t)(NS * kp + n0), v[4]);
        }
        tc::tmem_wait_ld();
#pragma unroll
        for (int b = 0; b < Q; ++b) {
          T val;
          if constexpr (NS == 4) {
            float x = __uint_as_float(v[3][b]);
            if (no > NS) x = fmaf(__uint_as_float(v[4][b]), 0.00390625f, x);
            x = fmaf(x, 0.00390625f, __uint_as_float(v[2][b]));
            x = fmaf(x, 0.00390625f, __uint_as_float(v[1][b]));
            x = fmaf(x, 0.00390625f, __uint_as_float(v[0][b]));
            const int es = min(max(r + we[n0 + b] - 10, -252), 252), e1 = es >> 1;
            val = x * __int_as_float((127 + e1) << 23) * __int_as_float((127 + es - e1) << 23);
          } else {
            long long hi = 0, lo = 0;
#pragma unroll
            for (int o = 0; o < 4; ++o) {
              hi += (long long)__float2int_rn(__uint_as_float(v[o][b])) << (8 * (3 - o));
              lo += (long long)__float2int_rn(__uint_as_float(v[4 + o][b])) << (8 * (3 - o));
            }
            // hi 2^32 + lo, every bit of it: cut to 64 bits (a unit of 2^-47 to 2^-50 of the row's largest
            // possible product) outputs of nine columns were off by 6 to 16 times an FP64 sum's error
            val = ud_make(hi + (lo >> 32), (unsigned)lo, r + we[n0 + b] - 66);
          }
          if constexpr (Epi::kDot) js[b & 3] = fma(val, vJs[n0 + b], js[b & 3]);
          O[(size_t)lane * (kp + 1) + n0 + b] = val;
        }
      }
      tc::fence_before_sync();
      __syncwarp();
      if (lane == 0) tc::mbar_arrive(&dempty[buf]);
      if constexpr (Epi::kDot) {
        if (h) jps[32 * q + lane] = (js[0] + js[1]) + (js[2] + js[3]);
      }
      tc::pair_sync(1 + q);
      if (!h && k < nrows) {
        double sc = 0.0, ex = 0.0, e0 = 0.0, e1 = 0.0;
        double j0 = 0.0;
        if constexpr (Epi::kDot) j0 = (double)(((js[0] + js[1]) + (js[2] + js[3])) + jps[32 * q + lane]);
        epi.prep(k, j0, sc, ex, e0, e1);
        e0t += e0;
        e1t += e1;
        if constexpr (Epi::kExtra) {
          scs[32 * q + lane] = (T)sc;
          const SO o = (SO)ex;
          if (!isfinite(o)) bad = true;
          epi.out[k * epi.ld + kcap] = o;
        }
      }
      if constexpr (Epi::kExtra) tc::pair_sync(1 + q);
      // rows 16 h .. of the quarter
      const int nr = (int)(nrows - k0 < 16 * (h + 1) ? nrows - k0 : 16 * (h + 1));
      for (int j = lane; j < kcap; j += 32) {
#pragma unroll 4
        for (int row = 16 * h; row < nr; ++row) {
          T o = O[(size_t)row * (kp + 1) + j];
          if constexpr (Epi::kExtra) o *= scs[32 * q + row];
          const SO os = (SO)o;
          bad = bad || !isfinite(os);
          epi.out[(k0 + row) * epi.ld + j] = os;
        }
      }
      tc::pair_sync(1 + q);
    }
    if (bad) latch(epi.status, TT_ERR_NONFINITE);
  } else if (warp < kUdEpi + kUdProd) {
    // ---- digits: warp p takes the rows 32 (p % 4) .. of every kStep-th K step
    const int p = warp - kUdEpi, m = 32 * (p & 3) + (lane >> 2), c2 = 2 * (lane & 3);
    unsigned char* at0 = ring + (size_t)(p & 3) * 512 + (size_t)(lane >> 2) * 16 + (size_t)(lane & 3) * 4;
    constexpr int kStep = kUdProd / 4;  // K steps in work at a time
    long tile_it = -1, k0 = 0;
    int inf[4] = {0, 0, 0, 0};
    int u = (p >> 2) % nunit, sl = (p >> 2) % nslot;
    long it = (p >> 2) / nunit;
    uint32_t ph = 1;
    bool first = true;
    for (long tile = blockIdx.x + it * (long)gridDim.x; tile < ntiles; tile = blockIdx.x + it * (long)gridDim.x) {
      if (it != tile_it) {
        tile_it = it;
        k0 = tile * 128 + m;
#pragma unroll
        for (int g = 0; g < 4; ++g) inf[g] = k0 + 8 * g < nrows ? rinfo[k0 + 8 * g] : 0;
      }
      UdRaw<S> raw;
      ud_load(src, lp, u, k0, nrows, inf, c2, vec, raw);
      __syncwarp();
      if (!first && !tc::wait_warp(&empty[sl], ph)) {
        lost = true;
        break;
      }
      ud_digits<NS>(src, lp, u, k0, nrows, inf, c2, raw, as + 16 * u, at0 + (size_t)sl * kStage, bad);
      tc::fence_smem_to_async();
      __syncwarp();
      if (lane == 0) tc::mbar_arrive(&full[sl]);
      sl += kStep;
      if (sl >= nslot) {  // nslot >= 3 >= kStep
        sl -= nslot;
        first = false;
        ph ^= 1u;
      }
      u += kStep;
      while (u >= nunit) {
        u -= nunit;
        ++it;
      }
    }
    if (bad) latch(epi.status, TT_ERR_NONFINITE);
  } else if (lane == 0) {
    // ---- the weights' digits, then the MMAs
    tc::mbar_expect(&bbar, bbytes);
    for (uint32_t o = 0; o < bbytes; o += 16384u) {
      const uint32_t n = bbytes - o < 16384u ? bbytes - o : 16384u;
      tc::bulk_g2s(tc::smem_u32(Bs) + o, reinterpret_cast<const unsigned char*>(B) + o, n, &bbar);
    }
    const uint32_t nr8 = (uint32_t)(NS * kp / 8) * 128u;
    const uint64_t a0 = tc::smem_desc(tc::smem_u32(ring), 2048u, 128u);
    const uint64_t b0 = tc::smem_desc(tc::smem_u32(Bs), nr8, 128u);
    const bool have_b = tc::mbar_wait(&bbar, 0);
    lost = !have_b;
    // descriptors are formed once: the loop is an add per operand (with index arithmetic between them an
    // MMA took 320 cycles instead of 50 to 85)
    uint32_t idesc[NS];
#pragma unroll
    for (int j = 0; j < NS; ++j) idesc[j] = tc::idesc_f16(128, (NS < no - j ? NS : no - j) * kp);
    const uint32_t idx = tc::idesc_f16(128, kp), id1 = tc::idesc_f16(128, (NS - 1) * kp);
    const uint64_t btop = (uint64_t)((uint32_t)((NS - 1) * kp / 8) * 128u >> 4);
    int sl = 0, it = 0;
    uint32_t ph = 0;
    for (long tile = blockIdx.x; tile < ntiles && !lost; tile += gridDim.x, ++it) {
      const int buf = it & 1;
      if (it >= 2 && !tc::mbar_wait(&dempty[buf], (uint32_t)(((it >> 1) - 1) & 1))) {
        lost = true;
        break;
      }
      tc::fence_after_sync();
      const uint32_t d = tmem + (uint32_t)(buf * 256);
      uint64_t bu = b0;
      for (int u = 0; u < nunit; ++u) {
        if (!tc::mbar_wait(&full[sl], ph)) {
          lost = true;
          break;
        }
        tc::fence_after_sync();
        const uint64_t au = a0 + (uint64_t)((uint32_t)sl * (kStage >> 4));
        // rows' digit j against the weights' digits 0 .. min(NS, no - j) - 1: orders j ..; the extra order
        // is written for the first time by j = 1
        tc::mma_f16(d, au, bu, idesc[0], u ? 1u : 0u);
        if (u == 0 && no > NS) {
          tc::mma_f16(d + (uint32_t)kp, au + 256u, bu, id1, 1u);
          tc::mma_f16(d + (uint32_t)(NS * kp), au + 256u, bu + btop, idx, 0u);
        } else {
          tc::mma_f16(d + (uint32_t)kp, au + 256u, bu, idesc[1], 1u);
        }
#pragma unroll
        for (int j = 2; j < NS; ++j) tc::mma_f16(d + (uint32_t)(j * kp), au + (uint64_t)(j * 256), bu, idesc[j], 1u);
        tc::mma_commit(&empty[sl]);
        bu += bstep >> 4;
        if (++sl == nslot) {
          sl = 0;
          ph ^= 1u;
        }
      }
      if (!lost) tc::mma_commit(&dfull[buf]);
    }
    // nothing of this thread's is in flight past here (bounded)
    if (!have_b) {
      (void)tc::mbar_wait(&bbar, 0, 1L << 14);
    } else {
      tc::mma_commit(&bbar);
      if (!tc::mbar_wait(&bbar, 1)) lost = true;
    }
  }
  tc::fence_before_sync();
  if (__syncthreads_or(lost) && tid == 0) latch(status, TT_ERR_TIMEOUT);
  if (partials) {
    // energy partials: the epilogue's first four warps have them, in a fixed order
    double* red = reinterpret_cast<double*>(ring);
    e0t = warp_sum(e0t);
    e1t = warp_sum(e1t);
    if (warp < 4 && lane == 0) {
      red[2 * warp] = e0t;
      red[2 * warp + 1] = e1t;
    }
    __syncthreads();
    if (tid < 2) partials[2 * (size_t)blockIdx.x + tid] = (red[tid] + red[2 + tid]) + (red[4 + tid] + red[6 + tid]);
  }
  if (warp == kUdEpi + kUdProd) {
    tc::fence_after_sync();
    tc::tmem_dealloc(tmem, kCols);
  }
}

// Whether the digit update takes a pass of nrows rows: outputs within the accumulators (two sets of 256
// columns), K steps and stages within shared memory.
template <typename T, class Src>
inline bool update_dig_fits(const Src& src, const LivePattern& lp, long nrows, int kcap) {
  constexpr int NS = sizeof(T) == 4 ? 4 : 8;
  if (kcap < 1 || nrows < kUdMinRows || nrows >= (1L << 31)) return false;
  const int kp = ud_kp(kcap), nunit = ud_units(src, lp);
  if (NS * kp > 256 || nunit > kUdMaxUnits || ud_slots<T>(nunit, kp) < 3) return false;
  if constexpr (XgElem<Src>::stencil) {
    if (src.nax < 1 || src.nax > 3 || src.rcap != lp.rcap || lp.nextra > 6) return false;
    // differences are scaled with the row's centre columns: past this weight their digits would fall short
    for (int t = 0; t < src.nterm; ++t)
      if (!(src.lam[t] <= 64.0 && src.lam[t] >= -64.0)) return false;
  }
  return true;
}
template <typename T, class Src>
inline size_t update_dig_wbytes(const Src& src, const LivePattern& lp, int kcap) {
  constexpr int NS = sizeof(T) == 4 ? 4 : 8;
  const int kp = ud_kp(kcap), nunit = ud_units(src, lp);
  return ud_b_bytes(nunit, NS, kp) + sizeof(int) * (size_t)(kp + 16 * nunit);
}

// Columns of the storage matrix of a pass, and where its inflow columns stand.
template <typename S>
inline int ud_storage_cols(const SrcStencil<S>& s, const LivePattern&) { return s.rcap; }
template <typename S>
inline int ud_storage_cols(const SrcRows<S>&, const LivePattern& lp) { return lp.ncap(); }

// Column sizes, called before launch_update_dig.  From RZ (ncap x ncap row-major, before it is overwritten) where
// it is the triangular factor of the pass's columns to their own accuracy (R^T R = A^T A column by column):
inline tt_status launch_ud_scales(cudaStream_t s, const double* RZ, int n, const UdBufs& ub) {
  k_ud_colexp<<<(unsigned)n, 128, 0, s>>>(RZ, n, ub.cexp);
  count_launch();
  return cudaGetLastError() == cudaSuccess ? TT_OK : TT_ERR_CUDA;
}

// From the columns themselves where it is not: a Gram matrix's factor ends at pivots of 4 n eps of its largest
// diagonal entry and a sketch's keeps the columns' parts in its range, so a column may be far larger than RZ says; a
// row's scale follows that column, and the other columns of the row lost as many bits (nine orthogonal columns
// graded 1 to 1e-12: the state to 1 %).  One more pass over the storage (1,048,576 x 32 FP64: 0.05 ms).
template <class Src>
tt_status launch_ud_scales_cols(cudaStream_t s, int num_sms, const Src& src, const LivePattern& lp, long nrows,
                                const UdBufs& ub) {
  using S = typename XgElem<Src>::type;
  const int ncol = ud_storage_cols(src, lp);
  int nextra = 0, extra0 = 0, G = 1;
  const double* bc = nullptr;
  const S* A = nullptr;
  long ld = 0;
  if constexpr (XgElem<Src>::stencil) {
    nextra = lp.nextra;
    extra0 = (src.nterm + 1) * src.rcap;
    G = src.G;
    bc = src.bcval;
    A = src.Z;
    ld = src.ldz;
  } else {
    A = src.A;
    ld = src.ld;
  }
  if (cudaMemsetAsync(ub.slots, 0, sizeof(unsigned long long) * (size_t)(ncol + nextra), s) != cudaSuccess)
    return TT_ERR_CUDA;
  k_xg_colmax<S><<<xg_colmax_grid(num_sms, ncol, nrows), 256, 0, s>>>(A, ncol, ld, 1, nrows, ub.slots, bc, nextra, G,
                                                                      nullptr);
  count_launch();
  k_ud_slotexp<<<1, 256, 0, s>>>(ncol, extra0, nextra, ub.slots, ub.cexp);
  count_launch();
  return cudaGetLastError() == cudaSuccess ? TT_OK : TT_ERR_CUDA;
}

template <typename T, class Src, class Epi>
tt_status launch_update_dig(cudaStream_t s, int num_sms, const Src& src, LivePattern lp, const UdBufs& ub, long nrows,
                            const double* W, int kcap, const Epi& epi, double* partials, long* grid_out, int cat) {
  constexpr int NS = sizeof(T) == 4 ? 4 : 8;
  using S = typename XgElem<Src>::type;
  const int kp = ud_kp(kcap), nunit = ud_units(src, lp), nslot = ud_slots<T>(nunit, kp);
  const size_t bb = ud_b_bytes(nunit, NS, kp);
  size_t smem = (size_t)nslot * NS * 4096 + bb + ud_misc_bytes<T>(nunit, kp);
  if (smem < 117 * 1024) smem = 117 * 1024;  // one CTA per SM: its accumulators never wait for another's
  auto kern = k_update_dig<NS, Src, Epi>;
  if (const tt_status a = smem_optin(kern, smem); a != TT_OK) return a;
  unsigned short* B = reinterpret_cast<unsigned short*>(ub.w);
  int* wexp = reinterpret_cast<int*>(ub.w + bb);
  int* aexp = wexp + kp;
  TimerScope scope(cat, s);
  k_ud_weights<NS, Src><<<(unsigned)kp, 256, 0, s>>>(src, lp, W, kcap, kp, ub.cexp, B, wexp, aexp, epi.status);
  count_launch();
  const long rb = (nrows + 127) / 128, gr = rb < 16L * num_sms ? rb : 16L * num_sms;
  if constexpr (XgElem<Src>::stencil) {
    LivePattern lz{lp.r_ptr, lp.rcap, 1, 0};
    k_ud_rows<S, short><<<(unsigned)gr, 256, 0, s>>>(src.Z, src.ldz, lz, src.rcap, nrows, ub.cexp, ub.rho, false);
    count_launch();
    k_ud_info<S><<<(unsigned)((nrows + 255) / 256), 256, 0, s>>>(src, lp, nrows, ub.cexp, ub.rho, ub.rinfo, NS == 4 && sizeof(S) == 4);
    count_launch();
  } else {
    k_ud_rows<S, int><<<(unsigned)gr, 256, 0, s>>>(src.A, src.ld, lp, lp.ncap(), nrows, ub.cexp, ub.rinfo,
                                                          NS == 4 && sizeof(S) == 4);
    count_launch();
  }
  const long ntiles = (nrows + 127) / 128, grid = num_sms < ntiles ? num_sms : ntiles;
  if (grid_out) *grid_out = grid;
  kern<<<(unsigned)grid, ud_threads(NS), smem, s>>>(src, lp, nrows, ub.rinfo, B, wexp, aexp, kcap, nslot, ud_vec(src), epi,
                                               partials, epi.status);
  count_launch();
  return cudaGetLastError() == cudaSuccess ? TT_OK : TT_ERR_CUDA;
}

}  // namespace ttk
