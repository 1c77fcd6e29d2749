// Exact Gram products of tall column blocks on the tensor cores, and the triangular factor of the
// merged core's columns from them (the L->R orthogonalisation of the rounding, Sec. 3.1 footnote).
//
// Every storage column c is held in fixed point, v = round(x 2^-U_c) with one power of two per column,
// and v is written in balanced digits of base 512,
//   v = sum_j d_j 512^(NS-1-j),   -256 <= d_j <= 255,
// NS = 4 digits (34 bits and sign) for FP32 passes and NS = 7 (61 bits and sign) for FP64 passes.
// Digits are exact in FP16, products of two digits are integers up to 2^16, and the FP32
// accumulators of tcgen05.mma.kind::f16 sum 256 rows of them without any rounding (every partial sum is
// an integer of at most 2^24).  The digit products of a chunk are then folded into 64-bit integers.
// So sum_k v_a v_b comes out exactly, for columns whose entries carry a fixed-point rounding of at most
// 2^-(9 NS - 1) of their column's largest entry (FP32 2^-35, FP64 2^-62; the storage's own rounding of
// entries near that size is 2^-25 and 2^-54).  The columns of the transport sum are integer
// combinations of a row and its neighbours (C - L, H - C, H - L, H - 2 C + L), so their Gram matrix is an
// integer combination of the products of the neighbour blocks, formed without rounding or
// cancellation (k_xg_combine); the operators' coefficients scale the factor's columns at the end.
//
// The factor R with R^T R = G is a Cholesky factor in 128-bit fixed point (xchol.cuh): G is exact and
// columns are resolved down to about 2^-57 of their norm, as a Householder QR in FP64 resolves them.
//
// Why: a Householder TSQR is a chain of reflectors behind block barriers on the FMA pipes; measured
// at 1,048,576 rows x 160 columns it took 5.3 ms (FP32 leaf) + 2.1 ms (merges) and 91.9 + 17 ms in
// FP64, whose FMA pipe runs at 1/64 of the FP32 rate on this part.  Here the digits of the storage
// columns are written once (k_xg_digits, bound by memory) in the layout of the MMA operands, so that the
// product kernel (k_xg_mma) only moves 16-byte rows with bulk copies: a neighbour block is the same
// digits at another cell, a missing neighbour a page of zeros.  Measured for both roundings of a step
// at 1,048,576 rows, rank 32: FP32 digits 0.19, products 0.87, Cholesky 0.41 ms (leaves and merges before:
// 6.0 + 2.1 ms); FP64 0.25, 3.06, 0.41 ms (before 99.6 + 14 ms).
#pragma once
#include <map>

#include "bigpass.cuh"
#include "instr.cuh"
#include "small.cuh"
#include "tc.cuh"
#include "xchol.cuh"

namespace ttk {

constexpr int kXgThreads = 576;   // 16 folding warps, a copying warp, an MMA warp
constexpr int kXgTiles = 4;       // output tiles a CTA accumulates (TMEM: 4 x 128 columns)
constexpr int kXgMaxBlk = 6;      // operand blocks a CTA stages
constexpr int kXgMaxSub = 56;     // column groups of a pass
constexpr int kXgMaxNb = 24;      // operand blocks of a pass
constexpr int kXgMaxCta = 80;     // CTAs that share a row range
constexpr int kXgMaxStage = 6;
constexpr long kXgMaxOct = 2048L * 32;  // row octets per CTA: the 64-bit sums stay below 2^62
constexpr int kXgMaxRaw = 448;          // storage columns of all neighbour blocks

template <int NS>
struct XgCfg {
  static constexpr int W = NS == 4 ? 32 : 16;  // columns per operand block (NS * W <= 128 rows)
  static constexpr int H = NS == 4 ? 1 : 2;    // 64-bit sums per entry (digit groups of 4 and 3)
};

// A row-major storage matrix whose rows are the groups of cells (row = g + G cell), or plain rows
// (G = 8, ncell = ceil(nrows / 8)).  Its digits are kept per octet of rows (a cell's groups padded to a
// multiple of 8): record = for each column group, for digit j, for column a: eight rows in 16 bytes.
struct XgArray {
  int ncol, G, oc;  // columns, rows per cell, octets per cell
  long ncell;
  int rec;          // bytes of an octet's record
  long sr, sc;      // element strides of rows and columns
};

// One column group of the products: `w` columns (a multiple of 8, the last ones padding) of an array, at
// the cell itself (nb = 0), its lower (1 + 2 axis) or upper (2 + 2 axis) neighbour, or the inflow column
// of a face (nb = 8 + face).
struct XgSub {
  short raw0;        // first raw column
  unsigned char cnt, w, arr, nb;
  int off;           // byte offset in the array's record
};

struct XgPlan {
  int ns, nsub, nb, ncta, ntile, nraw;
  XgSub sub[kXgMaxSub];
  unsigned char bsub0[kXgMaxNb], bnsub[kXgMaxNb];  // operand block -> its column groups (equal widths)
  unsigned char ctiles[kXgMaxCta], cblks[kXgMaxCta];
  unsigned char tp[kXgMaxCta][kXgTiles], tq[kXgMaxCta][kXgTiles];  // tile -> local block of p, q
  unsigned char blk[kXgMaxCta][kXgMaxBlk];                         // local block -> operand block
  short tile0[kXgMaxCta];                                          // first tile of the CTA
  unsigned char gp[kXgMaxCta * kXgTiles], gq[kXgMaxCta * kXgTiles];
};

// What the product kernel reads beside the plan.
struct XgArgs {
  const unsigned char* dig[2];  // digit records of the arrays
  const unsigned char* bc;      // digit records of one cell of the inflow columns: [face slot][octet]
  const unsigned char* zero;    // a page of zeros
  int oc, rec[2], bcrec;
  long noct, opg;               // octets in all, and per row group
  int nax, ext[3];
  int cstr[3];                  // cell strides of the axes
  unsigned char face[6];        // inflow column -> 2 axis + (upper face)
  int nstage;
  size_t stage_bytes;
};

__host__ __device__ inline int xg_block_rows(const XgPlan& pl, int b) {
  return pl.ns * pl.sub[pl.bsub0[b]].w * pl.bnsub[b];
}

// Adds the column groups of `ncol` columns to the plan: whole operand blocks of W columns, then the rest
// rounded up to 8; groups of equal width are made adjacent by xg_tiles.
template <int NS>
inline bool xg_add(XgPlan& pl, int ncol, int raw0, int arr, int nb) {
  constexpr int W = XgCfg<NS>::W;
  int off = 0;
  for (int c = 0; c < ncol; c += W) {
    if (pl.nsub == kXgMaxSub) return false;
    const int cnt = ncol - c < W ? ncol - c : W, w = (cnt + 7) & ~7;
    pl.sub[pl.nsub++] = XgSub{(short)(raw0 + c), (unsigned char)cnt, (unsigned char)w, (unsigned char)arr,
                              (unsigned char)nb, off};
    off += NS * w * 16;
  }
  return true;
}
template <int NS>
inline int xg_record(int ncol) {
  constexpr int W = XgCfg<NS>::W;
  int off = 0;
  for (int c = 0; c < ncol; c += W) off += NS * (((ncol - c < W ? ncol - c : W) + 7) & ~7) * 16;
  return off;
}

// Operand blocks (column groups of one width side by side, at most W columns; with 7 digits always 16, a
// padding group where one is missing, since an MMA's N is a multiple of 16), and the output tiles of each
// CTA: the upper triangle of the blocks, or (arrays: split) blocks of array 0 x blocks of array 1.  A CTA
// takes up to four tiles that share blocks: the next tile is one that adds the fewest.
template <int NS>
inline bool xg_tiles(XgPlan& pl, bool split) {
  constexpr int W = XgCfg<NS>::W;
  XgSub in[kXgMaxSub];
  const int n = pl.nsub;
  for (int i = 0; i < n; ++i) in[i] = pl.sub[i];
  pl.ns = NS;
  pl.nsub = pl.nb = 0;
  int nleft = 0;
  for (int arr = 0; arr < (split ? 2 : 1); ++arr) {
    for (int w = W; w >= 8; w -= 8) {
      int room = 0;
      for (int i = 0; i < n; ++i) {
        if (in[i].w != w || (split && in[i].arr != arr)) continue;
        if (pl.nsub == kXgMaxSub) return false;
        if (room < w) {
          if (pl.nb == kXgMaxNb) return false;
          pl.bsub0[pl.nb] = (unsigned char)pl.nsub;
          pl.bnsub[pl.nb++] = 0;
          room = W;
        }
        pl.sub[pl.nsub++] = in[i];
        ++pl.bnsub[pl.nb - 1];
        room -= w;
      }
      if (NS == 7 && w == 8 && room == 8) {
        if (pl.nsub == kXgMaxSub) return false;
        pl.sub[pl.nsub++] = XgSub{0, 0, 8, 0, 255, 0};  // padding: zeros
        ++pl.bnsub[pl.nb - 1];
      }
    }
    if (arr == 0) nleft = pl.nb;
  }
  const int q0 = split ? nleft : 0, np = split ? nleft : pl.nb;
  bool done[kXgMaxNb][kXgMaxNb] = {};
  int open = 0;
  for (int p = 0; p < np; ++p)
    for (int q = (split ? q0 : p); q < pl.nb; ++q) ++open;
  pl.ncta = pl.ntile = 0;
  while (open > 0) {
    if (pl.ncta == kXgMaxCta) return false;
    const int k = pl.ncta++;
    int nblk = 0, nt = 0;
    unsigned char blk[kXgMaxBlk];
    pl.tile0[k] = (short)pl.ntile;
    auto local = [&](int b) {
      for (int i = 0; i < nblk; ++i)
        if (blk[i] == b) return i;
      return -1;
    };
    while (nt < kXgTiles && open > 0) {
      int bp = -1, bq = -1, best = 3;
      for (int p = 0; p < np; ++p)
        for (int q = (split ? q0 : p); q < pl.nb; ++q) {
          if (done[p][q]) continue;
          const int add = (local(p) < 0) + (p != q && local(q) < 0);
          if (add < best) {
            best = add;
            bp = p;
            bq = q;
          }
        }
      if (nblk + best > kXgMaxBlk || (nt > 0 && best == 2)) break;
      if (local(bp) < 0) blk[nblk++] = (unsigned char)bp;
      if (local(bq) < 0) blk[nblk++] = (unsigned char)bq;
      done[bp][bq] = true;
      --open;
      pl.tp[k][nt] = (unsigned char)local(bp);
      pl.tq[k][nt] = (unsigned char)local(bq);
      pl.gp[pl.ntile] = (unsigned char)bp;
      pl.gq[pl.ntile] = (unsigned char)bq;
      ++pl.ntile;
      ++nt;
    }
    pl.ctiles[k] = (unsigned char)nt;
    pl.cblks[k] = (unsigned char)nblk;
    for (int i = 0; i < nblk; ++i) pl.blk[k][i] = blk[i];
  }
  return true;
}

// Bytes of a stage (64 rows of every operand block of the CTA that stages most).
inline size_t xg_stage_bytes(const XgPlan& pl) {
  size_t most = 0;
  for (int k = 0; k < pl.ncta; ++k) {
    size_t b = 0;
    for (int i = 0; i < pl.cblks[k]; ++i) b += (size_t)xg_block_rows(pl, pl.blk[k][i]) * 128;
    if (b > most) most = b;
  }
  return most;
}
constexpr size_t kXgPad = 128 * 16;  // an M = 128 operand of a narrower block reads past its last octet
inline int xg_stages(const XgPlan& pl) {
  const int n = (int)((226 * 1024 - kXgPad) / xg_stage_bytes(pl));
  return n < kXgMaxStage ? n : kXgMaxStage;
}

// ---- fixed point ---------------------------------------------------------------------------------
// Unit exponent U of a column with largest magnitude `maxbits` (an FP64 bit pattern): every entry is
// below 2^E, and 2^E maps to 2^(9 NS - 2), inside the digits' range.
__host__ __device__ inline int xg_unit(unsigned long long maxbits, int NS) {
  return ((int)((maxbits >> 52) & 0x7ff) - 1022) - (9 * NS - 2);
}
// round(x 2^-U), U folded into the shift constant K (see xg_shift_const).  An exponent field of zero
// (zero, denormals) gives 0; Inf and NaN give some in-range integer.
__device__ __forceinline__ long long xg_fix(double x, int K) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(x);
  const int e = (int)((b >> 52) & 0x7ff);
  const unsigned long long m = e ? (((b & 0xfffffffffffffull) | 0x10000000000000ull) << 10) : 0ull;
  const int sh = min(max(K - e, 1), 63);
  const long long r = (long long)(((m >> sh) + 1ull) >> 1);
  return (long long)b < 0 ? -r : r;
}
__device__ __forceinline__ long long xg_fix(float x, int K) {
  const unsigned b = __float_as_uint(x);
  const int e = (int)((b >> 23) & 0xff);
  const unsigned long long m = e ? ((unsigned long long)((b & 0x7fffffu) | 0x800000u) << 39) : 0ull;
  const int sh = min(max(K - e, 1), 63);
  const long long r = (long long)(((m >> sh) + 1ull) >> 1);
  return (int)b < 0 ? -r : r;
}
__device__ __forceinline__ int xg_shift_const(double, int U) { return 1084 + U; }
__device__ __forceinline__ int xg_shift_const(float, int U) { return 188 + U; }

// sum of 256 * 512^s over the NS digits: v + bias has the biased digits 0..511
template <int NS>
__host__ __device__ constexpr unsigned long long xg_bias() {
  unsigned long long b = 0;
  for (int s = 0; s < NS; ++s) b |= 256ull << (9 * s);
  return b;
}
// Digits of two rows of one column packed as FP16 pairs: dig[j] = (row 0, row 1) for digit j.
template <int NS>
__device__ __forceinline__ void xg_digits2(long long v0, long long v1, unsigned (&dig)[NS]) {
  const unsigned long long u0 = (unsigned long long)v0 + xg_bias<NS>(), u1 = (unsigned long long)v1 + xg_bias<NS>();
#pragma unroll
  for (int j = 0; j < NS; ++j) {
    const int s = 9 * (NS - 1 - j);
    const unsigned a = (unsigned)(u0 >> s), b = (unsigned)(u1 >> s);
    unsigned x = (__byte_perm(a, b, 0x5410) & 0x01ff01ffu) | 0x64006400u;  // 1024 + biased digit
    asm("sub.rn.f16x2 %0, %0, %1;" : "+r"(x) : "r"(0x65006500u));          // - 1280
    dig[j] = x;
  }
}

// Column maxima |x| (as FP64 bit patterns, over the finite entries: Inf and NaN are latched where the
// rows are rewritten) of a matrix of ncol <= 256 columns: a CTA takes whole rows, a thread always the
// same column, eight loads in flight.
template <typename S>
__global__ void __launch_bounds__(256) k_xg_colmax(const S* __restrict__ A, int ncol, long sr, long sc, long nrows,
                                                   unsigned long long* __restrict__ slots,
                                                   const double* __restrict__ bc, int nbc, int G) {
  __shared__ unsigned long long sm[256];
  constexpr S kMax = sizeof(S) == 4 ? (S)3.402823466e+38f : (S)1.7976931348623157e308;
  const int rpb = 256 / ncol, tid = threadIdx.x;
  const int col = tid % ncol, sub = tid / ncol;
  for (int i = tid; i < ncol; i += blockDim.x) sm[i] = 0ull;
  __syncthreads();
  if (sub < rpb) {
    S m = S(0);
    const long step = (long)gridDim.x * rpb;
    long k = (long)blockIdx.x * rpb + sub;
    for (; k + 7 * step < nrows; k += 8 * step) {
      S v[8];
#pragma unroll
      for (int u = 0; u < 8; ++u) v[u] = A[(k + u * step) * sr + col * sc];
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        const S a = fabs(v[u]);
        m = (a > m && a <= kMax) ? a : m;
      }
    }
    for (; k < nrows; k += step) {
      const S a = fabs(A[k * sr + col * sc]);
      m = (a > m && a <= kMax) ? a : m;
    }
    atomicMax(&sm[col], (unsigned long long)__double_as_longlong((double)m));
  }
  __syncthreads();
  for (int i = tid; i < ncol; i += blockDim.x) atomicMax(&slots[i], sm[i]);
  if (blockIdx.x == 0)
    for (int i = tid; i < nbc * G; i += blockDim.x)
      atomicMax(&slots[ncol + i / G], (unsigned long long)__double_as_longlong(fabs(bc[i])));
}

// Digit records of an array (and, in the CTAs past its octets, of the inflow columns: one cell, one
// column each): a thread forms one column of one octet, eight rows, and writes 16 bytes per digit.
// Bound by memory: N r (sizeof(S) + 2 NS) bytes.
template <int NS, typename S>
__global__ void __launch_bounds__(256) k_xg_digits(const S* __restrict__ A, XgArray ar, LivePattern lp, long nrows,
                                                   const unsigned long long* __restrict__ slots,
                                                   unsigned char* __restrict__ out, const double* __restrict__ bc,
                                                   int nbc, unsigned char* __restrict__ bcout) {
  constexpr int W = XgCfg<NS>::W;
  const int r = lp.r_ptr ? *lp.r_ptr : lp.rcap;
  const int cpad = ar.rec / (NS * 16);  // columns with padding
  const long noct = ar.ncell * ar.oc;
  const long tot = noct * cpad;
  long i = blockIdx.x * (long)blockDim.x + threadIdx.x;
  for (; i < tot; i += (long)gridDim.x * blockDim.x) {
    const long oct = tot < (1L << 31) ? (long)((unsigned)i / (unsigned)cpad) : i / cpad;
    const int c = (int)(i - oct * cpad);
    const long cell = (long)((unsigned)oct / (unsigned)ar.oc);
    const int g0 = (int)(oct - cell * ar.oc) * 8;
    const long k0 = cell * ar.G + g0;
    // column groups are full blocks of W and then the rest: the width of this column's group
    const int blk = c / W, a = c - blk * W;
    const int w = cpad - blk * W < W ? cpad - blk * W : W;
    const bool ok = c < ar.ncol && lp.live(c, r);
    S x[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) x[u] = (ok && g0 + u < ar.G && k0 + u < nrows) ? A[(k0 + u) * ar.sr + c * ar.sc] : S(0);
    const int K = xg_shift_const(S(0), ok ? xg_unit(slots[c], NS) : 0);
    unsigned dig[4][NS];
#pragma unroll
    for (int u = 0; u < 4; ++u) xg_digits2<NS>(xg_fix(x[2 * u], K), xg_fix(x[2 * u + 1], K), dig[u]);
    unsigned char* o = out + oct * ar.rec + (size_t)(blk * W * NS) * 16;
#pragma unroll
    for (int j = 0; j < NS; ++j)
      *reinterpret_cast<uint4*>(o + (j * w + a) * 16) = make_uint4(dig[0][j], dig[1][j], dig[2][j], dig[3][j]);
  }
  if (blockIdx.x == 0 && nbc > 0) {
    const int bcw = NS * 8 * 16;  // record of one inflow column: a group of 8, seven of them padding
    for (int e = threadIdx.x; e < nbc * ar.oc * 8; e += blockDim.x) {
      const int f = e / (ar.oc * 8), rem = e - f * ar.oc * 8, o = rem / 8, a = rem - o * 8;
      const int K = xg_shift_const(0.0, xg_unit(slots[ar.ncol + f], NS));
      unsigned dig[4][NS];
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int g = 8 * o + 2 * u;
        const double x0 = (a == 0 && g < ar.G) ? bc[f * ar.G + g] : 0.0;
        const double x1 = (a == 0 && g + 1 < ar.G) ? bc[f * ar.G + g + 1] : 0.0;
        xg_digits2<NS>(xg_fix(x0, K), xg_fix(x1, K), dig[u]);
      }
      unsigned char* dst = bcout + (size_t)(f * ar.oc + o) * bcw;
#pragma unroll
      for (int j = 0; j < NS; ++j)
        *reinterpret_cast<uint4*>(dst + (j * 8 + a) * 16) = make_uint4(dig[0][j], dig[1][j], dig[2][j], dig[3][j]);
    }
  }
}

namespace tc {
// F16 x F16 -> F32, both operands K-major
__host__ __device__ constexpr uint32_t idesc_f16(int M, int N) {
  return (1u << 4) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}
__device__ __forceinline__ void mma_f16(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc, uint32_t idesc,
                                        uint32_t accumulate) {
  asm volatile(
      "{\n.reg .pred p;\nsetp.ne.b32 p, %4, 0;\n"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(d_tmem),
      "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accumulate)
      : "memory");
}
// eight consecutive FP32 columns of this warp's quarter of TMEM
__device__ __forceinline__ void tmem_ld8(uint32_t taddr, uint32_t* r) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];\n"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
               : "r"(taddr));
}
__device__ __forceinline__ void mbar_expect(uint64_t* bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n" ::"r"(smem_u32(bar)), "r"(bytes) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint64_t* bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];\n" ::"r"(smem_u32(bar)) : "memory");
}
// bulk copy of `bytes` (16-byte multiples, aligned) from global memory, completing on the mbarrier
__device__ __forceinline__ void bulk_g2s(uint32_t dst, const void* src, uint32_t bytes, uint64_t* bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];\n" ::"r"(dst),
               "l"(src), "r"(bytes), "r"(smem_u32(bar))
               : "memory");
}
}  // namespace tc

// Folds an accumulator tile into this thread's 64-bit sums: TMEM row m = this lane, columns of the right
// block in groups of width WD: column n = (s NS + j) WD + b; acc[h][s WD + b] += 512^(..) value, digits
// j < 4 into h = 0 and the rest into h = 1.
template <int NS, int WD>
__device__ __forceinline__ void xg_fold(uint32_t ta, int nsub, long long* acc) {
  constexpr int W = XgCfg<NS>::W;
#pragma unroll
  for (int s = 0; s < W / WD; ++s) {
    if (s >= nsub) continue;
#pragma unroll
    for (int j = 0; j < NS; ++j) {
      constexpr int CH = WD % 16 == 0 ? 16 : 8;  // columns in flight (registers hold the sums)
      const int h = j / 4;
      const int wgt = 1 << (9 * ((h == 0 ? 3 : NS - 1) - j));
#pragma unroll
      for (int b0 = 0; b0 < WD; b0 += CH) {
        uint32_t v[CH];
#pragma unroll
        for (int b = 0; b < CH; b += 8) tc::tmem_ld8(ta + (uint32_t)((s * NS + j) * WD + b0 + b), v + b);
        tc::tmem_wait_ld();
#pragma unroll
        for (int b = 0; b < CH; ++b)
          asm("mad.wide.s32 %0, %1, %2, %0;"
              : "+l"(acc[h * W + s * WD + b0 + b])
              : "r"(__float2int_rn(__uint_as_float(v[b]))), "r"(wgt));
      }
    }
  }
}

// The digit products of a row range: CTA (group, k) accumulates the tiles of plan entry k over its row
// group and writes its 64-bit sums to part[group][tile][h][column n][row m].  One warp copies the
// operand blocks of 64 rows into a ring of stages (one bulk copy per column group and octet), one
// thread issues the MMAs, and four warps per tile fold its accumulators every 256 rows; the tiles' fold
// points are staggered by 64 rows, so the MMAs of the other tiles run while one is folded.
template <int NS>
__global__ void __launch_bounds__(kXgThreads, 1)
    k_xg_mma(const __grid_constant__ XgPlan pl, const __grid_constant__ XgArgs ar, long long* __restrict__ part,
             int* __restrict__ status) {
  constexpr int W = XgCfg<NS>::W, H = XgCfg<NS>::H, NSW = NS * W;
  extern __shared__ __align__(1024) unsigned char xg_smem[];
  __shared__ uint64_t full[kXgMaxStage], empty[kXgMaxStage], acc_full[kXgTiles], acc_empty[kXgTiles];
  __shared__ uint32_t tbase, boff[kXgMaxBlk];
  __shared__ int nsubs;
  __shared__ struct {
    uint32_t dst, ldo;  // smem offset of the group in its stage, bytes per octet of its block
    int off, bytes, arr, nb;
  } csub[kXgMaxBlk * 4];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int kcta = blockIdx.x % pl.ncta;
  const long group = blockIdx.x / pl.ncta;
  const int nblk = pl.cblks[kcta], nt = pl.ctiles[kcta], nst = ar.nstage;
  const uint32_t ncols = tc::tmem_cols(nt * NSW);
  if (warp == 0) {
    tc::tmem_alloc(&tbase, ncols);
    tc::tmem_relinquish();
  }
  if (tid == 32) {
    for (int i = 0; i < nst; ++i) {
      tc::mbar_init(&full[i], 1);
      tc::mbar_init(&empty[i], 1);
    }
    for (int i = 0; i < kXgTiles; ++i) {
      tc::mbar_init(&acc_full[i], 1);
      tc::mbar_init(&acc_empty[i], 4);
    }
    uint32_t o = 0;
    int n = 0;
    for (int i = 0; i < nblk; ++i) {
      const int b = pl.blk[kcta][i], rows = xg_block_rows(pl, b);
      boff[i] = o;
      for (int u = 0; u < pl.bnsub[b]; ++u) {
        const XgSub& sb = pl.sub[pl.bsub0[b] + u];
        csub[n].dst = o + (uint32_t)(u * NS * sb.w) * 16u;
        csub[n].ldo = (uint32_t)rows * 16u;
        csub[n].off = sb.off;
        csub[n].bytes = NS * sb.w * 16;
        csub[n].arr = sb.arr;
        csub[n].nb = sb.nb;
        ++n;
      }
      o += (uint32_t)rows * 128u;
    }
    nsubs = n;
  }
  // what an M = 128 operand may read past the last stage
  for (int i = tid; i < (int)kXgPad / 16; i += kXgThreads)
    reinterpret_cast<uint4*>(xg_smem + nst * ar.stage_bytes)[i] = make_uint4(0, 0, 0, 0);
  tc::fence_before_sync();
  __syncthreads();
  tc::fence_after_sync();
  const uint32_t tmem = tbase;
  const uint32_t sbase = tc::smem_u32(xg_smem);
  const long ob = group * ar.opg;
  const long oe = (ob + ar.opg < ar.noct) ? ob + ar.opg : ar.noct;
  const int ntile = (int)((oe - ob + 7) / 8);
  bool lost = false;  // a bounded wait of this thread ran out

  if (warp < 16) {
    // ---- fold
    const int q = warp >> 2;
    if (q < nt) {
      long long acc[W * H];
#pragma unroll
      for (int i = 0; i < W * H; ++i) acc[i] = 0;
      const int bq = pl.blk[kcta][pl.tq[kcta][q]];
      const int w = pl.sub[pl.bsub0[bq]].w, ns = pl.bnsub[bq];
      const uint32_t ta = tmem + ((uint32_t)(32 * (warp & 3)) << 16) + (uint32_t)(q * NSW);
      int f = 0;
      for (int t = 0; t < ntile && !lost; ++t) {
        if (!((t + 1 - q) % 4 == 0 || t == ntile - 1)) continue;
        if (!tc::mbar_wait(&acc_full[q], f & 1)) {
          lost = true;
          break;
        }
        ++f;
        tc::fence_after_sync();
        if constexpr (NS == 4) {
          if (w == 32) xg_fold<NS, 32>(ta, ns, acc);
          else if (w == 24) xg_fold<NS, 24>(ta, ns, acc);
          else if (w == 16) xg_fold<NS, 16>(ta, ns, acc);
          else xg_fold<NS, 8>(ta, ns, acc);
        } else {
          if (w == 16) xg_fold<NS, 16>(ta, ns, acc);
          else xg_fold<NS, 8>(ta, ns, acc);
        }
        tc::fence_before_sync();
        __syncwarp();
        if (lane == 0) tc::mbar_arrive(&acc_empty[q]);
      }
      long long* out = part + ((size_t)group * pl.ntile + pl.tile0[kcta] + q) * (size_t)(H * W * 128);
      const int m = 32 * (warp & 3) + lane;
#pragma unroll
      for (int i = 0; i < W * H; ++i) out[(size_t)i * 128 + m] = acc[i];
    }
  } else if (warp == 16) {
    // ---- copies
    const int n8 = nsubs * 8;
    uint32_t total = 0;
    for (int i = 0; i < nsubs; ++i) total += (uint32_t)csub[i].bytes * 8u;
    for (int t = 0; t < ntile; ++t) {
      const int st = t % nst, ph = t / nst;
      if (t >= nst && !tc::mbar_wait(&empty[st], (ph - 1) & 1)) {
        lost = true;
        break;
      }
      if (lane == 0) tc::mbar_expect(&full[st], total);
      __syncwarp();
      const uint32_t stage = sbase + (uint32_t)(st * ar.stage_bytes);
      for (int i = lane; i < n8; i += 32) {
        const int u = i >> 3, o = i & 7;
        const long oct = ob + (long)t * 8 + o;
        const int nb = csub[u].nb;
        const unsigned char* src = ar.zero;
        if (oct < oe && nb != 255) {
          long from = oct;
          bool ok = true;
          if (nb != 0) {
            const unsigned cell = (unsigned)oct / (unsigned)ar.oc;
            if (nb < 8) {
              const int ax = (nb - 1) >> 1, up = (nb - 1) & 1;
              const int idx = (int)((cell / (unsigned)ar.cstr[ax]) % (unsigned)ar.ext[ax]);
              ok = up ? idx < ar.ext[ax] - 1 : idx > 0;
              from += (up ? 1L : -1L) * ar.cstr[ax] * ar.oc;
            } else {
              const int face = ar.face[nb - 8], ax = face >> 1;
              const int idx = (int)((cell / (unsigned)ar.cstr[ax]) % (unsigned)ar.ext[ax]);
              ok = (face & 1) ? idx == ar.ext[ax] - 1 : idx == 0;
              from = (long)(nb - 8) * ar.oc + (oct - (long)cell * ar.oc);
            }
          }
          if (ok)
            src = nb >= 8 ? ar.bc + from * ar.bcrec
                          : (csub[u].arr ? ar.dig[1] + from * ar.rec[1] : ar.dig[0] + from * ar.rec[0]) + csub[u].off;
        }
        tc::bulk_g2s(stage + csub[u].dst + (uint32_t)o * csub[u].ldo, src, (uint32_t)csub[u].bytes, &full[st]);
      }
    }
    // the copies in flight land before the CTA ends (their stages were all consumed otherwise)
    if (__any_sync(0xffffffffu, lost))
      for (int st = 0; st < nst; ++st)
        if (st < ntile) (void)tc::mbar_wait(&full[st], 0, 1L << 16);
  } else if (lane == 0) {
    // ---- MMAs
    int used[kXgTiles] = {0, 0, 0, 0};  // chunks folded so far
    for (int t = 0; t < ntile; ++t) {
      const int st = t % nst;
      if (!tc::mbar_wait(&full[st], (t / nst) & 1)) {
        lost = true;
        break;
      }
      tc::fence_after_sync();
      const uint32_t stage = sbase + (uint32_t)(st * ar.stage_bytes);
#pragma unroll
      for (int i = 0; i < kXgTiles; ++i) {
        const int q = (t + 1 + i) & 3;  // the tile that starts a chunk here comes last
        if (q >= nt) continue;
        const bool start = t == 0 || (t - q) % 4 == 0;
        if (start && t > 0 && !lost) {
          int u = 0;
#pragma unroll
          for (int x = 0; x < kXgTiles; ++x)
            if (x == q) u = used[x]++;
          if (!tc::mbar_wait(&acc_empty[q], u & 1)) lost = true;
          tc::fence_after_sync();
        }
        if (lost) break;
        const int lp = pl.tp[kcta][q], lq = pl.tq[kcta][q];
        const int rp = xg_block_rows(pl, pl.blk[kcta][lp]), rq = xg_block_rows(pl, pl.blk[kcta][lq]);
        const uint32_t ldp = (uint32_t)rp * 16u, ldq = (uint32_t)rq * 16u;
        const uint32_t ap = stage + boff[lp], bp = stage + boff[lq];
        const uint32_t idesc = tc::idesc_f16(128, rq);
#pragma unroll
        for (int kk = 0; kk < 4; ++kk)
          tc::mma_f16(tmem + (uint32_t)(q * NSW), tc::smem_desc(ap + 2u * kk * ldp, ldp, 128u),
                      tc::smem_desc(bp + 2u * kk * ldq, ldq, 128u), idesc, (start && kk == 0) ? 0u : 1u);
        if ((t + 1 - q) % 4 == 0 || t == ntile - 1) tc::mma_commit(&acc_full[q]);
      }
      if (lost) break;
      tc::mma_commit(&empty[st]);
    }
    if (lost) {
      // MMAs may still run: wait for them (bounded) before the accumulators are released
      tc::mma_commit(&empty[0]);
      (void)tc::mbar_wait(&empty[0], 0, 1L << 16);
    }
  }
  tc::fence_before_sync();
  if (__syncthreads_or(lost) && tid == 0) latch(status, TT_ERR_TIMEOUT);
  if (warp == 0) {
    tc::fence_after_sync();
    tc::tmem_dealloc(tmem, ncols);
  }
}

// ---- sum of the partial sums ---------------------------------------------------------------------
// 192-bit two's complement integers (three 64-bit words, low first).
struct Int192 {
  unsigned long long w[3];
};
__device__ __forceinline__ void add192(Int192& a, unsigned long long x0, unsigned long long x1, unsigned long long x2) {
  const unsigned long long s0 = a.w[0] + x0;
  const unsigned long long t1 = a.w[1] + x1;
  const unsigned long long s1 = t1 + (s0 < x0 ? 1ull : 0ull);
  const unsigned long long carry = (t1 < x1 ? 1ull : 0ull) + (s1 < t1 ? 1ull : 0ull);
  a.w[0] = s0;
  a.w[1] = s1;
  a.w[2] = a.w[2] + x2 + carry;
}
__device__ __forceinline__ void add_shifted(Int192& a, __int128 v, int sh) {  // a += v 2^sh, 0 <= sh < 128
  const unsigned long long lo = (unsigned long long)v;
  const long long hi = (long long)(v >> 64);
  if (sh == 0) {
    add192(a, lo, (unsigned long long)hi, (unsigned long long)(hi >> 63));
  } else if (sh >= 64) {
    const int t = sh - 64;
    add192(a, 0ull, lo << t, (t ? lo >> (64 - t) : 0ull) | ((unsigned long long)hi << t));
  } else {
    add192(a, lo << sh, (lo >> (64 - sh)) | ((unsigned long long)hi << sh), (unsigned long long)(hi >> (64 - sh)));
  }
}

// Raw products as 192-bit integers, summed over the row groups, the left digits i and the digit groups of
// the right column: gint[word plane][row a][column b], row-major with ldg.  Upper triangle of blocks: the
// mirrored entry is written too; split: columns of array 1 start at ldg's column 0.  One thread per entry.
template <int NS>
__global__ void __launch_bounds__(256) k_xg_sum(const __grid_constant__ XgPlan pl, int ngroups, int split, int ldg,
                                                size_t plane, const long long* __restrict__ part,
                                                unsigned long long* __restrict__ gint) {
  constexpr int W = XgCfg<NS>::W, H = XgCfg<NS>::H;
  const int tile = blockIdx.x;
  const int p = pl.gp[tile], q = pl.gq[tile];
  const int idx = blockIdx.y * blockDim.x + threadIdx.x;
  const int ia = idx % W, ib = idx / W;
  if (ib >= W) return;
  const int wp = pl.sub[pl.bsub0[p]].w, wq = pl.sub[pl.bsub0[q]].w;
  const int sp = ia / wp, sq = ib / wq;
  if (sp >= pl.bnsub[p] || sq >= pl.bnsub[q]) return;
  const XgSub& up = pl.sub[pl.bsub0[p] + sp];
  const XgSub& uq = pl.sub[pl.bsub0[q] + sq];
  const int a = ia - sp * wp, b = ib - sq * wq;
  if (a >= up.cnt || b >= uq.cnt) return;
  const size_t gstride = (size_t)pl.ntile * (H * W * 128);
  const long long* base = part + (size_t)tile * (H * W * 128);
  Int192 g{{0ull, 0ull, 0ull}};
#pragma unroll
  for (int i = 0; i < NS; ++i) {
#pragma unroll
    for (int h = 0; h < H; ++h) {
      const long long* ptr = base + (size_t)(h * W + ib) * 128 + (sp * NS + i) * wp + a;
      __int128 s = 0;
      int gr = 0;
      for (; gr + 7 < ngroups; gr += 8) {
        long long v[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) v[u] = ptr[(gr + u) * gstride];
#pragma unroll
        for (int u = 0; u < 8; ++u) s += v[u];
      }
      for (; gr < ngroups; ++gr) s += ptr[gr * gstride];
      add_shifted(g, s, 9 * (NS - 1 - i) + ((H == 2 && h == 0) ? 9 * (NS - 4) : 0));
    }
  }
  const int ra = up.raw0 + a, rb = uq.raw0 + b - split;
  const size_t o = (size_t)ra * ldg + rb;
  gint[o] = g.w[0];
  gint[plane + o] = g.w[1];
  gint[2 * plane + o] = g.w[2];
  if (split == 0 && p != q) {
    const size_t m = (size_t)rb * ldg + ra;
    gint[m] = g.w[0];
    gint[plane + m] = g.w[1];
    gint[2 * plane + m] = g.w[2];
  }
}

// A column of the transport sum in raw columns: sum_i al[i] raw[i] (|al| <= 2), times coef.
struct XgComb {
  int n, raw[3], al[3], slot;
  double coef;
};
template <typename S>
__device__ __forceinline__ XgComb xg_comb(const SrcStencil<S>& s, int c) {
  XgComb x{};
  const auto cc = s.col(c);
  x.coef = cc.kind == 1 ? -cc.lam : cc.kind == 4 ? -0.5 * cc.lam : cc.kind == 5 ? 0.5 * cc.lam : 1.0;
  if (cc.kind == 2) {
    x.n = 1;
    x.raw[0] = (1 + 2 * s.nax) * s.rcap + cc.b;
    x.al[0] = 1;
    x.slot = s.rcap + cc.b;
    return x;
  }
  x.slot = cc.q;
  const int C = cc.q, L = (1 + 2 * cc.ax) * s.rcap + cc.q, Hh = L + s.rcap;
  auto put = [&](int raw, int al) {
    x.raw[x.n] = raw;
    x.al[x.n++] = al;
  };
  if (cc.kind == 0) put(C, 1);
  else if (cc.kind == 4) { put(Hh, 1); put(L, -1); }
  else if (cc.kind == 5) { put(Hh, 1); put(C, -2); put(L, 1); }
  else if (cc.w > 0) { put(C, 1); put(L, -1); }
  else { put(Hh, 1); put(C, -1); }
  return x;
}
template <class Src>
__device__ __forceinline__ XgComb xg_comb(const Src&, int c) {
  return XgComb{1, {c, 0, 0}, {1, 0, 0}, c, 1.0};
}

// Upper triangle of the Gram matrix of the sum's columns from the raw products (exact), and each
// column's unit and coefficient.
template <int NS, class Src>
__global__ void __launch_bounds__(256) k_xg_combine(const __grid_constant__ Src src, int n, int nraw,
                                                    const unsigned long long* __restrict__ raw,
                                                    const unsigned long long* __restrict__ slots,
                                                    unsigned long long* __restrict__ gint, int* __restrict__ unit,
                                                    double* __restrict__ coef) {
  const int idx = blockIdx.x * blockDim.x + threadIdx.x;
  const int a = idx / n, b = idx - (idx / n) * n;
  if (a >= n) return;
  if (a == b) {
    const XgComb x = xg_comb(src, a);
    unit[a] = xg_unit(slots[x.slot], NS);
    coef[a] = x.coef;
  }
  if (b < a) return;
  const XgComb x = xg_comb(src, a), y = xg_comb(src, b);
  const size_t rp = (size_t)nraw * nraw, plane = (size_t)n * n;
  Int192 g{{0ull, 0ull, 0ull}};
  for (int i = 0; i < x.n; ++i)
    for (int j = 0; j < y.n; ++j) {
      const size_t o = (size_t)x.raw[i] * nraw + y.raw[j];
      unsigned long long w0 = raw[o], w1 = raw[rp + o], w2 = raw[2 * rp + o];
      int al = x.al[i] * y.al[j];
      if (al < 0) {  // two's complement negation
        w0 = ~w0 + 1ull;
        w1 = ~w1 + (w0 == 0ull ? 1ull : 0ull);
        w2 = ~w2 + ((w0 | w1) == 0ull ? 1ull : 0ull);
        al = -al;
      }
      for (int k = 0; k < al; ++k) add192(g, w0, w1, w2);
    }
  const size_t o = (size_t)a * n + b;
  gint[o] = g.w[0];
  gint[plane + o] = g.w[1];
  gint[2 * plane + o] = g.w[2];
}

// ---- host drivers --------------------------------------------------------------------------------
// Row groups of a pass: one CTA per SM over ncta CTAs a group (`sms` SMs for this pass), at least 128
// rows each, and at most kXgMaxOct octets.
inline void xg_groups(long noct, int ncta, int sms, long& groups, long& opg) {
  groups = sms / ncta;
  const long most = (noct + 15) / 16, least = (noct + kXgMaxOct - 1) / kXgMaxOct;
  if (groups > most) groups = most;
  if (groups < least) groups = least;
  if (groups < 1) groups = 1;
  opg = (noct + groups - 1) / groups;
  opg = (opg + 7) / 8 * 8;
  groups = (noct + opg - 1) / opg;
}

template <class Src>
struct XgElem;
template <typename S>
struct XgElem<SrcRows<S>> { using type = S; };
template <typename S>
struct XgElem<SrcCols<S>> { using type = S; };
template <typename S>
struct XgElem<SrcStencil<S>> { using type = S; };

// Plan of a source's columns.
template <int NS, typename S>
inline bool xg_make_plan(const SrcRows<S>&, const LivePattern& lp, XgPlan& pl) {
  const int n = lp.ncap();
  pl.nsub = 0;
  pl.nraw = n;
  return n <= kXcMaxN && xg_add<NS>(pl, n, 0, 0, 0) && xg_tiles<NS>(pl, false) && xg_stages(pl) >= 2;
}
template <int NS, typename S>
inline bool xg_make_plan(const SrcCols<S>&, const LivePattern& lp, XgPlan& pl) {
  return xg_make_plan<NS>(SrcRows<S>{nullptr, 0}, lp, pl);
}
template <int NS, typename S>
inline bool xg_make_plan(const SrcStencil<S>& s, const LivePattern& lp, XgPlan& pl) {
  pl.nsub = 0;
  const int nsh = 1 + 2 * s.nax;
  pl.nraw = nsh * s.rcap + lp.nextra;
  if (lp.ncap() > kXcMaxN || pl.nraw > kXgMaxRaw || s.rcap > 256 || lp.nextra > 6) return false;
  for (int i = 0; i < nsh; ++i)
    if (!xg_add<NS>(pl, s.rcap, i * s.rcap, 0, i)) return false;
  for (int e = 0; e < lp.nextra; ++e)
    if (!xg_add<NS>(pl, 1, nsh * s.rcap + e, 0, 8 + e)) return false;
  return xg_tiles<NS>(pl, false) && xg_stages(pl) >= 2;
}
template <typename S>
inline bool xg_array(const SrcRows<S>& s, int n, long nrows, int NS, XgArray& ar, const S** A) {
  ar = XgArray{n, 8, 1, (nrows + 7) / 8, NS == 4 ? xg_record<4>(n) : xg_record<7>(n), s.ld, 1};
  *A = s.A;
  return ar.ncell < (1L << 31);
}
template <typename S>
inline bool xg_array(const SrcCols<S>& s, int n, long nrows, int NS, XgArray& ar, const S** A) {
  ar = XgArray{n, 8, 1, (nrows + 7) / 8, NS == 4 ? xg_record<4>(n) : xg_record<7>(n), 1, s.ld};
  *A = s.A;
  return ar.ncell < (1L << 31);
}
template <typename S>
inline bool xg_array(const SrcStencil<S>& s, int, long nrows, int NS, XgArray& ar, const S** A) {
  ar = XgArray{s.rcap, s.G, (s.G + 7) / 8, nrows / s.G, NS == 4 ? xg_record<4>(s.rcap) : xg_record<7>(s.rcap),
               s.ldz, 1};
  *A = s.Z;
  return ar.ncell * ar.oc < (1L << 31);
}
template <class Src>
inline LivePattern xg_array_live(const Src&, const LivePattern& lp) { return lp; }
template <typename S>
inline LivePattern xg_array_live(const SrcStencil<S>&, const LivePattern& lp) {
  return LivePattern{lp.r_ptr, lp.rcap, 1, 0};
}
template <class Src>
inline void xg_geometry(const Src&, XgArgs& a, const double** bc, int*) {
  a.nax = 0;
  *bc = nullptr;
}
template <typename S>
inline void xg_geometry(const SrcStencil<S>& s, XgArgs& a, const double** bc, int* nbc) {
  a.nax = s.nax;
  for (int i = 0; i < 3; ++i) {
    a.ext[i] = s.ext[i];
    a.cstr[i] = (int)(s.stride[i] / s.G);
  }
  *bc = s.bcval;
  for (int e = 0; e < *nbc; ++e) a.face[e] = (unsigned char)(2 * s.axis[s.bc_term[e]] + (s.w[s.bc_term[e]] > 0 ? 0 : 1));
}

// The plan of a source's columns, kept per shape and host thread (a pure function of the shape: the
// greedy assignment takes some microseconds, and a step asks several times).
template <class Src>
inline long xg_plan_key(const Src&, const LivePattern& lp) { return lp.ncap(); }
template <typename S>
inline long xg_plan_key(const SrcStencil<S>& s, const LivePattern& lp) {
  return 1000000L * (1 + s.nax) + 1000L * s.rcap + 10L * lp.nextra + 100000000L * lp.nblk;
}
template <int NS, class Src>
inline const XgPlan* xg_plan_of(const Src& src, const LivePattern& lp) {
  struct Entry {
    bool ok;
    XgPlan pl;
  };
  if (lp.rcap > 999 || lp.nextra > 6) return nullptr;
  static thread_local std::map<long, Entry> cache;
  const long key = xg_plan_key(src, lp);
  auto it = cache.find(key);
  if (it == cache.end()) {
    if (cache.size() >= 64) cache.clear();
    it = cache.emplace(key, Entry{}).first;
    it->second.ok = xg_make_plan<NS>(src, lp, it->second.pl);
  }
  return it->second.ok ? &it->second.pl : nullptr;
}

// Whether a pass of the source over nrows rows can take the exact Gram kernels.
template <typename T, class Src>
inline bool xg_fits(const Src& src, const LivePattern& lp, long nrows) {
  constexpr int NS = sizeof(T) == 4 ? 4 : 7;
  XgArray ar;
  const typename XgElem<Src>::type* A = nullptr;
  return xg_plan_of<NS>(src, lp) != nullptr && xg_array(src, lp.ncap(), nrows, NS, ar, &A);
}

// Launches the product kernels of a plan whose digit records are in place.
template <int NS>
tt_status xg_launch_products(cudaStream_t s, const XgPlan& pl, XgArgs& args, long groups, long long* part, int split,
                             int ldg, size_t plane, unsigned long long* gint, int* status) {
  constexpr int W = XgCfg<NS>::W;
  args.stage_bytes = xg_stage_bytes(pl);
  args.nstage = xg_stages(pl);
  size_t smem = args.stage_bytes * args.nstage + kXgPad;
  if (smem < 117 * 1024) smem = 117 * 1024;  // one CTA per SM: its accumulators never wait for another's
  auto kern = k_xg_mma<NS>;
  if (const tt_status a = smem_optin(kern, smem); a != TT_OK) return a;
  kern<<<(unsigned)(groups * pl.ncta), kXgThreads, smem, s>>>(pl, args, part, status);
  count_launch();
  k_xg_sum<NS><<<dim3((unsigned)pl.ntile, (W * W + 255) / 256), 256, 0, s>>>(pl, (int)groups, split, ldg, plane, part,
                                                                           gint);
  count_launch();
  return cudaGetLastError() == cudaSuccess ? TT_OK : TT_ERR_CUDA;
}
template <int NS, typename S>
void xg_launch_digits(cudaStream_t s, int num_sms, const S* A, const XgArray& ar, LivePattern lp, long nrows,
                      unsigned long long* slots, unsigned char* dig, const double* bc, int nbc, unsigned char* bcdig) {
  const long rpb = 256 / ar.ncol, need = (nrows + 8 * rpb - 1) / (8 * rpb);
  long grid = need < 8L * num_sms ? need : 8L * num_sms;
  k_xg_colmax<S><<<(unsigned)(grid > 0 ? grid : 1), 256, 0, s>>>(A, ar.ncol, ar.sr, ar.sc, nrows, slots, bc, nbc, ar.G);
  count_launch();
  const long tot = ar.ncell * ar.oc * (ar.rec / (NS * 16));
  grid = (tot + 255) / 256;
  if (grid > 16L * num_sms) grid = 16L * num_sms;
  k_xg_digits<NS, S><<<(unsigned)(grid > 0 ? grid : 1), 256, 0, s>>>(A, ar, lp, nrows, slots, dig, bc, nbc, bcdig);
  count_launch();
}

// Triangular factor RZ (ncap x ncap, row-major; R^T R = A^T A) of the source's columns.  sms: SMs this
// pass may take.  Dry runs take the workspace only; everything but RZ is released on return (later
// work on the stream may overwrite it).
template <typename T, class Src>
tt_status xg_factor(cudaStream_t s, int num_sms, int sms, const Src& src, LivePattern lp, long nrows, Bump& ws,
                    double** RZ_out, int* status, int leaf_cat = kTsqrLeaf) {
  using S = typename XgElem<Src>::type;
  constexpr int NS = sizeof(T) == 4 ? 4 : 7;
  constexpr int W = XgCfg<NS>::W, H = XgCfg<NS>::H;
  const int n = lp.ncap();
  const XgPlan* plan = xg_plan_of<NS>(src, lp);
  XgArray ar;
  const S* A = nullptr;
  if (!plan || !xg_array(src, n, nrows, NS, ar, &A)) return TT_ERR_UNSUPPORTED;
  const XgPlan& pl = *plan;
  double* R = ws.take<double>((size_t)n * n);
  *RZ_out = R;
  const size_t mark = ws.off;
  XgArgs args{};
  int nbc = lp.nextra;
  const double* bc = nullptr;
  xg_geometry(src, args, &bc, &nbc);
  if (!bc) nbc = 0;
  args.oc = ar.oc;
  args.noct = ar.ncell * ar.oc;
  args.rec[0] = ar.rec;
  args.bcrec = NS * 8 * 16;
  long groups;
  xg_groups(args.noct, pl.ncta, sms > 0 ? sms : num_sms, groups, args.opg);
  const size_t zbytes = (size_t)NS * W * 16;
  // zeroed: column maxima and the page of zeros
  unsigned char* zeroed = ws.take<unsigned char>(zbytes + 8 * (size_t)(n + kMaxTerms));
  unsigned long long* slots = reinterpret_cast<unsigned long long*>(zeroed + zbytes);
  unsigned char* dig = ws.take<unsigned char>((size_t)args.noct * ar.rec);
  unsigned char* bcdig = ws.take<unsigned char>((size_t)nbc * ar.oc * args.bcrec);
  long long* part = ws.take<long long>((size_t)groups * pl.ntile * (H * W * 128));
  unsigned long long* raw = ws.take<unsigned long long>(3 * (size_t)pl.nraw * pl.nraw);
  unsigned long long* gint = ws.take<unsigned long long>(3 * (size_t)n * n);
  int* unit = ws.take<int>(n);
  double* coef = ws.take<double>(n);
  ws.release(mark);
  if (ws.dry) return TT_OK;
  {
    TimerScope scope(leaf_cat, s);
    cudaMemsetAsync(zeroed, 0, zbytes + 8 * (size_t)(n + kMaxTerms), s);
    xg_launch_digits<NS>(s, num_sms, A, ar, xg_array_live(src, lp), nrows, slots, dig, bc, nbc, bcdig);
    args.dig[0] = args.dig[1] = dig;
    args.rec[1] = ar.rec;
    args.bc = bcdig;
    args.zero = zeroed;
    const tt_status st = xg_launch_products<NS>(s, pl, args, groups, part, 0, pl.nraw,
                                                (size_t)pl.nraw * pl.nraw, raw, status);
    if (st != TT_OK) return st;
    k_xg_combine<NS, Src><<<(unsigned)((n * n + 255) / 256), 256, 0, s>>>(src, n, pl.nraw, raw, slots, gint, unit, coef);
    count_launch();
  }
  TimerScope scope(kTsqrMerge, s);
  return launch_xg_chol(s, n, gint, unit, coef, R);
}
}  // namespace ttk
