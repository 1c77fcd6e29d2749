// Exact Gram products of tall column blocks on the tensor cores, and the triangular factor of the
// merged core's columns from them (the L->R orthogonalisation of the rounding, Sec. 3.1 footnote).
//
// Every storage column c is held in fixed point, v = round(x 2^-U_c) with one power of two per column,
// and v is written in balanced digits of base 256,
//   v = sum_j d_j 256^(NS-1-j),   -128 <= d_j <= 127,
// NS = 4 digits (30 bits and sign) for FP32 passes and NS = 8 (62 bits and sign) for FP64 passes.
// Digits are exact in FP16, products of two digits are integers up to 2^14, and the FP32
// accumulators of tcgen05.mma.kind::f16 sum 1,024 rows of them without any rounding (every partial sum is
// an integer of at most 2^24: the limit, a longer chunk would round).  The digit products of a chunk are then
// folded into 64-bit integers.
// So sum_k v_a v_b comes out exactly, for columns whose entries carry a fixed-point rounding of at most
// 2^-(8 NS - 1) of their column's largest entry (FP32 2^-31, FP64 2^-63; the storage's own rounding of
// entries near that size is 2^-25 and 2^-54).  The columns of the transport sum are integer
// combinations of a row and its neighbours (C - L, H - C, H - L, H - 2 C + L), so their Gram matrix is an
// integer combination of the products of the neighbour blocks, formed without rounding or
// cancellation (k_xg_combine); the operators' coefficients scale the factor's columns at the end.
//
// The factor R with R^T R = G is a Cholesky factor in fixed point (xchol.cuh), 128 bits for FP64 passes and 64 for
// FP32 ones: G is exact and columns are resolved down to about 2^-57 (2^-27) of their norm, as a Householder QR in
// FP64 (FP32) resolves them.
//
// Why: a Householder TSQR is a chain of reflectors behind block barriers on the FMA pipes; measured
// at 1,048,576 rows x 160 columns it took 5.3 ms (FP32 leaf) + 2.1 ms (merges) and 91.9 + 17 ms in
// FP64, whose FMA pipe runs at 1/64 of the FP32 rate on this part.  Here the digits of the storage
// columns are written once (k_xg_digits, bound by memory) in the layout of the MMA operands, so that the
// product kernel (k_xg_mma) only moves 16-byte rows with bulk copies: a neighbour block is the same
// digits at another cell, a missing neighbour a page of zeros.  Measured for both roundings of a step
// at 1,048,576 rows, rank 32: FP32 digits 0.18, products 0.64 ms (leaves and merges before: 6.0 + 2.1 ms);
// FP64 0.28, 1.7 ms (before 99.6 + 14 ms).  With base 512 and MMAs of N = 128 columns over octets copied one by
// one the products took 0.87 and 3.06 ms.
#pragma once
#include <cmath>
#include <map>
#include <vector>

#include "bigpass.cuh"
#include "instr.cuh"
#include "small.cuh"
#include "tc.cuh"
#include "xchol.cuh"

namespace ttk {

constexpr int kXgCopy = 2;        // copying warps
constexpr int kXgThreads = 32 * (16 + kXgCopy + 1);  // 16 folding warps, the copying warps, an MMA warp
constexpr int kXgGroups = 2;      // MMA groups of a CTA: one block of rows x up to two blocks (N <= 256)
constexpr int kXgTiles = 4;       // output tiles of a CTA (TMEM: 4 x 128 columns)
// Octets of rows of a stage (and at most of a piece): 64 rows.  A stage costs its hand-over beside its MMAs: with 32
// rows the products of the 1,048,576 x 160 pass took 1.03 ms instead of 0.68 (FP64 2.80, 1.80).
constexpr int kXgStageOct = 8;
constexpr int kXgChunkTiles = 128 / kXgStageOct;  // stages between two folds: 1024 rows * 2^14 = 2^24 is exact
constexpr int kXgMaxBlk = 6;      // operand blocks a CTA stages
constexpr int kXgMaxSub = 56;     // column groups of a pass
constexpr int kXgMaxNb = 24;      // operand blocks of a pass
constexpr int kXgMaxCta = 80;     // CTAs that share a row range
constexpr int kXgMaxStage = 8;
constexpr long kXgMaxPieces = 512L * 16;  // pieces per CTA: at most 512 chunks, the 64-bit sums stay below 2^58
constexpr int kXgMaxRaw = 448;          // storage columns of all neighbour blocks

template <int NS>
struct XgCfg {
  static constexpr int W = NS == 4 ? 32 : 16;  // columns per operand block (NS * W <= 128 rows)
  static constexpr int H = NS / 4;             // 64-bit sums per entry (groups of 4 digits)
};

// A storage matrix whose rows are the groups of cells (row = g + G cell), or plain rows (cells of 64).  Its
// digits are kept in pieces: a cell's rows (padded) in `parts` pieces of `po` octets, po even and at most
// kXgStageOct, so that a piece is a run of K for the MMAs and every neighbour's rows are pieces too.  One plane per
// column group: [cell][part][rows j w + a of the operand in eights][octet][8 rows x 16 bytes].
struct XgArray {
  int ncol, G, po, parts;
  long ncell, npiece;  // npiece = ncell * parts
  int cpad;            // columns with the groups' padding
  long sr, sc;         // element strides of rows and columns
};
inline void xg_pieces(XgArray& ar) {
  const int oc = (ar.G + 7) / 8;
  ar.parts = (oc + kXgStageOct - 1) / kXgStageOct;
  ar.po = ((oc + ar.parts - 1) / ar.parts + 1) & ~1;
  ar.npiece = ar.ncell * ar.parts;
}

// One column group of the products: `w` columns (a multiple of 8, the last ones padding) of an array, at
// the cell itself (nb = 0), its lower (1 + 2 axis) or upper (2 + 2 axis) neighbour, or the inflow column
// of a face (nb = 8 + face).
struct XgSub {
  short raw0;        // first raw column
  unsigned char cnt, w, arr, nb;
  int c0;            // columns (with padding) in the planes before
};

struct XgPlan {
  int ns, nsub, nb, ncta, nraw;
  XgSub sub[kXgMaxSub];
  unsigned char bsub0[kXgMaxNb], bnsub[kXgMaxNb];  // operand block -> its column groups (equal widths)
  unsigned char cgroups[kXgMaxCta], cblks[kXgMaxCta];
  unsigned char blk[kXgMaxCta][kXgMaxBlk];           // local block -> operand block, in the stage's order
  unsigned char gm[kXgMaxCta][kXgGroups];            // MMA group: local block of the rows,
  unsigned char gn[kXgMaxCta][kXgGroups], gnn[kXgMaxCta][kXgGroups];  // first local block of the columns, and how many
  unsigned char tp[kXgMaxCta * kXgTiles], tq[kXgMaxCta * kXgTiles];   // tile 4 cta + 2 group + h: blocks (p, q);
                                                                      // p = 255: unused
};

// What the product kernel reads beside the plan.
struct XgArgs {
  const unsigned char* dig[2];  // digit records of the arrays
  const unsigned char* bc;      // digit pieces of one cell of the inflow columns: [face slot][part]
  const unsigned char* zero;    // a page of zeros
  int po, parts, nc;            // octets of a piece, pieces of a cell, pieces of a stage
  long npiece, ppg;             // pieces in all, and per row group
  int nax, ext[3];
  int cstr[3];                  // cell strides of the axes
  unsigned char face[6];        // inflow column -> 2 axis + (upper face)
  int nstage;
  size_t stage_bytes;
  const int* skip;              // (nullable) no products where it is set
};

__host__ __device__ inline int xg_block_rows(const XgPlan& pl, int b) {
  return pl.ns * pl.sub[pl.bsub0[b]].w * pl.bnsub[b];
}

// Adds the column groups of `ncol` columns to the plan: whole operand blocks of W columns, then the rest
// rounded up to 8; groups of equal width are made adjacent by xg_tiles.
template <int NS>
inline bool xg_add(XgPlan& pl, int ncol, int raw0, int arr, int nb) {
  constexpr int W = XgCfg<NS>::W;
  int c0 = 0;
  for (int c = 0; c < ncol; c += W) {
    if (pl.nsub == kXgMaxSub) return false;
    const int cnt = ncol - c < W ? ncol - c : W, w = (cnt + 7) & ~7;
    pl.sub[pl.nsub++] = XgSub{(short)(raw0 + c), (unsigned char)cnt, (unsigned char)w, (unsigned char)arr,
                              (unsigned char)nb, c0};
    c0 += w;
  }
  return true;
}

// Operand blocks (column groups of one width side by side, at most W columns), and the MMA groups of each
// CTA: the upper triangle of the blocks, or (arrays: split) blocks of array 0 x blocks of array 1.  A group
// is one block of rows times an aligned pair of blocks (N = 256: an MMA of N = 128 takes as long as one
// of 256, measured 1,930 against 1,070 cycles for 16 products of 128 x 128 x 16); an odd last block takes
// the rows against every pair.  A CTA has two groups (512 TMEM columns), the second one chosen to share
// most blocks with the first.
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
    }
    if (arr == 0) nleft = pl.nb;
  }
  struct Group {
    int m, n0, nn;
  };
  std::vector<Group> gr;
  const int q0 = split ? nleft : 0, np = split ? nleft : pl.nb, nq = pl.nb - q0;
  if (split) {
    for (int j = 0; j < nq; j += 2)
      for (int p = 0; p < np; ++p) gr.push_back({p, q0 + j, j + 1 < nq ? 2 : 1});
  } else {
    for (int j = 0; j + 1 < nq; j += 2)
      for (int p = 0; p <= j + 1; ++p) gr.push_back({p, j, 2});
    if (nq & 1) {
      for (int j = 0; j + 1 < nq; j += 2) gr.push_back({nq - 1, j, 2});
      gr.push_back({nq - 1, nq - 1, 1});
    }
  }
  pl.ncta = 0;
  while (!gr.empty()) {
    if (pl.ncta == kXgMaxCta) return false;
    const int k = pl.ncta++;
    int nblk = 0;
    unsigned char* blk = pl.blk[k];
    auto local = [&](int b) {
      for (int i = 0; i < nblk; ++i)
        if (blk[i] == b) return i;
      return -1;
    };
    auto added = [&](const Group& g) {  // blocks a group adds
      int a = 0;
      for (int i = 0; i < g.nn; ++i) a += local(g.n0 + i) < 0;
      return a + (local(g.m) < 0 && (g.m < g.n0 || g.m >= g.n0 + g.nn));
    };
    Group mine[kXgGroups];
    int ng = 0;
    while (ng < kXgGroups && !gr.empty()) {
      size_t best = 0;
      for (size_t i = 1; i < gr.size(); ++i)
        if (added(gr[i]) < added(gr[best])) best = i;
      const Group g = gr[best];
      gr.erase(gr.begin() + best);
      mine[ng++] = g;
      // a pair's blocks lie side by side in the stage: aligned pairs are always added whole
      if (local(g.n0) < 0 || (g.nn == 2 && local(g.n0 + 1) != local(g.n0) + 1))
        for (int i = 0; i < g.nn; ++i) blk[nblk++] = (unsigned char)(g.n0 + i);
      if (local(g.m) < 0) blk[nblk++] = (unsigned char)g.m;
    }
    pl.cgroups[k] = (unsigned char)ng;
    pl.cblks[k] = (unsigned char)nblk;
    for (int g = 0; g < kXgGroups; ++g)
      for (int h = 0; h < 2; ++h) {
        const int t = kXgTiles * k + 2 * g + h;
        pl.tp[t] = pl.tq[t] = 255;
        if (g >= ng || h >= mine[g].nn) continue;
        const int p = mine[g].m, q = mine[g].n0 + h;
        // the entry below the diagonal of a diagonal pair, and an odd last block's row against itself
        // through a pair, have their mirror elsewhere
        if (!split && p > q && !((nq & 1) && p == nq - 1)) continue;
        pl.tp[t] = (unsigned char)p;
        pl.tq[t] = (unsigned char)q;
      }
    for (int g = 0; g < ng; ++g) {
      pl.gm[k][g] = (unsigned char)local(mine[g].m);
      pl.gn[k][g] = (unsigned char)local(mine[g].n0);
      pl.gnn[k][g] = (unsigned char)mine[g].nn;
    }
  }
  return true;
}

// Bytes of a stage (every operand block of the CTA that stages most).
inline size_t xg_stage_bytes(const XgPlan& pl, int oct = kXgStageOct) {
  size_t most = 0;
  for (int k = 0; k < pl.ncta; ++k) {
    size_t b = 0;
    for (int i = 0; i < pl.cblks[k]; ++i) b += (size_t)xg_block_rows(pl, pl.blk[k][i]) * (16 * oct);
    if (b > most) most = b;
  }
  return most;
}
constexpr size_t kXgPad = 16 * 1024;  // an M = 128 operand of a narrower block reads past its piece
inline int xg_stages(const XgPlan& pl, int oct = kXgStageOct) {
  const int n = (int)((226 * 1024 - kXgPad) / xg_stage_bytes(pl, oct));
  return n < kXgMaxStage ? n : kXgMaxStage;
}

// ---- fixed point ---------------------------------------------------------------------------------
// Unit exponent U of a column with largest magnitude `maxbits` (an FP64 bit pattern): every entry is
// below 2^E, and 2^E maps to 2^(8 NS - 2), inside the digits' range.
__host__ __device__ inline int xg_unit(unsigned long long maxbits, int NS) {
  return ((int)((maxbits >> 52) & 0x7ff) - 1022) - (8 * NS - 2);
}
// round(x 2^-U), U folded into the shift constant K (see xg_shift_const).  Zero and FP64's subnormal numbers (an
// exponent field of zero; their squares vanish in FP64) give 0, FP32's are taken as FP64 numbers; Inf and NaN give
// some in-range integer.
__device__ __forceinline__ long long xg_fix(double x, int K) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(x);
  const int e = (int)((b >> 52) & 0x7ff);
  const unsigned long long m = e ? (((b & 0xfffffffffffffull) | 0x10000000000000ull) << 10) : 0ull;
  const int sh = min(max(K - e, 0), 63);
  const long long r = (long long)(((m >> sh) + 1ull) >> 1);
  return (long long)b < 0 ? -r : r;
}
__device__ __forceinline__ long long xg_fix(float x, int K) {
  const unsigned b = __float_as_uint(x);
  const int e = (int)((b >> 23) & 0xff);
  if (e == 0) return b << 1 ? xg_fix((double)x, K + 896) : 0;
  const unsigned long long m = (unsigned long long)((b & 0x7fffffu) | 0x800000u) << 39;
  const int sh = min(max(K - e, 0), 63);
  const long long r = (long long)(((m >> sh) + 1ull) >> 1);
  return (int)b < 0 ? -r : r;
}
__device__ __forceinline__ int xg_shift_const(double, int U) { return 1084 + U; }
__device__ __forceinline__ int xg_shift_const(float, int U) { return 188 + U; }

// Digits of two rows of one column packed as FP16 pairs: dig[j] = (row 0, row 1) for digit j.  v + bias
// (128 in every byte) has the biased digits 0..255 as its bytes.
template <int NS>
__device__ __forceinline__ void xg_digits2(long long v0, long long v1, unsigned (&dig)[NS]) {
  constexpr unsigned long long kBias = 0x8080808080808080ull >> (64 - 8 * NS);
  const unsigned long long u0 = (unsigned long long)v0 + kBias, u1 = (unsigned long long)v1 + kBias;
#pragma unroll
  for (int j = 0; j < NS; ++j) {
    const int byte = NS - 1 - j;
    const unsigned a = (unsigned)(u0 >> (32 * (byte / 4))), b = (unsigned)(u1 >> (32 * (byte / 4)));
    const unsigned k = (unsigned)(byte % 4);
    unsigned x = (__byte_perm(a, b, k | (4u + k) << 8) & 0x00ff00ffu) | 0x64006400u;  // 1024 + biased digit
    asm("sub.rn.f16x2 %0, %0, %1;" : "+r"(x) : "r"(0x64806480u));                     // - 1152
    dig[j] = x;
  }
}

// Column maxima |x| (FP64 bit patterns of which the exponent counts, over the finite entries: Inf and NaN are
// latched where the rows are rewritten, or set *nonfinite where none are) of a matrix of ncol <= 256 columns: a
// CTA takes whole rows, a thread always the same column, eight loads in flight.  Compared as the integers of
// their upper 32 bits: FP64 comparisons run on the FP64 pipe (1,048,576 x 32 FP64: 0.21 ms, now 0.05).
__device__ __forceinline__ unsigned xg_high(double x) { return (unsigned)__double2hiint(x) & 0x7fffffffu; }
__device__ __forceinline__ unsigned xg_high(float x) { return __float_as_uint(x) & 0x7fffffffu; }
template <typename S>
__global__ void __launch_bounds__(256) k_xg_colmax(const S* __restrict__ A, int ncol, long sr, long sc, long nrows,
                                                   unsigned long long* __restrict__ slots,
                                                   const double* __restrict__ bc, int nbc, int G,
                                                   int* __restrict__ nonfinite) {
  __shared__ unsigned sm[256];
  constexpr unsigned kInf = sizeof(S) == 4 ? 0x7f800000u : 0x7ff00000u;
  const int rpb = 256 / ncol, tid = threadIdx.x;
  const int col = tid % ncol, sub = tid / ncol;
  for (int i = tid; i < ncol; i += blockDim.x) sm[i] = 0u;
  __syncthreads();
  if (sub < rpb) {
    unsigned m = 0u, top = 0u;
    const long step = (long)gridDim.x * rpb;
    long k = (long)blockIdx.x * rpb + sub;
    for (; k + 7 * step < nrows; k += 8 * step) {
      S v[8];
#pragma unroll
      for (int u = 0; u < 8; ++u) v[u] = A[(k + u * step) * sr + col * sc];
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        const unsigned a = xg_high(v[u]);
        top = max(top, a);
        m = max(m, a < kInf ? a : 0u);
      }
    }
    for (; k < nrows; k += step) {
      const unsigned a = xg_high(A[k * sr + col * sc]);
      top = max(top, a);
      m = max(m, a < kInf ? a : 0u);
    }
    if (nonfinite && top >= kInf) *nonfinite = 1;
    atomicMax(&sm[col], m);
  }
  __syncthreads();
  for (int i = tid; i < ncol; i += blockDim.x) {
    const unsigned m = sm[i];
    atomicMax(&slots[i], sizeof(S) == 4 ? (unsigned long long)__double_as_longlong((double)__uint_as_float(m))
                                        : (unsigned long long)m << 32);
  }
  if (blockIdx.x == 0)
    for (int i = tid; i < nbc * G; i += blockDim.x)
      atomicMax(&slots[ncol + i / G], (unsigned long long)__double_as_longlong(fabs(bc[i])));
}

// Byte offset of row m's octet in a plane of groups of w columns (NS w rows) at piece `piece`.
template <int NS>
__device__ __forceinline__ size_t xg_dig_off(long piece, int po, int w, int m, int oct) {
  return ((size_t)piece * (NS * w / 8) + (m >> 3)) * (size_t)(po * 128) + oct * 128 + (m & 7) * 16;
}

// Digits of an array (and, in the first CTA, of the inflow columns: one cell, one column each): a thread
// forms one column of one octet, eight rows, and writes 16 bytes per digit.  Bound by memory:
// N r (sizeof(S) + 2 NS) bytes.
template <int NS, typename S>
__global__ void __launch_bounds__(256) k_xg_digits(const S* __restrict__ A, XgArray ar, LivePattern lp, long nrows,
                                                   const unsigned long long* __restrict__ slots,
                                                   unsigned char* __restrict__ out, const double* __restrict__ bc,
                                                   int nbc, unsigned char* __restrict__ bcout,
                                                   const int* __restrict__ skip) {
  constexpr int W = XgCfg<NS>::W;
  const bool off = skip && *skip != 0;  // (tested behind the loads below, which hide it)
  const int r = lp.r_ptr ? *lp.r_ptr : lp.rcap;
  const int cpad = ar.cpad;
  const long noct = ar.npiece * ar.po;
  const long tot = noct * cpad;
  long i = blockIdx.x * (long)blockDim.x + threadIdx.x;
  for (; i < tot; i += (long)gridDim.x * blockDim.x) {
    const long oct = tot < (1L << 31) ? (long)((unsigned)i / (unsigned)cpad) : i / cpad;
    const int c = (int)(i - oct * cpad);
    const unsigned piece = (unsigned)oct / (unsigned)ar.po;
    const int oin = (int)((unsigned)oct - piece * (unsigned)ar.po);
    const unsigned cell = ar.parts == 1 ? piece : piece / (unsigned)ar.parts;
    const int g0 = ((int)(piece - cell * (unsigned)ar.parts) * ar.po + oin) * 8;
    const long k0 = (long)cell * ar.G + g0;
    // column groups are full blocks of W and then the rest: the width of this column's group
    const int blk = c / W, a = c - blk * W;
    const int w = cpad - blk * W < W ? cpad - blk * W : W;
    const bool ok = c < ar.ncol && lp.live(c, r);
    S x[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) x[u] = (ok && g0 + u < ar.G && k0 + u < nrows) ? A[(k0 + u) * ar.sr + c * ar.sc] : S(0);
    const int K = xg_shift_const(S(0), ok ? xg_unit(slots[c], NS) : 0);
    if (off) return;
    unsigned dig[4][NS];
#pragma unroll
    for (int u = 0; u < 4; ++u) xg_digits2<NS>(xg_fix(x[2 * u], K), xg_fix(x[2 * u + 1], K), dig[u]);
    unsigned char* o = out + (size_t)(blk * W) * noct * (NS * 16);
#pragma unroll
    for (int j = 0; j < NS; ++j)
      *reinterpret_cast<uint4*>(o + xg_dig_off<NS>(piece, ar.po, w, j * w + a, oin)) =
          make_uint4(dig[0][j], dig[1][j], dig[2][j], dig[3][j]);
  }
  if (blockIdx.x == 0 && nbc > 0) {
    // one inflow column: a group of 8, seven of them padding
    const int co = ar.parts * ar.po;
    for (int e = threadIdx.x; e < nbc * co * 8; e += blockDim.x) {
      const int f = e / (co * 8), rem = e - f * co * 8, o = rem / 8, a = rem - o * 8;
      const int K = xg_shift_const(0.0, xg_unit(slots[ar.ncol + f], NS));
      unsigned dig[4][NS];
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int g = 8 * o + 2 * u;
        const double x0 = (a == 0 && g < ar.G) ? bc[f * ar.G + g] : 0.0;
        const double x1 = (a == 0 && g + 1 < ar.G) ? bc[f * ar.G + g + 1] : 0.0;
        xg_digits2<NS>(xg_fix(x0, K), xg_fix(x1, K), dig[u]);
      }
#pragma unroll
      for (int j = 0; j < NS; ++j)
        *reinterpret_cast<uint4*>(bcout + xg_dig_off<NS>((long)f * ar.parts + o / ar.po, ar.po, 8, j * 8 + a, o % ar.po)) =
            make_uint4(dig[0][j], dig[1][j], dig[2][j], dig[3][j]);
    }
  }
}

// Column maxima and digit records of a small explicit matrix in one launch: a CTA takes eight columns, all
// rows (at most kXgSmallRows).  The small cores' matrices are a chain of short kernels, bound by
// launches: this one stands for a memset and two kernels.  The first CTA zeroes the page of zeros.
constexpr long kXgSmallRows = 4096;
template <int NS, typename S>
__global__ void __launch_bounds__(256) k_xg_small_digits(const S* __restrict__ A, XgArray ar, LivePattern lp, long nrows,
                                                         unsigned long long* __restrict__ slots,
                                                         unsigned char* __restrict__ out, uint4* __restrict__ zero,
                                                         int nzero) {
  constexpr int W = XgCfg<NS>::W;
  __shared__ unsigned long long sm[8];
  constexpr S kMax = sizeof(S) == 4 ? (S)3.402823466e+38f : (S)1.7976931348623157e308;
  const int tid = threadIdx.x;
  const int r = lp.r_ptr ? *lp.r_ptr : lp.rcap;
  const int c0 = blockIdx.x * 8;
  if (blockIdx.x == 0)
    for (int i = tid; i < nzero; i += blockDim.x) zero[i] = make_uint4(0, 0, 0, 0);
  if (tid < 8) sm[tid] = 0ull;
  __syncthreads();
  // maxima: the faster of rows and columns in memory goes along the lanes
  const bool rowmajor = ar.sc == 1;
  const int cl = rowmajor ? tid & 7 : tid >> 5, rl = rowmajor ? tid >> 3 : tid & 31;
  {
    const int c = c0 + cl;
    S m = S(0);
    if (c < ar.ncol && lp.live(c, r)) {
#pragma unroll 8
      for (long k = rl; k < nrows; k += 32) {
        const S a = fabs(A[k * ar.sr + c * ar.sc]);
        m = (a > m && a <= kMax) ? a : m;
      }
    }
    atomicMax(&sm[cl], (unsigned long long)__double_as_longlong((double)m));
  }
  __syncthreads();
  if (tid < 8 && c0 + tid < ar.ncol) slots[c0 + tid] = sm[tid];
  const int cpad = ar.cpad;
  const int noct = (int)ar.npiece * ar.po;  // octets of rows, pieces one after the other
  const int a8 = rowmajor ? tid & 7 : (tid >> 2) & 7;  // column of the slab
  const int o0 = rowmajor ? tid >> 3 : (tid & 3) | ((tid >> 5) << 2);
  const int c = c0 + a8;
  const bool ok = c < ar.ncol && lp.live(c, r);
  const int K = xg_shift_const(S(0), ok ? xg_unit(sm[a8], NS) : 0);
  const int blk = c / W, a = c - blk * W;
  const int w = cpad - blk * W < W ? cpad - blk * W : W;
  for (int o = o0; o < noct; o += 32) {
    S x[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) x[u] = (ok && 8l * o + u < nrows) ? A[(8l * o + u) * ar.sr + c * ar.sc] : S(0);
    unsigned dig[4][NS];
#pragma unroll
    for (int u = 0; u < 4; ++u) xg_digits2<NS>(xg_fix(x[2 * u], K), xg_fix(x[2 * u + 1], K), dig[u]);
    unsigned char* dst = out + (size_t)(blk * W) * noct * (NS * 16);
#pragma unroll
    for (int j = 0; j < NS; ++j)
      *reinterpret_cast<uint4*>(dst + xg_dig_off<NS>(o / ar.po, ar.po, w, j * w + a, o % ar.po)) =
          make_uint4(dig[0][j], dig[1][j], dig[2][j], dig[3][j]);
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
__device__ __forceinline__ void tmem_ld4(uint32_t taddr, uint32_t* r) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0, %1, %2, %3}, [%4];\n"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
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

// Columns of an operand block that one of the four folding warpgroups takes.
template <int NS>
struct XgFold {
  static constexpr int Q = XgCfg<NS>::W / 4;
};
// Folds this warpgroup's columns of an accumulator tile into its 64-bit sums: TMEM row m = this lane, the
// block's column c = s w + b at TMEM column (s NS + j) w + b for digit j (ta: at j = 0 of the first of Q
// columns); acc[h][..] += 256^(..) value, digits j < 4 into h = 0 and the rest into h = 1.  All loads are in
// flight at once; release (nullable): arrive there as soon as they have landed.
template <int NS>
__device__ __forceinline__ void xg_fold(uint32_t ta, int w, uint64_t* release, long long* acc) {
  constexpr int Q = XgFold<NS>::Q;
  uint32_t v[NS][Q];
#pragma unroll
  for (int j = 0; j < NS; ++j) {
    if constexpr (Q == 8) tc::tmem_ld8(ta + (uint32_t)(j * w), v[j]);
    else tc::tmem_ld4(ta + (uint32_t)(j * w), v[j]);
  }
  tc::tmem_wait_ld();
  if (release) {
    tc::fence_before_sync();
    __syncwarp();
    if ((threadIdx.x & 31) == 0) tc::mbar_arrive(release);
  }
#pragma unroll
  for (int j = 0; j < NS; ++j) {
    const int wgt = 1 << (8 * (3 - j % 4));
#pragma unroll
    for (int b = 0; b < Q; ++b)
      asm("mad.wide.s32 %0, %1, %2, %0;"
          : "+l"(acc[(j / 4) * Q + b])
          : "r"(__float2int_rn(__uint_as_float(v[j][b]))), "r"(wgt));
  }
}

// The ring of stages after `issued` tiles: tiles first .. issued - 1 are the last ones of their stages, and tile u's
// copies complete the phase of parity (u / nst) & 1 of its stage's mbarrier.
__host__ __device__ __forceinline__ int xg_last_first(int issued, int nst) { return issued > nst ? issued - nst : 0; }
__host__ __device__ __forceinline__ unsigned xg_fill_parity(int u, int nst) { return (unsigned)(u / nst) & 1u; }

// Whether MMA group g ends a chunk with tile t (of ntile): the two groups' chunks are half a chunk apart.
__device__ __forceinline__ bool xg_ends(int g, int t, int ntile) {
  return (t + 1 + g * (kXgChunkTiles / 2)) % kXgChunkTiles == 0 || t == ntile - 1;
}

// The digit products of a row range: CTA (group, k) accumulates the tiles of plan entry k over its row
// group and writes its 64-bit sums to part[group][tile][h][column n][row m].  Two warps copy the
// operand blocks of up to 64 rows into a ring of stages (one bulk copy per column group and piece: copies
// an octet at a time, 2 KB, took 1.6 times as long), one thread issues the MMAs, and sixteen warps fold a
// group's accumulators every 16 stages (at most 1024 rows; each warp a quarter of the rows and of the
// columns, all its loads in flight) while the MMAs of the other group run.  A stage of eight MMAs (1,024 cycles at
// the tensor cores' rate) takes about 1,800: the copies share the L2 (7 to 8 TB/s) and each stage is handed over.
template <int NS>
__global__ void __launch_bounds__(kXgThreads, 1)
    k_xg_mma(const __grid_constant__ XgPlan pl, const __grid_constant__ XgArgs ar, long long* __restrict__ part,
             int* __restrict__ status) {
  constexpr int W = XgCfg<NS>::W, H = XgCfg<NS>::H;
  extern __shared__ __align__(1024) unsigned char xg_smem[];
  __shared__ uint64_t full[kXgMaxStage], empty[kXgMaxStage], acc_full[kXgGroups], acc_empty[kXgGroups], done;
  __shared__ uint32_t tbase, rows_s;
  __shared__ int nsubs, off;
  __shared__ struct {
    uint64_t a, b;
    uint32_t idesc;
  } ginfo[kXgGroups];
  __shared__ struct {
    uint32_t dst;  // offset of the group in a piece of the stage
    int c0, bytes, arr, nb;
  } csub[kXgMaxBlk * 4];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int kcta = blockIdx.x % pl.ncta;
  const long group = blockIdx.x / pl.ncta;
  const int nblk = pl.cblks[kcta], ng = pl.cgroups[kcta], nst = ar.nstage;
  constexpr uint32_t kCols = 512;
  if (warp == 0) {
    tc::tmem_alloc(&tbase, kCols);
    tc::tmem_relinquish();
  }
  if (tid == 32) {
    for (int i = 0; i < nst; ++i) {
      tc::mbar_init(&full[i], 1);
      tc::mbar_init(&empty[i], 1);
    }
    for (int i = 0; i < kXgGroups; ++i) {
      tc::mbar_init(&acc_full[i], 1);
      tc::mbar_init(&acc_empty[i], 16);
    }
    tc::mbar_init(&done, 1);
    // a piece of a stage: the rows (digits of columns) of the CTA's blocks one after the other, in eights
    // of po octets each (K-major core matrices without swizzle: LBO 128, SBO 128 po)
    const uint32_t po16 = (uint32_t)ar.po * 16u;
    uint32_t rows = 0, boff[kXgMaxBlk];
    int n = 0;
    for (int i = 0; i < nblk; ++i) {
      const int b = pl.blk[kcta][i];
      boff[i] = rows;
      for (int u = 0; u < pl.bnsub[b]; ++u) {
        const XgSub& sb = pl.sub[pl.bsub0[b] + u];
        csub[n].dst = (rows + (uint32_t)(u * NS * sb.w)) * po16;
        csub[n].c0 = sb.c0;
        csub[n].bytes = NS * sb.w * (int)po16;
        csub[n].arr = sb.arr;
        csub[n].nb = sb.nb;
        ++n;
      }
      rows += (uint32_t)xg_block_rows(pl, b);
    }
    nsubs = n;
    rows_s = rows;
    // operands of the MMA groups: descriptors at stage 0 (the address field counts 16 bytes) and the
    // instruction descriptor, read by the issuing thread for every stage (from the plan in constant
    // memory the chain of dependent loads took longer than the MMAs)
    const uint32_t s0 = tc::smem_u32(xg_smem);
    for (int g = 0; g < ng; ++g) {
      const int m = pl.gm[kcta][g], n0 = pl.gn[kcta][g];
      int nrow = 0;
      for (int i = 0; i < pl.gnn[kcta][g]; ++i) nrow += xg_block_rows(pl, pl.blk[kcta][n0 + i]);
      ginfo[g].a = tc::smem_desc(s0 + boff[m] * po16, 128u, 8u * po16);
      ginfo[g].b = tc::smem_desc(s0 + boff[n0] * po16, 128u, 8u * po16);
      ginfo[g].idesc = tc::idesc_f16(128, nrow);
    }
  }
  if (tid == 64) off = ar.skip ? *ar.skip : 0;
  // what an M = 128 operand may read past the last piece
  for (int i = tid; i < (int)kXgPad / 16; i += kXgThreads)
    reinterpret_cast<uint4*>(xg_smem + nst * ar.stage_bytes)[i] = make_uint4(0, 0, 0, 0);
  tc::fence_before_sync();
  __syncthreads();
  tc::fence_after_sync();
  const uint32_t tmem = tbase;
  const uint32_t sbase = tc::smem_u32(xg_smem);
  const uint32_t pieceb = rows_s * (uint32_t)ar.po * 16u;  // bytes of a piece of the stage
  const int nc = ar.nc;
  const long pb = group * ar.ppg;
  const long pe = (pb + ar.ppg < ar.npiece) ? pb + ar.ppg : ar.npiece;
  const int ntile = off ? 0 : (int)((pe - pb + nc - 1) / nc);
  bool lost = false;  // a bounded wait of this thread ran out

  if (warp < 16) {
    // ---- fold: warpgroup v takes the columns [v Q, v Q + Q) of every tile's right block
    constexpr int Q = XgFold<NS>::Q;
    const int v = warp >> 2;
    long long acc[kXgTiles][H * Q];
    uint32_t ta[kXgTiles];
    int wd[kXgTiles];
#pragma unroll
    for (int q = 0; q < kXgTiles; ++q) {
#pragma unroll
      for (int i = 0; i < H * Q; ++i) acc[q][i] = 0;
      wd[q] = 0;
      ta[q] = 0;
      if (pl.tp[kXgTiles * kcta + q] != 255) {
        const int bq = pl.tq[kXgTiles * kcta + q];
        const int w = pl.sub[pl.bsub0[bq]].w, sb = (v * Q) / w;
        if (sb < pl.bnsub[bq]) wd[q] = w;  // 0: no such columns
        const int first = (q & 1) ? xg_block_rows(pl, bq - 1) : 0;  // the pair's first block
        ta[q] = tmem + ((uint32_t)(32 * (warp & 3)) << 16) + (uint32_t)((q >> 1) * 256 + first + sb * NS * w + (v * Q - sb * w));
      }
    }
    int f[kXgGroups] = {0, 0};
    for (int t = 0; t < ntile && !lost; ++t) {
#pragma unroll
      for (int g = 0; g < kXgGroups; ++g) {
        if (g >= ng || lost || !xg_ends(g, t, ntile)) continue;
        if (!tc::mbar_wait(&acc_full[g], f[g] & 1)) {
          lost = true;
          continue;
        }
        ++f[g];
        tc::fence_after_sync();
        if (wd[2 * g] > 0) xg_fold<NS>(ta[2 * g], wd[2 * g], wd[2 * g + 1] > 0 ? nullptr : &acc_empty[g], acc[2 * g]);
        if (wd[2 * g + 1] > 0) xg_fold<NS>(ta[2 * g + 1], wd[2 * g + 1], &acc_empty[g], acc[2 * g + 1]);
        if (wd[2 * g] == 0 && wd[2 * g + 1] == 0 && lane == 0) tc::mbar_arrive(&acc_empty[g]);
      }
    }
    const int m = 32 * (warp & 3) + lane;
#pragma unroll
    for (int q = 0; q < kXgTiles; ++q) {
      if (pl.tp[kXgTiles * kcta + q] == 255) continue;
      long long* out = part + ((size_t)group * pl.ncta * kXgTiles + kXgTiles * kcta + q) * (size_t)(H * W * 128);
#pragma unroll
      for (int h = 0; h < H; ++h)
#pragma unroll
        for (int b = 0; b < Q; ++b) out[(size_t)(h * W + v * Q + b) * 128 + m] = acc[q][h * Q + b];
    }
  } else if (warp < 16 + kXgCopy) {
    // ---- copies: a lane keeps some of a stage's copies, their sources and cells advanced from stage to
    // stage (formed anew each time, with divisions and indexed parameters, the addresses of a stage took
    // some 3,000 cycles: 8.3 ms of products at 3,538,944 x 242, then 6.6)
    const int ncopy = nsubs * nc;
    constexpr int kPer = (kXgMaxBlk * 4 * (kXgStageOct / 2) + 32 * kXgCopy - 1) / (32 * kXgCopy);
    const int first = lane * kXgCopy + (warp - 16);
    const unsigned char* src[kPer];
    uint32_t dst[kPer];
    int bytes[kPer], kind[kPer], cs[kPer], ex[kPer], cpart[kPer], low[kPer], idx[kPer];
    long piece[kPer];
#pragma unroll
    for (int k = 0; k < kPer; ++k) {
      const int i = first + 32 * kXgCopy * k, u = i < ncopy ? i / nc : 0, c = i < ncopy ? i - u * nc : 0;
      const int nb = csub[u].nb;
      const int ax = nb == 0 ? 0 : nb < 8 ? (nb - 1) >> 1 : ar.face[nb - 8] >> 1;
      bytes[k] = csub[u].bytes;
      dst[k] = (uint32_t)c * pieceb + csub[u].dst;
      // 0 the cell, 1 lower and 2 upper neighbour, 3 lower and 4 upper face
      kind[k] = nb == 0 ? 0 : nb < 8 ? 1 + ((nb - 1) & 1) : 3 + (ar.face[nb - 8] & 1);
      cs[k] = nb == 0 ? 1 : ar.cstr[ax];
      ex[k] = nb == 0 ? 1 : ar.ext[ax];
      piece[k] = i < ncopy ? pb + c : pe;
      const long cell = piece[k] / ar.parts;
      cpart[k] = (int)(piece[k] - cell * ar.parts);
      low[k] = (int)(cell % cs[k]);
      idx[k] = (int)((cell / cs[k]) % ex[k]);
      const long shift = kind[k] == 1 ? -(long)cs[k] * ar.parts : kind[k] == 2 ? (long)cs[k] * ar.parts : 0;
      src[k] = nb >= 8 ? ar.bc + (size_t)(nb - 8) * ar.parts * bytes[k]
                       : (csub[u].arr ? ar.dig[1] : ar.dig[0]) + (size_t)csub[u].c0 * ar.npiece * (ar.po * NS * 16) +
                             (piece[k] + shift) * bytes[k];
    }
    int st = -1, t = 0;
    uint32_t ph = 1;
    for (; t < ntile; ++t) {
      if (++st == nst) {
        st = 0;
        ph ^= 1u;
      }
      if (t >= nst && !tc::mbar_wait(&empty[st], ph)) {
        lost = true;
        break;
      }
      if (warp == 16 && lane == 0) tc::mbar_expect(&full[st], pieceb * (uint32_t)nc);
      __syncwarp();
      const uint32_t stage = sbase + (uint32_t)(st * ar.stage_bytes);
#pragma unroll
      for (int k = 0; k < kPer; ++k) {
        if (first + 32 * kXgCopy * k >= ncopy) continue;
        const bool low_ = idx[k] == 0, up_ = idx[k] == ex[k] - 1;
        const bool ok = piece[k] < pe && (kind[k] == 0 || (kind[k] == 1 && !low_) || (kind[k] == 2 && !up_) ||
                                          (kind[k] == 3 && low_) || (kind[k] == 4 && up_));
        const unsigned char* from = kind[k] >= 3 ? src[k] + (size_t)cpart[k] * bytes[k] : src[k];
        tc::bulk_g2s(stage + dst[k], ok ? from : ar.zero, (uint32_t)bytes[k], &full[st]);
        piece[k] += nc;
        if (kind[k] < 3) src[k] += (long)nc * bytes[k];
        cpart[k] += nc;
        while (cpart[k] >= ar.parts) {
          cpart[k] -= ar.parts;
          if (++low[k] == cs[k]) {
            low[k] = 0;
            if (++idx[k] == ex[k]) idx[k] = 0;
          }
        }
      }
    }
    // the copies in flight land before the CTA ends, whoever gave up (bounded)
    for (int u = xg_last_first(t, nst); u < t; ++u) (void)tc::mbar_wait(&full[u % nst], xg_fill_parity(u, nst), 1L << 16);
  } else if (lane == 0) {
    // ---- MMAs
    // K steps of two octets; pieces of 1, 2, 3 or 4 steps (3 and 4: one piece a stage)
    // (operands in registers, and everything a stage does not change formed before: with them read and computed
    // between the MMAs a stage took some 1,900 cycles, of 1,024 for its eight MMAs)
    const int pk = ar.po / 2, ksteps = nc * pk;
    uint32_t ko[4];
#pragma unroll
    for (int kk = 0; kk < 4; ++kk) {
      const int c = kk / pk;
      ko[kk] = ((uint32_t)c * pieceb + (uint32_t)(kk - c * pk) * 256u) >> 4;
    }
    uint64_t ga[kXgGroups], gb[kXgGroups];
    uint32_t gi[kXgGroups];
#pragma unroll
    for (int g = 0; g < kXgGroups; ++g) {
      ga[g] = ginfo[g < ng ? g : 0].a;
      gb[g] = ginfo[g < ng ? g : 0].b;
      gi[g] = ginfo[g < ng ? g : 0].idesc;
    }
    const uint32_t sstep = (uint32_t)(ar.stage_bytes >> 4);
    uint32_t folds[kXgGroups] = {0, 0};   // chunks ended so far
    bool fresh[kXgGroups] = {true, true}; // the next MMA of the group starts a chunk
    auto issue = [&](int g, uint64_t da, uint64_t db, uint32_t idesc, uint32_t so, bool start) {
      const uint32_t d = tmem + (uint32_t)(g * 256);
      da += so;
      db += so;
      tc::mma_f16(d, da + ko[0], db + ko[0], idesc, start ? 0u : 1u);
      if (ksteps > 1) tc::mma_f16(d, da + ko[1], db + ko[1], idesc, 1u);
      if (ksteps > 2) tc::mma_f16(d, da + ko[2], db + ko[2], idesc, 1u);
      if (ksteps > 3) tc::mma_f16(d, da + ko[3], db + ko[3], idesc, 1u);
    };
    auto ready = [&](int g, uint32_t done) {  // the accumulators of group g have been folded
      const bool ok = tc::mbar_wait(&acc_empty[g], (done - 1) & 1);
      tc::fence_after_sync();
      return ok;
    };
    int st = -1;
    uint32_t ph = 0, so = 0;
    for (int t = 0; t < ntile; ++t) {
      if (++st == nst) {
        st = 0;
        ph ^= 1u;
        so = 0;
      }
      if (!tc::mbar_wait(&full[st], ph)) {
        lost = true;
        break;
      }
      tc::fence_after_sync();
      // a group whose accumulators are being folded comes last
      const bool swap = ng > 1 && fresh[0] && folds[0] > 0;
      const bool e0 = xg_ends(0, t, ntile), e1 = xg_ends(1, t, ntile);
      if (!swap) {
        if (fresh[0] && folds[0] > 0 && !ready(0, folds[0])) lost = true;
        if (lost) break;
        issue(0, ga[0], gb[0], gi[0], so, fresh[0]);
        if (e0) tc::mma_commit(&acc_full[0]);
      }
      if (ng > 1) {
        if (fresh[1] && folds[1] > 0 && !ready(1, folds[1])) lost = true;
        if (lost) break;
        issue(1, ga[1], gb[1], gi[1], so, fresh[1]);
        if (e1) tc::mma_commit(&acc_full[1]);
        fresh[1] = e1;
        folds[1] += e1;
      }
      if (swap) {
        if (!ready(0, folds[0])) lost = true;
        if (lost) break;
        issue(0, ga[0], gb[0], gi[0], so, true);
        if (e0) tc::mma_commit(&acc_full[0]);
      }
      fresh[0] = e0;
      folds[0] += e0;
      so += sstep;
      if (lost) break;
      tc::mma_commit(&empty[st]);
    }
    // the MMAs end before the accumulators are released, whoever gave up (bounded)
    tc::mma_commit(&done);
    if (!tc::mbar_wait(&done, 0, 1L << 16)) lost = true;
  }
  tc::fence_before_sync();
  if (__syncthreads_or(lost) && tid == 0) latch(status, TT_ERR_TIMEOUT);
  if (warp == 0) {
    tc::fence_after_sync();
    tc::tmem_dealloc(tmem, kCols);
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
// mirrored entry is written too; split: columns of array 1 start at ldg's column 0.
// unit, coef (nullable): the columns' units and coefficients where the raw columns are the columns.  add: to what
// is there (rows in several passes).
template <int NS>
__global__ void __launch_bounds__(256) k_xg_sum(const __grid_constant__ XgPlan pl, int ngroups, int split, int ldg,
                                                size_t plane, const long long* __restrict__ part,
                                                unsigned long long* __restrict__ gint,
                                                const unsigned long long* __restrict__ slots, int* __restrict__ unit,
                                                double* __restrict__ coef, int add) {
  constexpr int W = XgCfg<NS>::W, H = XgCfg<NS>::H;
  if (unit && blockIdx.x == 0 && blockIdx.y == 0 && (int)threadIdx.x < ldg) {
    unit[threadIdx.x] = xg_unit(slots[threadIdx.x], NS);
    coef[threadIdx.x] = 1.0;
  }
  __shared__ unsigned long long red[3][256];
  const int tile = blockIdx.x;
  const int p = pl.tp[tile], q = pl.tq[tile];
  if (p == 255) return;
  // 32 entries of a CTA, the row groups shared by its eight warps
  const int lane = threadIdx.x & 31, prt = threadIdx.x >> 5;
  const int idx = blockIdx.y * 32 + lane;
  const int ia = idx % W, ib = idx / W;
  const int wp = pl.sub[pl.bsub0[p]].w, wq = pl.sub[pl.bsub0[q]].w;
  const int sp = ia / wp, sq = ib / wq;
  bool ok = ib < W && sp < pl.bnsub[p] && sq < pl.bnsub[q];
  const XgSub& up = pl.sub[pl.bsub0[p] + (ok ? sp : 0)];
  const XgSub& uq = pl.sub[pl.bsub0[q] + (ok ? sq : 0)];
  const int a = ia - sp * wp, b = ib - sq * wq;
  ok = ok && a < up.cnt && b < uq.cnt;
  const size_t gstride = (size_t)pl.ncta * kXgTiles * (H * W * 128);
  const long long* base = part + (size_t)tile * (H * W * 128);
  Int192 g{{0ull, 0ull, 0ull}};
  if (ok) {
#pragma unroll
    for (int i = 0; i < NS; ++i) {
#pragma unroll
      for (int h = 0; h < H; ++h) {
        const long long* ptr = base + (size_t)(h * W + ib) * 128 + (sp * NS + i) * wp + a;
        __int128 s = 0;
        int gr = prt;
        for (; gr + 24 < ngroups; gr += 32) {
          long long v[4];
#pragma unroll
          for (int u = 0; u < 4; ++u) v[u] = ptr[(gr + 8 * u) * gstride];
#pragma unroll
          for (int u = 0; u < 4; ++u) s += v[u];
        }
        for (; gr < ngroups; gr += 8) s += ptr[gr * gstride];
        add_shifted(g, s, 8 * (NS - 1 - i) + 8 * 4 * (H - 1 - h));
      }
    }
  }
#pragma unroll
  for (int i = 0; i < 3; ++i) red[i][threadIdx.x] = g.w[i];
  __syncthreads();
  if (prt != 0 || !ok) return;
  for (int u = 1; u < 8; ++u) add192(g, red[0][32 * u + lane], red[1][32 * u + lane], red[2][32 * u + lane]);
  const int ra = up.raw0 + a, rb = uq.raw0 + b - split;
  const size_t o = (size_t)ra * ldg + rb;
  if (add) add192(g, gint[o], gint[plane + o], gint[2 * plane + o]);
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
// Row groups of a pass: one CTA per SM over ncta CTAs a group (`sms` SMs for this pass), at least two
// stages each, and at most kXgMaxPieces.
inline void xg_groups(long npiece, int nc, int ncta, int sms, long& groups, long& ppg) {
  groups = sms / ncta;
  const long most = (npiece + 2 * nc - 1) / (2 * nc), least = (npiece + kXgMaxPieces - 1) / kXgMaxPieces;
  if (groups > most) groups = most;
  if (groups < least) groups = least;
  if (groups < 1) groups = 1;
  ppg = (npiece + groups - 1) / groups;
  ppg = (ppg + nc - 1) / nc * nc;
  groups = (npiece + ppg - 1) / ppg;
}

template <class Src>
struct XgElem;
template <typename S>
struct XgElem<SrcRows<S>> { using type = S; static constexpr bool stencil = false; };
template <typename S>
struct XgElem<SrcCols<S>> { using type = S; static constexpr bool stencil = false; };
template <typename S>
struct XgElem<SrcStencil<S>> { using type = S; static constexpr bool stencil = true; };

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
inline int xg_cpad(int n) { return (n + 7) & ~7; }
template <typename S>
inline bool xg_array(const SrcRows<S>& s, int n, long nrows, XgArray& ar, const S** A) {
  ar = XgArray{n, 64, 0, 0, (nrows + 63) / 64, 0, xg_cpad(n), s.ld, 1};
  xg_pieces(ar);
  *A = s.A;
  return ar.npiece < (1L << 28);
}
template <typename S>
inline bool xg_array(const SrcCols<S>& s, int n, long nrows, XgArray& ar, const S** A) {
  ar = XgArray{n, 64, 0, 0, (nrows + 63) / 64, 0, xg_cpad(n), 1, s.ld};
  xg_pieces(ar);
  *A = s.A;
  return ar.npiece < (1L << 28);
}
template <typename S>
inline bool xg_array(const SrcStencil<S>& s, int, long nrows, XgArray& ar, const S** A) {
  ar = XgArray{s.rcap, s.G, 0, 0, nrows / s.G, 0, xg_cpad(s.rcap), s.ldz, 1};
  xg_pieces(ar);
  *A = s.Z;
  return ar.npiece < (1L << 28);
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
  constexpr int NS = sizeof(T) == 4 ? 4 : 8;
  XgArray ar{};
  const typename XgElem<Src>::type* A = nullptr;
  return xg_plan_of<NS>(src, lp) != nullptr && xg_array(src, lp.ncap(), nrows, ar, &A);
}

// Launches the product kernels of a plan whose digit records are in place.
template <int NS>
tt_status xg_launch_products(cudaStream_t s, const XgPlan& pl, XgArgs& args, long groups, long long* part, int split,
                             int ldg, size_t plane, unsigned long long* gint, const unsigned long long* slots, int* unit,
                             double* coef, int* status, bool add = false) {
  constexpr int W = XgCfg<NS>::W;
  args.stage_bytes = xg_stage_bytes(pl, args.nc * args.po);
  args.nstage = xg_stages(pl, args.nc * args.po);
  size_t smem = args.stage_bytes * args.nstage + kXgPad;
  if (smem < 117 * 1024) smem = 117 * 1024;  // one CTA per SM: its accumulators never wait for another's
  auto kern = k_xg_mma<NS>;
  if (const tt_status a = smem_optin(kern, smem); a != TT_OK) return a;
  kern<<<(unsigned)(groups * pl.ncta), kXgThreads, smem, s>>>(pl, args, part, status);
  count_launch();
  k_xg_sum<NS><<<dim3((unsigned)(pl.ncta * kXgTiles), W * W / 32), 256, 0, s>>>(pl, (int)groups, split, ldg, plane, part,
                                                                           gint, slots, unit, coef, add);
  count_launch();
  return cudaGetLastError() == cudaSuccess ? TT_OK : TT_ERR_CUDA;
}
// CTAs of k_xg_colmax over nrows rows of ncol <= 256 columns.
inline unsigned xg_colmax_grid(int num_sms, int ncol, long nrows) {
  const long rpb = 256 / ncol, need = (nrows + 8 * rpb - 1) / (8 * rpb);
  const long grid = need < 8L * num_sms ? need : 8L * num_sms;
  return (unsigned)(grid > 0 ? grid : 1);
}
template <int NS, typename S>
void xg_launch_digits(cudaStream_t s, int num_sms, const S* A, const XgArray& ar, LivePattern lp, long nrows,
                      unsigned long long* slots, unsigned char* dig, const double* bc, int nbc, unsigned char* bcdig,
                      int* nonfinite = nullptr) {
  k_xg_colmax<S><<<xg_colmax_grid(num_sms, ar.ncol, nrows), 256, 0, s>>>(A, ar.ncol, ar.sr, ar.sc, nrows, slots, bc, nbc,
                                                                         ar.G, nonfinite);
  count_launch();
  const long tot = ar.npiece * ar.po * ar.cpad;
  long grid = (tot + 255) / 256;
  if (grid > 16L * num_sms) grid = 16L * num_sms;
  k_xg_digits<NS, S><<<(unsigned)(grid > 0 ? grid : 1), 256, 0, s>>>(A, ar, lp, nrows, slots, dig, bc, nbc, bcdig, nullptr);
  count_launch();
}

// 192-bit integer times 2^e, rounded.
__device__ __forceinline__ double real192(Int192 g, int e) {
  const bool neg = (long long)g.w[2] < 0;
  if (neg) {
    const Int192 one{{1ull, 0ull, 0ull}};
    g = Int192{{~g.w[0], ~g.w[1], ~g.w[2]}};
    add192(g, one.w[0], one.w[1], one.w[2]);
  }
  // the top 64 bits and a sticky bit
  int up = 128;
  unsigned long long hi = g.w[2], mid = g.w[1], lo = g.w[0];
  if (hi == 0ull) {
    hi = mid;
    mid = lo;
    lo = 0ull;
    up = 64;
  }
  if (hi == 0ull) {
    hi = mid;
    mid = 0ull;
    up = 0;
  }
  if (hi == 0ull) return 0.0;
  const int lz = __clzll((long long)hi);
  unsigned long long top = lz ? (hi << lz) | (mid >> (64 - lz)) : hi;
  const unsigned long long rest = lz ? (mid << lz) | (lo >> (64 - lz)) : (mid | lo);
  if (rest | lo) top |= 1ull;
  const double v = ldexp(__ull2double_rn(top), up - lz + e);
  return neg ? -v : v;
}
// Gram matrix in FP64 from its integers (upper triangle), units and coefficients applied.
template <int NS>
__global__ void __launch_bounds__(256) k_xg_real(int n, const unsigned long long* __restrict__ gint,
                                                 const int* __restrict__ unit, const double* __restrict__ coef,
                                                 double* __restrict__ out) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n * n) return;
  const int a = i / n, b = i - a * n;
  const size_t plane = (size_t)n * n, o = a <= b ? i : (size_t)b * n + a;
  const Int192 g{{gint[o], gint[plane + o], gint[2 * plane + o]}};
  out[i] = coef[a] * coef[b] * real192(g, unit[a] + unit[b]);
}
template <int NS>
__global__ void __launch_bounds__(256) k_xg_real_cols(int rows, int cols, size_t plane, const unsigned long long* __restrict__ gint,
                                                      const unsigned long long* __restrict__ sa,
                                                      const unsigned long long* __restrict__ sb, double* __restrict__ out) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= rows * cols) return;
  const int a = i / cols, b = i - a * cols;
  const Int192 g{{gint[i], gint[plane + i], gint[2 * plane + i]}};
  out[i] = real192(g, xg_unit(sa[a], NS) + xg_unit(sb[b], NS));
}

// Triangular factor RZ (ncap x ncap, row-major; R^T R = A^T A) of the source's columns.  sms: SMs this
// pass may take.  Dry runs take the workspace only; everything but RZ is released on return (later
// work on the stream may overwrite it).
// gram: R is the Gram matrix itself instead.
template <typename T, class Src>
tt_status xg_factor(cudaStream_t s, int num_sms, int sms, const Src& src, LivePattern lp, long nrows, Bump& ws,
                    double** RZ_out, int* status, int leaf_cat = kTsqrLeaf, bool gram = false) {
  using S = typename XgElem<Src>::type;
  constexpr int NS = sizeof(T) == 4 ? 4 : 8;
  constexpr int W = XgCfg<NS>::W, H = XgCfg<NS>::H;
  const int n = lp.ncap();
  const XgPlan* plan = xg_plan_of<NS>(src, lp);
  XgArray ar;
  const S* A = nullptr;
  if (!plan || !xg_array(src, n, nrows, ar, &A)) return TT_ERR_UNSUPPORTED;
  const XgPlan& pl = *plan;
  double* R = ws.take<double>((size_t)n * n);
  *RZ_out = R;
  const size_t mark = ws.off;
  XgArgs args{};
  int nbc = lp.nextra;
  const double* bc = nullptr;
  xg_geometry(src, args, &bc, &nbc);
  if (!bc) nbc = 0;
  args.po = ar.po;
  args.parts = ar.parts;
  args.nc = kXgStageOct / ar.po;
  args.npiece = ar.npiece;
  long groups;
  xg_groups(args.npiece, args.nc, pl.ncta, sms > 0 ? sms : num_sms, groups, args.ppg);
  constexpr bool direct = !XgElem<Src>::stencil;  // the raw columns are the columns
  const bool small = direct && nrows <= kXgSmallRows;
  const size_t zbytes = (size_t)8 * NS * W * 16;  // the largest piece of a column group
  // zeroed: column maxima and the page of zeros
  unsigned char* zeroed = ws.take<unsigned char>(zbytes + 8 * (size_t)(n + kMaxTerms));
  unsigned long long* slots = reinterpret_cast<unsigned long long*>(zeroed + zbytes);
  unsigned char* dig = ws.take<unsigned char>((size_t)ar.npiece * ar.po * ar.cpad * (NS * 16));
  unsigned char* bcdig = ws.take<unsigned char>((size_t)nbc * ar.parts * ar.po * (NS * 8 * 16));
  long long* part = ws.take<long long>((size_t)groups * pl.ncta * kXgTiles * (H * W * 128));
  unsigned long long* gint = ws.take<unsigned long long>(3 * (size_t)n * n);
  unsigned long long* raw = direct ? gint : ws.take<unsigned long long>(3 * (size_t)pl.nraw * pl.nraw);
  int* unit = ws.take<int>(n);
  double* coef = ws.take<double>(n);
  ws.release(mark);
  if (ws.dry) return TT_OK;
  {
    TimerScope scope(leaf_cat, s);
    if (small) {
      k_xg_small_digits<NS, S><<<(unsigned)((n + 7) / 8), 256, 0, s>>>(A, ar, lp, nrows, slots, dig,
                                                                       reinterpret_cast<uint4*>(zeroed), (int)(zbytes / 16));
      count_launch();
    } else {
      cudaMemsetAsync(zeroed, 0, zbytes + 8 * (size_t)(n + kMaxTerms), s);
      xg_launch_digits<NS>(s, num_sms, A, ar, xg_array_live(src, lp), nrows, slots, dig, bc, nbc, bcdig);
    }
    args.dig[0] = args.dig[1] = dig;
    args.bc = bcdig;
    args.zero = zeroed;
    const tt_status st =
        xg_launch_products<NS>(s, pl, args, groups, part, 0, pl.nraw, (size_t)pl.nraw * pl.nraw, raw, slots,
                               direct ? unit : nullptr, direct ? coef : nullptr, status);
    if (st != TT_OK) return st;
    if constexpr (!direct) {
      k_xg_combine<NS, Src><<<(unsigned)((n * n + 255) / 256), 256, 0, s>>>(src, n, pl.nraw, raw, slots, gint, unit, coef);
      count_launch();
    }
  }
  if (gram) {
    k_xg_real<NS><<<(unsigned)((n * n + 255) / 256), 256, 0, s>>>(n, gint, unit, coef, R);
    count_launch();
    return cudaGetLastError() == cudaSuccess ? TT_OK : TT_ERR_CUDA;
  }
  TimerScope scope(kTsqrMerge, s);
  return launch_xg_chol<(NS == 4 ? 1 : 2)>(s, n, gint, unit, coef, R);
}

// Products of the columns of two matrices over the same rows (explicit rows, FP64 digits).
template <typename S>
struct XgPair {
  const S *A, *B;
  int na, nb;
};
template <typename S>
struct XgElem<XgPair<S>> { using type = S; static constexpr bool stencil = false; };
constexpr int kXgPairCols = 256;  // columns of either matrix
template <int NS, typename S>
inline bool xg_make_plan(const XgPair<S>& s, const LivePattern&, XgPlan& pl) {
  pl.nsub = 0;
  pl.nraw = s.na + s.nb;
  return s.na <= kXgPairCols && s.nb <= kXgPairCols && xg_add<NS>(pl, s.na, 0, 0, 0) && xg_add<NS>(pl, s.nb, s.na, 1, 0) &&
         xg_tiles<NS>(pl, true) && xg_stages(pl) >= 2;
}
template <typename S>
inline long xg_plan_key(const XgPair<S>& s, const LivePattern&) { return ((long)s.na << 32) | (long)s.nb; }

// Whether the fixed point holds an inner product as well as FP64 sums do.  A column's rounding is 2^-62 of its
// largest entry, so a product of N rows is off by about 2^-62 sqrt(N) max|a| max|b|, an FP64 sum by 2^-53 of
// sum |a||b| or more: where the columns are large on different rows (sum |a||b| below 2^-9 sqrt(N) max|a| max|b|),
// the FP64 sums are the better ones.  sum |a||b| is bounded from below by one row of every `stride` (a hashed one: a
// fixed one would meet the same group in every cell): a CTA takes 16 x 16 pairs and 64 of these rows at a time, in
// units of the columns' powers of two; the sums are integers (2^-20), so that the decision does not depend on the
// order.  About 25 us of a product of 1,048,576 x 32 x 32 columns (0.74 ms in all; 0.72 ms without); with FP64
// conversions instead of integers and twice the rows 55 us.
constexpr long kXgCoverRows = 1L << 15;
__device__ __forceinline__ int xg_cover_exp(unsigned long long slot) { return (int)(slot >> 52); }
// |x| in units of 2^(ex - 1022), cut to FP32 (integers: the conversion runs on the FP64 pipe); ex: exponent field of
// the column's largest entry as FP64.
__device__ __forceinline__ float xg_cover_val(int e, unsigned m23, int ex) {
  const int f = min(e - ex + 126, 126);
  return e > 0 && f > 0 ? __uint_as_float(((unsigned)f << 23) | m23) : 0.0f;
}
__device__ __forceinline__ float xg_cover_abs(double x, int ex) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(x);
  return xg_cover_val((int)((b >> 52) & 0x7ffu), (unsigned)(b >> 29) & 0x7fffffu, ex);
}
__device__ __forceinline__ float xg_cover_abs(float x, int ex) {
  const unsigned b = __float_as_uint(x);
  return xg_cover_val((int)((b >> 23) & 0xffu), b & 0x7fffffu, ex - 896);
}
template <typename S>
__global__ void __launch_bounds__(256) k_xg_cover(const S* __restrict__ A, const S* __restrict__ B, int na, int nb,
                                                  long nrows, long stride, const unsigned long long* __restrict__ sa,
                                                  const unsigned long long* __restrict__ sb,
                                                  unsigned long long* __restrict__ cover) {
  __shared__ float va[64][17], vb[64][17];
  const int ta = (nb + 15) / 16, a0 = (int)blockIdx.y / ta * 16, b0 = (int)blockIdx.y % ta * 16;
  const int tid = threadIdx.x, ia = tid >> 4, ib = tid & 15;
  const long nsamp = (nrows + stride - 1) / stride;
  const bool la = a0 + ib < na, lb = b0 + ib < nb;
  const int fa = la ? xg_cover_exp(sa[a0 + ib]) : 0, fb = lb ? xg_cover_exp(sb[b0 + ib]) : 0;
  float sum = 0.0f;
  for (long m0 = (long)blockIdx.x * 64; m0 < nsamp; m0 += (long)gridDim.x * 64) {
    __syncthreads();
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int m = ia + 16 * u;
      const long k = (m0 + m) * stride + (long)((((unsigned)(m0 + m) * 2654435761u) >> 8) % (unsigned)stride);
      const bool in = m0 + m < nsamp && k < nrows;
      va[m][ib] = in && la ? xg_cover_abs(A[k * na + a0 + ib], fa) : 0.0f;
      vb[m][ib] = in && lb ? xg_cover_abs(B[k * nb + b0 + ib], fb) : 0.0f;
    }
    __syncthreads();
#pragma unroll 16
    for (int m = 0; m < 64; ++m) sum = fmaf(va[m][ia], vb[m][ib], sum);
  }
  if (a0 + ia < na && lb)
    atomicAdd(&cover[(size_t)(a0 + ia) * nb + b0 + ib], (unsigned long long)(sum * 1048576.0f));
}
// Sets *nonfinite for a pair that is not covered, or whose columns are so small that the storage's subnormal
// numbers (dropped from the fixed point) would count.
template <typename S>
__global__ void __launch_bounds__(256) k_xg_cover_check(int na, int nb, double least,
                                                        const unsigned long long* __restrict__ sa,
                                                        const unsigned long long* __restrict__ sb,
                                                        const unsigned long long* __restrict__ cover,
                                                        int* __restrict__ nonfinite) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= na * nb) return;
  const unsigned long long ma = sa[i / nb], mb = sb[i % nb];
  if (ma == 0ull || mb == 0ull) return;
  constexpr int kLow = sizeof(S) == 4 ? 1023 - 63 : 64;
  if (xg_cover_exp(ma) < kLow || xg_cover_exp(mb) < kLow || (double)cover[i] < least) *nonfinite = 1;
}

// Rows per pass of xg_cross: the workspace (256 MB of digits at 2 x 32 columns) does not grow with the rows;
// 65,536 rows a pass spent half of the time in k_xg_sum.
constexpr long kXgCrossRows = 1L << 18;
template <typename S>
inline bool xg_cross_same(const XgPair<S>& pr) { return pr.A == pr.B && pr.na == pr.nb; }
template <typename S>
inline const XgPlan* xg_cross_plan(const XgPair<S>& pr) {
  if (pr.na > kXgPairCols || pr.nb > kXgPairCols) return nullptr;
  // a matrix with itself: the upper triangle
  if (xg_cross_same(pr)) return xg_plan_of<8>(SrcRows<S>{pr.A, pr.na}, LivePattern{nullptr, pr.na, 1, 0});
  return xg_plan_of<8>(pr, LivePattern{nullptr, 1, 1, 0});
}
template <typename S>
inline bool xg_cross_fits(const XgPair<S>& pr) { return xg_cross_plan(pr) != nullptr; }

// W (na x nb, row-major) = A^T B of two row-major matrices, from exact products of their columns' fixed
// points; *nonfinite is set (or cleared) for an Inf or NaN and for columns that the fixed point does not hold as well
// as FP64 sums (k_xg_cover), and W is then to be formed otherwise: digits and products are left out (1,048,576 x 32 x
// 32 columns that are large on different rows: 3.06 ms with the sums, now 2.59).  An entry's
// error is its columns' rounding, 2^-62 of their largest entries: an FP64 sum rounds by 2^-53 of its
// terms, and ran at the rate of the FP64 pipe: three products of 1,048,576 x 32 x 32 columns 6.5 ms, now 2.2.
template <typename S>
tt_status xg_cross(cudaStream_t s, int num_sms, const XgPair<S>& pr, long nrows, Bump& ws, double* W, int* nonfinite,
                   int* status) {
  constexpr int NS = 8, H = XgCfg<NS>::H, Wd = XgCfg<NS>::W;
  const LivePattern la{nullptr, pr.na, 1, 0}, lb{nullptr, pr.nb, 1, 0};
  const XgPlan& pl = *xg_cross_plan(pr);
  const int nmat = xg_cross_same(pr) ? 1 : 2;
  const long rows = nrows < kXgCrossRows ? nrows : kXgCrossRows;
  XgArray aa, ab;
  const S* p = nullptr;
  if (!xg_array(SrcRows<S>{pr.A, pr.na}, pr.na, rows, aa, &p) || !xg_array(SrcRows<S>{pr.B, pr.nb}, pr.nb, rows, ab, &p))
    return TT_ERR_UNSUPPORTED;
  const size_t mark = ws.off;
  const int n = pr.na + pr.nb;
  const size_t zbytes = (size_t)8 * NS * Wd * 16, plane = (size_t)pr.na * pr.nb;
  unsigned char* zeroed = ws.take<unsigned char>(zbytes + 8 * (size_t)n);
  unsigned long long* slots = reinterpret_cast<unsigned long long*>(zeroed + zbytes);
  unsigned char* da = ws.take<unsigned char>((size_t)aa.npiece * aa.po * aa.cpad * (NS * 16));
  unsigned char* db = nmat == 1 ? da : ws.take<unsigned char>((size_t)ab.npiece * ab.po * ab.cpad * (NS * 16));
  unsigned long long* gint = ws.take<unsigned long long>(3 * plane);
  unsigned long long* cover = ws.take<unsigned long long>(plane);
  XgArgs args{};
  args.po = aa.po;
  args.parts = aa.parts;
  args.nc = kXgStageOct / aa.po;
  args.npiece = aa.npiece;
  long groups;
  xg_groups(args.npiece, args.nc, pl.ncta, num_sms, groups, args.ppg);
  long long* part = ws.take<long long>((size_t)groups * pl.ncta * kXgTiles * (H * Wd * 128));
  ws.release(mark);
  if (ws.dry) return TT_OK;
  cudaMemsetAsync(zeroed, 0, zbytes + 8 * (size_t)n, s);
  cudaMemsetAsync(nonfinite, 0, sizeof(int), s);
  for (int i = 0; i < nmat; ++i) {
    const XgArray& ar = i ? ab : aa;
    k_xg_colmax<S><<<xg_colmax_grid(num_sms, ar.ncol, nrows), 256, 0, s>>>(i ? pr.B : pr.A, ar.ncol, ar.sr, ar.sc, nrows,
                                                                           slots + (i ? pr.na : 0), nullptr, 0, ar.G,
                                                                           nonfinite);
    count_launch();
  }
  {
    const unsigned long long* sb = slots + (nmat == 1 ? 0 : pr.na);
    const long stride = nrows / kXgCoverRows | 1, need = (nrows / stride + 64) / 64;
    cudaMemsetAsync(cover, 0, 8 * plane, s);
    k_xg_cover<S><<<dim3((unsigned)(need < 2L * num_sms ? need : 2L * num_sms), (unsigned)((pr.na + 15) / 16 * ((pr.nb + 15) / 16))),
                    256, 0, s>>>(pr.A, pr.B, pr.na, pr.nb, nrows, stride, slots, sb, cover);
    count_launch();
    k_xg_cover_check<S><<<(unsigned)((plane + 255) / 256), 256, 0, s>>>(
        pr.na, pr.nb, 1048576.0 / 512.0 * sqrt((double)nrows), slots, sb, cover, nonfinite);
    count_launch();
  }
  args.dig[0] = da;
  args.dig[1] = db;
  args.bc = nullptr;
  args.zero = zeroed;
  args.skip = nonfinite;
  for (long r0 = 0; r0 < nrows; r0 += rows) {
    const long m = nrows - r0 < rows ? nrows - r0 : rows;
    for (int i = 0; i < nmat; ++i) {
      const XgArray& ar = i ? ab : aa;
      const long tot = ar.npiece * ar.po * ar.cpad;
      long grid = (tot + 255) / 256;
      if (grid > 16L * num_sms) grid = 16L * num_sms;
      // rows past m: zero digits
      k_xg_digits<NS, S><<<(unsigned)grid, 256, 0, s>>>((i ? pr.B : pr.A) + r0 * ar.sr, ar, i ? lb : la, m,
                                                        slots + (i ? pr.na : 0), i ? db : da, nullptr, 0, nullptr, nonfinite);
      count_launch();
    }
    const tt_status st = xg_launch_products<NS>(s, pl, args, groups, part, nmat == 1 ? 0 : pr.na, pr.nb, plane, gint, slots,
                                                nullptr, nullptr,
                                                status, r0 > 0);
    if (st != TT_OK) return st;
  }
  k_xg_real_cols<NS><<<(unsigned)((plane + 255) / 256), 256, 0, s>>>(pr.na, pr.nb, plane, gint, slots,
                                                                       slots + (nmat == 1 ? 0 : pr.na), W);
  count_launch();
  return cudaGetLastError() == cudaSuccess ? TT_OK : TT_ERR_CUDA;
}
}  // namespace ttk
