// FP64 GEMM emulated on the BF16 tensor cores (tcgen05), for the FP64 matrix products.
//
// GB300 executes FP64 at ~1 TFLOP/s (DMMA and DFMA alike) but BF16 at ~1.9 PFLOP/s, so an FP64
// product is formed from exact BF16 pieces (an error-free splitting in the manner of Ozaki, Ogita,
// Oishi and Rump):
//
//   row i of op(A) is scaled by 2^-(E_i+1), column j of op(B) by 2^-(F_j+1) (E, F: the smallest
//   exponents with |x| < 2^E over the row / column), so every scaled entry lies in (-1/2, 1/2);
//   X = x 2^(55-E) truncated to an integer (|X| < 2^55) is written in balanced radix 2^7,
//   X = sum_{p=1..8} a_p 2^(56-7p) with integer digits |a_p| <= 64 (integer arithmetic only), stored as
//   BF16, exactly.
//
//   A B = 2^(E_i+F_j+2) sum_{p,q} a_p b_q 2^-7(p+q); pairs with p + q >= 10 (each below 2^-58
//   of the scale) are dropped.  For d = p + q <= 7 the products of diagonal d are integers of
//   magnitude <= 2^12; summed over a K chunk of 512 with at most 6 pairs they stay below
//   2^24, so the FP32 tensor-memory accumulator holds them exactly.  After each chunk the six exact
//   sums are added, in units of 2^-49, to one 64-bit integer accumulator per output
//   (exact; integer operations are cheap on GB300 while FP64 additions are not).  The diagonals
//   d = 8, 9 have an FP32 accumulator each over all of K; its roundings stay near 2^-51 of the scale.
//
// Data flow: a split pass writes the 8 digit planes of op(A) and op(B) to global memory in the
// order the MMAs consume them (one 16-deep k-slice of a 128-row A tile = 8 planes x 4 KB,
// contiguous; of a 64-column B tile = 8 x 2 KB), so the GEMM kernel moves them with plain bulk
// asynchronous copies into a 4-stage shared-memory ring.  Warp roles: warp 16 issues the copies,
// warp 17 issues the MMAs (tcgen05, accumulators in TMEM: 8 diagonals of 64 columns, all of it), warps
// 0-15 (one TMEM lane per output row, a quarter of its 64 columns
// each) drain the exact accumulators at every chunk end and write C.  The kernel is persistent for
// short K, and its epilogue uses integer arithmetic only (see to_fp64).  8192^3 takes 24 ms (40 at first),
// 6144 x 6144 x 128 0.33 ms (1.16), back-transform 2 at n = 10240, k = 2560 137 ms (365).  Every mbarrier wait is bounded; on expiry the kernel records ST_TIMEOUT, waits (bounded) for
// its copies and MMAs in flight, frees TMEM and returns.
#include <cuda_bf16.h>

#include <algorithm>
#include <cmath>

#include "common.cuh"
#include "int_sums.cuh"
#include "tcgen05.cuh"

namespace gev {

namespace {

using namespace tc;

constexpr int OM = 128, ON = 64, KS = 16, NSTAGE = 4, NSLICE = 8, DMAX = 9, DEXACT = 7;
constexpr int CHUNK = 32;                  // k-slices per exact chunk (512 of K)
constexpr int KMAX = 32768;                // K per launch: the int64 sums stay below 2^63
constexpr int A_TILE = OM * KS * 2;        // one plane of a 128 x 16 slice: 4 KB
constexpr int B_TILE = ON * KS * 2;        // one plane of a 64 x 16 slice: 2 KB
constexpr int A_STAGE = NSLICE * A_TILE;   // 32 KB
constexpr int B_STAGE = NSLICE * B_TILE;   // 16 KB
constexpr int STAGE = A_STAGE + B_STAGE;   // 48 KB
constexpr int SMEM_OZ = NSTAGE * STAGE + 1024;
constexpr int NEPI_W = 16;                 // epilogue warps: TMEM lanes 32 (w % 4), columns 16 (w / 4)
constexpr int HC = ON / 4;                  // output columns per epilogue thread
constexpr int NTH = 32 * (NEPI_W + 2);      // + copy warp 16 + MMA warp 17
constexpr int TMEM_COLS_OZ = 512;          // diagonal d at columns (d - 2) ON
constexpr int GROUP_M = 16;                // raster: 16 row tiles share their B slices in L2
constexpr int EXP_BAD = 1 << 20;           // exponent marking a non-finite entry
constexpr int EXP_ZERO = -4000;            // exponent of an all-zero vector

// exponent e with |x| < 2^e for a finite x != 0; EXP_ZERO for 0, EXP_BAD for Inf / NaN
__device__ __forceinline__ int exp_above(double x) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(x);
  const int be = (int)((b >> 52) & 0x7FF);
  if (be == 0x7FF) return EXP_BAD;
  if (be == 0) return (b << 1) ? -1022 : EXP_ZERO;
  return be - 1022;
}


// One operand of a product as the exponent and split passes see it: vectors r (rows of op(A) or
// columns of op(B)) of elements k.  Real data: element (r, k) at X[r sr + k sk].  Complex data
// (double2 elements, strides in elements) enters through the real embedding of C = op(A) op(B):
//   cx 1 (A side): vector r = 2i + a, element k = 2l + b of the 2 x 2 block [[x, -y], [y, x]] of
//                  op(A)_il = x + iy;
//   cx 2 (B side): vector j, element k = 2l + c: x (c = 0) or y (c = 1) of op(B)_lj = x + iy;
// so that the real product of the two embedded operands is C with its real and imaginary parts in
// rows 2i and 2i + 1.  conj negates y (conjugate transposes).  The zero pattern (keep 1: l <= i,
// 2: l >= i; absolute l = local l + koff) refers to the complex indices.
struct Opnd {
  const void* X;
  long long sr, sk;
  int keep, cx, conj, koff;
};

__device__ __forceinline__ double opnd_at(const Opnd& o, long long r, long long k) {
  if (o.cx == 0) {
    if (!kept(o.keep, r, k + o.koff)) return 0.0;
    return static_cast<const double*>(o.X)[r * o.sr + k * o.sk];
  }
  const long long ri = (o.cx == 1) ? (r >> 1) : r, ki = k >> 1;
  if (!kept(o.keep, ri, ki + o.koff)) return 0.0;
  const double2 z = static_cast<const double2*>(o.X)[ri * o.sr + ki * o.sk];
  const double y = o.conj ? -z.y : z.y;
  if (o.cx == 2) return (k & 1) ? y : z.x;
  const long long a = r & 1, b = k & 1;
  return (a == b) ? z.x : (a == 0 ? -y : y);
}

// The two operands of one product, for the passes that handle both in one launch.
struct Opnd2 {
  Opnd o[2];
  int R[2];     // vectors: rows of op(A), columns of op(B)
  int fast[2];  // 1: consecutive vectors are adjacent in memory
  int* E[2];    // their exponents
  int TR[2];    // rows of a plane tile (OM, ON)
  int RT[2];    // row tiles
  unsigned char* out[2];
  int nblk0;    // grid blocks of operand 0 (the rest: operand 1)
};

// E[r] = max exponent over the kept entries of vector r, both operands in one launch; grid.y covers K
// in slabs.  Blocks of 256 threads take 32 vectors: a warp reads across 32 vectors (fast) or along one.
// One slab: E is written; several: atomicMax into a very negative initial value.
__global__ void __launch_bounds__(256) k_vec_exp(Opnd2 q, int K, int slab, int slabs) {
  const int w = blockIdx.x < q.nblk0 ? 0 : 1, blk = blockIdx.x - (w ? q.nblk0 : 0);
  const Opnd o = q.o[w];
  const int R = q.R[w], lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int k_lo = blockIdx.y * slab, k_hi = min(K, k_lo + slab);
  int* E = q.E[w];
  if (q.fast[w]) {
    __shared__ int red[8][32];
    const int r = blk * 32 + lane;
    int e = EXP_ZERO;
    if (r < R) {
#pragma unroll 8
      for (int k = k_lo + warp; k < k_hi; k += 8) e = max(e, exp_above(opnd_at(o, r, k)));
    }
    red[warp][lane] = e;
    __syncthreads();
    if (warp == 0 && r < R) {
#pragma unroll
      for (int u = 1; u < 8; ++u) e = max(e, red[u][lane]);
      if (slabs == 1) E[r] = e;
      else if (e != EXP_ZERO) atomicMax(&E[r], e);
    }
  } else {
#pragma unroll 1
    for (int u = 0; u < 4; ++u) {
      const int r = blk * 32 + warp * 4 + u;
      if (r >= R) return;  // uniform across the warp
      int e = EXP_ZERO;
#pragma unroll 8
      for (int k = k_lo + lane; k < k_hi; k += 32) e = max(e, exp_above(opnd_at(o, r, k)));
      e = __reduce_max_sync(0xffffffffu, e);
      if (lane == 0) {
        if (slabs == 1) E[r] = e;
        else if (e != EXP_ZERO) atomicMax(&E[r], e);
      }
    }
  }
}

__device__ __forceinline__ int clamp_exp(int e) { return e < -1100 ? EXP_ZERO : e; }

// the balanced radix-2^7 digits a_p of x 2^(55-E) (|x| < 2^E), as floats.  X + sum_p 2^6 2^(56-7p)
// has the digits a_p + 64 in its plain 7-bit fields (the top one may reach 128), so a digit is a shift, a
// mask that also sets the exponent of 1.5 2^23, and one exact subtraction: no carries, no integer conversion.
__device__ __forceinline__ void digits(double x, int E, float out[NSLICE]) {
  const unsigned long long bits = (unsigned long long)__double_as_longlong(x);
  const int be = (int)((bits >> 52) & 0x7FF);
  long long X = 0;
  if (E < EXP_BAD && (be != 0 || (bits << 1) != 0)) {
    unsigned long long m = bits & 0xFFFFFFFFFFFFFull;
    int ex;
    if (be == 0) { ex = -1022; } else { m |= (1ull << 52); ex = be - 1023; }
    const int s = ex + 3 - E;  // X = m 2^(ex - 52 + 55 - E); s <= 2 since |x| < 2^E
    unsigned long long u = 0;
    if (s >= 0) u = m << s;
    else if (s > -64) u = m >> (-s);  // bits below 2^-55 of the scale are dropped
    X = (bits >> 63) ? -(long long)u : (long long)u;
  }
  constexpr unsigned long long BIAS = (64ull << 49) | (64ull << 42) | (64ull << 35) | (64ull << 28) | (64ull << 21) |
                                      (64ull << 14) | (64ull << 7) | 64ull;
  const unsigned long long Y = (unsigned long long)(X + (long long)BIAS);  // >= 0
#pragma unroll
  for (int p = 1; p <= NSLICE; ++p) {
    const uint32_t f = (uint32_t)(Y >> (56 - 7 * p)) & (p == 1 ? 0xFFu : 0x7Fu);
    out[p - 1] = __int_as_float(0x4B400000 | f) - (12582912.0f + 64.0f);  // exact
  }
}

__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi) {
  const __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);  // exact: |a_p| <= 64
  return *reinterpret_cast<const uint32_t*>(&v);
}

// the digits of two neighbouring elements into the 8 planes (4 bytes each)
__device__ __forceinline__ void store_pair(double x0, double x1, int E, unsigned char* dst, int tile_bytes) {
  float a[NSLICE], b[NSLICE];
  digits(x0, E, a);
  digits(x1, E, b);
#pragma unroll
  for (int p = 0; p < NSLICE; ++p)
    *reinterpret_cast<uint32_t*>(dst + (long long)p * tile_bytes) = pack_bf16(a[p], b[p]);
}

// Digit planes of both operands in one launch.  A warp takes 8 vectors x 16 elements (one slice of one
// 8-row group): lane = 4 (row) + pair, so that every plane receives two contiguous 128-byte rows of core
// matrices and global memory is read in 64-byte runs whichever index is contiguous.
__device__ __forceinline__ void split_tile(const Opnd2& q, int w, long long u, int K, int KT) {
  const Opnd o = q.o[w];
  const int R = q.R[w], TR = q.TR[w], lane = threadIdx.x & 31;
  const long long RG = (long long)q.RT[w] * (TR / 8);
  if (u >= RG * KT) return;
  long long rg, kt;
  if (q.fast[w]) { rg = u % RG; kt = u / RG; } else { kt = u % KT; rg = u / KT; }
  const long long r = rg * 8 + (lane >> 2);
  const int Er = (r < R) ? (q.E[w] ? clamp_exp(q.E[w][r]) : 1) : EXP_ZERO;  // (no exponents: every entry below 2)
  double x[4];
#pragma unroll
  for (int h = 0; h < 4; ++h) {
    const long long k = kt * 16 + (h >> 1) * 8 + (lane & 3) * 2 + (h & 1);
    x[h] = (r < R && k < K) ? opnd_at(o, r, k) : 0.0;
  }
  const int tile_bytes = TR * KS * 2;
  unsigned char* base = q.out[w] + (((r / TR) * KT + kt) * NSLICE) * (long long)tile_bytes;
#pragma unroll
  for (int h = 0; h < 2; ++h)
    store_pair(x[2 * h], x[2 * h + 1], Er, base + toff16((int)(r % TR), h * 8 + (lane & 3) * 2), tile_bytes);
}
__global__ void __launch_bounds__(256) k_split(Opnd2 q, int K, int KT) {
  const int w = blockIdx.x < q.nblk0 ? 0 : 1;
  split_tile(q, w, (long long)(blockIdx.x - (w ? q.nblk0 : 0)) * 8 + (threadIdx.x >> 5), K, KT);
}

// The same for K <= 16 NS in one pass: the warp holds its 8 vectors entirely, so the exponents come out
// of the registers and no separate exponent pass (nor an initialised E) is needed.
template <int NS>
__global__ void __launch_bounds__(128) k_split_short(Opnd2 q, int K, int KT) {
  const int w = blockIdx.x < q.nblk0 ? 0 : 1;
  const long long blk = blockIdx.x - (w ? q.nblk0 : 0);
  const Opnd o = q.o[w];
  const int R = q.R[w], TR = q.TR[w], lane = threadIdx.x & 31;
  const long long rg = blk * 4 + (threadIdx.x >> 5);
  if (rg >= (long long)q.RT[w] * (TR / 8)) return;
  const long long r = rg * 8 + (lane >> 2);
  double x[NS * 4];
  int e = EXP_ZERO;
#pragma unroll
  for (int h = 0; h < NS * 4; ++h) {
    const long long k = (h >> 1) * 8 + (lane & 3) * 2 + (h & 1);
    x[h] = (r < R && k < K) ? opnd_at(o, r, k) : 0.0;
  }
#pragma unroll
  for (int h = 0; h < NS * 4; ++h) e = max(e, exp_above(x[h]));
  e = max(e, __shfl_xor_sync(0xffffffffu, e, 1));
  e = max(e, __shfl_xor_sync(0xffffffffu, e, 2));
  if ((lane & 3) == 0 && r < R) q.E[w][r] = e;
  const int Er = clamp_exp(e);
  const int tile_bytes = TR * KS * 2;
  unsigned char* base = q.out[w] + ((r / TR) * KT * NSLICE) * (long long)tile_bytes + toff16((int)(r % TR), (lane & 3) * 2);
#pragma unroll
  for (int h = 0; h < 2 * NS; ++h)
    if ((h >> 1) < KT)
      store_pair(x[2 * h], x[2 * h + 1], Er, base + (long long)(h >> 1) * NSLICE * tile_bytes + (h & 1) * 128, tile_bytes);
}

// K slices of a row tile of a block-diagonal op(A): the first slice of the tile's K range and the
// count (bm, bk multiples of 16 that divide / are multiples of the 128-row tile)
__host__ __device__ __forceinline__ void bd_range(int bm, int bk, int mt, int* first, int* count) {
  if (bm <= OM) {
    const int per = OM / bm;
    *first = mt * per * bk / KS;
    *count = per * bk / KS;
  } else {
    *first = (mt / (bm / OM)) * bk / KS;
    *count = bk / KS;
  }
}

// Entry (i, kk) (embedded units for complex data) of a block-diagonal back-transform-2 operand.
__device__ __forceinline__ double bd_at(const BdOp& o, long long i, long long kk) {
  const long long ir = o.cx ? (i >> 1) : i, kr = o.cx ? (kk >> 1) : kk;
  const int b = o.b;
  double x = 0.0, y = 0.0;
  if (o.kind == 1) {  // V_j^H: row q of block j, column r of the block's window
    const long long j = ir / b, q = ir % b, r = kr - 2LL * b * j;
    if (r < 0 || r >= 2 * b || j >= o.nblk) return 0.0;
    const long long g = o.g_lo + j, t = o.L - (o.ngroups - 1 - g), sw = g * b + q, rel = r - q;
    if (sw > o.n - 3 || rel < 0 || rel >= b || o.w00 + 2LL * b * j + r >= o.n) return 0.0;
    const long long rid = sw * o.ntask + t;
    if (o.cx) {
      const double2 tau = static_cast<const double2*>(o.tau2)[rid];
      if (tau.x == 0.0 && tau.y == 0.0) return 0.0;
      const double2 v = static_cast<const double2*>(o.V2)[rid * b + rel];
      x = v.x;
      y = -v.y;  // conjugate: op(A) = V^H
    } else {
      if (static_cast<const double*>(o.tau2)[rid] == 0.0) return 0.0;
      return static_cast<const double*>(o.V2)[rid * b + rel];
    }
  } else {  // W_j: row r of block j, column q
    const long long j = ir / (2 * b), r = ir % (2 * b), q = kr - (long long)b * j;
    if (q < 0 || q >= b || j >= o.nblk) return 0.0;
    const long long off = j * 2LL * b * b + r + q * 2LL * b;
    if (o.cx) {
      const double2 w = static_cast<const double2*>(o.W)[off];
      x = w.x;
      y = w.y;
    } else {
      return static_cast<const double*>(o.W)[off];
    }
  }
  const long long a = i & 1, c = kk & 1;  // the 2 x 2 block [[x, -y], [y, x]]
  return (a == c) ? x : (a == 0 ? -y : y);
}

// Row exponents and digit planes of a block-diagonal op(A) in the compact layout: row tile mt holds
// only the slices of its K range (bd_range).  One warp per row of the padded MT x 128 rows; lane l
// takes 8 consecutive columns of the range and writes 16 bytes to each plane.
__device__ __forceinline__ void split_bd_row(long long i, int M, const BdOp& o, int bm, int bk, int* E, unsigned char* out) {
  const int lane = threadIdx.x & 31;
  const int mt = (int)(i / OM);
  int f = 0, c = 0;
  bd_range(bm, bk, mt, &f, &c);
  const bool act = lane * 8 < c * KS;
  double v[8];
  int e = EXP_ZERO;
#pragma unroll
  for (int q = 0; q < 8; ++q) {
    const long long kk = (long long)f * KS + lane * 8 + q;
    v[q] = (act && i < M) ? bd_at(o, i, kk) : 0.0;
    e = max(e, exp_above(v[q]));
  }
  e = __reduce_max_sync(0xffffffffu, e);
  if (lane == 0) E[i] = e;
  if (!act) return;
  const int Er = clamp_exp(e);
  float dg[8][NSLICE];
#pragma unroll
  for (int q = 0; q < 8; ++q) digits(v[q], Er, dg[q]);
  const int tile_bytes = OM * KS * 2;
  unsigned char* base = out + (((long long)mt * c + (lane >> 1)) * NSLICE) * tile_bytes + toff16((int)(i % OM), (lane & 1) * 8);
#pragma unroll
  for (int p = 0; p < NSLICE; ++p) {
    *reinterpret_cast<uint4*>(base + (long long)p * tile_bytes) =
        make_uint4(pack_bf16(dg[0][p], dg[1][p]), pack_bf16(dg[2][p], dg[3][p]), pack_bf16(dg[4][p], dg[5][p]),
                   pack_bf16(dg[6][p], dg[7][p]));
  }
}

__global__ void __launch_bounds__(256) k_split_bd(int M, BdOp o, int bm, int bk, int MT, int* E, unsigned char* out) {
  const long long i = (blockIdx.x * 256ll + threadIdx.x) >> 5;
  if (i < (long long)MT * OM) split_bd_row(i, M, o, bm, bk, E, out);  // uniform per warp
}

// What the two products of a back-transform-2 level read, in one launch: the planes of both block-diagonal
// operands and of the level's rows of Y.
struct BdSide {
  BdOp o;
  int M, bm, bk, MT, nblk;  // nblk: grid blocks
  int* E;
  unsigned char* out;
};
__global__ void __launch_bounds__(256) k_level_prep(BdSide a1, BdSide a2, Opnd2 y, int K, int KT) {
  int blk = blockIdx.x;
  const int warp = threadIdx.x >> 5;
  if (blk < a1.nblk) {
    const long long i = blk * 8ll + warp;
    if (i < (long long)a1.MT * OM) split_bd_row(i, a1.M, a1.o, a1.bm, a1.bk, a1.E, a1.out);
    return;
  }
  blk -= a1.nblk;
  if (blk < a2.nblk) {
    const long long i = blk * 8ll + warp;
    if (i < (long long)a2.MT * OM) split_bd_row(i, a2.M, a2.o, a2.bm, a2.bk, a2.E, a2.out);
    return;
  }
  split_tile(y, 0, (blk - a2.nblk) * 8ll + warp, K, KT);
}

struct OzP {
  int M, N, K, koff, c_lower, tri_a, tri_b, cx;  // cx: complex product in the real embedding
  int MT, NT, KT, ksplit;
  double alpha, beta;
  double* C;
  long long ldc;
  double* ws;  // split-K partials (ksplit > 1): ws[z M N + i + j M]
  const unsigned char* Ap;
  const unsigned char* Bp;
  const int* E;
  const int* F;  // null: 1 for every column (entries below 2)
  int* status;
  // block-diagonal op(A) (0: off): block j has rows [j bd_bm, (j+1) bd_bm) and its non-zero columns
  // [j bd_bk, (j+1) bd_bk); the A planes then hold, per row tile, only that tile's K range (compact)
  int bd_bm, bd_bk;
  // alpha: 0 general, 1, -1; beta: 0, 1, 2 general (a comparison of doubles is an FP64 instruction)
  int amode, bmode;
};

int alpha_mode(double a) { return a == 1.0 ? 1 : (a == -1.0 ? -1 : 0); }
int beta_mode(double b) { return b == 0.0 ? 0 : (b == 1.0 ? 1 : 2); }

// One work item of the product kernel: an output tile (a share of its k-slices when K is split).
struct OzItem {
  int m0, n0, z, s_lo, nst, nt;
  long long a_tile;  // A-plane slice kt of the tile is slice a_tile + kt
  bool skip;         // nothing of the tile is wanted (c_lower)
};
__device__ __forceinline__ OzItem oz_item(const OzP& p, int it) {
  OzItem w;
  const int tiles = p.MT * p.NT;
  w.z = it / tiles;
  const int t = it % tiles;
  // grouped raster: GROUP_M row tiles sweep the column tiles together
  const int per_group = GROUP_M * p.NT;
  const int first = (t / per_group) * GROUP_M;
  const int gm = min(p.MT - first, GROUP_M);
  const int within = t % per_group;
  const int mt = first + within % gm;
  w.nt = within / gm;
  w.m0 = mt * OM;
  w.n0 = w.nt * ON;
  // complex products: rows 2i, 2i + 1 and elements 2l, 2l + 1 belong to complex row i / element l
  const int rs = p.cx ? 1 : 0;
  const long long mr0 = w.m0 >> rs, mrn = OM >> rs;
  w.skip = p.c_lower && w.n0 > mr0 + mrn - 1;
  // k-slices holding non-zero products for this tile (absolute k = local k + koff)
  long long kb = 0, ke = p.K >> rs;
  if (p.tri_a == 1) ke = std::min<long long>(ke, mr0 + mrn - p.koff);
  else if (p.tri_a == 2) kb = std::max<long long>(kb, mr0 - p.koff);
  if (p.tri_b == 1) kb = std::max<long long>(kb, (long long)w.n0 - p.koff);
  else if (p.tri_b == 2) ke = std::min<long long>(ke, (long long)w.n0 + ON - p.koff);
  kb <<= rs;
  ke <<= rs;
  int s_lo = (int)(kb / KS), s_hi = (int)(ke > 0 ? (ke + KS - 1) / KS : 0);
  if (s_hi < s_lo) s_hi = s_lo;
  w.a_tile = (long long)mt * p.KT;
  if (p.bd_bm) {
    int f = 0, c = 0;
    bd_range(p.bd_bm, p.bd_bk, mt, &f, &c);
    s_lo = min(f, p.KT);
    s_hi = min(f + c, p.KT);
    w.a_tile = (long long)mt * c - f;
  }
  if (p.ksplit > 1) {  // this item's share of the slices
    const int tot = s_hi - s_lo;
    const int a = s_lo + (int)((long long)tot * w.z / p.ksplit);
    const int b = s_lo + (int)((long long)tot * (w.z + 1) / p.ksplit);
    s_lo = a;
    s_hi = b;
  }
  w.s_lo = s_lo;
  w.nst = s_hi - s_lo;
  return w;
}

// Persistent: a CTA per SM walks over the work items.  The copy warp runs ahead into the next item's
// slices while the epilogue works, and the epilogue first drains all sums of an item into registers and
// releases the tensor memory, so the conversion to FP64, the loads of C and the stores overlap the next
// item's MMAs: an item costs max(MMAs + drain, epilogue) instead of their sum plus a launch and the first
// copies.  Sixteen epilogue warps of 16 columns: the conversion is a chain of integer instructions and
// needs warps in flight more than it needs registers (18 warps: at most 112 registers per thread).
__global__ void __launch_bounds__(NTH, 1) ozaki_kernel(OzP p) {
  extern __shared__ __align__(1024) unsigned char smem[];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int items = p.MT * p.NT * p.ksplit, rs = p.cx ? 1 : 0;

  unsigned char* ctrl = smem + NSTAGE * STAGE;
  uint64_t* full = reinterpret_cast<uint64_t*>(ctrl);  // [NSTAGE]: slice landed
  uint64_t* empty = full + NSTAGE;                      // [NSTAGE]: slice consumed by the MMAs
  uint64_t* cfull = empty + NSTAGE;                     // chunk accumulated
  uint64_t* cempty = cfull + 1;                         // chunk drained by the epilogue warps
  uint64_t* done = cempty + 1;                          // all MMAs complete
  uint32_t* tslot = reinterpret_cast<uint32_t*>(ctrl + 256);
  volatile int* err = reinterpret_cast<volatile int*>(ctrl + 320);
  int* issued = reinterpret_cast<int*>(ctrl + 384);
  int* consumed = reinterpret_cast<int*>(ctrl + 448);
  if (tid == 0) {
    for (int s = 0; s < NSTAGE; ++s) {
      mbar_init(su32(&full[s]), 1);
      mbar_init(su32(&empty[s]), 1);
    }
    mbar_init(su32(cfull), 1);
    mbar_init(su32(cempty), NEPI_W);
    mbar_init(su32(done), 1);
    asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
    *err = 0;
    *issued = 0;
    *consumed = 0;
  }
  if (warp == 0) tmem_alloc(su32(tslot), TMEM_COLS_OZ);
  fence_before();
  __syncthreads();
  fence_after();
  const uint32_t tmem = *tslot;

  if (warp == NEPI_W) {
    // ---- copy warp: digit-plane slices into the stage ring
    if (lane == 0) {
      int sg = 0;  // slices issued, over all items
      for (int it = blockIdx.x; it < items && !*err; it += gridDim.x) {
        const OzItem w = oz_item(p, it);
        if (w.skip) continue;
        const unsigned char* a_src = p.Ap + (w.a_tile + w.s_lo) * A_STAGE;
        const unsigned char* b_src = p.Bp + ((long long)w.nt * p.KT + w.s_lo) * B_STAGE;
        for (int s = 0; s < w.nst; ++s, ++sg) {
          const int slot = sg % NSTAGE;
          if (sg >= NSTAGE && !bar_wait(su32(&empty[slot]), ((sg / NSTAGE) - 1) & 1, err)) {
            if (!*err) *err = 411;
            break;
          }
          const uint32_t fb = su32(&full[slot]);
          mbar_expect_tx(fb, STAGE);
          const uint32_t dst = su32(smem + slot * STAGE);
          bulk_g2s(dst, a_src + (long long)s * A_STAGE, A_STAGE, fb);
          bulk_g2s(dst + A_STAGE, b_src + (long long)s * B_STAGE, B_STAGE, fb);
          *issued = sg + 1;
        }
      }
    }
  } else if (warp == NEPI_W + 1) {
    // ---- MMA warp: the 36 digit-pair products of a 16-deep slice in 13 MMAs of up to 256 columns (an MMA of
    // 64 columns took about 75 cycles for its 32 of tensor work, also with A kept in the collector buffer; 36 of
    // them per slice ran 8192^3 in 41.9 ms, these 13 in 24.0 ms, 0.87 of the BF16 peak)
    if (lane == 0) {
      int sg = 0, cg = 0;  // slices and chunks, over all items
      for (int it = blockIdx.x; it < items && !*err; it += gridDim.x) {
        const OzItem w = oz_item(p, it);
        if (w.skip) continue;
        for (int s = 0; s < w.nst; ++s, ++sg) {
          const int slot = sg % NSTAGE;
          const bool chunk_start = (s % CHUNK) == 0;
          if (chunk_start && cg > 0 && !bar_wait(su32(cempty), (cg - 1) & 1, err)) {
            if (!*err) *err = 412;
            break;
          }
          if (!bar_wait(su32(&full[slot]), (sg / NSTAGE) & 1, err)) {
            if (!*err) *err = 413;
            break;
          }
          *consumed = sg + 1;
          fence_after();
          const uint32_t a0 = su32(smem + slot * STAGE);
          const uint64_t ad = sdesc16(a0), bd = sdesc16(a0 + A_STAGE);
          // plane pa of A against planes qb .. qb + w - 1 of B in one MMA (64 w columns): the planes are
          // adjacent in shared memory and their diagonals d = pa + qb .. in tensor memory.  pa = 1 touches
          // every diagonal first: it restarts the exact ones (d <= 7) at a chunk start and the last two at
          // the item's start.
          auto mma = [&](int pa, int qb, int w, int en) {
            mma_bf16(tmem + (pa + qb - 2) * ON, ad + ((pa - 1) * A_TILE >> 4), bd + ((qb - 1) * B_TILE >> 4),
                     idesc_bf16(OM, w * ON), en);
          };
          const int en = chunk_start ? 0 : 1;
          mma(1, 1, 4, en);
          mma(1, 5, 2, en);
          mma(1, 7, 2, s > 0 ? 1 : 0);
          mma(2, 1, 4, 1);
          mma(2, 5, 3, 1);
          mma(3, 1, 3, 1);
          mma(3, 4, 3, 1);
          mma(4, 1, 3, 1);
          mma(4, 4, 2, 1);
          mma(5, 1, 4, 1);
          mma(6, 1, 3, 1);
          mma(7, 1, 2, 1);
          mma(8, 1, 1, 1);
          commit(su32(&empty[slot]));
          if ((s % CHUNK) == CHUNK - 1 || s == w.nst - 1) {
            commit(su32(cfull));
            ++cg;
          }
        }
      }
      commit(su32(done));
      if (!bar_wait_plain(su32(done), 0) && !*err) *err = 414;
    }
  } else {
    // ---- epilogue warps: drain the sums per chunk, then convert and write C
    const int quarter = warp & 3, col0 = (warp >> 2) * HC;
    const uint32_t lane_base = tmem + ((uint32_t)(quarter * 32) << 16) + (uint32_t)col0;
    const bool read_c = p.ksplit == 1 && p.bmode != 0;
    int cg = 0;
    for (int it = blockIdx.x; it < items; it += gridDim.x) {
      const OzItem w = oz_item(p, it);
      if (w.skip) continue;
      long long acc[HC];
      float sh[HC];
#pragma unroll
      for (int c = 0; c < HC; ++c) {
        acc[c] = 0;
        sh[c] = 0.f;
      }
      const int nchunk = (w.nst + CHUNK - 1) / CHUNK;
      bool good = true;
      for (int c = 0; c < nchunk; ++c, ++cg) {
        if (!bar_wait(su32(cfull), cg & 1, err)) {
          if (!*err) *err = 415;
          good = false;
          break;
        }
        fence_after();
        if (c == nchunk - 1) {
#pragma unroll
          for (int d = DEXACT + 1; d <= DMAX; ++d) {
            uint32_t r[16];
            tmem_ld16(lane_base + (uint32_t)((d - 2) * ON), r);
            tmem_wait_ld();
            const float sc = __int_as_float((127 - 7 * d) << 23);  // 2^-7d
#pragma unroll
            for (int q = 0; q < HC; ++q) sh[q] = fmaf(__uint_as_float(r[q]), sc, sh[q]);
          }
        }
        // the sums of diagonal d are integers below (d - 1) 512 2^12: two neighbouring diagonals make one 32-bit
        // integer (2^7 S_d + S_{d+1} < 2^31), and a wide multiply-add puts it in units of 2^-49
#pragma unroll
        for (int d = 2; d <= DEXACT; d += 2) {
          uint32_t r[16];
          int t[HC];
          tmem_ld16(lane_base + (uint32_t)((d - 2) * ON), r);
          tmem_wait_ld();
#pragma unroll
          for (int q = 0; q < HC; ++q) t[q] = __float2int_rn(__uint_as_float(r[q])) << 7;
          tmem_ld16(lane_base + (uint32_t)((d - 1) * ON), r);
          tmem_wait_ld();
#pragma unroll
          for (int q = 0; q < HC; ++q)
            acc[q] += (long long)(t[q] + __float2int_rn(__uint_as_float(r[q]))) * (1 << (49 - 7 * (d + 1)));
        }
        fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(su32(cempty));
      }
      if (!good) break;
      const int gi = w.m0 + quarter * 32 + lane;
      const bool any = nchunk > 0, row_ok = gi < p.M;
      const int Ei = (any && row_ok) ? p.E[gi] : EXP_ZERO;
      const int cmax = p.c_lower ? min(p.N, (gi >> rs) + 1) : p.N;  // columns [0, cmax) of this row are wanted
      double* crow = p.ksplit > 1 ? p.ws + (long long)w.z * p.M * p.N + gi : p.C + gi;
      const long long ld = p.ksplit > 1 ? p.M : p.ldc;
      // Every exponent of the warp's rows and columns in the middle of the range, alpha = +-1, beta = 0 or 1 (or
      // partial sums): the short conversion, with nothing else in its loop (one FP64 addition per output when C
      // is added; a choice among multiplications and additions is evaluated in full otherwise).
      {
        const int gq = w.n0 + col0 + (lane & (HC - 1));
        const int fl = (any && gq < p.N) ? (p.F ? p.F[gq] : 1) : 0;
        const bool mid = any && (!row_ok || (Ei > -400 && Ei < 400)) && fl > -400 && fl < 400;
        if (__all_sync(0xffffffffu, mid) && (p.ksplit > 1 || (p.amode != 0 && p.bmode != 2))) {
          const uint32_t flip = (p.ksplit == 1 && p.amode == -1) ? 0xFFFFFFFFu : 0u;
          const int nc = row_ok ? min(HC, cmax - (w.n0 + col0)) : 0;  // outputs of this thread
          double* cp = crow + (long long)(w.n0 + col0) * ld;
#pragma unroll
          for (int h = 0; h < HC; h += 8) {
            double cin[8];
#pragma unroll
            for (int u = 0; u < 8; ++u) cin[u] = (read_c && h + u < nc) ? cp[(h + u) * ld] : 0.0;
#pragma unroll
            for (int u = 0; u < 8; ++u) {
              const int fj = __shfl_sync(0xffffffffu, fl, h + u);
              double v = to_fp64_fast(acc[h + u], sh[h + u], Ei + fj + 2, flip);
              if (read_c) v += cin[u];
              if (h + u < nc) cp[(h + u) * ld] = v;
            }
          }
          continue;
        }
      }
      if (row_ok) {
#pragma unroll
        for (int h = 0; h < HC; h += 4) {
          // the loads of 4 outputs (column exponents, C) first, so that they overlap
          double cin[4];
          int fj[4];
#pragma unroll
          for (int u = 0; u < 4; ++u) {
            const int gj = w.n0 + col0 + h + u;
            fj[u] = (any && gj < cmax) ? (p.F ? p.F[gj] : 1) : EXP_ZERO;
            cin[u] = (read_c && gj < cmax) ? crow[gj * ld] : 0.0;
          }
#pragma unroll
          for (int u = 0; u < 4; ++u) {
            const int gj = w.n0 + col0 + h + u;
            if (gj >= cmax) continue;
            double v = 0.0;
            if (Ei >= -1100 && fj[u] >= -1100) v = to_fp64(acc[h + u], sh[h + u], Ei + fj[u] + 2);
            // an Inf / NaN entry reached this output
            if (any && (Ei >= EXP_BAD || fj[u] >= EXP_BAD)) v = __longlong_as_double(0x7FF8000000000000ll);
            if (p.ksplit == 1) {
              // (a sign bit: negation is an FP64 instruction here)
              if (p.amode == -1) v = __longlong_as_double(__double_as_longlong(v) ^ (long long)(1ull << 63));
              else if (p.amode == 0) v = p.alpha * v;
              if (p.bmode == 1) v += cin[u];
              else if (p.bmode == 2) v = fma(p.beta, cin[u], v);
            }
            crow[gj * ld] = v;
          }
        }
      }
    }
  }
  __syncthreads();
  if (tid == 0 && *err) {
    // a wait gave up: let the copies already issued land before the shared memory is released
    for (int s = *consumed; s < *issued; ++s) bar_wait_plain(su32(&full[s % NSTAGE]), (s / NSTAGE) & 1);
    atomicCAS(&p.status[ST_TIMEOUT], 0, *err);
  }
  fence_before();
  __syncthreads();
  if (warp == 0) tmem_dealloc(tmem, TMEM_COLS_OZ);
}

// C = alpha sum_z ws[z] + beta C in a fixed order (deterministic)
// (rs = 1: complex product in the real embedding, rows 2i, 2i + 1 belong to complex row i)
__global__ void k_oz_reduce(int M, int N, int ks, int c_lower, int rs, double alpha, const double* ws, double beta,
                            double* C, long long ldc) {
  const long long total = (long long)M * N;
  for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < total;
       t += (long long)gridDim.x * blockDim.x) {
    const int i = (int)(t % M), j = (int)(t / M);
    if (c_lower && (i >> rs) < j) continue;
    double s = 0.0;
    for (int z = 0; z < ks; ++z) s += ws[(long long)z * total + t];
    double* c = &C[i + (long long)j * ldc];
    const double o = alpha * s;
    *c = (beta != 0.0) ? o + beta * (*c) : o;
  }
}

size_t rup(size_t x, size_t a) { return (x + a - 1) / a * a; }

struct OzLayout {
  size_t Mp, Np, Kp, f_off, a_off, b_off, total;
};

OzLayout oz_layout(int M, int N, int K) {
  OzLayout L;
  L.Mp = rup(std::max(M, 1), OM);
  L.Np = rup(std::max(N, 1), ON);
  L.Kp = rup(std::max(std::min(K, KMAX), 1), KS);
  L.f_off = rup(L.Mp * sizeof(int), 256);
  L.a_off = L.f_off + rup(L.Np * sizeof(int), 256);
  L.b_off = L.a_off + L.Mp * L.Kp * 2 * NSLICE;
  L.total = L.b_off + L.Np * L.Kp * 2 * NSLICE;
  return L;
}

}  // namespace

size_t gemm_f64_emulated_scratch(int M, int N, int K) { return oz_layout(M, N, K).total; }

namespace {

// K range of an exponent block: short enough for about six blocks per SM (a block is a chain of loads: with one
// block per 32 vectors the pass over a 1500 x 32 operand took 40 us), at most 512, at least 64
int exp_slab(const Sys& s, int nblk, int K) {
  const int want = (int)cdiv(6 * s.sms, nblk);
  return std::min(512, std::max(64, (int)(cdiv(cdiv(K, want), 64) * 64)));
}

// Exponents and digit planes of both operands.  K <= 128 (the thin products of the panels): one launch
// that holds whole vectors in registers; else an exponent pass and a split pass, each over both operands.
// (For a 1500 x 32 x 32 product the former two exponent and two split launches with their two memsets
// took about 36 us.)
void split_both(Sys& s, int M, int N, int K, const Opnd& a, const Opnd& b, int fast_a, int fast_b, int* E, int* F,
                unsigned char* Ap, unsigned char* Bp, int MT, int NT, int KT) {
  Opnd2 q{};
  q.o[0] = a; q.o[1] = b;
  q.R[0] = M; q.R[1] = N;
  q.fast[0] = fast_a; q.fast[1] = fast_b;
  q.E[0] = E; q.E[1] = F;
  q.TR[0] = OM; q.TR[1] = ON;
  q.RT[0] = MT; q.RT[1] = NT;
  q.out[0] = Ap; q.out[1] = Bp;
  const long long ga = (long long)MT * (OM / 8), gb = (long long)NT * (ON / 8);  // 8-row groups
  if (K <= 128) {
    q.nblk0 = (int)cdiv(ga, 4);
    const unsigned nb = q.nblk0 + cdiv(gb, 4);
    GEV_COUNT(s);
    if (K <= 64) k_split_short<4><<<nb, 128, 0, s.stream>>>(q, K, KT);
    else k_split_short<8><<<nb, 128, 0, s.stream>>>(q, K, KT);
    return;
  }
  q.nblk0 = (int)cdiv(M, 32);
  const int nblk = q.nblk0 + (int)cdiv(N, 32), slab = exp_slab(s, nblk, K), slabs = (int)cdiv(K, slab);
  if (slabs > 1) cudaMemsetAsync(E, 0x80, (size_t)((unsigned char*)(F + NT * ON) - (unsigned char*)E), s.stream);
  GEV_COUNT(s);
  k_vec_exp<<<dim3(nblk, slabs), 256, 0, s.stream>>>(q, K, slab, slabs);
  q.nblk0 = (int)cdiv(ga * KT, 8);
  GEV_COUNT(s);
  k_split<<<q.nblk0 + cdiv(gb * KT, 8), 256, 0, s.stream>>>(q, K, KT);
}

// C (M x N, real, ldc) = alpha op(A) op(B) + beta C with op(A) = the M x K operand a and op(B) the
// N x K operand b (vectors = columns of op(B)), K in the operands' element units (embedded for
// complex data); ka / kb: bytes of one underlying element step along K of a / b, to offset the
// K pieces of one launch; rs = 1 for complex products.
void emulate(Sys& s, int M, int N, int K, Opnd a, size_t a_kstep, Opnd b, size_t b_kstep, int tri_a, int tri_b,
             int c_lower, int rs, double alpha, double beta, double* C, long long ldc) {
  const OzLayout L = oz_layout(M, N, K);
  int site = 0;
  if (s.ozws == nullptr || L.total > s.ozws_bytes) {  // internal sizing error: fail the call loudly
    fprintf(stderr, "gev: emulated FP64 GEMM scratch too small (%zu < %zu bytes)\n", s.ozws_bytes, L.total);
    site = 499;
  } else if (allow_dyn_smem(ozaki_kernel, SMEM_OZ) != 0) {
    site = 498;
  }
  if (site) {  // recorded in the status words: the caller's next status check returns GEV_ERR_CUDA
    if (s.status) cudaMemcpyAsync(s.status + ST_CONFIG, &site, sizeof(int), cudaMemcpyHostToDevice, s.stream);
    cudaStreamSynchronize(s.stream);
    return;
  }
  unsigned char* base = static_cast<unsigned char*>(s.ozws);
  int* E = reinterpret_cast<int*>(base);
  int* F = reinterpret_cast<int*>(base + L.f_off);
  unsigned char* Ap = base + L.a_off;
  unsigned char* Bp = base + L.b_off;
  const int fast_a = a.sr == 1, fast_b = b.sr == 1;
  const int MT = (int)(L.Mp / OM), NT = (int)(L.Np / ON);
  for (int k0 = 0; k0 < std::max(K, 1); k0 += KMAX) {  // K pieces (k0 even: whole complex elements)
    const int Kc = std::max(0, std::min(KMAX, K - k0));
    const int KT = (Kc + KS - 1) / KS;
    const int ku = k0 >> rs;  // the piece's first underlying element along K
    Opnd ap = a, bp = b;
    ap.X = static_cast<const unsigned char*>(a.X) + (size_t)ku * a_kstep;
    bp.X = static_cast<const unsigned char*>(b.X) + (size_t)ku * b_kstep;
    ap.koff = bp.koff = ku;
    if (Kc > 0) split_both(s, M, N, Kc, ap, bp, fast_a, fast_b, E, F, Ap, Bp, MT, NT, KT);
    OzP p{};
    p.M = M; p.N = N; p.K = Kc; p.koff = ku; p.c_lower = c_lower;
    p.tri_a = tri_a; p.tri_b = tri_b; p.cx = rs;
    p.MT = MT; p.NT = NT; p.KT = KT;
    p.alpha = alpha; p.beta = (k0 == 0) ? beta : 1.0;
    p.C = C; p.ldc = ldc; p.Ap = Ap; p.Bp = Bp; p.E = E; p.F = F; p.status = s.status;
    // split K when the output has too few tiles to fill the GPU in whole rounds; a share is at least 8 slices.  The cost
    // in slices (0.6 us): rounds of items, each with its first copies, drain and epilogue, and the pass that sums the
    // shares (launch, and their bytes at 5 TB/s).
    long long tiles = (long long)MT * NT;
    if (c_lower) tiles = (tiles + MT) / 2;
    int ks = 1;
    if (tiles < 2 * s.sms && KT >= 16) {
      const double item = 14.0, sum0 = 8.0, sum1 = (double)M * N * sizeof(double) / 3e6;
      double best = cdiv(tiles, s.sms) * (KT + item);
      for (int c = 2; c <= std::min(64, KT / 8); ++c) {
        if ((size_t)c * M * N * sizeof(double) > s.splitws_bytes) break;
        const double cost = cdiv(tiles * c, s.sms) * ((double)KT / c + item) + sum0 + sum1 * c;
        if (cost < 0.97 * best) {
          best = cost;
          ks = c;
        }
      }
    }
    p.ksplit = ks;
    p.ws = ks > 1 ? static_cast<double*>(s.splitws) : nullptr;
    p.amode = alpha_mode(p.alpha);
    p.bmode = beta_mode(p.beta);
    // long items: one CTA each, scheduled by the hardware as SMs come free (triangular tiles differ in
    // length, and the epilogue is a small part); short ones: persistent CTAs (8192^3 and the triangular
    // products of n = 10240 ran 8 - 15 % slower persistent, 8192 x 8192 x 128 1.9 times faster)
    const long long work = (long long)MT * NT * ks;
    GEV_COUNT(s);
    ozaki_kernel<<<KT >= 48 * ks ? work : std::min<long long>(work, s.sms), NTH, SMEM_OZ, s.stream>>>(p);
    if (ks > 1) {
      const long long total = (long long)M * N;
      unsigned blocks = cdiv(total, 256);
      if (blocks > 8u * s.sms) blocks = 8u * s.sms;
      GEV_COUNT(s);
      k_oz_reduce<<<blocks, 256, 0, s.stream>>>(M, N, ks, c_lower, rs, p.alpha, p.ws, p.beta, C, ldc);
    }
  }
}

int keep_a_of(int tri_a) { return tri_a == 1 ? 1 : (tri_a == 2 ? 2 : 0); }
int keep_b_of(int tri_b) { return tri_b == 1 ? 2 : (tri_b == 2 ? 1 : 0); }

}  // namespace

// FP64 GEMM on the tensor cores (real data); scratch s.ozws of s.ozws_bytes >= gemm_f64_emulated_scratch.
// Zero patterns: op(A)[i,k] = 0 for k > i (tri_a 1) or k < i (tri_a 2); op(B)[k,j] = 0 for k < j
// (tri_b 1) or k > j (tri_b 2).
void gemm_f64_emulated(Sys& s, const GemmP<double>& q) {
  if (q.M <= 0 || q.N <= 0) return;
  // op(A) row i, element k: A[i + k lda] (ta 0) or A[k + i lda]; op(B) column j, element k:
  // B[k + j ldb] (tb 0) or B[j + k ldb]
  Opnd a{q.A, q.ta ? q.lda : 1, q.ta ? 1 : q.lda, keep_a_of(q.tri_a), 0, 0, 0};
  Opnd b{q.B, q.tb ? 1 : q.ldb, q.tb ? q.ldb : 1, keep_b_of(q.tri_b), 0, 0, 0};
  emulate(s, q.M, q.N, q.K, a, sizeof(double) * (size_t)a.sk, b, sizeof(double) * (size_t)b.sk, q.tri_a, q.tri_b,
          q.c_lower, 0, q.alpha, q.beta, q.C, q.ldc);
}

// Complex FP64 GEMM on the tensor cores through the real embedding (2M x 2K) (2K x N): the
// result's real and imaginary parts are rows 2i and 2i + 1 of the real view of C (leading
// dimension 2 ldc).  alpha and beta must be real (the caller checks).  ta / tb 2: conjugate
// transposes.
void gemm_c128_emulated(Sys& s, const GemmP<zd>& q) {
  if (q.M <= 0 || q.N <= 0) return;
  Opnd a{q.A, q.ta ? q.lda : 1, q.ta ? 1 : q.lda, keep_a_of(q.tri_a), 1, q.ta == 2 ? 1 : 0, 0};
  Opnd b{q.B, q.tb ? 1 : q.ldb, q.tb ? q.ldb : 1, keep_b_of(q.tri_b), 2, q.tb == 2 ? 1 : 0, 0};
  emulate(s, 2 * q.M, q.N, 2 * q.K, a, sizeof(zd) * (size_t)a.sk, b, sizeof(zd) * (size_t)b.sk, q.tri_a, q.tri_b,
          q.c_lower, 1, q.alpha.x, q.beta.x, reinterpret_cast<double*>(q.C), 2 * q.ldc);
}

namespace {

struct BdLayout {
  size_t Mp, Np, f_off, a_off, b_off, total;
  int MT, NT, KT, acount;
};

// scratch of a block-diagonal product (embedded units): row exponents, column exponents, the compact
// A planes (acount slices per row tile) and the B planes over the whole K (no piece limit: a tile
// sums at most 16 slices, far below the int64 accumulator's range)
BdLayout bd_layout(int Me, int N, int Ke, int bme, int bke) {
  BdLayout L;
  L.Mp = rup(std::max(Me, 1), OM);
  L.Np = rup(std::max(N, 1), ON);
  L.MT = (int)(L.Mp / OM);
  L.NT = (int)(L.Np / ON);
  L.KT = (std::max(Ke, 1) + KS - 1) / KS;
  int f = 0;
  bd_range(bme, bke, 0, &f, &L.acount);
  L.f_off = rup(L.Mp * sizeof(int), 256);
  L.a_off = L.f_off + rup(L.Np * sizeof(int), 256);
  L.b_off = L.a_off + (size_t)L.MT * L.acount * A_STAGE;
  L.total = L.b_off + (size_t)L.NT * L.KT * B_STAGE;
  return L;
}

// the product launch of a block-diagonal product (embedded units; blocks bme x bke)
void launch_bdiag(Sys& s, const BdLayout& L, int Me, int N, int Ke, int rs, int bme, int bke, const int* E, const int* F,
                  const unsigned char* Ap, const unsigned char* Bp, double alpha, double beta, void* C, long long ldc) {
  OzP p{};
  p.M = Me; p.N = N; p.K = Ke; p.koff = 0; p.c_lower = 0;
  p.tri_a = 0; p.tri_b = 0; p.cx = rs;
  p.MT = L.MT; p.NT = L.NT; p.KT = L.KT; p.ksplit = 1;
  p.alpha = alpha; p.beta = beta;
  p.C = static_cast<double*>(C);
  p.ldc = ldc << rs;
  p.ws = nullptr;
  p.Ap = Ap; p.Bp = Bp; p.E = E; p.F = F; p.status = s.status;
  p.bd_bm = bme;
  p.bd_bk = bke;
  p.amode = alpha_mode(alpha);
  p.bmode = beta_mode(beta);
  GEV_COUNT(s);
  ozaki_kernel<<<std::min<long long>((long long)L.MT * L.NT, s.sms), NTH, SMEM_OZ, s.stream>>>(p);
}

}  // namespace

size_t gemm_f64_bdiag_scratch(int M, int N, int K, int bm, int bk, int cx) {
  const int e = cx ? 2 : 1;
  return bd_layout(e * M, N, e * K, e * bm, e * bk).total;
}

bool gemm_f64_bdiag(Sys& s, int M, int N, int K, const BdOp& a, int bm, int bk, const void* B, long long ldb,
                    double alpha, double beta, void* C, long long ldc, bool b_below_two) {
  if (M <= 0 || N <= 0) return true;
  const int rs = a.cx ? 1 : 0;
  const int Me = M << rs, Ke = K << rs, bme = bm << rs, bke = bk << rs;
  const BdLayout L = bd_layout(Me, N, Ke, bme, bke);
  if (!s.ozws || L.total > s.ozws_bytes) return false;
  if (allow_dyn_smem(ozaki_kernel, SMEM_OZ) != 0) return false;
  unsigned char* base = static_cast<unsigned char*>(s.ozws);
  int* E = reinterpret_cast<int*>(base);
  int* F = reinterpret_cast<int*>(base + L.f_off);
  unsigned char* Ap = base + L.a_off;
  unsigned char* Bp = base + L.b_off;
  // op(B) column j, element k: B[k + j ldb] (complex: the re / im parts of element k / 2)
  const Opnd b{B, ldb, 1, 0, a.cx ? 2 : 0, 0, 0};
  GEV_COUNT(s);
  k_split_bd<<<cdiv((long long)L.MT * OM * 32, 256), 256, 0, s.stream>>>(Me, a, bme, bke, L.MT, E, Ap);
  Opnd2 q{};
  q.o[0] = b;
  q.R[0] = N;
  q.E[0] = b_below_two ? nullptr : F;  // every entry of B below 2 in magnitude: exponent 1, no pass over B
  q.TR[0] = ON;
  q.RT[0] = L.NT;
  q.out[0] = Bp;
  if (!b_below_two && Ke > 0) {
    q.nblk0 = (int)cdiv(N, 32);
    const int slab = exp_slab(s, q.nblk0, Ke), slabs = (int)cdiv(Ke, slab);
    if (slabs > 1) cudaMemsetAsync(F, 0x80, L.Np * sizeof(int), s.stream);
    GEV_COUNT(s);
    k_vec_exp<<<dim3(q.nblk0, slabs), 256, 0, s.stream>>>(q, Ke, slab, slabs);
  }
  if (Ke > 0) {
    q.nblk0 = (int)cdiv((long long)L.NT * (ON / 8) * L.KT, 8);
    GEV_COUNT(s);
    k_split<<<q.nblk0, 256, 0, s.stream>>>(q, Ke, L.KT);
  }
  launch_bdiag(s, L, Me, N, Ke, rs, bme, bke, E, q.E[0], Ap, Bp, alpha, beta, C, ldc);
  return true;
}

// One level of back-transform 2 on columns whose entries stay below 2 in magnitude:
//   P (M1 x N) = op(A1) Y,  Y -= op(A2) P,   Y: rows x N, blocks b x 2b of A1 and 2b x b of A2 (complex units).
// Four launches: the planes of A1, A2 and Y, the first product, the planes of P, the second product.  (Two exponent
// fills, two launches for the A sides and two for the B sides before: 137 us a level at n = 4096, b = 32, k = 1229.)
// False, with nothing launched, when s.ozws is too small.
bool gemm_f64_bdiag_level(Sys& s, int M1, int rows, int N, const BdOp& a1, const BdOp& a2, int b, void* Y, long long ldy,
                          void* P, long long ldp) {
  if (M1 <= 0 || rows <= 0 || N <= 0) return true;
  const int rs = a1.cx ? 1 : 0, be = b << rs;
  const int Me = M1 << rs, Re = rows << rs;
  const BdLayout L1 = bd_layout(Me, N, Re, be, 2 * be), L2 = bd_layout(Re, N, Me, 2 * be, be);
  const size_t e2 = rup(L1.Mp * sizeof(int), 256), p1 = e2 + rup(L2.Mp * sizeof(int), 256);
  const size_t p2 = p1 + (size_t)L1.MT * L1.acount * A_STAGE, bp = p2 + (size_t)L2.MT * L2.acount * A_STAGE;
  if (!s.ozws || bp + (size_t)L1.NT * std::max(L1.KT, L2.KT) * B_STAGE > s.ozws_bytes) return false;
  if (allow_dyn_smem(ozaki_kernel, SMEM_OZ) != 0) return false;
  unsigned char* base = static_cast<unsigned char*>(s.ozws);
  int* E1 = reinterpret_cast<int*>(base);
  int* E2 = reinterpret_cast<int*>(base + e2);
  unsigned char* Bp = base + bp;
  const BdSide s1{a1, Me, be, 2 * be, L1.MT, (int)cdiv((long long)L1.MT * OM, 8), E1, base + p1};
  const BdSide s2{a2, Re, 2 * be, be, L2.MT, (int)cdiv((long long)L2.MT * OM, 8), E2, base + p2};
  Opnd2 q{};
  q.o[0] = Opnd{Y, ldy, 1, 0, a1.cx ? 2 : 0, 0, 0};  // column j, element k
  q.R[0] = N;
  q.TR[0] = ON;
  q.RT[0] = L1.NT;
  q.out[0] = Bp;
  GEV_COUNT(s);
  k_level_prep<<<s1.nblk + s2.nblk + cdiv((long long)L1.NT * (ON / 8) * L1.KT, 8), 256, 0, s.stream>>>(s1, s2, q, Re, L1.KT);
  launch_bdiag(s, L1, Me, N, Re, rs, be, 2 * be, E1, nullptr, base + p1, Bp, 1.0, 0.0, P, ldp);
  q.o[0].X = P;
  q.o[0].sr = ldp;
  q.nblk0 = (int)cdiv((long long)L2.NT * (ON / 8) * L2.KT, 8);
  GEV_COUNT(s);
  k_split<<<q.nblk0, 256, 0, s.stream>>>(q, Me, L2.KT);
  launch_bdiag(s, L2, Re, N, Me, rs, 2 * be, be, E2, nullptr, base + p2, Bp, -1.0, 1.0, Y, ldy);
  return true;
}

}  // namespace gev

extern "C" size_t gev_gemm_f64_scratch_bytes(int M, int N, int K) {
  if (M < 0 || N < 0 || K < 0) return 0;
  return ((gev::gemm_f64_emulated_scratch(M, N, K) + 255) & ~(size_t)255) + ((size_t)16 << 20);
}

extern "C" int gev_gemm_f64(int M, int N, int K, int ta, int tb, double alpha, const double* A, int lda,
                            const double* B, int ldb, double beta, double* C, int ldc, int engine, void* stream,
                            int* status_dev, void* scratch_dev, size_t scratch_bytes) {
  using namespace gev;
  if (M < 0) return -1;
  if (N < 0) return -2;
  if (K < 0) return -3;
  if (ta < 0 || ta > 1) return -4;
  if (tb < 0 || tb > 1) return -5;
  if (!A && M > 0 && K > 0) return -7;
  if (lda < std::max(1, ta ? K : M)) return -8;
  if (!B && K > 0 && N > 0) return -9;
  if (ldb < std::max(1, tb ? N : K)) return -10;
  if (!C && M > 0 && N > 0) return -12;
  if (ldc < std::max(1, M)) return -13;
  if (engine < 0 || engine > 1) return -14;
  if (!status_dev) return -16;
  if (engine == 1 && (!scratch_dev || scratch_bytes < gev_gemm_f64_scratch_bytes(M, N, K))) return -17;
  Sys s;
  s.stream = (cudaStream_t)stream;
  int dev = 0, sms = 0;
  GEV_CUDA_TRY(cudaGetDevice(&dev));
  GEV_CUDA_TRY(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
  s.sms = sms > 0 ? sms : 152;
  s.status = status_dev;
  s.emu_fp64 = engine;
  if (engine == 1) {  // planes first, then the split-K partials
    const size_t planes = (gemm_f64_emulated_scratch(M, N, K) + 255) & ~(size_t)255;
    s.ozws = scratch_dev;
    s.ozws_bytes = planes;
    s.splitws = static_cast<unsigned char*>(scratch_dev) + planes;
    s.splitws_bytes = scratch_bytes - planes;
  } else {
    s.splitws = nullptr;
    s.splitws_bytes = 0;
  }
  gemm<double>(s, gp<double>(M, N, K, ta, tb, alpha, A, lda, B, ldb, beta, C, ldc));
  GEV_TRY(last_error());
  GEV_CUDA_TRY(cudaStreamSynchronize(s.stream));
  return 0;
}
