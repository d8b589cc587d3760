// Float64 path: the m x n passes and the thin (m x r, n x r) kernels, with every inner product in
// fixed point on the integer units (fix64.cuh).  A float64 FMA loop over the same products ran at
// GB300's 1.2 TFLOP/s: at 4096 x 4096, r = 64 the sweep took 3.95 ms, the W pass 2.4 ms and the thin
// kernels 0.8 ms of a 7.3 ms iteration; now 1.21, 0.66 and 0.24 of 2.35 ms.  Element-wise float64 arithmetic (about eight
// operations per element of M) stays on the float64 units and bounds the sweep at small r: ncu, 4096 x 4096, float64
// pipe 64 % and wide-multiply pipe 33 % active at r = 10, 36 % and 66 % at r = 64 (W pass 19 % and 68 %).
//
// Exponents (fix64.cuh): the thin kernels and the sweep convert their operands themselves, each row of P, U, C and W
// and each column of an r x r factor or of a Gram operand with its own exponent; Delta is held in float64, and has
// one exponent per row and 64-column tile in Q = Delta V_bar, one per column and 64-row tile in
// W = Delta^T U_bar.  U_bar and V_bar as factors of those two sums are stored in fixed point once per iteration,
// row-major in the place of float64 values of the same size that are not needed at that time (U over P, V over W), with
// one exponent per 64-row tile (Buffers::ex).
#include <algorithm>
#include <type_traits>

#include "fix64.cuh"
#include "sfr_internal.h"

namespace sfr {
namespace {

constexpr int kNT = 512;        // two CTAs per SM where registers and shared memory allow
constexpr int kNW = kNT / 32;
constexpr int kTile = 64;       // rows of a thin tile = columns of a sweep tile = terms of a sum
constexpr int kLD = kTile + 1;  // row stride of [rank][64] operands: 16 rows on distinct banks (8-byte reads)
constexpr int kBM = 32;         // rows of a sweep CTA
constexpr int kLU = kBM + 2;
constexpr int kNonFinite = 0x7ff00000;  // upper word from which a value is infinite or NaN

__device__ __forceinline__ bool stopped(const DevState* st) { return *(volatile const int32_t*)&st->done != 0; }

__device__ __forceinline__ int abs_hi(double x) { return __double2hiint(x) & 0x7fffffff; }

template <typename T> __device__ __forceinline__ double ld_f64(const T* p) { return (double)*p; }
template <> __device__ __forceinline__ double ld_f64<__nv_bfloat16>(const __nv_bfloat16* p) {
  return (double)__bfloat162float(*p);
}

__device__ __forceinline__ double block_sum(double v, double* red) {
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  __syncthreads();
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
  __syncthreads();
  double t = 0.0;
  if (threadIdx.x == 0)
    for (int i = 0; i < kNT / 32; ++i) t += red[i];
  return t;  // thread 0 only
}

// How the threads share a small output block of units (4 x 2 outputs each): `units` of them times
// `groups` (a power of two, at most `most`), each group taking its part of the sum.
struct Split {
  int units, groups, u, g;
  __device__ __forceinline__ Split(int units_, int most) : units(units_) {
    groups = 1;
    while (groups * 2 <= most && groups * 2 * units <= kNT) groups *= 2;
    u = threadIdx.x % units;
    g = threadIdx.x / units;
  }
  __device__ __forceinline__ bool active() const { return g < groups; }
};

using Acc = long long[4][2];
__device__ __forceinline__ void zero(Acc& a) {
#pragma unroll
  for (int x = 0; x < 4; ++x) a[x][0] = a[x][1] = 0;
}

// hh, cx += sum over k in [0, K) of A[k][i0 + di x] B[k][j0 + dj y]  (both operands stored by terms)
__device__ __forceinline__ void mac_outer(const int2* A, int lda, int di, const int2* B, int ldb, int dj, int K, Acc& hh,
                                          Acc& cx) {
#pragma unroll 2
  for (int k = 0; k < K; ++k) {
    int2 a[4], b[2];
#pragma unroll
    for (int q = 0; q < 4; ++q) a[q] = A[k * lda + di * q];
    b[0] = B[k * ldb];
    b[1] = B[k * ldb + dj];
    fx::mac_block(a, b, hh, cx);
  }
}

// hh, cx += sum over k in [0, K) of A[i0 + di x][k] B[j0 + dj y][k]  (both stored by rows; A and B point at
// the first row's first term)
__device__ __forceinline__ void mac_inner(const int2* A, int di, const int2* B, int dj, int K, Acc& hh, Acc& cx) {
#pragma unroll 2
  for (int k = 0; k < K; ++k) {
    int2 a[4], b[2];
#pragma unroll
    for (int q = 0; q < 4; ++q) a[q] = A[di * q * kLD + k];
    b[0] = B[k];
    b[1] = B[dj * kLD + k];
    fx::mac_block(a, b, hh, cx);
  }
}

// ---------------------------------------------------------------- thin tiles
// Elements of a 64 x RP tile owned by a thread: e = t + 512 q, row e / RP, column e % RP, q < RP / 8;
// of an RP x RP matrix: the same numbering, q < NS.
template <int RP> struct Tile {
  static constexpr int NQ = kTile * RP / kNT, NS = (RP * RP + kNT - 1) / kNT;
  static __device__ __forceinline__ int row(int q) { return ((int)threadIdx.x + kNT * q) / RP; }
  static __device__ __forceinline__ int col(int q) { return ((int)threadIdx.x + kNT * q) % RP; }
};

template <int RP>
__device__ __forceinline__ void load_tile(const double* src, int64_t i0, int64_t rows, int r, double (&v)[Tile<RP>::NQ]) {
#pragma unroll
  for (int q = 0; q < Tile<RP>::NQ; ++q) {
    const int64_t i = i0 + Tile<RP>::row(q);
    const int a = Tile<RP>::col(q);
    v[q] = i < rows && a < r ? src[i * RP + a] : 0.0;
  }
}

// The leading r x r block of g, zero outside.
template <int RP>
__device__ __forceinline__ void load_square(const double* __restrict__ g, int r, double (&v)[Tile<RP>::NS]) {
#pragma unroll
  for (int q = 0; q < Tile<RP>::NS; ++q) {
    const int e = (int)threadIdx.x + kNT * q;
    v[q] = e < RP * RP && e / RP < r && e % RP < r ? g[e] : 0.0;
  }
}

template <int N> __device__ __forceinline__ int max_hi(const double (&v)[N]) {
  int h = 0;
#pragma unroll
  for (int q = 0; q < N; ++q) h = max(h, abs_hi(v[q]));
  return h;
}

// Exponents of one tile's operands, in shared memory.  Two sets take turns (by tile): a tile resets the other's
// between its barriers, when the tile before has been left by every thread and the next one has not begun.
struct TileExps {
  int rank[64];      // of the tile's columns (ranks): the factors taken out of them
  int row[kTile];    // of its rows after that
  int col[2][64];    // of the columns of the squares
  int gram[2][64];   // of the columns of the Gram operands
  __device__ __forceinline__ void reset() {
    if (threadIdx.x < 64) {
      const int t = threadIdx.x;
      rank[t] = row[t] = col[0][t] = col[1][t] = gram[0][t] = gram[1][t] = fx::kZero;
    }
  }
};
static_assert(kTile == 64, "one thread per entry");

// ex[column] = max(ex[column], e) for the thread's column t % RP of a tile or square (e: the maximum over its own
// entries); all threads call it.
template <int RP> __device__ __forceinline__ void col_max(int e, int* ex) {
  const int t = threadIdx.x;
  if constexpr (RP < 32) {
#pragma unroll
    for (int o = RP; o < 32; o *= 2) e = max(e, __shfl_xor_sync(0xffffffffu, e, o));
    if ((t & 31) < RP) atomicMax(ex + (t & 31), e);
  } else {
    atomicMax(ex + t % RP, e);
  }
}
// The same for row t / RP + 512 / RP q of a tile.
template <int RP> __device__ __forceinline__ void row_max(int e, int q, int* ex) {
  if constexpr (RP < 32) {
#pragma unroll
    for (int o = RP / 2; o; o /= 2) e = max(e, __shfl_xor_sync(0xffffffffu, e, o));
    if (threadIdx.x % RP == 0) atomicMax(ex + Tile<RP>::row(q), e);
  } else {
    e = __reduce_max_sync(0xffffffffu, e);
    if ((threadIdx.x & 31) == 0) atomicMax(ex + Tile<RP>::row(q), e);
  }
}

// Exponents of the rows of a tile (row i: the largest of its entries once rank k's factor 2^rank[k] is out)
// and of the columns of a square whose row k has taken that factor.  After a barrier on rank[].
template <int RP> __device__ __forceinline__ void row_exps(const double (&v)[Tile<RP>::NQ], TileExps& x) {
  const int d = x.rank[threadIdx.x % RP];
#pragma unroll
  for (int q = 0; q < Tile<RP>::NQ; ++q) {
    const int h = abs_hi(v[q]);
    row_max<RP>(h ? fx::value_exponent(h) - d : fx::kZero, q, x.row);
  }
}
template <int RP> __device__ __forceinline__ void square_exps(const double (&v)[Tile<RP>::NS], const TileExps& x, int* col) {
  int e = fx::kZero;
#pragma unroll
  for (int q = 0; q < Tile<RP>::NS; ++q) {
    const int at = (int)threadIdx.x + kNT * q;
    if (at < RP * RP) e = max(e, fx::value_exponent(abs_hi(v[q])) + x.rank[at / RP]);
  }
  col_max<RP>(e, col);
}

// X[column][row] (columns < r4) = the tile, X[k][c] (row stride RP) = the square, in the fixed point of those exponents.
template <int RP> __device__ __forceinline__ void fix_tile(const double (&v)[Tile<RP>::NQ], const TileExps& x, int r4, int2* X) {
  const int c = threadIdx.x % RP, d = x.rank[c];
  if (c < r4)
#pragma unroll
    for (int q = 0; q < Tile<RP>::NQ; ++q) X[c * kLD + Tile<RP>::row(q)] = fx::to_fix(v[q], d + x.row[Tile<RP>::row(q)]);
}
template <int RP>
__device__ __forceinline__ void fix_square(const double (&v)[Tile<RP>::NS], const TileExps& x, const int* col, int2* X) {
#pragma unroll
  for (int q = 0; q < Tile<RP>::NS; ++q) {
    const int at = (int)threadIdx.x + kNT * q;
    if (at < RP * RP) X[at] = fx::to_fix(v[q], col[at % RP] - x.rank[at / RP]);
  }
}
// X[column][row] = a Gram operand, each column in the fixed point of its own exponent.
template <int RP> __device__ __forceinline__ void fix_cols(const double (&v)[Tile<RP>::NQ], const int* col, int r4, int2* X) {
  const int c = threadIdx.x % RP;
  if (c < r4)
#pragma unroll
    for (int q = 0; q < Tile<RP>::NQ; ++q) X[c * kLD + Tile<RP>::row(q)] = fx::to_fix(v[q], col[c]);
}

// 64 x r product of a tile X and a square Y (r terms), 4 x 2 outputs per thread, handed to
// f(row, column, sum) (columns below the next even number).
template <int RP, typename F>
__device__ __forceinline__ void tile_product(const int2* X, const int2* Y, int r, F&& f) {
  const int nb = (r + 1) / 2;
  if ((int)threadIdx.x >= 16 * nb) return;
  const int i = threadIdx.x & 15, j = threadIdx.x >> 4;
  Acc hh, cx;
  zero(hh);
  zero(cx);
  mac_outer(X + i, kLD, 16, Y + j, RP, nb, r, hh, cx);
#pragma unroll
  for (int x = 0; x < 4; ++x)
#pragma unroll
    for (int y = 0; y < 2; ++y) f(i + 16 * x, j + nb * y, fx::total(hh[x][y], cx[x][y]));
}

// g[q] += entry t + 512 q of A^T B for two 64-row tiles (column exponents ea, eb; NaN if bad): units of 4 x 2
// entries, rows u % na + na x, columns u / na + nb y, the 64 terms split over the groups of sp, whose
// integer sums are added before the one conversion to float64.  Ends with `red` (8 x 512) in use.
template <int RP>
__device__ __forceinline__ void tile_gram(const int2* A, const int2* B, const int* ea, const int* eb, bool bad, const Split& sp,
                                          int r, long long* red, double (&g)[Tile<RP>::NS]) {
  const int na = (r + 3) / 4, nb = (r + 1) / 2;
  if (sp.active()) {
    const int a = sp.u % na, b = sp.u / na, K = kTile / sp.groups;
    Acc hh, cx;
    zero(hh);
    zero(cx);
    mac_inner(A + a * kLD + sp.g * K, na, B + b * kLD + sp.g * K, nb, K, hh, cx);
#pragma unroll
    for (int x = 0; x < 4; ++x)
#pragma unroll
      for (int y = 0; y < 2; ++y) red[(2 * x + y) * kNT + threadIdx.x] = fx::total(hh[x][y], cx[x][y]);
  }
  __syncthreads();
#pragma unroll
  for (int q = 0; q < Tile<RP>::NS; ++q) {
    const int at = (int)threadIdx.x + kNT * q, x = at / RP, y = at % RP;
    if (x < r && y < r) {
      const long long* p = red + (2 * (x / na) + y / nb) * kNT + x % na + na * (y % nb);
      long long T = 0;
      for (int k = 0; k < sp.groups; ++k) T += p[k * sp.units];
      g[q] = fx::add_total(T, fx::Scale(bad ? fx::kBad : ea[x] + eb[y]), g[q]);
    }
  }
}

template <int RP>
__device__ __forceinline__ void store_square(const double (&g)[Tile<RP>::NS], double* __restrict__ out) {
#pragma unroll
  for (int q = 0; q < Tile<RP>::NS; ++q)
    if ((int)threadIdx.x + kNT * q < RP * RP) out[(int)threadIdx.x + kNT * q] = g[q];
}

constexpr size_t kRed = 8 * 8 * kNT;  // bytes of the scratch of integer sums

// For every 64-row tile of this CTA: out = sum of the partials (nparts == 0: out as it is) (+ A H
// when A != nullptr), then the CTA's Gram partial, the sum over its rows of out^T out.
template <int RP>
__global__ void __launch_bounds__(kNT) f64_gram_kernel(const double* parts, int nparts, int64_t part_stride, double* out,
                                                       int64_t rows, const double* __restrict__ A,
                                                       const double* __restrict__ H, double* __restrict__ gpart, int r,
                                                       const DevState* st) {
  pdl_enter();
  if (stopped(st)) return;
  constexpr int NQ = Tile<RP>::NQ, NS = Tile<RP>::NS, LDO = RP + 1;
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ TileExps exps[2];
  const int r4 = (r + 3) / 4 * 4;
  long long* red = reinterpret_cast<long long*>(smem);         // Gram scratch, or the A H product's operands:
  int2* As = reinterpret_cast<int2*>(smem);                    // [r4][kLD]
  double* So = reinterpret_cast<double*>(As + r4 * kLD);       // [64][RP + 1]
  int2* Hs = reinterpret_cast<int2*>(So + kTile * LDO);        // [RP][RP]
  int2* X = reinterpret_cast<int2*>(smem + (A ? max(kRed, 8 * ((size_t)r4 * kLD + kTile * LDO + RP * RP)) : kRed));  // [r4][kLD]
  const Split sp((r + 3) / 4 * ((r + 1) / 2), 32);
  double g[NS];
#pragma unroll
  for (int q = 0; q < NS; ++q) g[q] = 0.0;
  exps[0].reset();
  __syncthreads();
  const int64_t ntiles = (rows + kTile - 1) / kTile;
  int turn = 0;
  for (int64_t tl = blockIdx.x; tl < ntiles; tl += gridDim.x, turn ^= 1) {
    const int64_t i0 = tl * kTile;
    TileExps& ex = exps[turn];
    double v[NQ];
    load_tile<RP>(nparts ? parts : out, i0, rows, r, v);
    auto add_parts = [&] {
#pragma unroll 4
      for (int s = 1; s < nparts; ++s) {
        double p[NQ];
        load_tile<RP>(parts + s * part_stride, i0, rows, r, p);
#pragma unroll
        for (int q = 0; q < NQ; ++q) v[q] += p[q];
      }
    };
    if (A) {
      double w[NQ], hv[NS];
      load_tile<RP>(A, i0, rows, r, w);
      load_square<RP>(H, r, hv);
      add_parts();
      const int hw = max_hi(w);
      col_max<RP>(fx::value_exponent(hw), ex.rank);
      const bool bad = __syncthreads_or(max(hw, max_hi(hv)) >= kNonFinite);  // (closes the previous tile's use of the scratch)
      row_exps<RP>(w, ex);
      square_exps<RP>(hv, ex, ex.col[0]);
      __syncthreads();
      fix_tile<RP>(w, ex, r4, As);
      fix_square<RP>(hv, ex, ex.col[0], Hs);
#pragma unroll
      for (int q = 0; q < NQ; ++q) So[Tile<RP>::row(q) * LDO + Tile<RP>::col(q)] = v[q];
      __syncthreads();
      tile_product<RP>(As, Hs, r, [&](int i, int j, long long T) {
        So[i * LDO + j] = fx::add_total(T, fx::Scale(bad ? fx::kBad : ex.row[i] + ex.col[0][j]), So[i * LDO + j]);
      });
      __syncthreads();
#pragma unroll
      for (int q = 0; q < NQ; ++q)
        v[q] = Tile<RP>::col(q) < r ? So[Tile<RP>::row(q) * LDO + Tile<RP>::col(q)] : 0.0;
    } else {
      add_parts();
    }
    const int hx = max_hi(v);
    col_max<RP>(fx::value_exponent(hx), ex.gram[0]);
    const bool bad = __syncthreads_or(hx >= kNonFinite);
    exps[turn ^ 1].reset();
    fix_cols<RP>(v, ex.gram[0], r4, X);
    if (nparts) {
#pragma unroll
      for (int q = 0; q < NQ; ++q) {
        const int64_t i = i0 + Tile<RP>::row(q);
        if (i < rows) out[i * RP + Tile<RP>::col(q)] = v[q];
      }
    }
    __syncthreads();
    tile_gram<RP>(X, X, ex.gram[0], ex.gram[0], bad, sp, r, red, g);
  }
  store_square<RP>(g, gpart + (int64_t)blockIdx.x * RP * RP);
}

// For every 64-row tile of this CTA: dst = src T, dst2 = src T2 (optional), hpart[cta] = the sum over
// its rows of old^T dst (optional, not with T2), and the fixed-point copy F of dst with its tile
// exponent (F may lie over src: each tile is read before it is written).
template <int RP>
__global__ void __launch_bounds__(kNT) f64_transform_kernel(const double* src, int64_t rows, const double* __restrict__ T,
                                                            double* __restrict__ dst, const double* __restrict__ T2,
                                                            double* __restrict__ dst2, const double* __restrict__ old,
                                                            double* __restrict__ hpart, int2* F, int* __restrict__ eF, int r,
                                                            const DevState* st) {
  pdl_enter();
  if (stopped(st)) return;
  constexpr int NQ = Tile<RP>::NQ, NS = Tile<RP>::NS, LDO = RP + 1;
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ TileExps exps[2];
  const int r4 = (r + 3) / 4 * 4;
  int2* X = reinterpret_cast<int2*>(smem);               // [r4][kLD] src tile, then the dst tile
  int2* O = X + r4 * kLD;                                // [r4][kLD] the old tile, or [RP][RP] T2
  int2* Ts = O + (hpart ? r4 * kLD : T2 ? RP * RP : 0);  // [RP][RP]
  double* So = reinterpret_cast<double*>(Ts + RP * RP);  // [64][RP + 1]
  long long* red = reinterpret_cast<long long*>(Ts);     // Gram scratch (T is converted again for the next tile)
  const Split sp((r + 3) / 4 * ((r + 1) / 2), 32);
  double g[NS];
#pragma unroll
  for (int q = 0; q < NS; ++q) g[q] = 0.0;
  exps[0].reset();
  __syncthreads();
  const int64_t ntiles = (rows + kTile - 1) / kTile;
  int turn = 0;
  for (int64_t tl = blockIdx.x; tl < ntiles; tl += gridDim.x, turn ^= 1) {
    const int64_t i0 = tl * kTile;
    TileExps& ex = exps[turn];
    double v[NQ];
    bool bad, bad_old = false;
    {
      double w[NQ], tv[NS], t2[NS];
      load_tile<RP>(src, i0, rows, r, v);
      load_square<RP>(T, r, tv);
      if (hpart) load_tile<RP>(old, i0, rows, r, w);
      if (T2) load_square<RP>(T2, r, t2);
      const int hv = max_hi(v), hs = max(max_hi(tv), T2 ? max_hi(t2) : 0);
      col_max<RP>(fx::value_exponent(hv), ex.rank);
      if (hpart) col_max<RP>(fx::value_exponent(max_hi(w)), ex.gram[0]);
      bad = __syncthreads_or(max(hv, hs) >= kNonFinite);  // (closes the previous tile's use of shared memory)
      if (hpart) bad_old = __syncthreads_or(max_hi(w) >= kNonFinite);
      row_exps<RP>(v, ex);
      square_exps<RP>(tv, ex, ex.col[0]);
      if (T2) square_exps<RP>(t2, ex, ex.col[1]);
      __syncthreads();
      fix_tile<RP>(v, ex, r4, X);
      fix_square<RP>(tv, ex, ex.col[0], Ts);
      if (hpart) fix_cols<RP>(w, ex.gram[0], r4, O);
      if (T2) fix_square<RP>(t2, ex, ex.col[1], O);
      exps[turn ^ 1].reset();
    }
    __syncthreads();
    for (int part = 0; part < (T2 ? 2 : 1); ++part) {
      tile_product<RP>(X, part ? O : Ts, r, [&](int i, int j, long long t) {
        So[i * LDO + j] = fx::add_total(t, fx::Scale(bad ? fx::kBad : ex.row[i] + ex.col[part][j]), 0.0);
      });
      __syncthreads();
#pragma unroll
      for (int q = 0; q < NQ; ++q)
        v[q] = Tile<RP>::col(q) < r ? So[Tile<RP>::row(q) * LDO + Tile<RP>::col(q)] : 0.0;
      double* o = part ? dst2 : dst;
#pragma unroll
      for (int q = 0; q < NQ; ++q) {
        const int64_t i = i0 + Tile<RP>::row(q);
        if (i < rows) o[i * RP + Tile<RP>::col(q)] = v[q];
      }
      if (part) break;  // (the next tile's first barrier comes before So and the operands are written again)
      const int h = max_hi(v);
      col_max<RP>(fx::value_exponent(h), ex.gram[1]);
      const bool bad_new = __syncthreads_or(h >= kNonFinite);
      const int lane = threadIdx.x & 31;
      int eD = max(ex.gram[1][lane], ex.gram[1][lane + 32]);
      eD = __reduce_max_sync(0xffffffffu, eD);
      if (threadIdx.x == 0) eF[tl] = bad_new ? fx::kBad : eD;
#pragma unroll
      for (int q = 0; q < NQ; ++q) {
        const int64_t i = i0 + Tile<RP>::row(q);
        if (i < rows) F[i * RP + Tile<RP>::col(q)] = fx::to_fix(v[q], eD);
      }
      if (hpart) {
        fix_cols<RP>(v, ex.gram[1], r4, X);  // src's copy is consumed
        __syncthreads();
        tile_gram<RP>(O, X, ex.gram[0], ex.gram[1], bad_old || bad_new, sp, r, red, g);
      }
    }
  }
  if (hpart) store_square<RP>(g, hpart + (int64_t)blockIdx.x * RP * RP);
}

size_t gram_smem(int rp, int r, bool add) {
  const size_t r4 = (r + 3) / 4 * 4, x = 8 * r4 * kLD;
  return x + (add ? std::max<size_t>(kRed, x + 8 * (size_t)(kTile * (rp + 1) + rp * rp)) : kRed);
}
size_t transform_smem(int rp, int r, bool hp, bool two) {
  const size_t r4 = (r + 3) / 4 * 4, x = 8 * r4 * kLD, sq = 8 * (size_t)rp * rp;
  return x + (hp ? x : two ? sq : 0) + std::max<size_t>(sq + 8 * (size_t)kTile * (rp + 1), hp ? kRed : 0);
}

// ---------------------------------------------------------------- sweep
// The outputs of a block of rows x ranks that a thread converts and keeps: e = t + 512 q, row(q) = e / RP, rank
// e % RP = t % RP; at(q) = their place among sums stored by units of DI interleaved rows: unit u has rows
// u % DI + DI x and ranks u / DI + nb y at word (2 x + y) 512 + u.
template <int RP, int DI> struct Own {
  int first;
  bool used;
  __device__ __forceinline__ Own(int rows, int nb, int r) {
    const int a = threadIdx.x % RP;
    first = a / nb * kNT + DI * (a % nb);
    used = a < r && row(0) < rows;  // (fewer outputs than threads: one per thread)
  }
  static __device__ __forceinline__ int row(int q) { return (int)threadIdx.x / RP + kNT / RP * q; }
  __device__ __forceinline__ int at(int q) const { return first + 2 * kNT * (row(q) / DI) + row(q) % DI; }
};

// ROWS rows of a row-major thin factor (stride RP, float64; rows from `valid` on are zeros) to dst[rank][row], each row in
// the fixed point of its own exponent ex[row].
template <int RP, int ROWS>
__device__ __forceinline__ void fix_rows(const double* __restrict__ src, int valid, int r, int r4, int2* dst, int ldd, int* ex) {
  constexpr int G = RP < 32 ? RP : 32, K = RP / G, PER = kNT / G, N = (ROWS + PER - 1) / PER;
  const int g = threadIdx.x % G, r0 = threadIdx.x / G;
  double v[N][K];
#pragma unroll
  for (int q = 0; q < N; ++q)
#pragma unroll
    for (int k = 0; k < K; ++k) {
      const int row = r0 + PER * q, a = g + 32 * k;
      v[q][k] = row < valid && a < r ? src[row * RP + a] : 0.0;
    }
#pragma unroll
  for (int q = 0; q < N; ++q) {
    const int row = r0 + PER * q;
    if (PER * N > ROWS && row >= ROWS) break;  // (whole warps)
    int h = max_hi(v[q]);
    if constexpr (G == 32) {
      h = __reduce_max_sync(0xffffffffu, h);
    } else {
#pragma unroll
      for (int o = G / 2; o; o /= 2) h = max(h, __shfl_xor_sync(0xffffffffu, h, o));
    }
    const int e = fx::exponent(h);
#pragma unroll
    for (int k = 0; k < K; ++k)
      if (g + 32 * k < r4) dst[(g + 32 * k) * ldd + row] = fx::to_fix(v[q][k], e);
    if (g == 0) ex[row] = e;
  }
}

// Algorithm 1's S- and Y-steps on 32 rows x the 64-column tiles of one column split:
//   L = U_bar C^T, z = M - L + Y_k / mu_k, Y_{k+1} = clip(mu_k z, -1, 1),
//   Delta = Y_{k+1} (1 / mu_k + 1 / mu_{k+1}) - Y_k / mu_k,
//   residual += (Y_{k+1} - Y_k)^2, Q += Delta V_bar
// (P_{k+1} = X_{k+1} V_bar = U_bar B_bar + Q, since L_{k+1} V_bar = U_bar B_bar V_bar^T V_bar).
// L: 2 rows x 2 columns per thread, sums over the r ranks.  Q: 4 rows x 2 ranks per thread and a part
// of the tile's 64 columns (Split); the parts' integer sums are added through shared memory (over
// the C tile), so that each output is converted to float64 once per tile.  A warp holds two whole rows of a tile, so
// that the exponent of a row of Delta is one reduction over its lanes.  U and C come in float64 and are converted here, by
// rows (C once per tile and CTA: r / 8 conversions per thread beside 24 r multiply-adds; 4096 x 4096, r = 64 1215 us,
// 1180 with fixed-point copies that shared an exponent among 64 rows).  Bounds: the integer units at
// 6 r multiply-adds per element and the float64 units at about 7 + r / 32 operations per element.
template <typename TMs, int RP>
__global__ void __launch_bounds__(kNT, 2) f64_sweep_kernel(const TMs* __restrict__ M, int64_t m, int64_t n, int64_t ldm,
                                                           const double* __restrict__ Yin, double* __restrict__ Yout,
                                                           double* __restrict__ D, int64_t ldy,
                                                           const double* __restrict__ U, const double* __restrict__ C,
                                                           const int2* __restrict__ V, const int* __restrict__ eV,
                                                           double* __restrict__ Qpart, int r, int cols_per_split,
                                                           double* __restrict__ resid_part, const DevState* st) {
  pdl_enter();
  if (stopped(st)) return;
  constexpr int LC = kLD;
  constexpr int rp = RP, NO = (kBM * RP + kNT - 1) / kNT;
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ double red[kNW];
  __shared__ int eu[kBM], ec[kTile], ed[kBM];  // exponents of the rows of U, C and Delta
  const int nb = (r + 1) / 2, r4 = (r + 3) / 4 * 4;
  int2* Us = reinterpret_cast<int2*>(smem);  // [r4][kLU]
  int2* Vs = Us + r4 * kLU;                  // [r4][kLD]
  int2* Ds = Vs + r4 * kLD;                  // [32][kLD]
  int2* Cs = Ds + kBM * kLD;                 // [r4][LC]
  long long* qs = reinterpret_cast<long long*>(Cs);  // [8][512]
  const double mu = st->mu, mu_next = fmin(st->mu_max, st->rho * mu);
  const double inv_mu = 1.0 / mu, dcoef = 1.0 / mu + 1.0 / mu_next;
  const int64_t i0 = (int64_t)blockIdx.x * kBM;
  const int64_t jbeg = (int64_t)blockIdx.y * cols_per_split, jend = min(n, jbeg + cols_per_split);
  const int t = threadIdx.x, ty = t >> 5, tx = t & 31;
  fix_rows<RP, kBM>(U + i0 * rp, (int)min((int64_t)kBM, m - i0), r, r4, Us, kLU, eu);
  const Split sp(8 * nb, 32);
  const int qk = kTile / sp.groups;
  const int2* qd = Ds + (sp.u & 7) * kLD + sp.g * qk;
  const int2* qv = Vs + (sp.u >> 3) * kLD + sp.g * qk;
  const Own<RP, 8> own(kBM, nb, r);
  double q[NO];
#pragma unroll
  for (int k = 0; k < NO; ++k) q[k] = 0.0;
  double resid = 0.0;
  const int64_t i = i0 + 2 * ty;  // this thread's elements: rows i + x, columns j0 + tx + 32 c
  const int nrow = m - i < 2 ? (int)(m - i) : 2;
  for (int64_t j0 = jbeg; j0 < jend; j0 += kTile) {
    const int64_t j = j0 + tx;
    const int left = jend - j < kTile ? (int)(jend - j) : kTile;  // columns 32 c < left are valid
    double mv[2][2], yv[2][2];
#pragma unroll
    for (int x = 0; x < 2; ++x) {
      const TMs* mp = M + (i + x) * ldm + j;
      const double* yp = Yin + (i + x) * ldy + j;
#pragma unroll
      for (int c = 0; c < 2; ++c) {
        const bool ok = x < nrow && 32 * c < left;
        mv[x][c] = ok ? ld_f64(mp + 32 * c) : 0.0;
        yv[x][c] = ok ? yp[32 * c] : 0.0;
      }
    }
    __syncthreads();  // the previous tile's Vs, Ds and sums are consumed
    fix_rows<RP, kTile>(C + j0 * rp, (int)min((int64_t)kTile, jend - j0), r, r4, Cs, LC, ec);
    for (int e = t; e < kTile * rp; e += kNT) {
      const int jj = e / rp, a = e % rp;
      if (a < r4) Vs[a * kLD + jj] = j0 + jj < jend ? V[j0 * rp + e] : make_int2(0, 0);
    }
    __syncthreads();
    {
      long long hh[2][2], cx[2][2];
#pragma unroll
      for (int x = 0; x < 2; ++x)
#pragma unroll
        for (int c = 0; c < 2; ++c) hh[x][c] = cx[x][c] = 0;
      const int2* up = Us + 2 * ty;
      const int2* cp = Cs + tx;
#pragma unroll 4
      for (int a = 0; a < r; ++a, up += kLU, cp += LC) {
        const int4 u = *reinterpret_cast<const int4*>(up);
        const int2 uv[2] = {make_int2(u.x, u.y), make_int2(u.z, u.w)};
        int2 cv[2];
#pragma unroll
        for (int c = 0; c < 2; ++c) cv[c] = cp[32 * c];
        fx::mac_block(uv, cv, hh, cx);
      }
#pragma unroll
      for (int x = 0; x < 2; ++x) {
        double* yo = Yout + (i + x) * ldy + j;
        double* dp = D + (i + x) * ldy + j;
        double d[2] = {0.0, 0.0};
#pragma unroll
        for (int c = 0; c < 2; ++c) {
          if (x < nrow && 32 * c < left) {
            const double y = yv[x][c];
            // mu_k z = mu_k (M - L) + Y_k
            const fx::Scale sl(eu[2 * ty + x] + ec[tx + 32 * c]);
            double yn = fma(mu, fx::add_total(-fx::total(hh[x][c], cx[x][c]), sl, mv[x][c]), y);
            yn = fabs(yn) > 1.0 ? copysign(1.0, yn) : yn;
            const double dy = yn - y;
            d[c] = fma(yn, dcoef, -(y * inv_mu));
            resid = fma(dy, dy, resid);
            yo[32 * c] = yn;
            dp[32 * c] = d[c];
          }
        }
        const int e = fx::exponent(__reduce_max_sync(0xffffffffu, max_hi(d)));
        if (tx == 0) ed[2 * ty + x] = e;
#pragma unroll
        for (int c = 0; c < 2; ++c) Ds[(2 * ty + x) * kLD + tx + 32 * c] = fx::to_fix(d[c], e);
      }
    }
    __syncthreads();
    if (sp.active()) {
      Acc hh, cx;
      zero(hh);
      zero(cx);
      mac_inner(qd, 8, qv, nb, qk, hh, cx);
#pragma unroll
      for (int x = 0; x < 4; ++x)
#pragma unroll
        for (int y = 0; y < 2; ++y) qs[(2 * x + y) * kNT + t] = fx::total(hh[x][y], cx[x][y]);
    }
    __syncthreads();
    const int ev = eV[j0 / kTile];
#pragma unroll
    for (int k = 0; k < NO; ++k)
      if (own.used) {
        long long T = 0;
        for (int g = 0; g < sp.groups; ++g) T += qs[own.at(k) + g * sp.units];
        q[k] = fx::add_total(T, fx::Scale(ed[own.row(k)] + ev), q[k]);
      }
  }
#pragma unroll
  for (int k = 0; k < NO; ++k) {
    if (own.used && i0 + own.row(k) < m) Qpart[((int64_t)blockIdx.y * m + i0) * rp + t + kNT * k] = q[k];
  }
  resid = block_sum(resid, red);
  if (t == 0) resid_part[(int64_t)blockIdx.y * gridDim.x + blockIdx.x] = resid;
}

size_t sweep_smem(int r) {
  const size_t r4 = (r + 3) / 4 * 4;
  return 8 * (r4 * kLU + r4 * kLD + kBM * kLD) + std::max<size_t>(8 * r4 * (kTile + 1), kRed);
}

// ---------------------------------------------------------------- W pass
__device__ __forceinline__ void cp_async8(void* dst, const void* src, int bytes) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;\n" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src),
               "r"(bytes)
               : "memory");
}

// Wpart[c][j][:] = sum over the rows i of chunk c of Delta[i][j] U_bar[i][:], U_bar in fixed point.
// CTA: 64 columns x a chunk of rows in stages, double-buffered by cp.async; 4 columns x 2
// ranks per thread and a part of each stage's rows (Split); after each 64-row tile (U's exponent) the
// parts' integer sums are added through shared memory and converted to float64 once per output.
// Delta arrives in float64 and is converted in place, a warp per column (lane = row): the exponent of a column is that of
// its stages so far in the 64-row tile, and when a second stage raises it the sums of the first are shifted.
// Stages of 64 rows up to rank 16, where the three barriers of a stage weigh more than its products (2000 x 2000, r = 10:
// 66 us in stages of 32, 59 in stages of 64; at ranks 13 to 16, where one CTA of 114 KB is left per SM, 79 us either way
// for 3000 x 1500); above, two CTAs per SM have room for 32.
// Bounded by the integer units at 3 r multiply-adds per element; 101 KB of shared memory at r = 64 lets
// two CTAs overlap on an SM.  With one exponent for all of Delta, stored in fixed point by the sweep, it took 606 us
// at 4096 x 4096, r = 64 (now 661) and 55 at 2000 x 2000, r = 10, but columns of M 1e10 smaller than the
// others lost 1e-6 of their own size.
template <int RP> constexpr int kWRows = RP <= 16 ? kTile : kBM;
template <int RP>
__global__ void __launch_bounds__(kNT, 2) f64_wpass_kernel(const double* __restrict__ D, int64_t ldy, int64_t m, int64_t n,
                                                           int rows_per_chunk, const int2* __restrict__ U,
                                                           const int* __restrict__ eU, double* __restrict__ Wpart,
                                                           int r, const DevState* st) {
  pdl_enter();
  if (stopped(st)) return;
  constexpr int rp = RP, NO = kTile * RP / kNT, W = kWRows<RP>, LU = W + 2, PER = kTile / W;  // PER stages per tile
  extern __shared__ __align__(16) unsigned char smem[];
  const int nb = (r + 1) / 2, r4 = (r + 3) / 4 * 4;
  const int stage = W * kLD + r4 * LU;  // 8-byte words per stage: Delta [W][kLD], U [r4][LU]
  int2* base = reinterpret_cast<int2*>(smem);
  __shared__ int ed[kTile], grown[kTile];  // exponents of Delta's columns, and by how much the last stage raised them
  long long* ws = reinterpret_cast<long long*>(base + 2 * stage);  // [8][512]
  const int64_t j0 = (int64_t)blockIdx.x * kTile;
  const int64_t r0 = (int64_t)blockIdx.y * rows_per_chunk, r1 = min(m, r0 + rows_per_chunk);
  const int nst = r1 > r0 ? (int)((r1 - r0 + W - 1) / W) : 0;
  const int t = threadIdx.x, warp = t >> 5, lane = t & 31;
  auto issue = [&](int k) {
    const int64_t it = r0 + (int64_t)k * W;
    const int nr = r1 - it < W ? (int)(r1 - it) : W;
    int2* ds = base + (k & 1) * stage;
    int2* us = ds + W * kLD;
    const bool col = j0 + (t & 63) < n;
    const double* src = D + it * ldy + j0 + (t & 63);
#pragma unroll
    for (int q = 0; q < W * kTile / kNT; ++q) {
      const int ii = (t >> 6) + kNT / kTile * q;
      const bool ok = col && ii < nr;
      cp_async8(ds + ii * kLD + (t & 63), ok ? src + ii * ldy : D, ok ? 8 : 0);
    }
    for (int e = t; e < W * rp; e += kNT) {
      const int ii = e / rp, a = e % rp;
      if (a < r4) cp_async8(us + a * LU + ii, ii < nr ? U + it * rp + e : U, ii < nr ? 8 : 0);
    }
    asm volatile("cp.async.commit_group;\n" ::: "memory");
  };
  // Delta of stage k to fixed point; second: not the first stage of a 64-row tile (chunks start at multiples of 64)
  auto convert = [&](int k, bool second) {
    int2* ds = base + (k & 1) * stage;
#pragma unroll
    for (int q = 0; q < kTile / kNW; ++q) {
      const int c = warp + kNW * q;
      double x[W / 32];
#pragma unroll
      for (int p = 0; p < W / 32; ++p) x[p] = *reinterpret_cast<const double*>(ds + (lane + 32 * p) * kLD + c);
      const int h = __reduce_max_sync(0xffffffffu, max_hi(x));
      const int old = second ? ed[c] : fx::kZero, e = max(old, h >= kNonFinite ? fx::kBad : fx::value_exponent(h));
#pragma unroll
      for (int p = 0; p < W / 32; ++p) ds[(lane + 32 * p) * kLD + c] = fx::to_fix(x[p], e);
      __syncwarp();  // every lane has read ed[c]
      if (lane == 0) ed[c] = e, grown[c] = second ? min(e - old, 63) : 0;
    }
  };
  const Split sp(16 * nb, 16);
  const int wk = W / sp.groups;
  const Own<RP, 16> own(kTile, nb, r);
  double w[NO];
#pragma unroll
  for (int k = 0; k < NO; ++k) w[k] = 0.0;
  Acc sum;  // of the 64-row tile so far, as fx::total
  zero(sum);
  if (nst > 0) issue(0);
  for (int k = 0; k < nst; ++k) {
    if (k + 1 < nst) issue(k + 1); else asm volatile("cp.async.commit_group;\n" ::: "memory");
    asm volatile("cp.async.wait_group 1;\n" ::: "memory");
    __syncthreads();
    const bool second = PER == 2 && (k & 1), last = PER == 1 || second || k + 1 == nst;  // last: the end of a 64-row tile
    convert(k, second);
    __syncthreads();
    if (sp.active()) {
      const int2* ds = base + (k & 1) * stage + sp.g * wk * kLD + (sp.u & 15);
      const int2* us = base + (k & 1) * stage + W * kLD + (sp.u >> 4) * LU + sp.g * wk;
      if (second) {
#pragma unroll
        for (int x = 0; x < 4; ++x) {
          const int g = grown[(sp.u & 15) + 16 * x];
          if (g > 0)
#pragma unroll
            for (int y = 0; y < 2; ++y) sum[x][y] >>= g;
        }
      }
      Acc cx;
      zero(cx);
#pragma unroll 2
      for (int i = 0; i < wk; ++i) {
        int2 a[4], b[2];
#pragma unroll
        for (int q = 0; q < 4; ++q) a[q] = ds[i * kLD + 16 * q];
        b[0] = us[i];
        b[1] = us[nb * LU + i];
        fx::mac_block(a, b, sum, cx);
      }
#pragma unroll
      for (int x = 0; x < 4; ++x)
#pragma unroll
        for (int y = 0; y < 2; ++y) {
          sum[x][y] = fx::total(sum[x][y], cx[x][y]);
          if (last) {
            ws[(2 * x + y) * kNT + t] = sum[x][y];
            sum[x][y] = 0;
          }
        }
    }
    __syncthreads();  // the stage is refilled by the next iteration's issue; the sums are complete
    if (last) {
      const int eu = eU[(r0 + (int64_t)k * W) / kTile];
#pragma unroll
      for (int q = 0; q < NO; ++q)
        if (own.used) {
          long long T = 0;
          for (int g = 0; g < sp.groups; ++g) T += ws[own.at(q) + g * sp.units];
          w[q] = fx::add_total(T, fx::Scale(ed[own.row(q)] + eu), w[q]);
        }  // (the next exponents and sums are stored after the next iteration's first barrier)
    }
  }
  asm volatile("cp.async.wait_group 0;\n" ::: "memory");
#pragma unroll
  for (int q = 0; q < NO; ++q) {
    if (own.used && j0 + own.row(q) < n) Wpart[((int64_t)blockIdx.y * n + j0) * rp + t + kNT * q] = w[q];
  }
}

size_t wpass_smem(int r, int rows) {
  const size_t r4 = (r + 3) / 4 * 4;
  return 2 * 8 * (rows * kLD + r4 * (rows + 2)) + kRed;
}

}  // namespace

// ---------------------------------------------------------------- launchers (called by sweep.cu's)
template <typename F>
static cudaError_t by_rank(int rp, F&& f) {
  switch (rp) {
    case 8: return f(std::integral_constant<int, 8>{});
    case 16: return f(std::integral_constant<int, 16>{});
    case 32: return f(std::integral_constant<int, 32>{});
    case 64: return f(std::integral_constant<int, 64>{});
    default: return cudaErrorInvalidValue;
  }
}

cudaError_t f64_gram(const Shape& s, const double* parts, int nparts, int64_t part_stride, double* out, int64_t rows,
                     int ctas, const double* A, const double* H, double* gpart, const DevState* dst, cudaStream_t st) {
  return by_rank(s.rp, [&](auto rpc) {
    auto kern = f64_gram_kernel<decltype(rpc)::value>;
    const size_t sm = gram_smem(s.rp, s.r, A != nullptr);
    cudaError_t e = set_smem_attr<&f64_gram_kernel<decltype(rpc)::value>>(sm);
    if (e != cudaSuccess) return e;
    return launch_pdl(kern, ctas, kNT, sm, st, parts, nparts, part_stride, out, rows, A, H, gpart, s.r, dst);
  });
}

cudaError_t f64_transform(const Shape& s, const double* src, int64_t rows, int ctas, const double* T, double* dst,
                          const double* T2, double* dst2, const double* old, double* hpart, void* F, int* eF,
                          const DevState* dstate, cudaStream_t st) {
  return by_rank(s.rp, [&](auto rpc) {
    auto kern = f64_transform_kernel<decltype(rpc)::value>;
    const size_t sm = transform_smem(s.rp, s.r, hpart != nullptr, T2 != nullptr);
    cudaError_t e = set_smem_attr<&f64_transform_kernel<decltype(rpc)::value>>(sm);
    if (e != cudaSuccess) return e;
    return launch_pdl(kern, ctas, kNT, sm, st, src, rows, T, dst, T2, dst2, old, hpart, static_cast<int2*>(F), eF,
                      s.r, dstate);
  });
}

cudaError_t f64_sweep(const Shape& s, const Buffers& b, int u_cur, cudaStream_t st) {
  const dim3 grid(s.sweep_grid_x, s.nsplit);
  const size_t sm = sweep_smem(s.r);
  const int64_t tu = (s.m + kTile - 1) / kTile;
  return by_rank(s.rp, [&](auto rpc) {
    auto go = [&](auto M) -> cudaError_t {
      using TMs = std::remove_const_t<std::remove_pointer_t<decltype(M)>>;
      auto kern = f64_sweep_kernel<TMs, decltype(rpc)::value>;
      cudaError_t e = set_smem_attr<&f64_sweep_kernel<TMs, decltype(rpc)::value>>(sm);
      if (e != cudaSuccess) return e;
      return launch_pdl(kern, grid, kNT, sm, st, M, s.m, s.n, s.ldm, static_cast<const double*>(b.Y[0]),
                        static_cast<double*>(b.Y[1]), static_cast<double*>(b.D), b.ldy, static_cast<const double*>(b.U[u_cur]),
                        static_cast<const double*>(b.C), static_cast<const int2*>(b.W), b.ex + tu, static_cast<double*>(b.Qpart), s.r, s.cols_per_split, b.resid_part, b.st);
    };
    if (b.m_dtype == SFR_F64) return go(static_cast<const double*>(b.M));
    if (b.m_dtype == SFR_F32) return go(static_cast<const float*>(b.M));
    return go(static_cast<const __nv_bfloat16*>(b.M));
  });
}

cudaError_t f64_wpass(const Shape& s, const Buffers& b, cudaStream_t st) {
  return by_rank(s.rp, [&](auto rpc) {
    const size_t sm = wpass_smem(s.r, kWRows<decltype(rpc)::value>);
    auto kern = f64_wpass_kernel<decltype(rpc)::value>;
    cudaError_t e = set_smem_attr<&f64_wpass_kernel<decltype(rpc)::value>>(sm);
    if (e != cudaSuccess) return e;
    return launch_pdl(kern, dim3(s.wpass_grid_x, s.nchunk64), kNT, sm, st, static_cast<const double*>(b.D), b.ldy, s.m, s.n,
                      s.rows_per_chunk64, static_cast<const int2*>(b.P), b.ex, static_cast<double*>(b.Wpart), s.r, b.st);
  });
}

}  // namespace sfr
