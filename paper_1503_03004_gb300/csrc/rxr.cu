// r x r steps of FixedRankOptStep (Algorithm 3), one CTA or cluster per problem.
//
// Stiefel projector (Sec. 4.1.1, Eq. 9): P_O[A] = A (A^T A)^{-1/2} for a full-rank
// m x r matrix A.  With A = P B (U side, P = X V) or A = W B (V side, W = X^T U),
//     A^T A = B G B,   G = P^T P  or  W^T W,
// so P_O[A] = P T with T = B (B G B)^{-1/2}: only r x r work, applied row-wise later.
// SPD projector (Sec. 4.1.2, Eq. 10): B_bar = Sym(U_bar^T X V_bar) = Sym(W^T V_bar)
//     = Sym(G_W T_V), and C = V_bar B_bar = W (T_V B_bar) so that L = U_bar C^T.
//
// The inverse square root Z = K^{-1/2} of K = B G B is computed in two stages:
//  1. cyclic parallel Jacobi in float32 (warm-started from the previous call's
//     eigenvectors) gives an approximate eigenbasis Q and eigenvalues lambda;
//  2. Newton's method for the symmetric solution of Z K Z = I in float64:
//     with R = I - Z K Z, the correction Delta solves Delta K Z + Z K Delta = R;
//     in the approximate eigenbasis K Z ~ Q diag(sqrt(lambda)) Q^T, so
//     Delta = Q [ (Q^T R Q)_pq / (sqrt(lambda_p) + sqrt(lambda_q)) ] Q^T.
//     The residual R is formed in float64; the small correction may be formed
//     in float32.  Each step contracts the error by roughly the eigenbasis error,
//     so two or three steps reach float64 round-off.
//
// GB300 runs float64 at about 2 FMA per clock per SM, so one r = 64 product (262k FMA)
// takes ~60 us on one SM.  The kernel therefore runs as a thread-block cluster: every
// CTA keeps full copies of the r x r matrices in shared memory, computes a slice of rows
// of each float64 product, and pushes its rows to the other CTAs through distributed
// shared memory.  Everything else (float32 Jacobi, element-wise steps, scalar decisions)
// is computed redundantly and identically by every CTA, so control flow stays uniform
// across the cluster; each CTA writes its own rows.
//
// The kernel is a chain of about thirty short dependent phases, so its time is barriers and load
// latency rather than arithmetic.  It is therefore built per padded rank (Dim): r <= 8 runs in one
// warp, r <= 16 in one CTA of 128 threads, r <= 32 in clusters of 256-thread CTAs, r <= 64 in clusters of 512,
// element-wise steps are done where a product's results are stored (Epi), and the statistics of the r
// eigenvalue estimates are taken by every warp for itself.  The mean call of a solve of 60 iterations (1536 x 1024, mixed path,
// partial sums included), one kernel of 512 threads for every rank -> now: r = 3 29.8 -> 20.6 us, r = 10 35.7 -> 24.2,
// r = 32 52.1 -> 40.4, r = 38 65.1 -> 63.2, r = 48 82.3 -> 77.4, r = 64 101.3 -> 89.7.
#include <cooperative_groups.h>

#include <type_traits>

#include "sfr_internal.h"

namespace cg = cooperative_groups;

namespace sfr {
namespace {

// Sizes of one padded rank RP: threads, the TM x TN outputs a thread takes of a float32 product, row strides of
// the float32 (16-byte aligned rows) and float64 (read along rows only) r x r arrays.
template <int RP_> struct Dim {
  static constexpr int RP = RP_, NT = RP == 64 ? 512 : RP == 32 ? 256 : RP == 16 ? 128 : 32;
  static constexpr int TM = RP == 64 ? 4 : RP == 32 ? 2 : 1, TN = RP == 64 ? 4 : 2;
  static constexpr int LD = RP + 4, LDD = RP;
  // One CTA per SM is all that is asked for: without that the registers of the functions the kernel calls were held to
  // 72 or 80, and the body kept its own on the stack around every call (grouped, padded rank 32: 88 bytes; with it 112 to
  // 140 registers and none).  FR-Nys 7805 x 7805, r = 21 10.6 -> 9.7 ms, 4096 x 2048, r = 32 from the host 10.2 -> 9.7.
  static constexpr int kBounds = per_sm(NT, 1);
};

__device__ __forceinline__ bool stopped(const DevState* st) { return *(volatile const int32_t*)&st->done != 0; }

// GB300 issues float64 arithmetic at about two operations per clock per SM, so every float64
// instruction that all 512 threads execute costs ~0.1 us.  The kernel therefore keeps float64 to
// the products and the few element-wise steps that need it, takes scalar float64 math on one
// thread, and does comparisons and float64 <-> float32 conversions with integer operations.

// |x| as an integer (ordered like |x| for non-NaN values; NaN sorts above +inf).
__device__ __forceinline__ long long abs_bits(double x) { return __double_as_longlong(x) & 0x7fffffffffffffffLL; }
constexpr long long kInfBits = 0x7ff0000000000000LL;

// float32 value of x 2^-e, rounded to nearest even, for |x 2^-e| < 2; results below the float32
// normal range flush to zero.  Integer operations only.
__device__ __forceinline__ float f64_to_f32_shift(double x, int e) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(x);
  const unsigned sign = (unsigned)(b >> 63) << 31;
  const int ex = (int)((b >> 52) & 0x7ff) - 1023 - e + 127;
  if (ex <= 0 || ((b >> 52) & 0x7ff) == 0) return __uint_as_float(sign);
  const unsigned long long mant = b & 0xfffffffffffffULL;
  const unsigned long long rest = mant & ((1ULL << 29) - 1);
  unsigned bits = ((unsigned)ex << 23) | (unsigned)(mant >> 29);
  if (rest > (1ULL << 28) || (rest == (1ULL << 28) && (bits & 1u))) bits += 1;  // carries into the exponent
  return __uint_as_float(bits | sign);
}

// Exact float64 value of f 2^e (f a normal float32 or zero; subnormals flush to zero).  Integer
// operations only.
__device__ __forceinline__ double f32_to_f64_shift(float f, int e) {
  const unsigned u = __float_as_uint(f);
  const unsigned ex = (u >> 23) & 0xff;
  const unsigned long long sign = (unsigned long long)(u >> 31) << 63;
  if (ex == 0) return __longlong_as_double((long long)sign);
  const unsigned long long b = sign | ((unsigned long long)(ex - 127 + 1023 + e) << 52) | ((unsigned long long)(u & 0x7fffffu) << 29);
  return __longlong_as_double((long long)b);
}
__device__ __forceinline__ double to_f64(double x) { return x; }
__device__ __forceinline__ double to_f64(float x) { return f32_to_f64_shift(x, 0); }

// C = epi(op(A) B) with float64 arithmetic, rows split across the cluster and broadcast through
// DSMEM.  A, B: float64 (row stride LDD).  C is float64 (LDD) or float (LD) and receives
// epi(i, j, (op(A) B)_ij).  C must not alias A or B.  On return every CTA holds the full product.
// PRE = false skips the barrier before the broadcast: allowed when no CTA has read C since the
// last cluster barrier.
template <typename DM, bool TA, bool PRE = true, typename TB, typename TCo, typename Epi>
__device__ __noinline__ void mm_dist(const double* A, const TB* B, TCo* C, int r, Epi epi) {
  constexpr int LDD = DM::LDD, ldb = sizeof(TB) == 8 ? DM::LDD : DM::LD, ldc = sizeof(TCo) == 8 ? DM::LDD : DM::LD;
  cg::cluster_group cl = cg::this_cluster();
  const int cs = (int)cl.num_blocks(), rank = (int)cl.block_rank();
  const int rpc = (r + cs - 1) / cs, i0 = min(r, rank * rpc), i1 = min(r, i0 + rpc);
  // (packed in r, not RP: a warp with idle lanes takes the float64 pipe as long as a full one: the kernel alone on
  // the float64 path, r = 5 23.6 -> 21.7 us, r = 10 34.5 -> 31.7)
  for (int e = threadIdx.x; e < (i1 - i0) * r; e += DM::NT) {
    const int i = i0 + e / r, j = e % r;
    // four independent chains (k mod 4) keep the float64 pipe busy with few warps per SM
    double acc[4] = {0.0, 0.0, 0.0, 0.0};
    int k = 0;
    for (; k + 4 <= r; k += 4)
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const double a = TA ? A[(k + q) * LDD + i] : A[i * LDD + k + q];
        acc[q] = fma(a, to_f64(B[(k + q) * ldb + j]), acc[q]);
      }
    for (; k < r; ++k) {
      const double a = TA ? A[k * LDD + i] : A[i * LDD + k];
      acc[0] = fma(a, to_f64(B[k * ldb + j]), acc[0]);
    }
    C[i * ldc + j] = epi(i, j, (acc[0] + acc[1]) + (acc[2] + acc[3]));
  }
  __syncthreads();
  if (cs > 1) {
    if (PRE) cl.sync();  // every CTA is past its earlier reads of C
    // push this CTA's rows to the other CTAs in 16-byte pieces (column pairs of float64 or quads of
    // float; the last piece of a row may carry columns >= r, which no product or loop reads)
    constexpr int per16 = 16 / sizeof(TCo);
    const int npc = (r + per16 - 1) / per16, per = (i1 - i0) * npc;
    for (int e = threadIdx.x; e < (cs - 1) * per; e += DM::NT) {
      const int q = 1 + e / per, w = e % per;
      const int i = i0 + w / npc, j = per16 * (w % npc);
      TCo* Cq = cl.map_shared_rank(C, (rank + q) % cs);
      *reinterpret_cast<float4*>(Cq + i * ldc + j) = *reinterpret_cast<const float4*>(C + i * ldc + j);
    }
    cl.sync();  // all rows have arrived everywhere
  }
}

// What a float32 product's value v at (i, j) becomes.
enum class Epi {
  kStore,      // C = v
  kScale,      // C = f v
  kAdd,        // C = X + v                         (Q <- Q + Q E)
  kOrtho,      // C = (3 I - v) / 2                 (Newton-Schulz factor)
  kBoth,       // C = v, Ct = v transposed          (the basis and its transpose)
  kLyapunov,   // C = v / (x_i + x_j)               (the Newton correction in the eigenbasis)
};
struct EpiArgs {
  float f = 1.f;
  const float* x = nullptr;  // kAdd: X (row stride LD); kLyapunov: x
  float* ct = nullptr;
};

// C = epi(op(A) diag(s) B) in float32 on the leading r4 x r4 blocks, r4 = r rounded up to 4 (s = nullptr: identity),
// TM x TN outputs per thread.  Operands move in 16-byte loads along k (A) and TN-wide ones (B); the sum over k
// runs in order.  Rows and columns r .. r4 of the operands are zeros (s, x finite there), and so are those of the
// result (kOrtho: 3/2 on the diagonal, which meets zeros only): the zero terms leave each sum as it is, and a rank that is
// no multiple of 4 needs neither a tail of the sum nor a second store path (r = 38, mean call of 60 iterations: 68.3 us with them,
// 64.0 without; r = 40: 63.7).
// C must not alias A or B.  One copy of the code for all steps (TA aside): the kernel runs each once
// or twice, and its instructions have to be fetched.
template <typename DM, bool TA>
__device__ __noinline__ void mmf(const float* A, const float* B, float* C, int r, Epi epi, const EpiArgs a_ = EpiArgs(),
                                 const float* s = nullptr) {
  constexpr int LD = DM::LD, TM = DM::TM, TN = DM::TN, NJ = DM::RP / TN;
  const int nb = (DM::RP / TM) * NJ;
  const int blk = threadIdx.x, i0 = TM * (blk / NJ), j0 = TN * (blk % NJ);
  const int r4 = (r + 3) & ~3;
  if (blk < nb && i0 < r4 && j0 < r4) {
    float acc[TM][TN];
#pragma unroll
    for (int x = 0; x < TM; ++x)
#pragma unroll
      for (int y = 0; y < TN; ++y) acc[x][y] = 0.f;
    auto load_a = [&](int k, float (&a)[TM][4]) {  // a[x][q] = op(A)(i0 + x, k + q) s(k + q)
      if constexpr (TA) {
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          if constexpr (TM == 4) {
            const float4 v = *reinterpret_cast<const float4*>(A + (k + q) * LD + i0);
            a[0][q] = v.x; a[1][q] = v.y; a[2][q] = v.z; a[3][q] = v.w;
          } else if constexpr (TM == 2) {
            const float2 v = *reinterpret_cast<const float2*>(A + (k + q) * LD + i0);
            a[0][q] = v.x; a[1][q] = v.y;
          } else {
            a[0][q] = A[(k + q) * LD + i0];
          }
        }
      } else {
#pragma unroll
        for (int x = 0; x < TM; ++x) {
          const float4 v = *reinterpret_cast<const float4*>(A + (i0 + x) * LD + k);
          a[x][0] = v.x; a[x][1] = v.y; a[x][2] = v.z; a[x][3] = v.w;
        }
      }
      if (s)
#pragma unroll
        for (int q = 0; q < 4; ++q)
#pragma unroll
          for (int x = 0; x < TM; ++x) a[x][q] *= s[k + q];
    };
    auto load_b = [&](int k, float (&b)[4][TN]) {
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        if constexpr (TN == 4) {
          const float4 v = *reinterpret_cast<const float4*>(B + (k + q) * LD + j0);
          b[q][0] = v.x; b[q][1] = v.y; b[q][2] = v.z; b[q][3] = v.w;
        } else {
          const float2 v = *reinterpret_cast<const float2*>(B + (k + q) * LD + j0);
          b[q][0] = v.x; b[q][1] = v.y;
        }
      }
    };
#pragma unroll(TM == 4 ? 1 : 2)
    for (int k = 0; k < r4; k += 4) {
      float a[TM][4], b[4][TN];
      load_a(k, a);
      load_b(k, b);
#pragma unroll
      for (int q = 0; q < 4; ++q)
#pragma unroll
        for (int x = 0; x < TM; ++x)
#pragma unroll
          for (int y = 0; y < TN; ++y) acc[x][y] = fmaf(a[x][q], b[q][y], acc[x][y]);
    }
    // (the step is chosen outside the loops: its code is fetched alone)
    auto each = [&](auto&& f) {
#pragma unroll
      for (int x = 0; x < TM; ++x) {
        float v[TN];
#pragma unroll
        for (int y = 0; y < TN; ++y) v[y] = acc[x][y] = f(i0 + x, j0 + y, acc[x][y]);
        float* c = C + (i0 + x) * LD + j0;
        if constexpr (TN == 4) *reinterpret_cast<float4*>(c) = make_float4(v[0], v[1], v[2], v[3]);
        else *reinterpret_cast<float2*>(c) = make_float2(v[0], v[1]);
      }
    };
    switch (epi) {
      case Epi::kStore: each([&](int, int, float v) { return v; }); break;
      case Epi::kScale: each([&](int, int, float v) { return v * a_.f; }); break;
      case Epi::kAdd: each([&](int i, int j, float v) { return a_.x[i * LD + j] + v; }); break;
      case Epi::kOrtho: each([&](int i, int j, float v) { return 0.5f * ((i == j ? 3.f : 0.f) - v); }); break;
      case Epi::kBoth:
        each([&](int, int, float v) { return v; });
#pragma unroll
        for (int y = 0; y < TN; ++y) {
          float* c = a_.ct + (j0 + y) * LD + i0;
          if constexpr (TM == 4) {
            *reinterpret_cast<float4*>(c) = make_float4(acc[0][y], acc[1][y], acc[2][y], acc[3][y]);
          } else {
#pragma unroll
            for (int x = 0; x < TM; ++x) c[x] = acc[x][y];
          }
        }
        break;
      case Epi::kLyapunov: each([&](int i, int j, float v) { return __fdividef(v, a_.x[i] + a_.x[j]); }); break;
    }
  }
  __syncthreads();
}

template <int RP> struct RxrSmem {  // 214 KB at RP = 64
  static constexpr int LD = Dim<RP>::LD, LDD = Dim<RP>::LDD;
  double G[RP * LDD];   // Gram of the thin factor (float64 sum of the partials); later B_bar
  double T[RP * LDD];   // T_hat = B Z_hat (Newton iterate); scratch vectors of the rank test
  double W[RP * LDD];   // B (until T_hat exists), then G T_hat
  float Gf[RP * LD];    // G 2^-eg (float32; the power of two keeps K = B G B finite)
  float Bf[RP * LD];    // B 2^-eb
  float QT[RP * LD];    // Q^T
  float Af[RP * LD];    // Q^T K Q / s (K = B G B), the Jacobi matrix, then the Newton correction in that basis
  float Q[RP * LD];     // approximate eigenbasis of K
  float F1[RP * LD];    // scratch
  float F2[RP * LD];    // scratch
  float lam[64], sq[64], isq[64];  // (all 64 read as two values per lane; entries past r unused)
  double red[64];
  unsigned mx[16];      // block-wide maxima, one slot each (bits of non-negative floats)
  float cs[RP / 2], sn[RP / 2];
  int pp[RP / 2], qq[RP / 2];
  double scale, inv_s, rs;  // s = trace(B G B) / r, 1 / s, 1 / sqrt(s)  (written by thread 0)
  float kn;                 // K's power-of-two scale over s
  int ok;
};

// Block-wide maxima of two 64-bit integers.
template <int NT>
__device__ __forceinline__ void block_max2_ll(long long& a, long long& b, double* red) {
  long long* rl = reinterpret_cast<long long*>(red);
  for (int o = 16; o > 0; o >>= 1) {
    a = max(a, __shfl_xor_sync(0xffffffffu, a, o));
    b = max(b, __shfl_xor_sync(0xffffffffu, b, o));
  }
  if (NT == 32) return;
  const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
  constexpr int NW = NT / 32;
  if (l == 0) rl[w] = a, rl[16 + w] = b;
  __syncthreads();
  a = l < NW ? rl[l] : 0LL;
  b = l < NW ? rl[16 + l] : 0LL;
  for (int o = 16; o > 0; o >>= 1) {
    a = max(a, __shfl_xor_sync(0xffffffffu, a, o));
    b = max(b, __shfl_xor_sync(0xffffffffu, b, o));
  }
}

// Block-wide maximum of non-negative floats through one shared slot (zero before); ends with a barrier.
__device__ __forceinline__ float block_max_f(float v, unsigned* slot) {
  const unsigned m = __reduce_max_sync(0xffffffffu, __float_as_uint(v));
  if ((threadIdx.x & 31) == 0) atomicMax(slot, m);
  __syncthreads();
  return __uint_as_float(*slot);
}

// Sum of x[0 .. r), r <= 64, by every warp for itself.
__device__ __forceinline__ float warp_sum64(const float* x, int stride, int r) {
  const int l = threadIdx.x & 31;
  float a = l < r ? x[l * stride] : 0.f, b = l + 32 < r ? x[(l + 32) * stride] : 0.f;
  for (int o = 16; o > 0; o >>= 1) {
    a += __shfl_xor_sync(0xffffffffu, a, o);
    b += __shfl_xor_sync(0xffffffffu, b, o);
  }
  return a + b;
}

// Statistics of the eigenvalue estimates, by every warp for itself: the largest (at least 0), the smallest
// (at most the largest), whether any is below f of the largest, whether any is not above 1e-14 of it.
struct LamStats {
  float hi, lo;
  bool small, bad;
};
__device__ __forceinline__ LamStats lam_stats(const float* lam, int r) {
  const int l = threadIdx.x & 31;
  const bool ia = l < r, ib = l + 32 < r;
  const float a = ia ? lam[l] : 0.f, b = ib ? lam[l + 32] : 0.f;
  LamStats s;
  s.hi = fmaxf(fmaxf(0.f, a), b);
  for (int o = 16; o > 0; o >>= 1) s.hi = fmaxf(s.hi, __shfl_xor_sync(0xffffffffu, s.hi, o));
  float n = -s.hi;
  if (ia) n = fmaxf(n, -a);
  if (ib) n = fmaxf(n, -b);
  for (int o = 16; o > 0; o >>= 1) n = fmaxf(n, __shfl_xor_sync(0xffffffffu, n, o));
  s.lo = -n;
  s.small = __any_sync(0xffffffffu, (ia && a < 1e-6f * s.hi) || (ib && b < 1e-6f * s.hi));
  s.bad = __any_sync(0xffffffffu, (ia && !(a > 1e-14f * s.hi)) || (ib && !(b > 1e-14f * s.hi))) || !(s.hi > 0.f);
  return s;
}

// Cyclic two-sided Jacobi on the symmetric n2 x n2 float matrix A (n2 even; rows/cols
// beyond r are zero), accumulating the rotations into Q (A_final = Q^T A_init Q).
// Round-robin ordering: n2/2 disjoint rotations per step, n2-1 steps per sweep.
template <typename DM>
__device__ __noinline__ void jacobi_f32(float* A, float* Q, int n2, int max_sweeps, double* red, float* cs, float* sn, int* pp,
                                        int* qq) {
  constexpr int LD = DM::LD, RPMAX = DM::RP, kThreads = DM::NT;
  const int np = n2 / 2;
  const bool pow2 = (np & (np - 1)) == 0;
  const int lg = 31 - __clz(np);
  for (int sweep = 0; sweep < max_sweeps; ++sweep) {
    // (summed by rows, a warp each, then over the rows by every warp: the sums decide how many sweeps run, so their order
    // must not depend on the number of threads, which differs between the kernels a rank may run in)
    const int lane_ = threadIdx.x & 31;
    float* rows = reinterpret_cast<float*>(red);  // [64] off-diagonal, [64] diagonal squares
    constexpr int NW_ = kThreads / 32, RPW = RPMAX / NW_;  // rows of a warp: their sums are taken side by side
    float v_[RPW];
#pragma unroll
    for (int u = 0; u < RPW; ++u) {
      const int i = (int)(threadIdx.x >> 5) + NW_ * u;
      const bool in = i < n2;
      const float a = in && lane_ < n2 ? A[i * LD + lane_] : 0.f;
      const float b = RPMAX > 32 && in && lane_ + 32 < n2 ? A[i * LD + lane_ + 32] : 0.f;
      v_[u] = lane_ == i ? 0.f : a * a;
      if (RPMAX > 32 && lane_ + 32 != i) v_[u] = fmaf(b, b, v_[u]);
      if (in && lane_ == (i & 31)) rows[64 + i] = i < 32 ? a * a : b * b;
    }
    for (int o = 16; o > 0; o >>= 1)
#pragma unroll
      for (int u = 0; u < RPW; ++u) v_[u] += __shfl_xor_sync(0xffffffffu, v_[u], o);
#pragma unroll
    for (int u = 0; u < RPW; ++u)
      if (lane_ == 0 && (int)(threadIdx.x >> 5) + NW_ * u < n2) rows[(threadIdx.x >> 5) + NW_ * u] = v_[u];
    __syncthreads();
    const float off = warp_sum64(rows, 1, n2), dia = warp_sum64(rows + 64, 1, n2);
    // off-diagonal mass below (1e-3)^2 of the diagonal: each float64 Newton step that follows
    // contracts the residual by about this factor (the next call refines the basis further)
    if (!(off > 1e-6 * dia)) break;
    if constexpr (RPMAX == 64) if (n2 == 64) {
      // 32 pairs: every warp computes all 32 rotations itself (lane k: pair k) and takes the
      // ones it needs by shuffles, so a step needs a single barrier; a thread rotates the two
      // 2 x 2 blocks (pair w + 16u, pair lane) of A and the four (row w + 16u v, pair lane)
      // entries pairs of Q, all loads first
      const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
      constexpr int NW = kThreads / 32;
      for (int step = 0; step < 63; ++step) {
        const int p = lane == 0 ? 63 : (step + lane) % 63, q = lane == 0 ? step : (step - lane + 63) % 63;
        const float apq = A[p * LD + q], app = A[p * LD + p], aqq = A[q * LD + q];
        float c = 1.f, sn_ = 0.f;
        if (apq * apq > 1e-18f * fabsf(app * aqq) && apq != 0.f) {
          // the angle only steers convergence (c^2 + s^2 = 1 holds for any t): fast approximations
          const float th = __fdividef(aqq - app, 2.f * apq);
          const float h = 1.f + th * th;
          const float t = fabsf(th) > 1e15f ? __fdividef(0.5f, th)
                                           : __fdividef(copysignf(1.f, th), fabsf(th) + h * rsqrtf(h));
          c = rsqrtf(1.f + t * t);
          sn_ = t * c;
        }
        float v[2][4], x[4][2];
        int k1p[2], k1q[2];
        float c1[2], s1[2];
#pragma unroll
        for (int u = 0; u < 2; ++u) {
          const int k1 = warp + NW * u;
          c1[u] = __shfl_sync(0xffffffffu, c, k1);
          s1[u] = __shfl_sync(0xffffffffu, sn_, k1);
          k1p[u] = __shfl_sync(0xffffffffu, p, k1);
          k1q[u] = __shfl_sync(0xffffffffu, q, k1);
        }
        __syncthreads();  // every warp has read the pivots of this step
#pragma unroll
        for (int u = 0; u < 2; ++u) {
          v[u][0] = A[k1p[u] * LD + p]; v[u][1] = A[k1p[u] * LD + q];
          v[u][2] = A[k1q[u] * LD + p]; v[u][3] = A[k1q[u] * LD + q];
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const int j = warp + NW * u;
          x[u][0] = Q[j * LD + p];
          x[u][1] = Q[j * LD + q];
        }
        if (sn_ != 0.f || s1[0] != 0.f || s1[1] != 0.f) {
#pragma unroll
          for (int u = 0; u < 2; ++u) {
            const float ra = c1[u] * v[u][0] - s1[u] * v[u][2], rb = c1[u] * v[u][1] - s1[u] * v[u][3];
            const float rc = s1[u] * v[u][0] + c1[u] * v[u][2], rd = s1[u] * v[u][1] + c1[u] * v[u][3];
            A[k1p[u] * LD + p] = c * ra - sn_ * rb;
            A[k1p[u] * LD + q] = sn_ * ra + c * rb;
            A[k1q[u] * LD + p] = c * rc - sn_ * rd;
            A[k1q[u] * LD + q] = sn_ * rc + c * rd;
          }
        }
        if (sn_ != 0.f) {
#pragma unroll
          for (int u = 0; u < 4; ++u) {
            const int j = warp + NW * u;
            Q[j * LD + p] = c * x[u][0] - sn_ * x[u][1];
            Q[j * LD + q] = sn_ * x[u][0] + c * x[u][1];
          }
        }
        __syncthreads();
      }
      continue;
    }
    for (int step = 0; step < n2 - 1; ++step) {
      if (threadIdx.x < np) {
        const int k = threadIdx.x;
        int p, q;
        if (k == 0) { p = n2 - 1; q = step; }
        else { p = (step + k) % (n2 - 1); q = (step - k + n2 - 1) % (n2 - 1); }
        const float apq = A[p * LD + q], app = A[p * LD + p], aqq = A[q * LD + q];
        float c = 1.f, s = 0.f;
        if (apq * apq > 1e-18f * fabsf(app * aqq) && apq != 0.f) {
          const float th = __fdividef(aqq - app, 2.f * apq);
          const float h = 1.f + th * th;
          float t;
          if (fabsf(th) > 1e15f) t = __fdividef(0.5f, th);
          else t = __fdividef(copysignf(1.f, th), fabsf(th) + h * rsqrtf(h));
          c = rsqrtf(1.f + t * t);
          s = t * c;
        }
        cs[k] = c; sn[k] = s; pp[k] = p; qq[k] = q;
      }
      __syncthreads();
      // A <- J^T A J in one phase: the pairs partition the indices, so each 2 x 2 block
      // (rows {p1, q1}, columns {p2, q2}) is touched by exactly one row and one column rotation.
      // Each thread takes up to four blocks, loads all of them, then rotates and stores.
      {
        constexpr int MB = ((RPMAX / 2) * (RPMAX / 2) + kThreads - 1) / kThreads;
        float v[MB][4];
        int pos[MB][4];
        float rc[MB][4];
        bool act[MB];
#pragma unroll
        for (int u = 0; u < MB; ++u) {
          const int e = threadIdx.x + u * kThreads;
          act[u] = e < np * np;
          if (!act[u]) continue;
          const int k1 = pow2 ? (e >> lg) : e / np, k2 = pow2 ? (e & (np - 1)) : e % np;
          rc[u][0] = cs[k1]; rc[u][1] = sn[k1];
          rc[u][2] = cs[k2];
          rc[u][3] = sn[k2];
          act[u] = !(rc[u][1] == 0.f && rc[u][3] == 0.f);
          const int p1 = pp[k1], q1 = qq[k1], p2 = pp[k2], q2 = qq[k2];
          pos[u][0] = p1 * LD + p2; pos[u][1] = p1 * LD + q2; pos[u][2] = q1 * LD + p2; pos[u][3] = q1 * LD + q2;
#pragma unroll
          for (int w = 0; w < 4; ++w) v[u][w] = A[pos[u][w]];
        }
#pragma unroll
        for (int u = 0; u < MB; ++u) {
          if (!act[u]) continue;
          const float c1 = rc[u][0], s1 = rc[u][1], c2 = rc[u][2], s2 = rc[u][3];
          const float ra = c1 * v[u][0] - s1 * v[u][2], rb = c1 * v[u][1] - s1 * v[u][3];
          const float rcc = s1 * v[u][0] + c1 * v[u][2], rd = s1 * v[u][1] + c1 * v[u][3];
          A[pos[u][0]] = c2 * ra - s2 * rb;
          A[pos[u][1]] = s2 * ra + c2 * rb;
          A[pos[u][2]] = c2 * rcc - s2 * rd;
          A[pos[u][3]] = s2 * rcc + c2 * rd;
        }
      }
      // Q <- Q J, up to eight (row, pair) items per thread, loads first
      {
        constexpr int MQ = (RPMAX / 2 * RPMAX + kThreads - 1) / kThreads;
        float x2[MQ][2], cq[MQ][2];
        int qp[MQ][2];
        bool act[MQ];
#pragma unroll
        for (int u = 0; u < MQ; ++u) {
          const int e = threadIdx.x + u * kThreads;
          act[u] = e < np * n2;
          if (!act[u]) continue;
          const int k = pow2 ? (e & (np - 1)) : e % np, j = pow2 ? (e >> lg) : e / np;
          cq[u][0] = cs[k];
          cq[u][1] = sn[k];
          act[u] = cq[u][1] != 0.f;
          qp[u][0] = j * LD + (pp[k]);
          qp[u][1] = j * LD + (qq[k]);
          x2[u][0] = Q[qp[u][0]]; x2[u][1] = Q[qp[u][1]];
        }
#pragma unroll
        for (int u = 0; u < MQ; ++u) {
          if (!act[u]) continue;
          const float c = cq[u][0], sv = cq[u][1];
          Q[qp[u][0]] = c * x2[u][0] - sv * x2[u][1];
          Q[qp[u][1]] = sv * x2[u][0] + c * x2[u][1];
        }
      }
      __syncthreads();
    }
  }
}

// A = (B Q)^T G (B Q) f = f Q^T K Q for the float32 copies Bf, Gf (three products; K itself is never formed).
template <typename DM>
__device__ __forceinline__ void gram_in_basis(const float* Bf, const float* Gf, const float* Q, float* A, float* F1, float* F2,
                                              int r, float f) {
  mmf<DM, false>(Bf, Q, F1, r, Epi::kStore);   // B Q
  mmf<DM, false>(Gf, F1, F2, r, Epi::kStore);  // G B Q
  EpiArgs e;
  e.f = f;
  mmf<DM, true>(F1, F2, A, r, Epi::kScale, e);  // (B Q)^T G B Q
}

// One first-order eigenbasis refinement round for a nearly diagonal f A = Q^T K Q / s (float32):
// Q <- Q (I + E), E_pq = A_pq / (A_qq - A_pp) for p != q (the small-angle Jacobi rotation of
// every pair at once), then one Newton-Schulz re-orthonormalisation, and the second-order
// eigenvalue estimates lam_p = f (A_pp - sum_q A_pq E_pq) (A itself is not recomputed; f is a power of two).  Pairs with
// (relative) gaps below 1e-5 are left alone, since any basis of a cluster serves the Newton
// preconditioner.  Returns max |E|; above 0.25 (A not close enough to diagonal for the
// first-order step) nothing is changed, else Q holds the refined basis and QT its transpose.
template <typename DM>
__device__ __noinline__ float refine_round(float* Q, float* QT, const float* A, float f, float* F1, float* F2,
                                           float* lam, int r, unsigned* slot) {
  constexpr int LD = DM::LD, RP = DM::RP;
  float big = 0.f;
  for (int e = threadIdx.x; e < r * RP; e += DM::NT) {
    const int p = e / RP, q = e % RP;
    if (q >= r) continue;
    float v = 0.f;
    if (p != q) {
      const float gap = A[q * LD + q] - A[p * LD + p];
      const float scl = fmaxf(fabsf(A[p * LD + p]), fabsf(A[q * LD + q]));
      if (fabsf(gap) > 1e-5f * scl) v = __fdividef(A[p * LD + q], gap);  // first-order term: 2 ulp is ample
    }
    F1[p * LD + q] = v;
    big = fmaxf(big, fabsf(v));
  }
  big = block_max_f(big, slot);
  if (!(big <= 0.25f)) return big;
  // lam_p = A_pp - sum_q A_pq E_pq: one warp per row
  const int lane = threadIdx.x & 31;
  for (int p = threadIdx.x >> 5; p < r; p += DM::NT / 32) {
    float acc = 0.f;
    for (int q = lane; q < r; q += 32) acc = fmaf(A[p * LD + q], F1[p * LD + q], acc);
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
    if (lane == 0) lam[p] = (A[p * LD + p] - acc) * f;
  }
  EpiArgs e;
  e.x = Q;
  mmf<DM, false>(Q, F1, F2, r, Epi::kAdd, e);       // Q (I + E)
  mmf<DM, true>(F2, F2, F1, r, Epi::kOrtho);        // (3 I - Q^T Q) / 2
  e.ct = QT;
  mmf<DM, false>(F2, F1, Q, r, Epi::kBoth, e);      // Q (3 I - Q^T Q) / 2
  return big;
}

static_assert(sizeof(RxrSmem<64>) <= 232448, "shared memory per CTA");

// Epilogues of mm_dist: the product itself, or I - product / s rounded to float32.
struct PlainEpi {
  __device__ double operator()(int, int, double v) const { return v; }
};
struct ResidEpi {
  double inv_s;
  __device__ float operator()(int i, int j, double v) const { return (float)((i == j ? 1.0 : 0.0) - v * inv_s); }
};

__device__ void fail(DevState* st, int code) {
  if (threadIdx.x == 0 && cg::this_cluster().block_rank() == 0) { st->status = code; st->done = 1; }
}

// Unbiased binary exponent of the largest |x| whose bits are `bits` (0 for 0).
__device__ __forceinline__ int exponent_of(long long bits) { return bits ? (int)(bits >> 52) - 1023 : 0; }

// v_side = false: T_U = B (B G_P B)^{-1/2}.
// v_side = true:  T_V = B (B G_W B)^{-1/2}, B <- Sym(G_W T_V), T_C = T_V B.
//
// With K = B G B and s = trace(K) / r, let Z be (K / s)^{-1/2}; then T = B Z / sqrt(s).  The kernel
// carries T_hat = B Z instead of Z: Newton's residual for Z K Z = I is
//     R = I - Z K Z = I - T_hat^T (G T_hat) / s,
// so float64 products form T_hat, W = G T_hat and T_hat^T W only, and K itself is needed in
// float32 alone (for the eigenbasis that preconditions Newton).  A Newton correction Delta of Z
// (float32, small) moves T_hat by B Delta and W by G B Delta, formed in float32: their rounding
// is float32-relative to the correction, and the next residual is formed in float64 again.
// float64: G, B, T_hat, W, R, B_bar, T_C.  float32: K, the eigenbasis, eigenvalue estimates, Z0
// and the Newton corrections, which only steer the iteration.  The mixed path also forms the
// starting T_hat = B Z0 and T_C in float32 (its U, V and C are float32).  Outputs are written by
// rows, each CTA of the cluster its own slice.
template <int RP>
__device__ __forceinline__ void rxr_body(const VGrid& vg__, const double* __restrict__ Gg, int rp, int r,
                                         double* __restrict__ Bg, double* __restrict__ Tout,
                                         double* __restrict__ TCout, const float* __restrict__ Qin,
                                         float* __restrict__ Qeig, int v_side, int mixed, DevState* st) {
  pdl_enter();
  SFR_VGRID(vg__);
  if (stopped(st)) return;
  using DM = Dim<RP>;
  constexpr int NT = DM::NT, LD = DM::LD, LDD = DM::LDD;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  RxrSmem<RP>& S = *reinterpret_cast<RxrSmem<RP>*>(smem_raw);
  cg::cluster_group cl = cg::this_cluster();
  const int tid = threadIdx.x;
  const int cs = (int)cl.num_blocks(), crank = (int)cl.block_rank();
  const bool writer = crank == 0;
  const int rpc = (r + cs - 1) / cs, row0 = min(r, crank * rpc), row1 = min(r, row0 + rpc);  // own rows
  const int n2 = (r + 1) & ~1;  // Jacobi works on an even size (row / column r zero when r is odd)
  float* Q = S.Q;
  // 1. G and B in float64 (B in W until T_hat exists), their power-of-two-scaled float32 copies,
  //    and the warm-start eigenbasis (Qin), all with zeros past r (mmf)
  constexpr int PER = RP * RP / NT;
  {
    double gv[PER], bv[PER];
    float qv[PER];
    long long gmax = 0, bmax = 0;
#pragma unroll
    for (int q = 0; q < PER; ++q) {
      const int e = tid + q * NT, i = e / RP, j = e % RP;
      const bool in = i < r && j < r;
      gv[q] = in ? Gg[i * rp + j] : 0.0;
      bv[q] = in ? Bg[i * rp + j] : 0.0;
      qv[q] = in ? Qin[i * rp + j] : 0.f;
    }
    if (tid < 16) S.mx[tid] = 0;
#pragma unroll
    for (int q = 0; q < PER; ++q) {
      gmax = max(gmax, abs_bits(gv[q]));
      bmax = max(bmax, abs_bits(bv[q]));
    }
    block_max2_ll<NT>(gmax, bmax, S.red);
    if (gmax >= kInfBits || bmax >= kInfBits || bmax == 0) { fail(st, SFR_E_NAN); return; }
    const int eg_ = exponent_of(gmax), eb_ = exponent_of(bmax);
    if (tid == 0) S.pp[0] = eg_, S.qq[0] = eb_;
#pragma unroll
    for (int q = 0; q < PER; ++q) {
      const int e = tid + q * NT, i = e / RP, j = e % RP;
      S.G[i * LDD + j] = gv[q];
      S.W[i * LDD + j] = bv[q];
      S.Gf[i * LD + j] = f64_to_f32_shift(gv[q], eg_);
      S.Bf[i * LD + j] = f64_to_f32_shift(bv[q], eb_);
      Q[i * LD + j] = qv[q];
    }
  }
  __syncthreads();
  const int eg = S.pp[0], eb = S.qq[0];
  // 2. A = Q^T K Q in the warm-start basis Q (float32, from the scaled copies: K 2^-(eg + 2 eb));
  //    s = trace(K) / r = trace(A) / r; A's scale over s is the power of two kn
  gram_in_basis<DM>(S.Bf, S.Gf, Q, S.Af, S.F1, S.F2, r, 1.f);
  const float trf = warp_sum64(S.Af, LD + 1, r);
  if (tid == 0) {
    // s = 2^(2k), the even power of two nearest below trace(B G B) / r (within a factor 4 of
    // it), so that 1 / s and 1 / sqrt(s) are exact and need no float64 division or square root;
    // A is scaled by K's power-of-two scale over s, exactly, so that its eigenvalues are those
    // of K / s.
    int e1 = 0;
    frexpf(trf / (float)r, &e1);  // trf / r = f 2^e1, f in [0.5, 1)
    const int tot = e1 + eg + 2 * eb, k = (tot >= 0 ? tot : tot - 1) / 2;  // floor(tot / 2)
    S.ok = trf > 0.f && trf < 3e38f && 2 * k > -1000 && 2 * k < 1000;
    auto pow2 = [](int e) { return __longlong_as_double((long long)(1023 + e) << 52); };
    S.scale = pow2(2 * k);
    S.inv_s = pow2(-2 * k);
    S.rs = pow2(-k);
    S.kn = ldexpf(1.f, eg + 2 * eb - 2 * k);
  }
  __syncthreads();
  if (!S.ok) { fail(st, SFR_E_NAN); return; }
  const float kn = S.kn;
  // 3. eigenbasis: refine the previous basis to first order (cheap) while its rotation is small;
  //    a round whose rotation is at most 1e-3 leaves the basis accurate to ~1e-6 and is the last,
  //    a larger one is followed by a fresh A; float32 Jacobi sweeps only when that does not converge
  bool accepted = false;
  float fa = kn;  // scale of A
  int slot = 0;
  for (int round = 0; round < 3 && !accepted; ++round) {
    const float big = refine_round<DM>(Q, S.QT, S.Af, fa, S.F1, S.F2, S.lam, r, S.mx + slot++);
    if (!(big <= 0.25f)) break;                      // A unchanged, Q unchanged
    accepted = big <= 1e-3f;
    if (!accepted) {
      gram_in_basis<DM>(S.Bf, S.Gf, Q, S.Af, S.F1, S.F2, r, kn);
      fa = 1.f;
    }
  }
  const bool rotated = !accepted;
  if (rotated) {
    // A in K / s's scale (row and column r of an odd rank are zeros in A and in Q: no rotation touches them)
    for (int e = tid; e < r * RP; e += NT) {
      const int i = e / RP, j = e % RP;
      if (j < r) S.Af[i * LD + j] *= fa;
    }
    __syncthreads();
    jacobi_f32<DM>(S.Af, Q, n2, 10, S.red, S.cs, S.sn, S.pp, S.qq);
    // re-orthonormalise the float basis: Q <- Q (3I - Q^T Q) / 2
    mmf<DM, true>(Q, Q, S.F1, r, Epi::kOrtho);
    EpiArgs ec;
    ec.ct = S.QT;
    mmf<DM, false>(Q, S.F1, S.F2, r, Epi::kBoth, ec);
    for (int e = tid; e < r * RP; e += NT)
      if (e / RP < r && e % RP < r) Q[(e / RP) * LD + e % RP] = S.F2[(e / RP) * LD + e % RP];
    // 4. eigenvalue estimates after Jacobi: the diagonal of A (Rayleigh quotients of the basis)
    for (int p = tid; p < r; p += NT) S.lam[p] = S.Af[p * LD + p];
    __syncthreads();
  }
  // (after a refinement round lam holds its second-order estimates); those far below the largest
  // are recomputed in float64 for the rank test (Eq. 9 needs rank r)
  LamStats ls = lam_stats(S.lam, r);
  if (ls.small) {
    if (rotated) {
      // Jacobi stopped at a 1e-3 off-diagonal, so a basis vector of a tiny eigenvalue still mixes
      // ~1e-3 of the large ones and its Rayleigh quotient sits near 1e-6 hi: two first-order rounds
      // (near-degenerate pairs are skipped) bring the mixing down to float32 rounding first.
      __syncthreads();
      for (int round = 0; round < 2; ++round) {
        gram_in_basis<DM>(S.Bf, S.Gf, Q, S.Af, S.F1, S.F2, r, kn);
        if (!(refine_round<DM>(Q, S.QT, S.Af, 1.f, S.F1, S.F2, S.lam, r, S.mx + slot++) <= 0.25f)) {
          for (int p = tid; p < r; p += NT) S.lam[p] = S.Af[p * LD + p];
          break;
        }
      }
      __syncthreads();
      ls.hi = lam_stats(S.lam, r).hi;
    }
    // A float32 eigenvector carries components of about 1e-7 along the large eigenvectors, which
    // alone would add ~1e-14 hi to its Rayleigh quotient (the rank threshold): project them out in
    // float64 first (q <- q - Q_L Q_L^T q over the columns of large eigenvalues), then take
    // q^T K q / (s q^T q) = (B q)^T G (B q) / (s q^T q) with float64 matrix-vector products.
    const float hi = ls.hi;
    double* qs = S.T;            // the vector (T_hat is free until step 6)
    double* cf = S.T + LDD;      // its coefficients on the large eigenvectors
    double* bq = S.T + 2 * LDD;  // B q
    __syncthreads();
    for (int p = 0; p < r; ++p) {
      if (!(S.lam[p] < 1e-6f * hi)) continue;  // uniform: lam is in shared memory
      if (tid < r) qs[tid] = (double)Q[tid * LD + p];
      if (tid < 4) S.red[tid] = 0.0;
      __syncthreads();
      if (tid < r) {
        double c = 0.0;
        if (!(S.lam[tid] < 1e-6f * hi))
          for (int k = 0; k < r; ++k) c = fma((double)Q[k * LD + tid], qs[k], c);
        cf[tid] = c;
      }
      __syncthreads();
      double qi = 0.0;
      if (tid < r) {
        qi = qs[tid];
        for (int q2 = 0; q2 < r; ++q2) qi = fma(-cf[q2], (double)Q[tid * LD + q2], qi);
      }
      __syncthreads();
      if (tid < r) qs[tid] = qi;
      __syncthreads();
      if (tid < r) {
        double v = 0.0;
        for (int k = 0; k < r; ++k) v = fma(S.W[tid * LDD + k], qs[k], v);  // (B q)_tid
        bq[tid] = v;
      }
      __syncthreads();
      double num = 0.0, den = 0.0;
      if (tid < r) {
        double gq = 0.0;
        for (int k = 0; k < r; ++k) gq = fma(S.G[tid * LDD + k], bq[k], gq);  // (G B q)_tid
        num = bq[tid] * gq;
        den = qi * qi;
      }
      if (tid < 64) {  // r <= 64: the first two warps hold every term
        for (int o = 16; o > 0; o >>= 1) {
          num += __shfl_xor_sync(0xffffffffu, num, o);
          den += __shfl_xor_sync(0xffffffffu, den, o);
        }
        if ((tid & 31) == 0) S.red[tid >> 4] = num, S.red[(tid >> 4) + 1] = den;
      }
      __syncthreads();
      if (tid == 0) S.lam[p] = (float)((S.red[0] + S.red[2]) / (S.red[1] + S.red[3]) * S.inv_s);
      __syncthreads();
    }
    const LamStats l2 = lam_stats(S.lam, r);
    // (thresholds against the estimate of the largest taken before the recomputation)
    ls.lo = fminf(hi, l2.lo);
    bool bad = false;
    for (int p = 0; p < r; ++p) bad |= !(S.lam[p] > 1e-14f * hi);
    ls.bad = bad || !(hi > 0.f);
  }
  if (writer && tid == 0) {
    if (v_side) st->lam_min_v = (double)ls.lo * S.scale; else st->lam_min_u = (double)ls.lo * S.scale;
  }
  if (ls.bad) { fail(st, SFR_E_RANK); return; }
  for (int p = tid; p < ((r + 3) & ~3); p += NT) {  // (past r: finite factors of zeros)
    const float sq = p < r ? sqrtf(S.lam[p]) : 1.f;
    S.sq[p] = sq;
    S.isq[p] = 1.f / sq;
  }
  float* QT = S.QT;
  __syncthreads();
  // 5. Z0 = Q diag(lambda^{-1/2}) Q^T (float32 start; Newton below brings it to float64 accuracy)
  mmf<DM, false>(Q, QT, S.F1, r, Epi::kStore, EpiArgs(), S.isq);
  for (int e = tid; e < r * RP; e += NT) {
    const int i = e / RP, j = e % RP;
    if (i < r && j < r) S.F2[i * LD + j] = 0.5f * (S.F1[i * LD + j] + S.F1[j * LD + i]);
  }
  __syncthreads();
  // 6. T_hat = B Z0.  Float64 path: float64 products of B with the float32 values of Z0, rows
  //    split across the cluster.  Mixed path: a float32 product of the scaled copy of B, in every
  //    CTA.  Newton below corrects the symmetric part of Z only, so the float32 rounding of T_hat
  //    stays as a rotation of the polar factor of about 1e-7, the size of the mixed path's own
  //    rounding of U and V.
  const PlainEpi plain;
  if (mixed) {
    mmf<DM, false>(S.Bf, S.F2, S.F1, r, Epi::kStore);  // B Z0 2^-eb
    for (int e = tid; e < r * RP; e += NT) {
      const int i = e / RP, j = e % RP;
      if (j < r) S.T[i * LDD + j] = f32_to_f64_shift(S.F1[i * LD + j], eb);
    }
    __syncthreads();
    if (cs > 1) cl.sync();  // every CTA is past its reads of W (still B) before W rows arrive
  } else {
    mm_dist<DM, false>(S.W, S.F2, S.T, r, plain);
  }
  // 7. Newton steps on Z K Z = I: R = I - T_hat^T (G T_hat) / s in float64, correction in float32
  bool w_stale = false;  // W lags T_hat by G (B Delta)
  for (int it = 0; it < 6; ++it) {
    // W was last read by the previous product (T_hat0 = B Z0 or the residual), F1 by this CTA
    // alone before that product's closing barrier: neither needs a barrier before its broadcast
    mm_dist<DM, false, false>(S.G, S.T, S.W, r, plain);               // W = G T_hat
    mm_dist<DM, true, false>(S.T, S.W, S.F1, r, ResidEpi{S.inv_s});  // I - Z K Z, rounded to float32
    w_stale = false;
    float rmax = 0.f;
    for (int e = tid; e < r * RP; e += NT) {  // R = Sym(I - Z K Z)
      const int i = e / RP, j = e % RP;
      if (j >= r) continue;
      const float v = S.F1[i * LD + j];
      rmax = fmaxf(rmax, fabsf(v));
      S.F2[i * LD + j] = 0.5f * (v + S.F1[j * LD + i]);
    }
    const float rm = block_max_f(rmax, S.mx + slot++);
    if (!(rm == rm)) { fail(st, SFR_E_NAN); return; }
    if (rm < 4e-16f * r) break;
    // The step below leaves a residual of about (eigenbasis error + float32 rounding of the
    // correction) x rm + O(rm^2): from rm < 3e-6 about 1e-11 (mixed path, whose Gram carries
    // float32 rounding), from rm < 1e-7 about 1e-14 (float64 path), so stop without forming it again
    // and update only this CTA's rows of T_hat (the rows it writes).
    const bool last = rm < (mixed ? 3e-6f : 1e-7f) || it == 5;
    EpiArgs el;
    el.x = S.sq;
    mmf<DM, false>(S.F2, Q, S.F1, r, Epi::kStore);            // R Q
    mmf<DM, true>(Q, S.F1, S.Af, r, Epi::kLyapunov, el);      // Dt = Q^T R Q / (sqrt(lam_p) + sqrt(lam_q))
    mmf<DM, false>(S.Af, QT, S.F2, r, Epi::kStore);           // Dt Q^T
    mmf<DM, false>(Q, S.F2, S.F1, r, Epi::kStore);            // Q Dt Q^T
    for (int e = tid; e < r * RP; e += NT) {
      const int i = e / RP, j = e % RP;
      if (j < r) S.F2[i * LD + j] = 0.5f * (S.F1[i * LD + j] + S.F1[j * LD + i]);  // Delta (symmetric)
    }
    __syncthreads();
    mmf<DM, false>(S.Bf, S.F2, S.F1, r, Epi::kStore);         // B Delta 2^-eb
    const int lo = last ? row0 : 0, hi = last ? row1 : r;
    for (int e = lo * RP + tid; e < hi * RP; e += NT) {
      const int i = e / RP, j = e % RP;
      if (j < r) S.T[i * LDD + j] += f32_to_f64_shift(S.F1[i * LD + j], eb);
    }
    __syncthreads();
    w_stale = true;
    if (last) break;
  }
  // 8. T = B (B G B)^{-1/2} = T_hat / sqrt(s): this CTA's rows, and its rows of the basis
  const double rs = S.rs;
  for (int e = row0 * rp + tid; e < row1 * rp; e += NT) {
    const int i = e / rp, j = e % rp;
    Tout[e] = j < r ? S.T[i * LDD + j] * rs : 0.0;
    Qeig[e] = j < r ? Q[i * LD + j] : (i == j ? 1.f : 0.f);
  }
  if (writer)
    for (int e = r * rp + tid; e < rp * rp; e += NT) {  // padding rows
      const int i = e / rp, j = e % rp;
      Tout[e] = 0.0;
      Qeig[e] = i == j ? 1.f : 0.f;
    }
  if (!v_side) return;
  // 9. B_bar = Sym(G_W T_V) (Eq. 10 with W = X^T U_bar) = Sym(G T_hat) / sqrt(s), T_C = T_V B_bar.
  //    W lags T_hat by the last correction: W + G (B Delta), the latter in float32.  Every CTA forms
  //    its rows of B_bar and sends them to the others (nobody reads G after the last W product).
  if (w_stale) mmf<DM, false>(S.Gf, S.F1, S.F2, r, Epi::kStore);  // G B Delta 2^-(eg + eb)
  for (int e = tid; e < (row1 - row0) * RP; e += NT) {
    const int i = row0 + e / RP, j = e % RP;
    if (j >= r) continue;
    double v = S.W[i * LDD + j] + S.W[j * LDD + i];
    if (w_stale) v += f32_to_f64_shift(S.F2[i * LD + j] + S.F2[j * LD + i], eg + eb);
    S.G[i * LDD + j] = 0.5 * rs * v;
  }
  __syncthreads();
  if (cs > 1) {
    const int npc = (r + 1) / 2, per = (row1 - row0) * npc;
    for (int e = tid; e < (cs - 1) * per; e += NT) {
      const int q = 1 + e / per, w = e % per;
      const int i = row0 + w / npc, j = 2 * (w % npc);
      double* Gq = cl.map_shared_rank(S.G, (crank + q) % cs);
      *reinterpret_cast<double2*>(Gq + i * LDD + j) = *reinterpret_cast<const double2*>(S.G + i * LDD + j);
    }
    cl.sync();
  }
  // this CTA's rows: B_bar, and T_C = T_V B_bar = (T_hat rows) B_bar / sqrt(s).  T_C only forms
  // C = W T_C, which the mixed path stores in float32: there float32 products suffice.
  if (mixed) {
    for (int e = tid; e < r * RP; e += NT) {
      const int i = e / RP, j = e % RP;
      if (j >= r) continue;
      S.Af[i * LD + j] = f64_to_f32_shift(S.G[i * LDD + j], 0);
      if (i >= row0 && i < row1) S.F2[i * LD + j] = f64_to_f32_shift(S.T[i * LDD + j], 0);
    }
    __syncthreads();
  }
  for (int e = row0 * rp + tid; e < row1 * rp; e += NT) {
    const int i = e / rp, j = e % rp;
    double tc = 0.0;
    if (j < r && mixed) {
      float acc[4] = {0.f, 0.f, 0.f, 0.f};
      int k = 0;
      for (; k + 4 <= r; k += 4)
#pragma unroll
        for (int q = 0; q < 4; ++q) acc[q] = fmaf(S.F2[i * LD + k + q], S.Af[(k + q) * LD + j], acc[q]);
      for (; k < r; ++k) acc[0] = fmaf(S.F2[i * LD + k], S.Af[k * LD + j], acc[0]);
      tc = f32_to_f64_shift((acc[0] + acc[1]) + (acc[2] + acc[3]), 0);
    } else if (j < r) {
      double acc[4] = {0.0, 0.0, 0.0, 0.0};
      int k = 0;
      for (; k + 4 <= r; k += 4)
#pragma unroll
        for (int q = 0; q < 4; ++q) acc[q] = fma(S.T[i * LDD + k + q], S.G[(k + q) * LDD + j], acc[q]);
      for (; k < r; ++k) acc[0] = fma(S.T[i * LDD + k], S.G[k * LDD + j], acc[0]);
      tc = (acc[0] + acc[1]) + (acc[2] + acc[3]);
    }
    Bg[e] = j < r ? S.G[i * LDD + j] : 0.0;
    TCout[e] = j < r ? tc * rs : 0.0;
  }
  if (writer)
    for (int e = r * rp + tid; e < rp * rp; e += NT) {
      Bg[e] = 0.0;
      TCout[e] = 0.0;
    }
}


}  // namespace

// Cluster size of the r x r kernel: one CTA for r <= 16 (a whole float64 product takes it about a
// microsecond, no more than the cluster barriers of a split one); above, 16 CTAs (non-portable
// size) when the device accepts it with this kernel's shared memory, else 8, else a single CTA.  The
// result does not depend on it (every float64 product element is one thread's loop; the float32 work is redundant).
template <int RP>
static int rxr_cluster_size() {
  if (RP <= 16) return 1;
  static const int best = [] {
    constexpr size_t smem = sizeof(RxrSmem<RP>);
    constexpr int NT = Dim<RP>::NT;
    auto kern = body_kernel_of<&rxr_body<RP>, Dim<RP>::kBounds>();
    if (cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess) cudaGetLastError();
    if (set_smem_attr<body_kernel_of<&rxr_body<RP>, Dim<RP>::kBounds>()>(smem) != cudaSuccess) cudaGetLastError();
    for (int cs : {16, 8}) {
      cudaLaunchConfig_t cfg = {};
      cfg.gridDim = dim3(cs);
      cfg.blockDim = dim3(NT);
      cfg.dynamicSmemBytes = smem;
      cudaLaunchAttribute at;
      at.id = cudaLaunchAttributeClusterDimension;
      at.val.clusterDim.x = cs;
      at.val.clusterDim.y = 1;
      at.val.clusterDim.z = 1;
      cfg.attrs = &at;
      cfg.numAttrs = 1;
      int nclusters = 0;
      if (cudaOccupancyMaxActiveClusters(&nclusters, kern, &cfg) == cudaSuccess && nclusters > 0) return cs;
      cudaGetLastError();
    }
    return 1;
  }();
  return best;
}

cudaError_t launch_rxr(const Shape& s, const Buffers& b, bool v_side, cudaStream_t st, bool fp64) {
  const double* parts = v_side ? b.GWpart : b.GPpart;
  const int count = v_side ? s.gw_blocks : s.gp_blocks;
  cudaError_t e = launch_reduce_parts(parts, count, s.rp * s.rp, b.Gsum, b.st, st);
  if (e != cudaSuccess) return e;
  // warm start: the U side from its own basis of the previous iteration; the V side from the U
  // side's basis of this iteration (both K share B, and their eigenbases meet as the iteration
  // settles, so the V side's first-order refinement holds from the fourth iteration on)
  auto go = [&](auto rpc) {
    constexpr int RP = decltype(rpc)::value, NT = Dim<RP>::NT;
    return launch_k_cluster<&rxr_body<RP>, Dim<RP>::kBounds>(rxr_cluster_size<RP>(), NT, sizeof(RxrSmem<RP>), st, (const double*)b.Gsum,
                                              s.rp, s.r, b.B, v_side ? b.TV : b.TU, v_side ? b.TCm : (double*)nullptr,
                                              (const float*)b.Qeig_u, v_side ? b.Qeig_v : b.Qeig_u, v_side ? 1 : 0,
                                              fp64 ? 0 : 1, b.st);
  };
  // grouped launches use one kernel for every rank up to 32, so that a step has one projector launch
  // per side whatever the ranks (which kernel runs a rank does not change its result)
  if (g_recorder && s.rp <= 32) return go(std::integral_constant<int, 32>{});
  switch (s.rp) {
    case 8: return go(std::integral_constant<int, 8>{});
    case 16: return go(std::integral_constant<int, 16>{});
    case 32: return go(std::integral_constant<int, 32>{});
    default: return go(std::integral_constant<int, 64>{});
  }
}

}  // namespace sfr
