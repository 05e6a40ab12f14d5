// The row passes of the CSR handles (block update, W/P update, Gram matrices) on the FP16 tensor cores
// with the precision of FP64 blocks (the bounds stand below), by digit splitting (Ozaki et al., "Error-free
// transformations of matrix multiplication by using fast routines of matrix multiplication and its
// applications", Numer. Algorithms 2012), from registers to registers (mma.sync.m16n8k16).
//
// Why. GB300 issues 2 FP64 lanes per clock per SM: at 16 columns a row of the block update is 768 + 144
// FP64 FMAs, and the FP64 pipe made these passes 10 times slower than their bytes. Here the contractions
// are integer digit products on the tensor cores, the splitting and recombination are integer
// operations, and the FP64 pipe keeps one add per output and the norms; the three pipes run side by
// side. What binds now is the integer work: about 50 operations per value split or combined. Measured (us per
// launch, FP64 pipe -> here; the block update with its Gram V^T V):
//                                    block update        W/P update     Gram P^T (A P) (in the product)
//   27-point 96^3, KP = 16          1357 -> 238 + 65     408 -> 147      239 -> 108 (102 without balancing)
//   diffusion 64^3, KP = 32         1619 -> 299 + 111    471 -> 165      280 -> 125
//   diffusion 100^3, KP = 8          455 -> 140 + 49     129 -> 85        78 -> 97 (kept fused)
//   diffusion 128^3, KP = 4          288 -> 152 + 50      77 -> 92 (kept)  58 -> 110 (kept fused)
// The same contractions in fixed point on the integer pipe (two 28-bit limbs, three IMAD.WIDE a term; 62
// lanes per clock per SM) took 383 + 115 and 205 us at KP = 16. The tile shapes (16 rows, 16 columns at most) are
// those of mma.sync: a warp holds its operands and results in registers in the layout in which it reads and
// writes them, so that there is no staging, no shared memory but the k x k matrices' digits, and no barrier in the
// loops (tcgen05.mma's smallest tile of 128 rows, with its operands in shared memory and results in tensor memory,
// needs all of these).
//
// Digits. A group of values (a row of a block, a column of a k x k matrix, a column of the rows that a
// warp sums) whose largest biased exponent is E is written x = 2^(E - 1022) 2^-B X, X the nearest
// integer (|X| <= 2^B: the group's largest value keeps all its bits, any other loses what lies below
// 2^-(B+1) of the scale), and X in 7 base-256 digits: six of -128..127 (X plus 128 in every digit, minus
// 128 digit by digit) and a leading one of at most 2^(B-48), all exact in FP16. Digit pairs (t, u) are kept
// for t + u <= 6 (28 products); what is dropped is random, 2^-60 of the two scales times the root of the number
// of terms at B = 57. (At B = 56 it is four times, at B = 55 sixteen times that: V zeta^-1 at KP = 32 was off by
// 8e-17 and 2.6e-16 of its norm, the FP64 pass by 5.2e-17 and B = 57 by 5.1e-17; at B = 57 no product of any
// width was further off than the FP64 pass on the Poisson, diffusion and 27-point systems, in an emulation.)
// (With one side's digits 0..255, two operations fewer per pair of digits, what is dropped has a mean
// that is the same for every row of a column: a smooth error, which an elliptic operator magnifies. The
// state after 8 iterations of the 27-point stencil was 100 times further off.)
//   A level sum S_L = sum_{t+u=L} sum_l is exact in the FP32 accumulator: within 2^18 * 16 = 2^22 (level 0) and
// (2 * 2^16 + 5 * 2^14) * 16 < 2^22 over one mma step of a row product at B = 57 (KP = 32 takes the levels of its
// two steps out one after the other); below (2 * 2^15 + 5 * 2^14) * 112 rows < 2^24 in a Gram
// (B = 56) between two drains.
//   A row product is off by 2^-58 or so of max_l |x_il| max_l |m_lj|, an FP64 sum by 2^-53 of sum_l |x_il m_lj|.
// These differ where columns of the block differ in size and the matrix makes up for it. V is such a block (a
// column whose Cholesky factor is 10^-6 of the others'), so is R at the set-up with a graded U, and A P, where a
// smooth column of P has eigenvalues far below the others': there column l enters as 2^o of it, and row l of the
// matrix as 2^-o, with o from the norms of the columns. The k x k steps know them: zeta has the column norms of
// V, Sigma those of R, and P^T A P = W^T (A P) is A P projected on the orthonormal W (emulated, Poisson 183^2, one
// smooth column and three rough ones: (A P) T off by 7e-14 of its norm without and 5e-17 with them, FP64 sums
// 9e-17). P has none: its columns are W's, of norm 1, and what CG adds to them.
//
// Widths. The row products see the block as rows of KV = max(KP, 8) columns and a Gram as rows of 16: for
// a narrower block several rows make one, with the k x k matrix repeated on the diagonal (the diagonal
// blocks of the Gram summed). Every row of the block keeps a scale of its own: neighbouring unknowns may be in
// different units, and a row 10^6 below its neighbour would lose 20 bits to a common one.
//
// A group that holds an infinity or a NaN has E = kMxNaN, and what is formed from it is NaN. A group below
// 2^-958 counts as zero (the solver squares norms: it can use nothing below 2^-511).
#pragma once
#include <cuda_fp16.h>
#include <stdint.h>

#include <type_traits>

#include "int_to_fp64.cuh"
#include "mbpcg_device.cuh"

namespace mbpcg {

constexpr int kMxDigits = 7;
constexpr int kMxThreads = 256;  // threads per CTA
constexpr int kMxGramBits = 56;  // B of the Grams
constexpr unsigned kMxAll = 0xffffffffu;
constexpr int kMxTiny = 64;     // a group with a scale exponent below this one counts as zero
constexpr int kMxNaN = 0x4000;  // scale exponent of a group that is not finite

__device__ __forceinline__ int mx_exponent(double x) { return (__double2hiint(x) >> 20) & 0x7FF; }

// X of 2^o x in a group of scale exponent E (>= its own), to nearest (halves away from zero). A group with E below
// `tiny` is zero; tiny - o >= 64.
template <int B>
__device__ __forceinline__ long long mx_int(double x, int E, int o, int tiny) {
  const int h = __double2hiint(x), e = (h >> 20) & 0x7FF;
  // 53 bits moved up to B + 1 (one below the unit), then down to the group's scale;
  // shr.u64 gives 0 from 64 on, which a zero or subnormal x (e = 0) reaches since E - o >= 64
  const unsigned long long m = (((unsigned long long)(unsigned)((h & 0xFFFFF) | 0x100000) << 32) |
                                (unsigned)__double2loint(x)) << (B - 52);
  unsigned long long r;
  asm("shr.u64 %0, %1, %2;" : "=l"(r) : "l"(m), "r"((E < tiny ? 4096 : E) - e - o));
  r = (r + 1) >> 1;
  const long long s = h >> 31;
  return (long long)(r ^ (unsigned long long)s) - s;
}

__device__ __forceinline__ uint32_t mx_prmt(uint32_t a, uint32_t b, uint32_t sel) {
  uint32_t r;
  asm("prmt.b32 %0, %1, %2, %3;" : "=r"(r) : "r"(a), "r"(b), "r"(sel));
  return r;
}
// The 7 digits of the two integers a and b as FP16 pairs (a in the low half).
__device__ __forceinline__ void mx_digits(long long a, long long b, uint32_t (&d)[kMxDigits]) {
  constexpr long long kBias = 0x6600808080808080LL;  // 128 in every digit but the first, which becomes an FP16 1536 + d
  const unsigned long long ua = (unsigned long long)(a + kBias), ub = (unsigned long long)(b + kBias);
  const uint32_t w[3] = {mx_prmt((uint32_t)ua, (uint32_t)ub, 0x5140u), mx_prmt((uint32_t)ua, (uint32_t)ub, 0x7362u),
                         mx_prmt((uint32_t)(ua >> 32), (uint32_t)(ub >> 32), 0x5140u)};
  {
    const uint32_t v = mx_prmt((uint32_t)(ua >> 32), (uint32_t)(ub >> 32), 0x7632u);
    const __half2 r = __hsub2(*reinterpret_cast<const __half2*>(&v), __half2half2(__ushort_as_half(0x6600)));
    d[0] = *reinterpret_cast<const uint32_t*>(&r);
  }
#pragma unroll
  for (int t = 1; t < kMxDigits; ++t) {
    const int byte = kMxDigits - 1 - t;
    const uint32_t v = mx_prmt(w[byte >> 1], 0x64646464u, (byte & 1) ? 0x4342u : 0x4140u);  // 1024 + 128 + digit
    const __half2 r = __hsub2(*reinterpret_cast<const __half2*>(&v), __half2half2(__ushort_as_half(0x6480)));
    d[t] = *reinterpret_cast<const uint32_t*>(&r);
  }
}

// D += A B, one warp: A 16 x 16 (or 16 x 8) by rows, B 16 x 8 (8 x 8) by columns, FP16 with FP32 sums.
__device__ __forceinline__ void mx_mma16(float (&d)[4], const uint32_t* a, uint32_t b0, uint32_t b1) {
  asm("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3},{%4,%5,%6,%7},{%8,%9},{%0,%1,%2,%3};"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
__device__ __forceinline__ void mx_mma8(float (&d)[4], const uint32_t* a, uint32_t b0) {
  asm("mma.sync.aligned.m16n8k8.row.col.f32.f16.f16.f32 {%0,%1,%2,%3},{%4,%5},{%6},{%0,%1,%2,%3};"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a[0]), "r"(a[1]), "r"(b0));
}

// t 2^k as FP64, rounded to nearest (half up), by integer operations; below 2^-1022: zero.
__device__ __forceinline__ double mx_double(long long t, int k) {
  const int s = (int)(t >> 32) >> 31;
  unsigned long long u = (unsigned long long)((t ^ (long long)s) - (long long)s);
  int top = 1023 + 62 + k;  // exponent of bit 63, less one
  if ((unsigned)(u >> 32) == 0) {  // rare, but for zeros (padded columns)
    if (u == 0) return 0.0;
    u <<= 32;
    top -= 32;
  }
  const int lz = __clz((int)(u >> 32));
  u <<= lz;
  // the leading one of the rounded significand raises the exponent field by one, a carry by two
  const unsigned long long m = (u >> 11) + ((u >> 10) & 1ull);
  const int e = top - lz;
  double v = __hiloint2double(((int)(m >> 32) + (e << 20)) | (s & (int)0x80000000), (int)m);
  if (e < 0) v = 0.0;
  if (e > 2044) v = __hiloint2double(0x7FF00000 | (s & (int)0x80000000), 0);
  return v;
}
__device__ __forceinline__ double mx_nan() { return __hiloint2double(0x7FF80000, 0); }

// ------------------------------------------------------------------------------------ row products

// Widths of the row products: view rows of KV columns in NB blocks of 8; lane (g, t) = (lane / 4,
// lane % 4) of a warp holds columns 8 c + 2 t, + 1 (c < NB) of the view rows g and g + 8 of its 16.
template <int KP>
struct MxRows {
  static constexpr int KV = KP < 8 ? 8 : KP;
  static constexpr int REP = KV / KP;  // rows of the block in a view row
  static constexpr int NB = KV / 8;
  static constexpr int KS = KV < 16 ? 1 : KV / 16;  // mma steps over the reduction index
  static constexpr int B = 57;
};

// A k x k matrix ready for the row products: the digits of each column in the fragment order of the
// mma (one 8-byte load per lane), and the columns' scale exponents.
template <int KP>
struct MxMatrix {
  using W = MxRows<KP>;
  uint2 b[kMxDigits][W::KS][W::NB][32];
  int e[KP];
};

// The accumulators of a row product start at 3 2^22, whose last bit is worth 1: their bits then count the
// level sum, which stays within 2^22 over one mma step. Level 6 starts 128 higher, which rounds it to level 5.
constexpr uint32_t kMxStart = 0x4B400000u;

// Weighted sum of the 7 levels' accumulators as integers, in units of 2^56 of the digits' product
// (level L weighs 2^(8 (12 - L))), with the start values' share kMxStartSum, modulo 2^64: a step's total is
// below 16 * 2^114 2^-56 = 2^62, that of two steps below 2^63 (the largest X is 2^57 - 2^4).
__device__ __forceinline__ unsigned long long mx_levels(const float (&d)[kMxDigits][4], int q) {
  unsigned long long r = __float_as_uint(d[6][q]) >> 8;
  r += __float_as_uint(d[5][q]);
  asm("mad.wide.u32 %0, %1, 256, %0;" : "+l"(r) : "r"(__float_as_uint(d[4][q])));
  asm("mad.wide.u32 %0, %1, 65536, %0;" : "+l"(r) : "r"(__float_as_uint(d[3][q])));
  asm("mad.wide.u32 %0, %1, 16777216, %0;" : "+l"(r) : "r"(__float_as_uint(d[2][q])));
  r += ((unsigned long long)(__float_as_uint(d[1][q]) + (__float_as_uint(d[0][q]) << 8))) << 32;
  return r;
}
constexpr unsigned long long kMxStartSum =
    (unsigned long long)(kMxStart >> 8) + (unsigned long long)kMxStart * (1ull + 256ull + 65536ull + 16777216ull) +
    ((unsigned long long)(uint32_t)(kMxStart + (kMxStart << 8)) << 32);

// Exponents o[l] (-63 to 0) that bring columns l of a block to like size, from a k x k matrix src(j, l) whose
// columns have the norms of the block's: the smallest column that is not zero has 0 (all threads; the caller
// synchronises before and after).
template <int KP, typename F>
__device__ void mx_column_exponents(F src, int (&o)[KP]) {
  __shared__ int c[KP];
  const int tid = threadIdx.x;
  if (tid < KP) {
    int e = 0;
#pragma unroll 8
    for (int j = 0; j < KP; ++j) e = max(e, mx_exponent(src(j, tid)));
    c[tid] = e;
  }
  __syncthreads();
  if (tid < KP) {
    int m = 0x7FF;
#pragma unroll 8
    for (int j = 0; j < KP; ++j) m = c[j] > 0 ? min(m, c[j]) : m;
    o[tid] = c[tid] > 0 ? max(m - c[tid], -63) : 0;
  }
}

// Fills M from src(l, j) (KP x KP; all threads; the caller synchronises before and after). o: row l enters as
// 2^-o[l] src(l, j), for blocks whose columns enter as 2^o[l] of theirs; or NULL.
template <int KP, typename F>
__device__ void mx_load_matrix(F src, const int* o, MxMatrix<KP>& M) {
  using W = MxRows<KP>;
  const int tid = threadIdx.x;
  if (tid < KP) {
    int e = 0;
    bool bad = false;
#pragma unroll 8
    for (int l = 0; l < KP; ++l) {
      const int x = mx_exponent(src(l, tid));
      bad |= x == 0x7FF;
      e = max(e, x > 0 && o != nullptr ? x - o[l] : x);
    }
    M.e[tid] = bad ? kMxNaN : e;
  }
  __syncthreads();
  for (int q = tid; q < W::KS * W::NB * 32; q += kMxThreads) {
    const int lane = q & 31, nb = (q >> 5) % W::NB, ks = (q >> 5) / W::NB;
    const int n = 8 * nb + (lane >> 2), k0 = 16 * ks + 2 * (lane & 3);
    // view matrix: KP x KP blocks on the diagonal
    auto at = [&](int k) {
      if (k >= W::KV || k / KP != n / KP) return 0LL;
      const double x = src(k % KP, n % KP);
      return mx_int<W::B>(x, M.e[n % KP], mx_exponent(x) > 0 && o != nullptr ? -o[k % KP] : 0, kMxTiny);
    };
    uint32_t d0[kMxDigits], d1[kMxDigits];
    mx_digits(at(k0), at(k0 + 1), d0);
    mx_digits(at(k0 + 8), at(k0 + 9), d1);
#pragma unroll
    for (int u = 0; u < kMxDigits; ++u) M.b[u][ks][nb][lane] = make_uint2(d0[u], d1[u]);
  }
}

// A warp's 16 view rows of a block: digits, and the scale exponents of the two rows whose columns this lane has.
template <int KP>
struct MxTile {
  using W = MxRows<KP>;
  uint32_t a[kMxDigits][2 * W::NB];
  int e[2];

  // the largest over the lanes of a row: at KP = 4 lanes t = 0, 1 hold one row of the block and t = 2, 3 the
  // next one, here and in the results
  static __device__ __forceinline__ int row_max(int m) {
    m = max(m, __shfl_xor_sync(kMxAll, m, 1));
    if constexpr (KP >= 8) m = max(m, __shfl_xor_sync(kMxAll, m, 2));
    return m;
  }

  // v[c][r]: columns 8 c + 2 t, + 1 of view row g + 8 r. o: column j enters as 2^o[j] of it; or NULL.
  __device__ __forceinline__ void split(const double2 (&v)[W::NB][2], const int* o) {
    int ox[W::NB], oy[W::NB];
#pragma unroll
    for (int c = 0; c < W::NB; ++c) {
      const int j = (8 * c + 2 * (threadIdx.x & 3)) % KP;
      ox[c] = o != nullptr ? o[j] : 0;
      oy[c] = o != nullptr ? o[j + 1] : 0;
    }
    auto largest = [&](int r, bool raw) {
      int m = 0;
#pragma unroll
      for (int c = 0; c < W::NB; ++c)
        m = max(m, max(mx_exponent(v[c][r].x) + (raw ? 0 : ox[c]), mx_exponent(v[c][r].y) + (raw ? 0 : oy[c])));
      return row_max(m);
    };
    e[0] = largest(0, false);
    e[1] = largest(1, false);
    if (o == nullptr) {
#pragma unroll
      for (int r = 0; r < 2; ++r)
        if (e[r] == 0x7FF) e[r] = kMxNaN;
    } else if (__any_sync(kMxAll, max(e[0], e[1]) >= 0x7FF - 63)) {  // not finite, which o may hide, or large
#pragma unroll
      for (int r = 0; r < 2; ++r)
        if (largest(r, true) == 0x7FF) e[r] = kMxNaN;
    }
#pragma unroll
    for (int r = 0; r < 2; ++r)
#pragma unroll
      for (int c = 0; c < W::NB; ++c) {
        uint32_t d[kMxDigits];
        mx_digits(mx_int<W::B>(v[c][r].x, e[r], ox[c], kMxTiny), mx_int<W::B>(v[c][r].y, e[r], oy[c], kMxTiny), d);
#pragma unroll
        for (int t = 0; t < kMxDigits; ++t) a[t][2 * c + r] = d[t];
      }
  }

  // Columns 8 nb + 2 t, + 1 of the two rows times M: y[r].
  __device__ __forceinline__ void times(const MxMatrix<KP>& M, int nb, double2 (&y)[2]) const {
    const int lane = threadIdx.x & 31;
    unsigned long long sum[4] = {0ull, 0ull, 0ull, 0ull};
#pragma unroll
    for (int ks = 0; ks < W::KS; ++ks) {
      float d[kMxDigits][4];
#pragma unroll
      for (int L = 0; L < kMxDigits; ++L)
#pragma unroll
        for (int q = 0; q < 4; ++q) d[L][q] = __uint_as_float(kMxStart + (L == kMxDigits - 1 ? 128u : 0u));
#pragma unroll
      for (int u = 0; u < kMxDigits; ++u) {
        const uint2 b = M.b[u][ks][nb][lane];
#pragma unroll
        for (int t = 0; t + u < kMxDigits; ++t) {
          if constexpr (W::KV >= 16) mx_mma16(d[t + u], a[t] + 4 * ks, b.x, b.y);
          else mx_mma8(d[t + u], a[t], b.x);
        }
      }
#pragma unroll
      for (int q = 0; q < 4; ++q) sum[q] += mx_levels(d, q) - kMxStartSum;
    }
    const int j = (8 * nb + 2 * (lane & 3)) % KP;
    double v[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int f = M.e[j + (q & 1)], er = e[q >> 1];
      v[q] = mx_double((long long)sum[q], er + f - 2044 - 2 * W::B + 56);
      if (max(f, er) == kMxNaN) v[q] = mx_nan();
    }
    y[0] = make_double2(v[0], v[1]);
    y[1] = make_double2(v[2], v[3]);
  }
};

// Loads v[c][r] from X, rows of the view up to nv (nf doubles in all: the last view row may be short).
template <int KP>
__device__ __forceinline__ void mx_load_rows(const double* X, size_t row, size_t nf, int t,
                                             double2 (&v)[MxRows<KP>::NB][2]) {
  using W = MxRows<KP>;
#pragma unroll
  for (int r = 0; r < 2; ++r)
#pragma unroll
    for (int c = 0; c < W::NB; ++c) {
      const size_t o = (row + 8 * r) * W::KV + 8 * c + 2 * t;
      v[c][r] = o < nf ? *reinterpret_cast<const double2*>(X + o) : make_double2(0.0, 0.0);
    }
}
template <int KP>
__device__ __forceinline__ void mx_store_rows(double* X, size_t row, size_t nf, int t,
                                              const double2 (&v)[MxRows<KP>::NB][2]) {
  using W = MxRows<KP>;
#pragma unroll
  for (int r = 0; r < 2; ++r)
#pragma unroll
    for (int c = 0; c < W::NB; ++c) {
      const size_t o = (row + 8 * r) * W::KV + 8 * c + 2 * t;
      if (o < nf) *reinterpret_cast<double2*>(X + o) = v[c][r];
    }
}

// Block update of Algorithm 1 (as k_axpy): X~ += P T, R -= (A P) T, V = W - (A P) Xi, and the CTA partials
// of nu at part[NPACK + j]. Gp: the upper triangle of P^T (A P). RFREE: R is neither read nor written, and there are
// no norms. Tiles of 16 view rows are dealt to the warps of the grid in turn (their sums do not depend on the order).
template <int KP, bool RFREE>
__global__ void __launch_bounds__(kMxThreads, KP >= 32 ? 1 : 2)
k_axpy_mx(int n, const double* __restrict__ P, const double* __restrict__ Q, const double* __restrict__ W,
          double* __restrict__ R, double* __restrict__ Xt, double* __restrict__ V, const double* __restrict__ Tg,
          const double* __restrict__ Xig, const double* __restrict__ Gp, const double* __restrict__ wdiag,
          double* __restrict__ part, int pstride, const SolveState* __restrict__ st) {
  using M = MxRows<KP>;
  if (st->done) return;
  __shared__ MxMatrix<KP> T, Xi;                                               // of P, of A P
  __shared__ typename std::conditional<RFREE, int, MxMatrix<KP>>::type Tq;     // T for A P
  __shared__ double red[RFREE ? 1 : kMxThreads / 32][KP];
  __shared__ int oq[KP];
  auto tg = [&](int l, int j) { return __ldg(Tg + l + j * KP); };
  mx_column_exponents<KP>([&](int j, int l) { return __ldg(Gp + pidx(min(j, l), max(j, l))); }, oq);
  mx_load_matrix<KP>(tg, nullptr, T);  // (its barrier stands before the first use of oq)
  mx_load_matrix<KP>([&](int l, int j) { return __ldg(Xig + l + j * KP); }, oq, Xi);
  if constexpr (!RFREE) mx_load_matrix<KP>(tg, oq, Tq);
  __syncthreads();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, g = lane >> 2, t = lane & 3;
  const size_t nf = (size_t)n * KP, nv = (nf + M::KV - 1) / M::KV;
  const size_t step = (size_t)gridDim.x * (kMxThreads / 32) * 16;
  double2 nu[M::NB];
#pragma unroll
  for (int c = 0; c < M::NB; ++c) nu[c] = make_double2(0.0, 0.0);
  for (size_t base = ((size_t)blockIdx.x * (kMxThreads / 32) + warp) * 16; base < nv; base += step) {
    const size_t row = base + g;
    MxTile<KP> tile;
    double2 v[M::NB][2], x[M::NB][2], y[2];
    mx_load_rows<KP>(P, row, nf, t, v);
    mx_load_rows<KP>(Xt, row, nf, t, x);
    tile.split(v, nullptr);
    mx_load_rows<KP>(Q, row, nf, t, v);
#pragma unroll
    for (int c = 0; c < M::NB; ++c) {
      tile.times(T, c, y);
#pragma unroll
      for (int r = 0; r < 2; ++r) {
        x[c][r].x += y[r].x;
        x[c][r].y += y[r].y;
      }
    }
    mx_store_rows<KP>(Xt, row, nf, t, x);
    mx_load_rows<KP>(W, row, nf, t, x);
    tile.split(v, oq);
    if constexpr (!RFREE) mx_load_rows<KP>(R, row, nf, t, v);
#pragma unroll
    for (int c = 0; c < M::NB; ++c) {
      tile.times(Xi, c, y);
#pragma unroll
      for (int r = 0; r < 2; ++r) {
        x[c][r].x -= y[r].x;
        x[c][r].y -= y[r].y;
      }
    }
    mx_store_rows<KP>(V, row, nf, t, x);
    if constexpr (!RFREE) {
#pragma unroll
      for (int c = 0; c < M::NB; ++c) {
        tile.times(Tq, c, y);
#pragma unroll
        for (int r = 0; r < 2; ++r) {
          v[c][r].x -= y[r].x;
          v[c][r].y -= y[r].y;
          double wx = v[c][r].x, wy = v[c][r].y;
          if (wdiag != nullptr) {
            const size_t i = ((row + 8 * r) * M::KV + 8 * c + 2 * t) / KP;
            const double w2 = i < (size_t)n ? __ldg(wdiag + i) : 0.0;
            wx *= w2;
            wy *= w2;
          }
          nu[c].x = fma(wx, v[c][r].x, nu[c].x);
          nu[c].y = fma(wy, v[c][r].y, nu[c].y);
        }
      }
      mx_store_rows<KP>(R, row, nf, t, v);
    }
  }
  if constexpr (!RFREE) {  // lanes of one column, view columns of one column, then the warps in order
#pragma unroll
    for (int c = 0; c < M::NB; ++c) {
#pragma unroll
      for (int off = 16; off >= 4; off >>= 1) {
        nu[c].x += __shfl_xor_sync(kMxAll, nu[c].x, off);
        nu[c].y += __shfl_xor_sync(kMxAll, nu[c].y, off);
      }
      if constexpr (KP == 4) {
        nu[c].x += __shfl_xor_sync(kMxAll, nu[c].x, 2);
        nu[c].y += __shfl_xor_sync(kMxAll, nu[c].y, 2);
      }
      const int j = 8 * c + 2 * t;
      if (g == 0 && j < KP) {
        red[warp][j] = nu[c].x;
        red[warp][j + 1] = nu[c].y;
      }
    }
    __syncthreads();
    if (threadIdx.x < KP) {
      double a = red[0][threadIdx.x];
      for (int w = 1; w < kMxThreads / 32; ++w) a += red[w][threadIdx.x];
      part[(size_t)blockIdx.x * pstride + npack(KP) + threadIdx.x] = a;
    }
  }
}

// W/P update of Algorithm 1 (as k_pw): W = V zeta^{-1}, P = W + P zeta^T (SETP: P = W; Zg is then Sigma, V is R).
// V = Q zeta with orthonormal Q, so that the columns of zeta have the norms of V's.
template <int KP, bool SETP>
__global__ void __launch_bounds__(kMxThreads, KP >= 32 ? 1 : 2)
k_pw_mx(int n, const double* __restrict__ V, double* __restrict__ W, double* __restrict__ P,
        const double* __restrict__ Zinvg, const double* __restrict__ Zg, const SolveState* __restrict__ st) {
  using M = MxRows<KP>;
  if (st != nullptr && st->pw_skip) return;
  __shared__ MxMatrix<KP> Zi;
  __shared__ typename std::conditional<SETP, int, MxMatrix<KP>>::type Zt;
  __shared__ int ov[KP];
  mx_column_exponents<KP>([&](int j, int l) { return __ldg(Zg + j + l * KP); }, ov);
  __syncthreads();
  mx_load_matrix<KP>([&](int l, int j) { return __ldg(Zinvg + l + j * KP); }, ov, Zi);
  if constexpr (!SETP) mx_load_matrix<KP>([&](int l, int j) { return __ldg(Zg + j + l * KP); }, nullptr, Zt);
  __syncthreads();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, g = lane >> 2, t = lane & 3;
  const size_t nf = (size_t)n * KP, nv = (nf + M::KV - 1) / M::KV;
  const size_t step = (size_t)gridDim.x * (kMxThreads / 32) * 16;
  for (size_t base = ((size_t)blockIdx.x * (kMxThreads / 32) + warp) * 16; base < nv; base += step) {
    const size_t row = base + g;
    MxTile<KP> tile;
    double2 v[M::NB][2], w[M::NB][2], y[2];
    mx_load_rows<KP>(V, row, nf, t, v);
    tile.split(v, ov);
    if constexpr (!SETP) mx_load_rows<KP>(P, row, nf, t, v);
#pragma unroll
    for (int c = 0; c < M::NB; ++c) tile.times(Zi, c, w[c]);
    mx_store_rows<KP>(W, row, nf, t, w);
    if constexpr (!SETP) {
      tile.split(v, nullptr);
#pragma unroll
      for (int c = 0; c < M::NB; ++c) {
        tile.times(Zt, c, y);
#pragma unroll
        for (int r = 0; r < 2; ++r) {
          w[c][r].x += y[r].x;
          w[c][r].y += y[r].y;
        }
      }
    }
    mx_store_rows<KP>(P, row, nf, t, w);
  }
}

// ------------------------------------------------------------------------------------ Gram matrices

// CTA partials of the upper triangle of X^T Y (Y = X when SYM). WT: of X^T D^2 X, with D in dw and as
// (D X)^T (D X) up to KP = 16, where that leaves one block to split (diffusion 77^3: 56 us against 80 for
// (D^2 X)^T X; D x is rounded once more than D^2 x, 2^-53 of each term), and D^2 in dw at KP = 32, where there are
// two anyway (FP64 products). A warp keeps its own column scales: the mma takes 16 view rows as its reduction
// index, so that a lane holds the view columns g and g + 8 of 4 rows, as the left operand and as the right one
// alike. The scales only grow; a tile that exceeds them (the first one, and then rarely: one bit of headroom)
// first has the sums turned into FP64. 56 bits of the scale: with 55 the Grams of unscaled diffusion were off by up
// to 1.5 times what FP64 sums are, with 56 by less than those on every system (in an emulation). KP = 32 is three
// problems of 16 columns (blockIdx.y: columns 0..15 with themselves, with 16..31, and 16..31 with themselves).
//   X^T Y of two blocks is P^T (A P). Where the diagonal of A varies, P is small where A P is large, and a scale over
// the rows would lose what their product does not: the rows are balanced by r = half the exponent of a_ii
// (rexp, k_row_exponents; or NULL), 2^r X against 2^-r Y. (Two unknowns per point in units 10^6 apart, 16 columns,
// emulated: off by 2e-12 of the largest entry without and 1e-16 with it, FP64 sums by 1e-15. The kernel takes 108
// us with it on the 27-point system, 102 without; 122 to 132 with the exponents taken from the diagonal on the way.)
constexpr int kMxDrainTiles = 7;  // 112 rows between two drains of the FP32 sums into FP64

template <int KP, bool SYM, bool WT = false>
__global__ void __launch_bounds__(kMxThreads, SYM && KP <= 16 ? 2 : 1)
k_gram_mx(int n, const double* __restrict__ X, const double* __restrict__ Y, const double* __restrict__ dw,
          const int* __restrict__ rexp, double* __restrict__ part, int pstride, const SolveState* __restrict__ st) {
  constexpr int KV = 16, WARPS = kMxThreads / 32;
  if (st != nullptr && st->done) return;
  constexpr bool BAL = !SYM;
  static_assert(SYM || KP >= KV, "a view row is a row of the block");
  __shared__ double red[WARPS][KV * KV];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, g = lane >> 2, t = lane & 3;
  // KP = 32: rows are 32 wide, this problem's columns start at xc (X) and yc (Y)
  constexpr int LD = KP > KV ? KP : KV;
  const int xc = KP > KV && blockIdx.y == 2 ? KV : 0, yc = KP > KV && blockIdx.y >= 1 ? KV : 0;
  const size_t nf = (size_t)n * KP, nv = (nf + LD - 1) / LD;
  const size_t step = (size_t)gridDim.x * WARPS * 16;

  float acc[kMxDigits][2][4];
  double f[2][4];
  int rs[BAL ? 4 : 1];  // r of the tile's rows
  constexpr int tiny = BAL ? kMxTiny + 64 : kMxTiny;
  int ex[2] = {0, 0}, ey[2] = {0, 0};  // scale exponents of view columns g, g + 8
  auto zero = [&]() {
#pragma unroll
    for (int L = 0; L < kMxDigits; ++L)
#pragma unroll
      for (int b = 0; b < 2; ++b)
#pragma unroll
        for (int q = 0; q < 4; ++q) acc[L][b][q] = 0.f;
  };
  // the FP32 sums into FP64, over an integer in units of 2^56 of the digits' product (level 5; level 6 rounded):
  // below 112 * 2^112 2^-56 < 2^63
  auto drain = [&]() {
#pragma unroll
    for (int b = 0; b < 2; ++b)
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        int s[kMxDigits];
#pragma unroll
        for (int L = 0; L < kMxDigits; ++L) s[L] = __float2int_rn(acc[L][b][q]);
        const long long sum = ((long long)s[0] << 40) + ((long long)s[1] << 32) + ((long long)s[2] << 24) +
                              ((long long)s[3] << 16) + ((long long)s[4] << 8) + s[5] + ((s[6] + 128) >> 8);
        // entry (g + 8 (q / 2), 8 b + 2 t + q % 2)
        const int el = ex[q >> 1];
        const int ej = __shfl_sync(kMxAll, SYM && KP <= KV ? ex[b] : ey[b], (2 * t + (q & 1)) * 4);
        bool ok;
        const int k = el + ej - 2044 - 2 * kMxGramBits + 56;
        double v = ll_to_double_scaled_rn(sum, k, ok);
        if (!ok) v = ldexp(ll_to_double_rn(sum), k);
        f[b][q] += max(el, ej) == kMxNaN ? mx_nan() : v;
      }
    zero();
  };
  zero();
#pragma unroll
  for (int b = 0; b < 2; ++b)
#pragma unroll
    for (int q = 0; q < 4; ++q) f[b][q] = 0.0;
  // x[h][c]: row 2 t + (h & 1) + 8 (h >> 1) of the tile, view column g + 8 c
  constexpr bool ONE = SYM && KP <= KV;  // both operands from one block
  double x[4][2], y[ONE ? 1 : 4][2];
  auto load = [&](size_t base) {
#pragma unroll
    for (int h = 0; h < 4; ++h) {
      const size_t r = base + 2 * t + (h & 1) + 8 * (h >> 1);
      if constexpr (BAL)
        rs[h] = rexp != nullptr && r < nv ? __ldg(rexp + r) : 0;
#pragma unroll
      for (int c = 0; c < 2; ++c) {
        const size_t o = r * LD + g + 8 * c;
        const bool in = r < nv && (KP >= KV || o < nf);
        x[h][c] = in ? __ldg(X + o + xc) : 0.0;
        if constexpr (!ONE) y[h][c] = in ? __ldg(Y + o + yc) : 0.0;
        if constexpr (WT) x[h][c] *= in ? __ldg(dw + (o / KP)) : 0.0;
      }
    }
  };
  // X takes part as 2^r X and Y as 2^-r Y
  auto off = [&](int h, int sign) { return BAL ? sign * rs[BAL ? h : 0] : 0; };
  auto grow = [&](const auto& v, int sign, const int (&e)[2], int (&ne)[2]) {
    bool over = false;
#pragma unroll
    for (int c = 0; c < 2; ++c) {
      int m = 0;
#pragma unroll
      for (int h = 0; h < 4; ++h) m = max(m, mx_exponent(v[h][c]) + off(h, sign));
      m = max(m, __shfl_xor_sync(kMxAll, m, 1));
      m = max(m, __shfl_xor_sync(kMxAll, m, 2));
      ne[c] = m > e[c] ? max(m, min(m + 1, 0x7FE)) : e[c];
      over |= ne[c] != e[c];
    }
    return over;
  };
  // the new scales; an infinity or a NaN, whose exponent is the largest, is looked for only here
  auto adopt = [&](const auto& v, const int (&ne)[2], int (&e)[2]) {
#pragma unroll
    for (int c = 0; c < 2; ++c) {
      int bad = e[c] == kMxNaN;
#pragma unroll
      for (int h = 0; h < 4; ++h) bad |= mx_exponent(v[h][c]) == 0x7FF;
      bad |= __shfl_xor_sync(kMxAll, bad, 1);
      bad |= __shfl_xor_sync(kMxAll, bad, 2);
      e[c] = bad ? kMxNaN : ne[c];
    }
  };
  auto split = [&](const auto& v, int sign, const int (&e)[2], uint32_t (&a)[kMxDigits][4]) {
#pragma unroll
    for (int hh = 0; hh < 2; ++hh)
#pragma unroll
      for (int c = 0; c < 2; ++c) {
        uint32_t d[kMxDigits];
        mx_digits(mx_int<kMxGramBits>(v[2 * hh][c], e[c], off(2 * hh, sign), tiny),
                  mx_int<kMxGramBits>(v[2 * hh + 1][c], e[c], off(2 * hh + 1, sign), tiny), d);
#pragma unroll
        for (int q = 0; q < kMxDigits; ++q) a[q][2 * hh + c] = d[q];
      }
  };
  int tiles = 0;
  size_t base = ((size_t)blockIdx.x * WARPS + warp) * 16;
  if (base < nv) load(base);
  for (; base < nv; base += step) {
    int nx[2], ny[2];
    bool over = grow(x, 1, ex, nx);
    if constexpr (!ONE) over |= grow(y, -1, ey, ny);
    if (__any_sync(kMxAll, over)) {
      drain();
      tiles = 0;
      adopt(x, nx, ex);
      if constexpr (!ONE) adopt(y, ny, ey);
    }
    uint32_t a[kMxDigits][4], b[ONE ? 1 : kMxDigits][4];
    split(x, 1, ex, a);
    if constexpr (!ONE) split(y, -1, ey, b);
    if (base + step < nv) load(base + step);
#pragma unroll
    for (int u = 0; u < kMxDigits; ++u) {
      const uint32_t* bu = ONE ? a[u] : b[ONE ? 0 : u];
#pragma unroll
      for (int q = 0; q + u < kMxDigits; ++q) {
        mx_mma16(acc[q + u][0], a[q], bu[0], bu[2]);
        mx_mma16(acc[q + u][1], a[q], bu[1], bu[3]);
      }
    }
    if (++tiles == kMxDrainTiles) {
      drain();
      tiles = 0;
    }
  }
  drain();
#pragma unroll
  for (int b = 0; b < 2; ++b)
#pragma unroll
    for (int q = 0; q < 4; ++q) red[warp][(g + 8 * (q >> 1)) * KV + 8 * b + 2 * t + (q & 1)] = f[b][q];
  __syncthreads();
  double* out = part + (size_t)blockIdx.x * pstride;
  constexpr int KB = KP < KV ? KP : KV;  // the diagonal blocks are KB wide
  for (int q = threadIdx.x; q < KB * KB; q += kMxThreads) {
    const int l = q / KB, j = q % KB;
    const int L = l + xc, J = j + yc;
    if (L > J) continue;
    double v = 0.0;
    for (int d = 0; d < KV / KB; ++d)
      for (int k = 0; k < WARPS; ++k) v += red[k][(l + d * KB) * KV + j + d * KB];
    out[pidx(L, J)] = v;
  }
}

}  // namespace mbpcg
