// The iteration loop of Algorithm 1 for a small CSR system (KP <= 8, FP64, explicit residual): many
// iterations in one launch of one thread-block cluster (sm_103a).
//
// What bounds a small system is not bytes or operations but the chain of launches: Poisson 64^2 at s = 4
// has 7 of them per iteration, each with a drain, a launch and loads from L2 at its start (31.8 us together;
// its 0.5 M FP64 FMAs would take the whole chip 0.9 us). Here 16 CTAs on 16 SMs stay for the whole loop
// (15.5 us): the rows of A, X~, R, W, P, A P and V of a CTA stay in its shared memory, the product reads the
// other CTAs' rows of P there (distributed shared memory: 1300 cycles for a row by row chain that took 2600
// through L2), the partial sums of the two Gram matrices are pushed into every CTA's shared memory, and
// every CTA repeats the k x k steps for itself: the same inputs in the same order, so the same bits and the
// same decisions. An iteration has three cluster barriers:
//   A P, partials of P^T A P | Xi, V = W - A P Xi, partials of V^T V | zeta, W, P |
// and what is not on that path goes beside the zeta step, whose chain leaves the FP64 units idle: X~ += P T
// and R -= A P T. The norms nu of the new R are summed with the next product, so the stopping test of an
// iteration falls beside the next Xi step (in the last iteration of a launch at once).
// Where the 15.5 us go (cycles, n = 4096, s = 4): product 5400, V 3900, W and P 3300 (FP64 pipe of 16 SMs),
// Xi 3300 and zeta 3100 (chains of FP64 latencies), 2 x 1700 for the sums inside a CTA, 3 barriers 2600,
// sums over the CTAs 1500.
// The cluster's CTAs are scheduled together by the hardware, so no wait here can miss its peer, and several
// small solves run side by side, one cluster each. 256 threads: 512 fill the FP64 pipe no better and double
// the additions of the sums (16.5 us).
#include <cooperative_groups.h>

#include <algorithm>
#include <cfloat>

#include "kernels.h"
#include "mbpcg_device.cuh"
#include "pivot.cuh"

namespace mbpcg {
namespace {

namespace cg = cooperative_groups;

constexpr int kLcCtas = 16;
constexpr int kLcThreads = 256;
constexpr int kLcWarps = kLcThreads / 32;
constexpr unsigned kAll = 0xffffffffu;

// Sums over the threads: a thread of column m = tid % KP holds ND products of a Gram, of (m, (m - d) mod KP)
// for d = 0 .. KP/2 (every pair once; the columns below KP/2 leave d = KP/2 to the others), then nu_m.
// The k x k steps run on KK threads, one entry each, which lie on the first KK / 32 of the SM's four
// sub-partitions (warp mod 4); the KG threads of those sub-partitions are the k x k group.
template <int KP>
struct LcCfg {
  static constexpr int NP = KP * (KP + 1) / 2;
  static constexpr int ND = KP / 2 + 1;
  static constexpr int NV = ND + 1;
  static constexpr int NE = NP + KP;
  static constexpr int KK = KP == 8 ? 64 : 32;
  static constexpr int KG = kLcThreads / 4 * (KK / 32);
};

template <int KP>
struct LcShared {
  using C = LcCfg<KP>;
  double part1[kLcCtas * C::NE];  // all CTAs' partials of P^T A P and nu, then of V^T V (pushed by their owners)
  double part2[kLcCtas * C::NP];
  double ra[C::NV * kLcThreads], rb[C::NV * kLcThreads / 4];
  double S[KP * KP], Lt[KP * KP], R[KP * KP], V[KP * KP];
  double d[KP], inv[KP], nu[KP];
  double Xi[KP * KP], T[KP * KP], Z[KP * KP], Zi[KP * KP], Sg[2][KP * KP];  // row-major
  double nh;
  int h, stop, bad, chunk;
};

__device__ __forceinline__ void bar_arrive(int id, int count) {
  asm volatile("bar.arrive %0, %1;" ::"r"(id), "r"(count) : "memory");
}
__device__ __forceinline__ void bar_sync(int id, int count) {
  asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(count) : "memory");
}
// named barriers: factor -> Sigma warp, k x k group, k x k threads
constexpr int kBarSigma = 1, kBarGroup = 2, kBarKk = 3;

__device__ __forceinline__ void lc_arrive() { asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory"); }
__device__ __forceinline__ double ld_cluster(uint32_t a) {
  double v;
  asm volatile("ld.shared::cluster.f64 %0, [%1];" : "=d"(v) : "r"(a) : "memory");
  return v;
}
__device__ __forceinline__ void lc_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }

// Packed entry of product v of the thread column m (v = ND: nu_m); -1 where another column has it.
template <int KP>
__device__ __forceinline__ int lc_entry(int v, int m) {
  if (v == LcCfg<KP>::ND) return LcCfg<KP>::NP + m;
  if (KP > 1 && 2 * v == KP && m < KP / 2) return -1;
  const int o = (m - v + KP) % KP;
  return pidx(min(o, m), max(o, m));
}

// CTA sums of val[0 .. NV) by column, pushed into slot `rank` of every CTA's part (ne entries a slot).
// A four-way tree: an FP64 addition holds its sub-partition's unit for ~70 cycles whatever the number of
// active lanes, so full warps of additions and few of them are what counts, not depth.
template <int KP, int NV>
__device__ __forceinline__ void lc_push(LcShared<KP>& sm, const double (&val)[LcCfg<KP>::NV], double* part, int ne,
                                        cg::cluster_group& cluster, int rank) {
  const int tid = threadIdx.x;
#pragma unroll
  for (int v = 0; v < NV; ++v) sm.ra[v * kLcThreads + tid] = val[v];
  __syncthreads();
  double *src = sm.ra, *dst = sm.rb;
  int cnt = kLcThreads;
#pragma unroll
  for (; cnt / 4 >= (KP > 4 ? KP : 4); cnt /= 4) {
    const int q = cnt / 4;
    for (int w = tid; w < NV * q; w += kLcThreads) {
      const int v = w / q, t = w % q;
      const double* p = src + v * cnt + t;
      dst[w] = (p[0] + p[q]) + (p[2 * q] + p[3 * q]);
    }
    __syncthreads();
    double* t = src;
    src = dst;
    dst = t;
  }
  for (int w = tid; w < NV * KP * kLcCtas; w += kLcThreads) {
    const int to = w / (NV * KP), v = w % (NV * KP) / KP, m = w % KP, e = lc_entry<KP>(v, m);
    if (e < 0) continue;
    double a = src[v * cnt + m];
    for (int t = m + KP; t < cnt; t += KP) a += src[v * cnt + t];
    cluster.map_shared_rank(part, to)[rank * ne + e] = a;
  }
}

// The sums over the CTAs, by nt threads (k: index of the caller): the Gram into sm.S (both triangles, the
// identity outside s x s), nu into sm.nu.
template <int KP>
__device__ __forceinline__ void lc_total(LcShared<KP>& sm, const double* part, int ne, int s, int k, int nt) {
  using C = LcCfg<KP>;
  for (int w = k; w - (k & 31) < 4 * ne; w += nt) {
    const int e = min(w / 4, ne - 1), q = w % 4;
    const double* p = part + 4 * q * ne + e;
    double a = (p[0] + p[ne]) + (p[2 * ne] + p[3 * ne]);
    a += __shfl_xor_sync(kAll, a, 1);
    a += __shfl_xor_sync(kAll, a, 2);
    if (q != 0 || w / 4 >= ne) continue;
    if (e < C::NP) {
      int l, m;
      punpack(e, l, m);
      sm.S[l * KP + m] = sm.S[m * KP + l] = m < s ? a : (l == m ? 1.0 : 0.0);
    } else {
      sm.nu[e - C::NP] = a;
    }
  }
}

template <int KP>
__device__ __forceinline__ void kk_sync() {
  if constexpr (LcCfg<KP>::KK == 32) __syncwarp();
  else bar_sync(kBarKk, LcCfg<KP>::KK);
}

// The k x k steps: thread k < KK has entry (a, b) = (k mod KP, k / KP) (more than one thread the same one
// below KP = 8), so a column lies in one warp.

// G = L D L^T of sm.S in the steps and with the pivot test of ldl_factor (small_warp.cu): afterwards S holds
// U = D L^T in its upper triangle, Lt[k][m] = L[m][k], d and inv the pivots. True on a bad pivot.
template <int KP>
__device__ __forceinline__ bool lc_factor(LcShared<KP>& sm, int s) {
  const int kt = threadIdx.x, a = kt % KP, b = kt / KP % KP, lo = min(a, b), hi = max(a, b);
  double x = sm.S[a * KP + b];
  long long mb = 0;
#pragma unroll
  for (int j = 0; j < KP; ++j)
    if (j < s) mb = max(mb, __double_as_longlong(sm.S[j * KP + j]));
  const long long thr = __double_as_longlong(64.0 * DBL_EPSILON * __longlong_as_double(mb));
  // Every thread has read the diagonal before step 0 changes it (at KP = 8 by two warps): one threshold, so
  // one decision, in all threads and all CTAs.
  kk_sync<KP>();
  bool bad = false;
  if (kt < KP && kt >= s) sm.d[kt] = sm.inv[kt] = 1.0;
  double linv = 1.0;  // 1/d of row a
#pragma unroll
  for (int k = 0; k < KP; ++k) {
    if (k >= s) break;
    double dk, u, w;
    if constexpr (LcCfg<KP>::KK == 32) {  // entry (i, j) is thread i + KP j's
      dk = __shfl_sync(kAll, x, k + KP * k);
      u = __shfl_sync(kAll, x, k + KP * lo);
      w = __shfl_sync(kAll, x, k + KP * hi);
    } else {
      dk = sm.S[k * KP + k];
      u = sm.S[k * KP + lo];
      w = sm.S[k * KP + hi];
    }
    const double uw = u * w;  // beside the reciprocal's chain
    const long long db = __double_as_longlong(dk);
    bad |= !(db > thr && db < 0x7E70000000000000LL);
    const double inv = rcp_pos(dk);
    if (lo > k) {
      x = fma(-uw, inv, x);
      if constexpr (LcCfg<KP>::KK != 32) sm.S[a * KP + b] = x;
    }
    if (a == k) linv = inv;
    if (kt == 0) {
      sm.d[k] = dk;
      sm.inv[k] = inv;
    }
    if constexpr (LcCfg<KP>::KK != 32) kk_sync<KP>();
  }
  if constexpr (LcCfg<KP>::KK == 32) sm.S[a * KP + b] = x;
  sm.Lt[a * KP + b] = x * linv;
  kk_sync<KP>();
  return bad;
}

// Xi = G^{-1} after lc_factor, in the sums of k_small_xi_x.
template <int KP>
__device__ __forceinline__ void lc_xi(LcShared<KP>& sm, int s) {
  const int kt = threadIdx.x, a = kt % KP, b = kt / KP % KP, seg = (kt & 31) - a;
  double x = a == b ? 1.0 : 0.0;
  double lt[KP];
#pragma unroll
  for (int k = 0; k < KP - 1; ++k) lt[k] = a > k && a < s ? -sm.Lt[k * KP + a] : 0.0;
#pragma unroll
  for (int k = 0; k < KP - 1; ++k) {  // column b of L^{-1}: x_k is final, the rows below take it
    const double xk = __shfl_sync(kAll, x, seg + k);
    if (a > k && a < s) x = fma(lt[k], xk, x);
  }
  sm.R[a * KP + b] = x;
  sm.V[a * KP + b] = sm.inv[a] * x;
  kk_sync<KP>();
  const int lo = min(a, b), hi = max(a, b);
  double v = 0.0;  // Xi[lo][hi] = sum_{j >= hi} R[j][lo] V[j][hi]
#pragma unroll
  for (int j = 0; j < KP; ++j)
    if (j >= hi && j < s) v = fma(sm.R[j * KP + lo], sm.V[j * KP + hi], v);
  sm.Xi[a * KP + b] = hi < s ? v : 0.0;
}

// T = Xi Sigma (Sigma upper triangular) by one warp.
template <int KP>
__device__ __forceinline__ void lc_t(LcShared<KP>& sm, const double* Sg) {
  for (int q = threadIdx.x & 31; q < KP * KP; q += 32) {
    const int a = q / KP, b = q % KP;
    double v = 0.0;
#pragma unroll
    for (int l = 0; l < KP; ++l)
      if (l <= b) v = fma(sm.Xi[a * KP + l], Sg[l * KP + b], v);
    sm.T[q] = v;
  }
}

// zeta = D^{1/2} L^T and zeta^{-1} after lc_factor, in the sums of k_small_zeta_x.
template <int KP>
__device__ __forceinline__ void lc_zeta(LcShared<KP>& sm, int s) {
  const int kt = threadIdx.x, a = kt % KP, b = kt / KP % KP, seg = (kt & 31) - a;
  const double ra = rsqrt_pos(sm.d[a]), rb = __shfl_sync(kAll, ra, (kt & ~(KP - 1) & 31) + b);
  const bool up = a <= b && b < s;
  sm.Z[a * KP + b] = up ? sm.S[a * KP + b] * ra : 0.0;
  double x = a == b ? 1.0 : 0.0;  // L^{-1}[b][a]: row b of L^{-1}, L^T x = e_b
  double lt[KP];
#pragma unroll
  for (int l = 1; l < KP; ++l) lt[l] = -sm.Lt[a * KP + l];
#pragma unroll
  for (int l = KP - 1; l >= 1; --l) {
    const double xl = __shfl_sync(kAll, x, seg + l);
    if (a < l && l <= b && b < s) x = fma(lt[l], xl, x);
  }
  sm.Zi[a * KP + b] = up ? x * rb : 0.0;
}

// Sn = zeta Sigma by one warp after lc_factor.
template <int KP>
__device__ __forceinline__ void lc_sigma(LcShared<KP>& sm, const double* Sg, double* Sn, int s) {
  for (int q = threadIdx.x & 31; q < KP * KP; q += 32) {
    const int a = q / KP, b = q % KP;
    const double ra = rsqrt_pos(sm.d[a]);
    double v = 0.0;
#pragma unroll
    for (int l = 0; l < KP; ++l)
      if (a <= l && l <= b) v = fma(sm.S[a * KP + l], Sg[l * KP + b], v);
    Sn[q] = (a < s && b < s) ? v * ra : 0.0;
  }
}

// h = argmin nu (lowest index on ties) and the stopping test, by one thread.
template <int KP>
__device__ __forceinline__ void lc_test(LcShared<KP>& sm, int s, int no_test, double tol_abs) {
  long long bb = __double_as_longlong(sm.nu[0]);  // nu >= 0: bit order = value order, NaN last
  int h = 0;
  for (int j = 1; j < s; ++j) {
    const long long v = __double_as_longlong(sm.nu[j]);
    if (v < bb) {
      bb = v;
      h = j;
    }
  }
  sm.nh = sqrt(__longlong_as_double(bb));
  sm.h = h;
  sm.stop = (!no_test && sm.nh < tol_abs) ? 1 : 0;
}

template <int KP>
__device__ __forceinline__ void lds_row(const double* p, double (&v)[KP]) {
  if constexpr (KP == 1) {
    v[0] = p[0];
  } else {
#pragma unroll
    for (int l = 0; l < KP; l += 2) {
      const double2 t = *reinterpret_cast<const double2*>(p + l);
      v[l] = t.x;
      v[l + 1] = t.y;
    }
  }
}

template <int KP>
__global__ void __launch_bounds__(kLcThreads, 1)
k_loop_cluster(int n, const int* __restrict__ rp, const int* __restrict__ ci, const double* __restrict__ av,
               double* Xg, double* Rg, double* Wg, double* Pg, const double* __restrict__ wdiag, double* Sigma,
               SolveState* st, int zcap, int iters, cudaGraphConditionalHandle cond, int use_cond) {
  using C = LcCfg<KP>;
  extern __shared__ __align__(16) double blocks[];
  __shared__ LcShared<KP> sm;
  cg::cluster_group cluster = cg::this_cluster();
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, rank = (int)cluster.block_rank();
  const bool lead = rank == 0 && tid == 0;
  if (st->done) {  // (the same for all CTAs: it is written only after the first barrier)
    if (lead) {
      st->pw_skip = 1;
      if (use_cond) cudaGraphSetConditional(cond, 0);
    }
    return;
  }
  const int s = st->s, maxit = st->maxit, no_test = st->no_test;
  const double tol_abs = st->tol_abs;
  int it = st->it;
  const int r0 = (int)((long long)n * rank / kLcCtas), r1 = (int)((long long)n * (rank + 1) / kLcCtas);
  const int tot = (r1 - r0) * KP, cap = ((n + kLcCtas - 1) / kLcCtas * KP + 1) & ~1;
  double *X = blocks, *R = X + cap, *W = R + cap, *P = W + cap, *Q = P + cap, *V = Q + cap;
  // the CTA's rows of A, the first zcap entries of them: values, the address of P's row in the CTA that owns
  // it; row starts
  const int p0 = __ldg(rp + r0), nz = __ldg(rp + r1) - p0;
  double* as = V + cap;
  uint32_t* ps = reinterpret_cast<uint32_t*>(as + zcap);
  int* rs = reinterpret_cast<int*>(ps + zcap);
  const uint32_t pbase = (uint32_t)__cvta_generic_to_shared(P);
  auto p_row = [&](int col) {
    const int own = (int)((unsigned)(kLcCtas * col + kLcCtas - 1) / (unsigned)n);  // the CTA whose rows have col
    uint32_t a;
    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"(pbase), "r"(own));
    return a + (uint32_t)(col - (int)((long long)n * own / kLcCtas)) * (KP * 8);
  };
  for (int p = tid; p < min(nz, zcap); p += kLcThreads) {
    ps[p] = p_row(__ldg(ci + p0 + p));
    as[p] = __ldg(av + p0 + p);
  }
  for (int i = tid; i <= r1 - r0; i += kLcThreads) rs[i] = __ldg(rp + r0 + i) - p0;
  const size_t g0 = (size_t)r0 * KP;
  for (int e = tid; e < tot; e += kLcThreads) {
    X[e] = Xg[g0 + e];
    R[e] = Rg[g0 + e];
    W[e] = Wg[g0 + e];
    P[e] = Pg[g0 + e];
  }
  for (int q = tid; q < KP * KP; q += kLcThreads) sm.Sg[0][q] = Sigma[q / KP + q % KP * KP];
  cluster.sync();  // every CTA runs and has read the state
  const int m = tid % KP;  // this thread's column of every row it meets
  int done = 0, status = -1, tested = 0, cur = 0;  // cur: which Sigma is the current one
  auto nu_term = [&](int e, double acc) {
    const double r = R[e];
    return fma(wdiag != nullptr ? r * __ldg(wdiag + r0 + e / KP) : r, r, acc);
  };
  for (int u = 0; u < iters; ++u) {
    double val[C::NV];
    // A P and the partials of P^T A P, and nu of the iteration before
#pragma unroll
    for (int v = 0; v < C::NV; ++v) val[v] = 0.0;
    for (int e = tid; e - lane < tot; e += kLcThreads) {
      double acc = 0.0, pm = 0.0;
      if (e < tot) {
        const int i = e / KP, pe = rs[i + 1];
        constexpr int kB = 8;  // entries of a row in flight together
        if (pe <= zcap) {
          for (int p = rs[i]; p < pe; p += kB) {
            double x[kB];
#pragma unroll
            for (int b = 0; b < kB; ++b) x[b] = p + b < pe ? ld_cluster(ps[p + b] + m * 8) : 0.0;
#pragma unroll
            for (int b = 0; b < kB; ++b)
              if (p + b < pe) acc = fma(as[p + b], x[b], acc);
          }
        } else {
          for (int p = rs[i]; p < pe; p += kB) {
            double x[kB], a[kB];
            int c[kB];
#pragma unroll
            for (int b = 0; b < kB; ++b) {
              const int q = p0 + min(p + b, pe - 1);
              c[b] = __ldg(ci + q);
              a[b] = __ldg(av + q);
            }
#pragma unroll
            for (int b = 0; b < kB; ++b) x[b] = ld_cluster(p_row(c[b]) + m * 8);
#pragma unroll
            for (int b = 0; b < kB; ++b)
              if (p + b < pe) acc = fma(a[b], x[b], acc);
          }
        }
        pm = P[e];
        Q[e] = acc;
        val[C::ND] = nu_term(e, val[C::ND]);
      }
#pragma unroll
      for (int v = 0; v < C::ND; ++v) {
        const int o = (m - v + KP) % KP, from = (lane & ~(KP - 1)) + o;
        const double po = v ? __shfl_sync(kAll, pm, from) : pm, qo = v ? __shfl_sync(kAll, acc, from) : acc;
        val[v] = fma(o <= m ? po : pm, o <= m ? acc : qo, val[v]);
      }
    }
    lc_push<KP, C::NV>(sm, val, sm.part1, C::NE, cluster, rank);
    cluster.sync();
    lc_total<KP>(sm, sm.part1, C::NE, s, tid, kLcThreads);
    __syncthreads();
    if (tid < C::KK) {
      const bool bad = lc_factor<KP>(sm, s);
      if (!bad) lc_xi<KP>(sm, s);
      if (tid == 0) {
        sm.bad = bad;
        sm.chunk = 0;
      }
    } else if (tid == kLcThreads - 1) {
      if (u > 0) lc_test<KP>(sm, s, no_test, tol_abs);
      else sm.stop = 0;
    }
    __syncthreads();
    if (sm.stop) {  // the iteration before met the tolerance
      done = 1;
      status = 0;
      break;
    }
    if (sm.bad) {
      done = 1;
      status = 6;
      break;
    }
    ++it;
    // V = W - (A P) Xi, partials of V^T V; T = Xi Sigma
    if (warp == kLcWarps - 1) lc_t<KP>(sm, sm.Sg[cur]);
#pragma unroll
    for (int v = 0; v < C::NV; ++v) val[v] = 0.0;
    {
      double Xi[KP];
#pragma unroll
      for (int l = 0; l < KP; ++l) Xi[l] = sm.Xi[l * KP + m];
      for (int e = tid; e - lane < tot; e += kLcThreads) {
        double vv = 0.0;
        if (e < tot) {
          double q[KP];
          lds_row<KP>(Q + (e - m), q);
          vv = W[e];
#pragma unroll
          for (int l = 0; l < KP; ++l) vv = fma(-q[l], Xi[l], vv);
          V[e] = vv;
        }
#pragma unroll
        for (int v = 0; v < C::ND; ++v) {
          const int o = (m - v + KP) % KP;
          const double vo = v ? __shfl_sync(kAll, vv, (lane & ~(KP - 1)) + o) : vv;
          val[v] = fma(vo, vv, val[v]);
        }
      }
    }
    lc_push<KP, C::ND>(sm, val, sm.part2, C::NP, cluster, rank);
    lc_arrive();
    // The k x k group waits for the other CTAs and takes the zeta step; X~ += P T and R -= (A P) T go on
    // beside it on the other sub-partitions, in chunks of a warp, and the group joins when it is through.
    if ((warp & 3) < C::KK / 32) {
      lc_wait();
      lc_total<KP>(sm, sm.part2, C::NP, s, (warp >> 2) * C::KK + (warp & 3) * 32 + lane, C::KG);
      bar_sync(kBarGroup, C::KG);
      if (tid < C::KK) {
        const bool bad = lc_factor<KP>(sm, s);
        if (tid == 0) sm.bad = bad;
        bar_arrive(kBarSigma, C::KK + 32);
        if (!bad) lc_zeta<KP>(sm, s);
      }
      bar_sync(kBarGroup, C::KG);
    } else if (warp == kLcWarps - 1) {
      bar_sync(kBarSigma, C::KK + 32);
      if (!sm.bad) lc_sigma<KP>(sm, sm.Sg[cur], sm.Sg[cur ^ 1], s);
    }
    {
      double T[KP];
#pragma unroll
      for (int l = 0; l < KP; ++l) T[l] = sm.T[l * KP + m];
      for (;;) {
        int c = 0;
        if (lane == 0) c = atomicAdd(&sm.chunk, 1);
        const int e = __shfl_sync(kAll, c, 0) * 32 + lane;
        if (e - lane >= tot) break;
        if (e < tot) {
          double p[KP], q[KP];
          lds_row<KP>(P + (e - m), p);
          lds_row<KP>(Q + (e - m), q);
          double xv = X[e], rv = R[e];
#pragma unroll
          for (int l = 0; l < KP; ++l) {
            xv = fma(p[l], T[l], xv);
            rv = fma(-q[l], T[l], rv);
          }
          X[e] = xv;
          R[e] = rv;
        }
      }
    }
    if ((warp & 3) >= C::KK / 32) lc_wait();
    __syncthreads();
    const bool zbad = sm.bad != 0;
    if (!zbad) {
      cur ^= 1;
      // W = V zeta^{-1}, P = W + P zeta^T. A thread has the columns ja and jb = KP - 1 - ja of a row: KP + 1
      // terms of each triangular product whatever ja is.
      if constexpr (KP >= 4) {
        constexpr int H = KP / 2;
        const int ja = tid % H, jb = KP - 1 - ja;
        double zi[KP + 1], z[KP + 1];
        int lw[KP + 1], lp[KP + 1];
#pragma unroll
        for (int t = 0; t <= KP; ++t) {
          const bool fw = t <= ja, fp = t < KP - ja;
          lw[t] = fw ? t : t - ja - 1;
          lp[t] = fp ? ja + t : jb + t - (KP - ja);
          zi[t] = sm.Zi[lw[t] * KP + (fw ? ja : jb)];
          z[t] = sm.Z[(fp ? ja : jb) * KP + lp[t]];
        }
        const int half = (r1 - r0) * H;
        for (int f = tid; f - lane < half; f += kLcThreads) {
          const int row = f / H * KP;
          double wa = 0.0, wb = 0.0, pa = 0.0, pb = 0.0;
          if (f < half) {
            double acc = 0.0;
#pragma unroll
            for (int t = 0; t <= KP; ++t) {
              acc = fma(V[row + lw[t]], zi[t], acc);
              if (t == ja) {
                wa = acc;
                acc = 0.0;
              }
            }
            wb = acc;
            acc = wa;
#pragma unroll
            for (int t = 0; t <= KP; ++t) {
              acc = fma(P[row + lp[t]], z[t], acc);
              if (t == KP - 1 - ja) {
                pa = acc;
                acc = wb;
              }
            }
            pb = acc;
          }
          __syncwarp();  // the row's lanes have read V and P
          if (f < half) {
            W[row + ja] = wa;
            W[row + jb] = wb;
            P[row + ja] = pa;
            P[row + jb] = pb;
          }
        }
      } else {
        double Zi[KP], Z[KP];
#pragma unroll
        for (int l = 0; l < KP; ++l) {
          Zi[l] = sm.Zi[l * KP + m];
          Z[l] = sm.Z[m * KP + l];
        }
        for (int e = tid; e - lane < tot; e += kLcThreads) {
          double w = 0.0, pn = 0.0;
          if (e < tot) {
            double v[KP], p[KP];
            lds_row<KP>(V + (e - m), v);
            lds_row<KP>(P + (e - m), p);
#pragma unroll
            for (int l = 0; l < KP; ++l)
              if (l <= m) w = fma(v[l], Zi[l], w);
            pn = w;
#pragma unroll
            for (int l = 0; l < KP; ++l)
              if (l >= m) pn = fma(p[l], Z[l], pn);
          }
          __syncwarp();  // the row's lanes have read V and P
          if (e < tot) {
            W[e] = w;
            P[e] = pn;
          }
        }
      }
    }
    if (!zbad && it < maxit && u + 1 < iters) {
      cluster.sync();  // the new P is complete; nu is tested with the next product
      continue;
    }
    // the last iteration of the launch, or of the solve: its test now
    __syncthreads();
#pragma unroll
    for (int v = 0; v < C::NV; ++v) val[v] = 0.0;
    for (int e = tid; e < tot; e += kLcThreads) val[C::ND] = nu_term(e, val[C::ND]);
    lc_push<KP, C::NV>(sm, val, sm.part1, C::NE, cluster, rank);
    cluster.sync();
    lc_total<KP>(sm, sm.part1, C::NE, s, tid, kLcThreads);
    __syncthreads();
    if (tid == 0) lc_test<KP>(sm, s, no_test, tol_abs);
    __syncthreads();
    tested = 1;
    if (sm.stop) {
      done = 1;
      status = 0;
    } else if (zbad || it >= maxit) {
      done = 1;
      status = zbad ? 6 : no_test ? 0 : 5;
    }
    break;
  }
  __syncthreads();
  for (int e = tid; e < tot; e += kLcThreads) {
    Xg[g0 + e] = X[e];
    Rg[g0 + e] = R[e];
    Wg[g0 + e] = W[e];
    Pg[g0 + e] = P[e];
  }
  if (rank != 0) return;
  for (int q = tid; q < KP * KP; q += kLcThreads) Sigma[q / KP + q % KP * KP] = sm.Sg[cur][q];
  if (tid != 0) return;
  if (it > st->it && !tested) tested = 1;  // left at the Xi step: the test of the iteration before is in sm
  st->it = it;
  if (tested) {
    st->best_col = sm.h;
    st->nu_h = sm.nh;
    st->r_from_v = 0;
  }
  if (sm.stop) st->converged = 1;
  if (done) {
    st->done = 1;
    st->pw_skip = 1;
    st->status = status;
  }
  if (use_cond) cudaGraphSetConditional(cond, done ? 0u : 1u);
}

// Entries of A in the largest of the CTAs' row ranges.
__global__ void k_lc_slice(int n, const int* __restrict__ rp, int* out) {
  int v = 0;
  if (threadIdx.x < kLcCtas)
    v = rp[(long long)n * (threadIdx.x + 1) / kLcCtas] - rp[(long long)n * threadIdx.x / kLcCtas];
  v = __reduce_max_sync(kAll, v);
  if (threadIdx.x == 0) *out = v;
}

size_t lc_smem(int kp, int n, int zcap) {
  const int rows = (n + kLcCtas - 1) / kLcCtas;
  return 6 * (size_t)((rows * kp + 1) & ~1) * sizeof(double) + (size_t)zcap * 12 + (size_t)(rows + 1) * 4;
}

using LcKernel = void (*)(int, const int*, const int*, const double*, double*, double*, double*, double*, const double*,
                          double*, SolveState*, int, int, cudaGraphConditionalHandle, int);

LcKernel lc_kernel(int kp) {
  switch (kp) {
    case 1: return k_loop_cluster<1>;
    case 2: return k_loop_cluster<2>;
    case 4: return k_loop_cluster<4>;
    default: return k_loop_cluster<8>;
  }
}

cudaLaunchConfig_t lc_config(int kp, int n, int zcap, cudaStream_t s, cudaLaunchAttribute* at) {
  cudaLaunchConfig_t c = {};
  c.gridDim = dim3(kLcCtas);
  c.blockDim = dim3(kLcThreads);
  c.dynamicSmemBytes = lc_smem(kp, n, zcap);
  c.stream = s;
  at->id = cudaLaunchAttributeClusterDimension;
  at->val.clusterDim.x = kLcCtas;
  at->val.clusterDim.y = at->val.clusterDim.z = 1;
  c.attrs = at;
  c.numAttrs = 1;
  return c;
}

}  // namespace

// The line: FP64 FMAs of one iteration (the 16 SMs do about 47 thousand a microsecond, 6 to 14 us besides),
// below which no size measured was slower. us per iteration, launches of the row kernels / this kernel:
//   Poisson, s = 1: n = 256 23.9 / 5.9, 16384 26.7 / 10.2, 32761 27.1 / 16.1, 44100 30.4 / 21.3;
//   s = 2: 4096 26.3 / 8.9, 16384 30.3 / 19.2, 25600 30.9 / 29.7; s = 4: 256 31.8 / 8.5, 4096 29.2 / 15.6,
//   8100 29.8 / 24.7, 10000 (1.28 M) 34.1 / 29.0; s = 8: 256 32.8 / 13.8, 2025 (0.91 M) 34.1 / 25.1, 3025
//   (1.35 M) 33.7 / 32.1, 4096 (1.83 M) 33.7 / 38.6; 27-point, s = 4: n = 1728 38.6 / 13.9, 5832 (1.21 M) 36.9 /
//   29.6; s = 8: 1728 (1.04 M) 37.9 / 28.7, 2197 (1.33 M) 37.7 / 34.7.
// From KP = 16 the k x k steps are larger than one warp's work (clusters of their own, small_warp.cu).
static long long lc_fmas(int kp, int n, long long nnz) {
  return nnz * kp + n * ((long long)kp * (2 * (kp / 2 + 1) + 5 * kp + 1));
}
bool loop_cluster_fits(int kp, int n, long long nnz) { return kp <= 8 && lc_fmas(kp, n, nnz) <= 1400000; }

// The same for the CTA with the most entries: where a few neighbouring rows have most of A, one SM does their
// part of the product. us per iteration, row kernels / this kernel, at 16 times the FMAs of that CTA: s = 8, n =
// 1500: 2.25 M 64 / 61, 3.13 M 77 / 95, 3.88 M 88 / 143; s = 4, n = 2000: 2.08 M 108 / 82.
static bool lc_balanced(int kp, int n, int slice) { return lc_fmas(kp, n, 16LL * slice) <= 2250000; }

void loop_cluster_slice(cudaStream_t s, int n, const int* rp, int* out) { k_lc_slice<<<1, 32, 0, s>>>(n, rp, out); }

int loop_cluster_ready(int kp, int n, int slice) {
  constexpr size_t kSmem = 227 * 1024;
  const LcKernel k = lc_kernel(kp);
  cudaFuncAttributes fa;
  cudaLaunchAttribute at;
  int clusters = 0, zcap = -1;
  if (!lc_balanced(kp, n, slice)) return -1;
  bool ok = cudaFuncGetAttributes(&fa, k) == cudaSuccess && lc_smem(kp, n, 0) + fa.sharedSizeBytes <= kSmem;
  if (ok) {
    zcap = (int)std::min((size_t)slice, (kSmem - fa.sharedSizeBytes - lc_smem(kp, n, 0)) / 12);
    const cudaLaunchConfig_t c = lc_config(kp, n, zcap, nullptr, &at);
    ok = cudaFuncSetAttribute(k, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess &&
         cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)(kSmem - fa.sharedSizeBytes)) ==
             cudaSuccess &&
         cudaOccupancyMaxActiveClusters(&clusters, k, &c) == cudaSuccess;
  }
  if (!ok) cudaGetLastError();  // a refusal here only means the launches of the row kernels
  return ok && clusters > 0 && 2 * (long long)zcap >= slice ? zcap : -1;
}

void launch_loop_cluster(cudaStream_t s, int kp, const LoopArgs& a, int iters, cudaGraphConditionalHandle cond,
                         int use_cond) {
  cudaLaunchAttribute at;
  const cudaLaunchConfig_t c = lc_config(kp, a.n, a.zcap, s, &at);
  // (a launch that is refused is the thread's last error, as with the other kernels)
  (void)cudaLaunchKernelEx(&c, lc_kernel(kp), a.n, a.rp, a.ci, a.av, a.X, a.R, a.W, a.P, a.wdiag, a.Sigma, a.st,
                           a.zcap, iters, cond, use_cond);
}

}  // namespace mbpcg
