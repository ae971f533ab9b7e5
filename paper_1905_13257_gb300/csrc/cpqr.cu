// Column-pivoted Householder QR of the small sketch W (l x n, FP64) and the
// solve for the interpolation matrix P.
//
// Algorithm 4 steps 4-8 (transposed): k pivots of a column-pivoted QR of W
// select the skeleton J; C = R11^{-1} R12 by back-substitution; P(:,J) = I,
// P(:,Jc) = C.  The paper's QR is pivoted modified Gram-Schmidt (mgsqr,
// Sec. 2.4); Householder reflections with the same pivot rule give the same
// pivots and R in exact arithmetic and are the stabler choice.
//
// Pivot rule: the largest residual column norm ||W^(s)(s:, j)||, recomputed
// from the updated matrix at every step (no downdating) and compared as its
// square, ties to the lowest column index.
//
// n <= 1024 and l <= 64, or n <= 512 and l <= 96 (cpqr_cluster_kernel, and
// cpqr_batch_kernel for a batch): a cluster of 8 CTAs, every column held in the
// registers of G lanes; one cluster barrier per step.
// Larger n (cpqr_small_kernel): one CTA of 1024 threads works in place on a
// copy of W held row-major in global memory (L2-resident); thread t owns
// columns t, t + 1024, ...
// In both, sums run in a fixed order.
//
// Candidates (the learned proposal's restricted ID).  The cluster form with cpos
// (one int per column): only the columns with cpos[j] >= 0 may become pivots,
// ties going to the lowest cpos, and the rank tolerance is that of the candidate
// columns; every column is updated, so that R11^{-1} R12 is the least-squares
// fit of all columns on W(:, J).  More columns than the cluster holds:
// launch_cpqr_columns.
#include <cooperative_groups.h>
#include <float.h>

#include <type_traits>

#include "cta_qr.cuh"
#include "df.cuh"
#include "idsk_internal.h"

namespace cg = cooperative_groups;

namespace idsk {
namespace {

constexpr int NT = 1024;
constexpr int QMAX = 32;   // columns per thread -> n <= 32768

__global__ void __launch_bounds__(NT, 1)
cpqr_small_kernel(double* __restrict__ M, int rows, int n, int ld, int k, double tol_factor,
                  double* __restrict__ R, int* __restrict__ J, int* __restrict__ colpos,
                  int* __restrict__ kout, qr::Reflectors refl) {
  __shared__ qr::QrShared sh;
  qr::cta_pivoted_qr<NT>(M, rows, n, ld, k, tol_factor, R, J, colpos, kout, sh, refl);
}


constexpr int CL_CTAS = 8;                    // CTAs of the cluster
constexpr int CL_WARPS = 8;                   // warps that hold columns
static_assert(CL_CTAS == 8 && CL_WARPS == 8, "best_of_8");
constexpr int CL_WORKERS = CL_WARPS * 32;
constexpr int CL_THREADS = CL_WORKERS + 32;   // and one warp for the step's scalars

// A candidate column: its residual norm as an ordered integer (0: none), its
// place in the tie order, its index, its rows.
struct Cand {
  double col[kLMaxW];
  unsigned long long key;
  int ord, j;
};

// Shared scratch of one QR.
struct ClusterQr {
  Cand inbox[2][CL_CTAS];   // every CTA's best candidate, by step parity
  Cand wbest[CL_WARPS];
  double fro_w[CL_WARPS], fro_in[CL_CTAS];
  double gamma, v0, beta;
};

__device__ __forceinline__ bool nonzero(double x) {   // on the integer units
  return ((unsigned long long)__double_as_longlong(x) << 1) != 0ull;
}

// The lanes that hold the largest key and, among these, the lowest order
// (whole warp; on the integer units).
__device__ __forceinline__ bool warp_best(unsigned long long key, int ord,
                                          unsigned long long* best, int* best_ord) {
  const unsigned hi = (unsigned)(key >> 32);
  const unsigned mh = __reduce_max_sync(0xffffffffu, hi);
  const unsigned lo = hi == mh ? (unsigned)key : 0u;
  const unsigned ml = __reduce_max_sync(0xffffffffu, lo);
  const bool top = hi == mh && lo == ml;
  const int o = __reduce_min_sync(0xffffffffu, top ? ord : 0x7fffffff);
  *best = ((unsigned long long)mh << 32) | ml;
  *best_ord = o;
  return top && ord == o;
}

// The best of 8 candidates (whole warp).
__device__ __forceinline__ int best_of_8(const Cand* c, int lane) {
  unsigned long long k;
  int o;
  const bool win = warp_best(c[lane & 7].key, c[lane & 7].ord, &k, &o);
  return (__ffs(__ballot_sync(0xffffffffu, win)) - 1) & 7;
}

// The matrix of a QR: W itself (row-major), or columns of it ...
struct MatrixSrc {
  const double* M;
  int64_t ld;
  const int* cols = nullptr;
  template <int G, int RPT>
  __device__ __forceinline__ void fill(double (&c)[RPT], int g, int j, int rows) const {
    if (cols) j = cols[j];
#pragma unroll
    for (int q = 0; q < RPT; ++q)
      if (g + G * q < rows) c[q] = M[(int64_t)(g + G * q) * ld + j];
  }
};
// ... or, in a batch, the sum of the work items' FP32 slabs in item order as
// FP32 pairs (deterministic), four slabs' rows in flight per lane.
struct SlabSrc {
  const BatchItem* items;   // the job's
  const float* slabs;
  int nitem, lw;
  template <int G, int RPT>
  __device__ __forceinline__ void fill(double (&c)[RPT], int g, int j, int rows) const {
    constexpr int AHEAD = 4;
    float hi[RPT], lo[RPT];
#pragma unroll
    for (int q = 0; q < RPT; ++q) hi[q] = lo[q] = 0.f;
    const float* src = slabs + slab_index(j, 0, lw);
    for (int i0 = 0; i0 < nitem; i0 += AHEAD) {
      float x[AHEAD][RPT];
#pragma unroll
      for (int u = 0; u < AHEAD; ++u) {
        const float* p = src + items[min(i0 + u, nitem - 1)].slab;
#pragma unroll
        for (int q = 0; q < RPT; ++q) x[u][q] = g + G * q < lw ? p[slab_index(0, g + G * q, lw)] : 0.f;
      }
#pragma unroll
      for (int u = 0; u < AHEAD; ++u)
        if (i0 + u < nitem) {
#pragma unroll
          for (int q = 0; q < RPT; ++q) df_add(hi[q], lo[q], x[u][q], 0.f);
        }
    }
#pragma unroll
    for (int q = 0; q < RPT; ++q)
      if (g + G * q < rows) c[q] = (double)hi[q] + (double)lo[q];
  }
};

// Column-pivoted Householder QR of M (rows x n row-major, rows <= LM, n <=
// 8 * 256 / G) by a cluster of 8 CTAs.  M is only read.
//
// What bounds it is not the arithmetic (60 x 1000, k = 50: 5 MFMA) but the
// chain of dependent phases of a step on narrow FP64 units (a warp's FP64
// instruction takes an SM sub-partition's pipe for about 64 cycles, also when
// it is predicated off).  So: a column's rows are spread over G lanes (row i
// in lane i mod G: 4 to 32 rows a lane, rows above the pivot row are skipped
// by branches that are uniform over the warp), G the largest that n allows;
// columns are dealt to the CTAs in turn; the next norms are summed while the
// columns are updated; every CTA pushes its best column with its norm into
// the other CTAs' shared memory, so that one cluster barrier per step is
// enough; the reflector is used unscaled, H = I - gamma v v^T with v = x,
// v_s = x_s - beta and gamma = 1 / (||x||^2 + |x_s| ||x||), so that the
// products v^T c start before the scalars, which a warp of their own forms
// meanwhile (one square root and one division).  Rounding differs from the
// scaled form by a few ulp only.
// Measured (k = 50, l = 60; before: one column per thread, two cluster
// barriers, every row in every step, 12.9 us a step for any n): n = 512 640 ->
// 248 us, n = 200 (k = 20, l = 30) 258 -> 86 us, n = 1000 1779 us in one CTA
// -> 387 us.
// LM: most rows (64 or 96).  src.fill(c, g, j, rows) loads a lane's rows g, g +
// G, ... of column j (rows past the last: zero).
// KEEP: the reflectors go to refl.
template <int G, int LM, bool KEEP = false, typename Src>
__device__ __forceinline__ void cluster_qr(const Src& src, int rows, int n, int k,
                                           double tol_factor,
                                           const int* __restrict__ cpos, double* __restrict__ R,
                                           int* __restrict__ J, int* __restrict__ colpos,
                                           int* __restrict__ kout, ClusterQr& sh,
                                           qr::Reflectors refl = {}) {
  constexpr int RPT = LM / G;   // rows per lane
  cg::cluster_group cl = cg::this_cluster();
  cl.barrier_arrive();   // waited for before the first write into another CTA
  auto& inbox = sh.inbox;
  auto& wbest = sh.wbest;
  const int rank = (int)cl.block_rank();
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
  const bool worker = warp < CL_WARPS;
  const int g = lane & (G - 1);
  const int j = (t / G) * CL_CTAS + rank;
  const bool have = worker && j < n;
  const bool busy = worker && ((t & ~31) / G) * CL_CTAS + rank < n;   // the warp holds a column
  const int kmax = min(k, min(rows, n));

  double c[RPT];
#pragma unroll
  for (int q = 0; q < RPT; ++q) c[q] = 0.0;
  if (have) src.template fill<G>(c, g, j, rows);
  int ord = 0x7fffffff;   // place in the tie order; past the last: never a pivot
  if (have) {
    ord = cpos ? cpos[j] : j;
    if (ord < 0) ord = 0x7fffffff;
    if (g == 0) colpos[j] = -1;
  }
  bool piv = false;

  // sum over the G lanes of a column (fixed tree)
  auto group_sum = [&](double v) {
#pragma unroll
    for (int o = 1; o < G; o <<= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
  };
  double ss = 0.0;   // the column's residual norm, squared
  if (busy) {
#pragma unroll
    for (int q = 0; q < RPT; ++q)
      if (G * q < rows) ss += c[q] * c[q];
    ss = group_sum(ss);
  }
  // ||W||_F of the candidates: columns of a warp, warps, CTAs in order
  if (worker) {
    double f = ord != 0x7fffffff ? ss : 0.0;
#pragma unroll
    for (int o = G; o < 32; o <<= 1) f += __shfl_xor_sync(0xffffffffu, f, o);
    if (lane == 0) sh.fro_w[warp] = f;
  }
  __syncthreads();
  cl.barrier_wait();
  if (t < CL_CTAS) {
    double f = 0.0;
    for (int w = 0; w < CL_WARPS; ++w) f += sh.fro_w[w];
    *cl.map_shared_rank(&sh.fro_in[rank], t) = f;   // read after step 0's cluster barrier
  }
  double tol2 = 0.0;

  int s = 0;
  for (; s < kmax; ++s) {
    const int b = s & 1;
    const int gs = s & (G - 1), qs = s / G;   // lane and register of the pivot row
    // the warp's candidate: largest norm, ties to the lowest order
    if (worker) {
      unsigned long long key = 0ull;
      if (ord != 0x7fffffff && !piv) key = (unsigned long long)__double_as_longlong(ss) + 1ull;
      unsigned long long wk;
      int o;
      const bool win = warp_best(key, ord, &wk, &o);
      if (lane == 0) {
        wbest[warp].key = wk;
        wbest[warp].ord = o;
      }
      if (wk != 0ull && win) {
#pragma unroll
        for (int q = 0; q < RPT; ++q)
          if (q >= qs) wbest[warp].col[g + G * q] = c[q];
        if (g == 0) wbest[warp].j = j;
      }
    }
    __syncthreads();
    // the CTA's candidate into every CTA's inbox
    {
      const int w = best_of_8(wbest, lane);
      for (int e = t; e < CL_CTAS * LM; e += CL_THREADS) {
        const int i = e % LM;
        if (i >= s && i < rows)
          cl.map_shared_rank(&inbox[b][rank], e / LM)->col[i] = wbest[w].col[i];
      }
      if (t < CL_CTAS) {
        Cand* dst = cl.map_shared_rank(&inbox[b][rank], t);
        dst->key = wbest[w].key;
        dst->ord = wbest[w].ord;
        dst->j = wbest[w].j;
      }
    }
    cl.sync();
    const int best = best_of_8(inbox[b], lane);
    const Cand& pc = inbox[b][best];
    double nrm2 = __longlong_as_double((long long)(pc.key - 1ull));
    if (s == 0) {
      double f = 0.0;
      for (int x = 0; x < CL_CTAS; ++x) f += sh.fro_in[x];
      const int e2 = (int)((unsigned long long)__double_as_longlong(f) >> 52) - 1023;
      if (f > 0.0 && e2 < 1024 && (e2 < -800 || e2 > 1000)) {   // uniform over the cluster
        // data of extreme scale, whose squares (or their reciprocals) leave
        // FP64's range or lose bits: go on with W times a power of two, which
        // J and P do not depend on (R is the solve's input only)
        const double scale = __longlong_as_double((long long)(1023 - e2 / 2) << 52);
        f = f * scale * scale;
        if (busy) {
          ss = 0.0;
#pragma unroll
          for (int q = 0; q < RPT; ++q) {
            c[q] *= scale;
            ss += c[q] * c[q];
          }
          ss = group_sum(ss);
        }
        for (int i = t; i < rows; i += CL_THREADS) inbox[b][best].col[i] *= scale;   // own copy
        __syncthreads();
        nrm2 = 0.0;
        for (int i = 0; i < rows; ++i) nrm2 += pc.col[i] * pc.col[i];
      }
      const double tol = tol_factor * DBL_EPSILON * sqrt(f);
      tol2 = tol * tol;
    }
    if (pc.key == 0ull || !(nrm2 > tol2)) break;   // uniform over the cluster
    const int p = pc.j;
    double x[RPT], d = 0.0, cs = 0.0;
    if (!worker) {
      // scalars of the reflector; below the pivot row all zero: H = I
      const double a0 = pc.col[s];
      const double x0 = s + 1 + lane < rows ? pc.col[s + 1 + lane] : 0.0;
      const double x1 = s + 33 + lane < rows ? pc.col[s + 33 + lane] : 0.0;
      const double x2 = (LM > 64 && s + 65 + lane < rows) ? pc.col[s + 65 + lane] : 0.0;
      const bool any = __any_sync(0xffffffffu, nonzero(x0) || nonzero(x1) || nonzero(x2));
      if (lane == 0) {
        double beta = a0, gamma = 0.0, v0 = 0.0;
        if (any) {
          const double nrm = sqrt(nrm2);
          beta = a0 >= 0.0 ? -nrm : nrm;
          v0 = a0 - beta;
          gamma = 1.0 / (nrm2 + fabs(a0) * nrm);
        }
        sh.beta = beta;
        sh.gamma = gamma;
        sh.v0 = v0;
        if (rank == 0) {
          J[s] = p;
          colpos[p] = s;
        }
      }
    } else if (busy) {
      // x = the pivot column below row s; d = x^T c, cs = row s of the column
#pragma unroll
      for (int q = 0; q < RPT; ++q) {
        x[q] = 0.0;
        if (q >= qs && G * q < rows) {
          if (g + G * q > s && g + G * q < rows) x[q] = pc.col[g + G * q];
          d += x[q] * c[q];
          if (q == qs) cs = c[q];
        }
      }
      d = group_sum(d);
      cs = __shfl_sync(0xffffffffu, cs, (lane & ~(G - 1)) + gs);
    }
    __syncthreads();
    if (KEEP && rank == 0 && !worker) {
      for (int i = s + lane; i < rows; i += 32)
        refl.V[(int64_t)s * rows + i] = i == s ? sh.v0 : pc.col[i];
      if (lane == 0) refl.gamma[s] = sh.gamma;
    }
    if (busy) {
      const double v0 = sh.v0;
      const double w = sh.gamma * (d + v0 * cs);
      ss = 0.0;
#pragma unroll
      for (int q = 0; q < RPT; ++q) {
        if (q >= qs && G * q < rows) {
          c[q] -= w * x[q];
          const double y = (q > qs || g > gs) ? c[q] : 0.0;   // rows below s
          ss += y * y;
        }
      }
      ss = group_sum(ss);
      if (j == p) piv = true;
      if (have && g == 0)
        R[(int64_t)s * n + j] = j == p ? sh.beta : (piv ? 0.0 : cs - w * v0);
    }
  }
  if (rank == 0) {
    if (t == 0) *kout = s;
    for (int q = s + t; q < k; q += CL_THREADS) J[q] = -1;
  }
}

template <int G, int LM>
__global__ void __cluster_dims__(CL_CTAS, 1, 1) __launch_bounds__(CL_THREADS, 1)
    cpqr_cluster_kernel(const double* __restrict__ M, int rows, int n, int64_t ld, int k,
                        double tol_factor, const int* __restrict__ cpos, double* __restrict__ R,
                        int* __restrict__ J, int* __restrict__ colpos, int* __restrict__ kout) {
  __shared__ ClusterQr sh;
  cluster_qr<G, LM>(MatrixSrc{M, ld}, rows, n, k, tol_factor, cpos, R, J, colpos, kout, sh);
}

// The QR of the columns cols[0 .. n) of M, its reflectors kept (rows <= 64).
template <int G>
__global__ void __cluster_dims__(CL_CTAS, 1, 1) __launch_bounds__(CL_THREADS, 1)
    cpqr_columns_kernel(const double* __restrict__ M, int rows, int n, int64_t ld,
                        const int* __restrict__ cols, int k, double tol_factor,
                        double* __restrict__ R, int* __restrict__ J, int* __restrict__ colpos,
                        int* __restrict__ kout, qr::Reflectors refl) {
  __shared__ ClusterQr sh;
  cluster_qr<G, kLMax, true>(MatrixSrc{M, ld, cols}, rows, n, k, tol_factor, nullptr, R, J, colpos,
                             kout, sh, refl);
}

// work = M(:, cols), row-major rows x n (the one-CTA QR works in place).
__global__ void gather_columns_kernel(const double* __restrict__ M, int rows, int n, int64_t ld,
                                      const int* __restrict__ cols, double* __restrict__ work) {
  const int j = blockIdx.x * blockDim.x + threadIdx.x;
  if (j >= n) return;
  const int c = cols[j];
  for (int i = blockIdx.y; i < rows; i += gridDim.y)
    work[(int64_t)i * n + j] = M[(int64_t)i * ld + c];
}

// R(:, j) = the first k_out rows of H_(k_out - 1) ... H_0 M(:, j) for every
// column j of M (rows <= 64), colpos, and J = cols[Jc]: 16 lanes a column (row i
// in lane i mod 16), the reflectors in shared memory.
constexpr int RA_THREADS = 256, RA_COLS = RA_THREADS / 16;
__global__ void __launch_bounds__(RA_THREADS) reflect_columns_kernel(
    const double* __restrict__ M, int rows, int n, int64_t ld, const double* __restrict__ V,
    const double* __restrict__ gamma, const int* __restrict__ cols, const int* __restrict__ Jc,
    const int* __restrict__ kout, int k, double* __restrict__ R, int* __restrict__ J,
    int* __restrict__ colpos) {
  extern __shared__ double vs[];   // k_out x 64, zero outside rows s .. rows - 1
  __shared__ double gs[kLMax];
  __shared__ int Js[kLMax];
  const int kk = *kout, t = threadIdx.x, g = t & 15;
  for (int e = t; e < kk * kLMax; e += RA_THREADS) {
    const int s = e / kLMax, i = e % kLMax;
    vs[e] = i >= s && i < rows ? V[(int64_t)s * rows + i] : 0.0;
  }
  for (int u = t; u < kk; u += RA_THREADS) {
    gs[u] = gamma[u];
    Js[u] = cols[Jc[u]];
  }
  __syncthreads();
  if (blockIdx.x == 0)
    for (int u = t; u < k; u += RA_THREADS) J[u] = u < kk ? Js[u] : -1;
  const int j = blockIdx.x * RA_COLS + (t >> 4);
  const bool in = j < n;
  double c[4];
#pragma unroll
  for (int q = 0; q < 4; ++q)
    c[q] = in && g + 16 * q < rows ? M[(int64_t)(g + 16 * q) * ld + j] : 0.0;
  int pos = -1;
  for (int u = g; u < kk; u += 16)
    if (Js[u] == j) pos = u;
#pragma unroll
  for (int o = 1; o < 16; o <<= 1) pos = max(pos, __shfl_xor_sync(0xffffffffu, pos, o));
  if (in && g == 0) colpos[j] = pos;
  for (int s = 0; s < kk; ++s) {
    const double* v = vs + s * kLMax + g;
    double d = 0.0;
#pragma unroll
    for (int q = 0; q < 4; ++q)
      if (q >= s >> 4) d += v[16 * q] * c[q];
#pragma unroll
    for (int o = 1; o < 16; o <<= 1) d += __shfl_xor_sync(0xffffffffu, d, o);
    const double w = gs[s] * d;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      if (q >= s >> 4) c[q] -= w * v[16 * q];
      if (in && 16 * q + g == s) R[(int64_t)s * n + j] = c[q];
    }
  }
}

// The slab sums and pivoted QRs of a batch, one cluster per job (n <= 512): all
// of them run at once, on up to 8 SMs each.
__global__ void __cluster_dims__(CL_CTAS, 1, 1) __launch_bounds__(CL_THREADS, 1)
    cpqr_batch_kernel(const QrJob* __restrict__ jobs, const BatchJob* __restrict__ bjobs,
                      const BatchItem* __restrict__ items, const float* __restrict__ slabs,
                      double tol_factor) {
  __shared__ ClusterQr sh;
  const QrJob q = jobs[blockIdx.x / CL_CTAS];
  const BatchJob& bj = bjobs[q.job];
  const SlabSrc src{items + bj.item0, slabs, bj.nitem, w_width(q.rows, false)};
  const int cols = (q.n + CL_CTAS - 1) / CL_CTAS;
  auto go = [&](auto g, auto lm) {
    cluster_qr<decltype(g)::value, decltype(lm)::value>(src, q.rows, q.n, q.k, tol_factor,
                                                        nullptr, q.R, q.J, q.colpos, q.kout, sh);
  };
  using L64 = std::integral_constant<int, 64>;
  using L96 = std::integral_constant<int, 96>;
  if (q.rows <= 64) {
    if (cols <= CL_WORKERS / 16)
      go(std::integral_constant<int, 16>(), L64());
    else if (cols <= CL_WORKERS / 8)
      go(std::integral_constant<int, 8>(), L64());
    else
      go(std::integral_constant<int, 4>(), L64());
  } else if (cols <= CL_WORKERS / 8) {
    go(std::integral_constant<int, 8>(), L96());
  } else {
    go(std::integral_constant<int, 4>(), L96());
  }
}


// P(:, j) for every column j: e_u when j = J[u]; otherwise the solution of
// R11 x = R(:, j) by back-substitution, R11(t, u) = R(t, J[u]).  One warp per
// column, column-oriented: x_t = b_t / R11(t, t) (by the diagonal's
// reciprocal, formed once per block), then b_u -= R11(u, t) x_t
// for u < t, lane u holding b_u and b_{u+32}.  R11 lives in shared memory.
constexpr int SP_WARPS = 8;
constexpr size_t kSolveSmem = sizeof(double) * kLMaxW * kLMaxW;   // R11, at most
__device__ __forceinline__ void solve_p_body(const double* __restrict__ R,
                                             const int* __restrict__ J,
                                             const int* __restrict__ colpos,
                                             const int* __restrict__ kout, int k, int n,
                                             double* __restrict__ P, int cblock) {
  extern __shared__ double r11[];   // kk x kk, row-major
  __shared__ int Js[kLMaxW];
  __shared__ double rdiag[kLMaxW];   // 1 / R11(t, t)
  const int kk = qr::solve_setup(R, J, kout, n, r11, Js, rdiag);
  const int j = cblock * SP_WARPS + (threadIdx.x >> 5);
  if (j < n) qr::solve_column(j, R, colpos, k, kk, n, P, r11, rdiag);
}

__global__ void __launch_bounds__(SP_WARPS * 32) solve_p_kernel(
    const double* __restrict__ R, const int* __restrict__ J, const int* __restrict__ colpos,
    const int* __restrict__ kout, int k, int n, double* __restrict__ P) {
  solve_p_body(R, J, colpos, kout, k, n, P, blockIdx.x);
}

__global__ void __launch_bounds__(SP_WARPS * 32) solve_batch_kernel(
    const QrJob* __restrict__ jobs) {
  const QrJob q = jobs[blockIdx.y];
  if ((int)blockIdx.x * SP_WARPS >= q.n) return;
  solve_p_body(q.R, q.J, q.colpos, q.kout, q.k, q.n, q.P, blockIdx.x);
}


}  // namespace

bool cpqr_cluster_ok(int rows, int64_t n) {
  return n <= (rows <= kLMax ? 1024 : 512) && rows <= kLMaxW;
}

// Up to 512 columns for 65 to 96 rows (24 or fewer rows a lane).
// The cluster form reads W itself; the one-CTA form works in place on a copy
// of W in `work` (rows x n).  G: the most lanes per column that n columns on 8
// CTAs of 256 threads allow.
cudaError_t launch_cpqr_small(const double* W, int64_t ldw, double* work, int rows, int n, int k,
                              double tol_factor, const int* cpos, double* R, int* J, int* colpos,
                              int* kout, cudaStream_t st, bool one_cta) {
  if (n > NT * QMAX || rows > kLMaxW || k > kLMaxW) return cudaErrorInvalidValue;
  if (cpos && !cpqr_cluster_ok(rows, n)) return cudaErrorInvalidValue;
  if (!one_cta && cpqr_cluster_ok(rows, n)) {
    const int cols = (n + CL_CTAS - 1) / CL_CTAS;   // columns per CTA
    auto go = [&](auto kern) {
      kern<<<CL_CTAS, CL_THREADS, 0, st>>>(W, rows, n, ldw, k, tol_factor, cpos, R, J, colpos,
                                           kout);
    };
    const bool wide = rows > kLMax;
    if (cols <= CL_WORKERS / 16)
      wide ? go(cpqr_cluster_kernel<16, 96>) : go(cpqr_cluster_kernel<16, 64>);
    else if (cols <= CL_WORKERS / 8)
      wide ? go(cpqr_cluster_kernel<8, 96>) : go(cpqr_cluster_kernel<8, 64>);
    else if (cols <= CL_WORKERS / 4)
      wide ? go(cpqr_cluster_kernel<4, 96>) : go(cpqr_cluster_kernel<4, 64>);
    else
      go(cpqr_cluster_kernel<2, 64>);
  } else {
    const cudaError_t e =
        cudaMemcpy2DAsync(work, sizeof(double) * n, W, sizeof(double) * ldw, sizeof(double) * n,
                          rows, cudaMemcpyDeviceToDevice, st);
    if (e != cudaSuccess) return e;
    cpqr_small_kernel<<<1, NT, 0, st>>>(work, rows, n, n, k, tol_factor, R, J, colpos, kout,
                                        qr::Reflectors{});
  }
  count_launches(1);
  return cudaGetLastError();
}

// Candidates of a W with more columns than a cluster holds: the QR of W(:, cand)
// alone (the cluster form up to 1024 candidates), its reflectors then applied to
// all columns, whose work spreads over the SMs; the masked QR of all n columns
// would run in one CTA, in time proportional to n.  Measured, with the solve and
// the copies of the call (k = 50, l = 60, 100 candidates): n = 4096 404 us in place of
// 5152 us masked, n = 16,384 786 and 16,848 us.
cudaError_t launch_cpqr_columns(const double* W, int64_t ldw, double* work, int rows, int n, int k,
                                double tol_factor, const int* cand, int ncand, double* refl,
                                double* R, int* Jc, int* J, int* colpos, int* kout,
                                cudaStream_t st) {
  if (ncand > NT * QMAX || rows > kLMax || k > kLMax) return cudaErrorInvalidValue;
  const qr::Reflectors rf{refl, refl + (size_t)k * rows};
  if (cpqr_cluster_ok(rows, ncand)) {
    const int per = (ncand + CL_CTAS - 1) / CL_CTAS;   // columns per CTA
    auto go = [&](auto kern) {
      kern<<<CL_CTAS, CL_THREADS, 0, st>>>(W, rows, ncand, ldw, cand, k, tol_factor, R, Jc, colpos,
                                           kout, rf);
    };
    if (per <= CL_WORKERS / 16)
      go(cpqr_columns_kernel<16>);
    else if (per <= CL_WORKERS / 8)
      go(cpqr_columns_kernel<8>);
    else if (per <= CL_WORKERS / 4)
      go(cpqr_columns_kernel<4>);
    else
      go(cpqr_columns_kernel<2>);
  } else {
    gather_columns_kernel<<<dim3((ncand + 255) / 256, 8), 256, 0, st>>>(W, rows, ncand, ldw, cand,
                                                                        work);
    cpqr_small_kernel<<<1, NT, 0, st>>>(work, rows, ncand, ncand, k, tol_factor, R, Jc, colpos,
                                        kout, rf);
    count_launches(1);
  }
  const cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  reflect_columns_kernel<<<(n + RA_COLS - 1) / RA_COLS, RA_THREADS, sizeof(double) * kLMax * k,
                           st>>>(W, rows, n, ldw, refl, rf.gamma, cand, Jc, kout, k, R, J, colpos);
  count_launches(2);
  return cudaGetLastError();
}

// The QRs of a batch and their solves, in job order (the caller puts the long
// ones first).
cudaError_t launch_qr_batch(const QrJob* jobs, int njobs, const BatchJob* bjobs,
                            const BatchItem* items, const float* slabs, int kmax, int nmax,
                            double tol_factor, cudaStream_t st) {
  if (njobs <= 0) return cudaSuccess;
  cpqr_batch_kernel<<<njobs * CL_CTAS, CL_THREADS, 0, st>>>(jobs, bjobs, items, slabs, tol_factor);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  const size_t sm = sizeof(double) * (size_t)kmax * kmax;
  e = allow_smem(solve_batch_kernel, kSolveSmem);
  if (e != cudaSuccess) return e;
  solve_batch_kernel<<<dim3((nmax + SP_WARPS - 1) / SP_WARPS, njobs), SP_WARPS * 32, sm, st>>>(
      jobs);
  count_launches(2);
  return cudaGetLastError();
}

cudaError_t launch_solve_p(const double* R, const int* J, const int* colpos, const int* kout,
                           int k, int n, double* P, cudaStream_t st) {
  const size_t sm = sizeof(double) * (size_t)k * k;
  if (sm > 48 * 1024) {
    const cudaError_t e = allow_smem(solve_p_kernel, kSolveSmem);
    if (e != cudaSuccess) return e;
  }
  solve_p_kernel<<<(n + SP_WARPS - 1) / SP_WARPS, SP_WARPS * 32, sm, st>>>(R, J, colpos, kout, k,
                                                                         n, P);
  count_launches(1);
  return cudaGetLastError();
}

}  // namespace idsk
