// The coarse-grid pivoted QR (Algorithm 5 steps 3-7, transposed) as one
// cooperative, persistent launch: all k steps of the left-looking Householder
// QR of A_c (m_c x n) in a single kernel, with grid-wide barriers between the
// dependent phases of a step instead of four dependent launches.
//
// Work split.  CTA b owns a fixed range of A_c's rows (at most 512) for the
// passes over rows, and a fixed range of columns for the per-column updates.
// Per step s, with pivot p:
//   A  pivot from the norms (every CTA, same data, same choice); scale
//      column s-1 of V into v_{s-1}; for the CTA's rows (one per thread)
//        u = A(:, p) - V_s F(p, :)^T     (rows >= s; kept as column s of V),
//      the CTA's partials of V_s^T u and ||u||^2 (rows > s), and its share
//      of A^T u: its rows of every column (warp w takes columns w, w + 16,
//      ..., loaded a column ahead of the sums, so that the warps stream A_c
//      independently of one another), one partial per (CTA, column);
//   -- grid barrier --
//   B  every CTA sums the partials (in CTA order) into the Householder
//      scalars alpha = u_s, beta, tau, den = alpha - beta and h = V_s^T v_s;
//   C  for the CTA's columns: g_j = A(s, j) + (A^T u)_j / den, F(j, s),
//      R(s, j) and the norm downdate (a norm that lost more than 20 bits is
//      recomputed from its definition, rows split over the CTAs);
//   -- grid barrier --
// A^T v_s = A(s, :)^T + (A^T u below row s) / (u_s - beta) lets the pass over
// A_c run before the scalars exist, so a step needs two grid barriers.
//
// A CTA's rows of V are needed by that CTA alone (but for row s of the step,
// which its owner publishes), so V lives in shared memory, 8 bytes an entry:
// 512 rows x 50 columns fill 205 KB; columns that do not fit stay in global
// memory.
// Arithmetic: the passes over rows and the sums of their per-CTA partials in
// FP32 pairs (about 48 bits) for FP32 data in whole row quads; FP32 data with
// an odd number of rows: FP32 pairs over a lane's rows, FP64 from there on and
// for the first norms; FP64 for the products of FP64 data (V is kept as FP32
// pairs for all); scalars, F, R and the norms in FP64; every sum in a fixed
// order.  GB300's FP64 pipe is narrow (a warp's FP64 instruction holds it for
// about 60 cycles), so nothing per row of the steps' passes over FP32 data runs
// in FP64.
//
// Number of CTAs: one per SM for large A_c, at least 16,384 entries each for
// small ones: a step of a small QR is a chain of latencies, and fewer CTAs
// make its barriers and partial sums cheaper.
//
// What bounds it: for large A_c the pass, one read of A_c per step (73,728 x
// 1000: 90K of a step's 123K cycles, 295 MB at 6.8 TB/s with the 50 MB that
// stay in L2), then the waiting for the slowest CTA (8K) and the chain of
// phases around it; for small A_c that chain (about 26K cycles).
// Measured (before: V in global memory, a reduction tree per column, branches
// around loads, one CTA per SM always; odd m_c and FP64 on four launches per
// step): 73,728 x 1000, k = 50 on 144 SMs 3.79 -> 3.07 ms; 42,075 x 333, k =
// 50 about 5.5 -> 1.26 ms with pair sums throughout, about 0.12 ms more with the
// wider sums of odd m_c; 1152 x 96, k = 8 196 -> 125 us; FP64 1536 x 200, k = 20
// about 1 ms -> 330 us.
// Two columns in registers per warp (three or four were slower: the longer
// loop costs more in instruction fetch than the loads ahead gain).
//
// Waits are bounded: a grid barrier that gives up raises the status word, and
// every CTA then leaves its step loop.
#include <float.h>
#include <stdlib.h>
#include <string.h>

#include <algorithm>
#include <type_traits>

#include "df.cuh"
#include "idsk_internal.h"
#include "tc_common.cuh"

namespace idsk {
namespace {

constexpr int CW = 16;               // warps
constexpr int CT = CW * 32;          // threads
constexpr int RMAX = 512;            // rows per CTA at most: one per thread
constexpr int HP = kLMax + 1;        // per-CTA partials: V^T u (kLMax), ||u||^2
constexpr double kRecomputeFrac = 1.0 / (1 << 20);
// cint slots (shared with coarse.cu's layout where the host reads them)
constexpr int CI_P = 0, CI_STOP = 1, CI_NREC = 2, CI_KOUT = 3, CI_BAR = 4, CI_NREC_ODD = 6;
// the recompute counter of step s: slot CI_NREC (even s) or CI_NREC_ODD (odd
// s); CTA 0 clears the slot of step s during step s, whose users all passed
// step s - 2's barriers long before
__device__ __forceinline__ int nrec_slot(int s) { return (s & 1) ? CI_NREC_ODD : CI_NREC; }

// Optional timeline of CTA 0 (clock64 at the phase boundaries of every step),
// compiled only when IDSK_CC_TRACE is defined by a profiling harness.
#ifdef IDSK_CC_TRACE
__device__ long long g_cc_trace[64 * 16];
#define CC_TRACE(s, point)                                                        \
  do {                                                                            \
    if (blockIdx.x == 0 && threadIdx.x == 0 && (s) < 64) g_cc_trace[(s) * 16 + (point)] = clock64(); \
  } while (0)
#else
#define CC_TRACE(s, point) \
  do {                     \
  } while (0)
#endif

struct CoopArgs {
  const void* Ac;       // mc x n, FP32 or FP64
  int64_t mc;
  int n, kmax, k;
  int64_t ldf;
  float2* V;            // mc x k FP32 pairs, column-major: the columns past vs_cols
  int vs_cols, vs_rows; // columns of V in shared memory, their leading dimension
  double* F;            // F[t * ldf + j]
  double* Rc;           // k x n
  double* nu2;          // residual norms squared, -1 once pivoted
  double* nu20;
  int* colpos;
  int* Jc;
  double* gpart;        // G x n: per-CTA column partials (FP32 pairs or FP64)
  float2* upart;        // G x HP
  float2* vrow;         // row s of V (t < s) and u_s (slot kLMax), from its owner
  int* rlist;
  int* cint;
  int* status;
  int keep_cols;        // leading columns whose loads are kept in L2 (evict_last)
  double tol_factor;
};

// Read-only loads with an L2 cache policy (createpolicy), zero where `on` is
// false: predicated inside, since a branch around a load costs more than the
// load and makes the next instruction wait for it.
__device__ __forceinline__ float4 ld_hint(const float4* p, uint64_t policy, bool on) {
  float4 v;
  asm volatile(
      "{\n .reg .pred q;\n setp.ne.b32 q, %6, 0;\n mov.f32 %0, 0f00000000;\n"
      " mov.f32 %1, 0f00000000;\n mov.f32 %2, 0f00000000;\n mov.f32 %3, 0f00000000;\n"
      " @q ld.global.nc.L2::cache_hint.v4.f32 {%0, %1, %2, %3}, [%4], %5;\n}"
      : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w)
      : "l"(p), "l"(policy), "r"((int)on));
  return v;
}
__device__ __forceinline__ float ld_hint(const float* p, uint64_t policy, bool on) {
  float v;
  asm volatile(
      "{\n .reg .pred q;\n setp.ne.b32 q, %3, 0;\n mov.f32 %0, 0f00000000;\n"
      " @q ld.global.nc.L2::cache_hint.f32 %0, [%1], %2;\n}"
      : "=f"(v)
      : "l"(p), "l"(policy), "r"((int)on));
  return v;
}
__device__ __forceinline__ double ld_hint(const double* p, uint64_t policy, bool on) {
  double v;
  asm volatile(
      "{\n .reg .pred q;\n setp.ne.b32 q, %3, 0;\n mov.f64 %0, 0d0000000000000000;\n"
      " @q ld.global.nc.L2::cache_hint.f64 %0, [%1], %2;\n}"
      : "=d"(v)
      : "l"(p), "l"(policy), "r"((int)on));
  return v;
}

__device__ __forceinline__ unsigned long long norm_key(double x) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(x);
  return (b >> 63) ? 0ull : b;
}

// Largest key of a warp, ties to the lowest index, in every lane.
__device__ __forceinline__ void warp_top(unsigned long long& key, int& idx) {
  const unsigned hi = (unsigned)(key >> 32);
  const unsigned mh = __reduce_max_sync(0xffffffffu, hi);
  const unsigned lo = hi == mh ? (unsigned)key : 0u;
  const unsigned ml = __reduce_max_sync(0xffffffffu, lo);
  idx = __reduce_min_sync(0xffffffffu, (hi == mh && lo == ml) ? idx : 0x7fffffff);
  key = ((unsigned long long)mh << 32) | ml;
}

// Grid-wide barrier (cooperative launch: all CTAs are resident) on a counter
// that only grows: barrier e is passed when every CTA has arrived e times.
// Bounded (LIMIT clock64 cycles): false when it gave up (or another CTA did),
// with the status word raised.  The arrival releases and the poll acquires at
// GPU scope, so what a CTA wrote before is visible to all after.
template <long long LIMIT = tc::kWaitCycles>
__device__ bool grid_sync(const CoopArgs& a, int* sflag, int& epoch) {
  ++epoch;
  __syncthreads();
  if (threadIdx.x == 0) {
    int* cnt = a.cint + CI_BAR;
    const int target = (int)gridDim.x * epoch;
    asm volatile("red.release.gpu.global.add.s32 [%0], 1;" ::"l"(cnt) : "memory");
    const long long t0 = clock64();
    for (uint32_t it = 0;; ++it) {
      int v;
      asm volatile("ld.acquire.gpu.global.s32 %0, [%1];" : "=r"(v) : "l"(cnt) : "memory");
      if (v - target >= 0) break;
      if ((it & 15) == 15) {
        if (*(volatile int*)a.status) {
          *sflag = 1;
          break;
        }
        if (clock64() - t0 > LIMIT) {
          atomicOr(a.status, 1);
          *sflag = 1;
          break;
        }
      }
    }
  }
  __syncthreads();
  return *(volatile int*)sflag == 0;
}

// Fixed-order sum of a double over the CTA (warp trees, then warps in order);
// the result is returned to every thread.
__device__ double cta_sum(double v, double* red) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  __syncthreads();
  if (lane == 0) red[warp] = v;
  __syncthreads();
  double s = 0.0;
  for (int w = 0; w < CW; ++w) s += red[w];
  return s;
}

__device__ __forceinline__ void warp_pair_sum(float& h, float& l) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const float oh = __shfl_xor_sync(0xffffffffu, h, o);
    const float ol = __shfl_xor_sync(0xffffffffu, l, o);
    df_add(h, l, oh, ol);
  }
}

// a += b, normalised: the low part of a running pair sum grows with every plain
// addition and loses bits.  For the sums over the CTAs: with plain additions, P
// of FP64 data was off by 3.0e-15 against 64 bits (11,520 x 200, k = 20; mean of
// 24 matrices); so 2.3e-15, the multi-launch form 2.4e-15.
__device__ __forceinline__ void pair_add(float2& a, float2 b) {
  df_add(a.x, a.y, b.x, b.y);
  a = df_norm(a.x, a.y);
}

// A column's running sum in a pass: an FP32 pair, or FP64 for FP64 data.
template <typename T>
struct Sum;
template <>
struct Sum<float> {
  float h = 0.f, l = 0.f;
  using U = float2;   // u as the pass holds it
  static __device__ __forceinline__ U u_of(float uh, float ul) { return make_float2(uh, ul); }
  __device__ __forceinline__ void mac(float x, U u) { df_acc(h, l, x, u.x, u.y); }
  __device__ __forceinline__ void sq(float x) { df_acc(h, l, x, x, 0.f); }
  __device__ __forceinline__ void add(const Sum& o) { df_add(h, l, o.h, o.l); }
  __device__ __forceinline__ Sum from(int mask) const {
    Sum r;
    r.h = __shfl_xor_sync(0xffffffffu, h, mask);
    r.l = __shfl_xor_sync(0xffffffffu, l, mask);
    return r;
  }
  __device__ __forceinline__ double bits() const {   // as one 8-byte partial
    return __longlong_as_double(((long long)__float_as_int(l) << 32) | (unsigned)__float_as_int(h));
  }
  static __device__ __forceinline__ Sum of_bits(double b) {
    Sum r;
    const long long x = __double_as_longlong(b);
    r.h = __int_as_float((int)x);
    r.l = __int_as_float((int)(x >> 32));
    return r;
  }
  __device__ __forceinline__ double value() const { return (double)h + (double)l; }
};
template <>
struct Sum<double> {
  double v = 0.0;
  using U = double;
  static __device__ __forceinline__ U u_of(float uh, float ul) { return (double)uh + (double)ul; }
  __device__ __forceinline__ void mac(double x, U u) { v = fma(x, u, v); }
  __device__ __forceinline__ void sq(double x) { v = fma(x, x, v); }
  __device__ __forceinline__ void add(const Sum& o) { v += o.v; }
  __device__ __forceinline__ Sum from(int mask) const {
    Sum r;
    r.v = __shfl_xor_sync(0xffffffffu, v, mask);
    return r;
  }
  __device__ __forceinline__ double bits() const { return v; }
  static __device__ __forceinline__ Sum of_bits(double b) {
    Sum r;
    r.v = b;
    return r;
  }
  __device__ __forceinline__ double value() const { return v; }
};

// What lanes' and CTAs' sums are added in, and the column norms formed in: FP32
// pairs for FP32 data in whole row quads, else FP64 (an odd number of rows: P
// against 64 bits 3.5e-15 for 42,075 x 333, k = 50, with pairs 5.2e-15).
template <typename T, bool VEC>
using Total = Sum<std::conditional_t<VEC, T, double>>;

template <typename S>
__device__ __forceinline__ void warp_reduce(S& s) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) s.add(s.from(o));
}

// Sums of four columns over the warp at once: two exchanges in which a lane
// keeps half of the columns, then three plain levels; lanes 0, 8, 16, 24 end
// with columns 0, 1, 2, 3 (a tree per column takes 20 pair additions, this 6).
template <typename S>
__device__ __forceinline__ S reduce4(S (&c)[4], int lane) {
  const bool up = lane & 16, odd = lane & 8;
#pragma unroll
  for (int p = 0; p < 2; ++p) {
    const S give = up ? c[p] : c[p + 2];
    S keep = up ? c[p + 2] : c[p];
    keep.add(give.from(16));
    c[p] = keep;
  }
  const S give = odd ? c[0] : c[1];
  S keep = odd ? c[1] : c[0];
  keep.add(give.from(8));
#pragma unroll
  for (int o = 4; o > 0; o >>= 1) keep.add(keep.from(o));
  return keep;
}

// Sums of four columns' FP32 pairs over the warp, in FP64 (reduce4's lanes), by
// error-free extraction (S. M. Rump, T. Ogita, S. Oishi, "Accurate
// floating-point summation", 2008): with 2^B above every lane's |h|, a pair is
// cut at 2^(B-17) and 2^(B-35) by adding and subtracting 1.5 times a power of
// two.  32 lanes' first and second slices add up in FP32 without rounding, the
// third ones within 2^(B-51): as good as FP64 sums of the pairs, whose 10
// operations hold the FP64 units longer than the pass itself (42,075 x 333, k =
// 50: a whole ID 3786 us with them, with pairs only 3238 us).
struct Slices {
  float a = 0.f, b = 0.f, c = 0.f;
  __device__ __forceinline__ void add(const Slices& o) { a += o.a, b += o.b, c += o.c; }
  __device__ __forceinline__ Slices from(int mask) const {
    Slices r;
    r.a = __shfl_xor_sync(0xffffffffu, a, mask);
    r.b = __shfl_xor_sync(0xffffffffu, b, mask);
    r.c = __shfl_xor_sync(0xffffffffu, c, mask);
    return r;
  }
};
__device__ __forceinline__ Sum<double> reduce4_wide(Sum<float> (&c)[4], int lane) {
  unsigned e[4];   // exponent of the largest |h|, in every lane
  bool big = false;
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const float h = c[q].h + c[q].l, t = h - c[q].h;   // h + l without rounding
    c[q].l = (c[q].h - (h - t)) + (c[q].l - t);
    c[q].h = h;
    e[q] = __reduce_max_sync(0xffffffffu, __float_as_uint(h) & 0x7fffffffu) >> 23;
    big = big || e[q] > 246u;
  }
  Sum<double> r;
  if (big) {   // (uniform) the first cut would overflow, or has: infinities, NaN
    Sum<double> d[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) d[q].v = c[q].value();
    return reduce4(d, lane);
  }
  Slices s[4];
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const float m1 = __uint_as_float((e[q] + 7u) << 23 | 0x400000u);
    const float m2 = __uint_as_float((e[q] > 11u ? e[q] - 11u : 1u) << 23 | 0x400000u);
    s[q].a = __fadd_rn(__fadd_rn(c[q].h, m1), -m1);
    const float r1 = c[q].h - s[q].a;
    const float h2 = __fadd_rn(__fadd_rn(r1, m2), -m2), l2 = __fadd_rn(__fadd_rn(c[q].l, m2), -m2);
    s[q].b = h2 + l2;
    s[q].c = (r1 - h2) + (c[q].l - l2);
  }
  const Slices t = reduce4(s, lane);
  r.v = (double)t.a + ((double)t.b + (double)t.c);
  return r;
}
// The lanes' sums of four columns, as what they are added in.
__device__ __forceinline__ void total4(Sum<float> (&c)[4], int lane, Sum<float>& r) {
  r = reduce4(c, lane);
}
__device__ __forceinline__ void total4(Sum<double> (&c)[4], int lane, Sum<double>& r) {
  r = reduce4(c, lane);
}
__device__ __forceinline__ void total4(Sum<float> (&c)[4], int lane, Sum<double>& r) {
  r = reduce4_wide(c, lane);
}

// One pass over A_c for the CTA's rows.  Lane l holds rows 4 (l + 32 e) + q
// (VEC: 128-bit loads, whole row quads) or l + 32 i of every column, RL rows
// (what the CTA's rows need: the products of lanes without a row cost as much
// as the others).  begin() loads the warp's first columns; run<MODE> takes the
// columns, MODE 0: sums of squares; MODE 1: A^T u with u from uhs / uls (zero
// past the CTA's rows).  The leading keep_cols columns are loaded with an
// evict-last L2 policy.  part: the CTA's n partials.
template <typename T, bool VEC, int RL>
struct Pass {
  using S = Sum<T>;              // a lane's rows
  using R = Total<T, VEC>;       // lanes and CTAs
  static constexpr int NB = 2;   // columns in registers
  const T* col0;      // the lane's first row in column 0
  int64_t mc;
  int nrows, row0, cnt, warp, keep_cols;   // cnt: the warp's columns
  uint64_t keep, stream;
  T x[NB][RL];

  static __device__ __forceinline__ int off(int i) {   // of a lane's row i
    return VEC ? 128 * (i >> 2) + (i & 3) : 32 * i;
  }
  __device__ __forceinline__ void init(const T* Ar, int64_t mc_, int n, int nrows_, int keep_c) {
    warp = threadIdx.x >> 5;
    row0 = (VEC ? 4 : 1) * (threadIdx.x & 31);
    col0 = Ar + row0;
    mc = mc_;
    nrows = nrows_;
    cnt = n > warp ? (n - warp + CW - 1) / CW : 0;
    keep_cols = keep_c;
    keep = tc::policy_evict_last();
    stream = tc::policy_evict_first();
  }
  // column i of the warp (the last one again past it)
  __device__ __forceinline__ void load(int i, T (&y)[RL]) const {
    const int j = warp + CW * min(i, cnt - 1);
    const T* col = col0 + (int64_t)j * mc;
    const uint64_t pol = j < keep_cols ? keep : stream;
    if constexpr (VEC) {
#pragma unroll
      for (int e = 0; e < RL / 4; ++e) {
        const float4 v = ld_hint(reinterpret_cast<const float4*>(col + 128 * e), pol,
                                 row0 + 128 * e < nrows);
        y[4 * e] = v.x, y[4 * e + 1] = v.y, y[4 * e + 2] = v.z, y[4 * e + 3] = v.w;
      }
    } else {
#pragma unroll
      for (int e = 0; e < RL; ++e) y[e] = ld_hint(col + 32 * e, pol, row0 + 32 * e < nrows);
    }
  }
  __device__ __forceinline__ void begin() {
    if (cnt == 0) return;
#pragma unroll
    for (int b = 0; b < NB - 1; ++b) load(b, x[b]);
  }
  template <int MODE>
  __device__ __forceinline__ void run(const float* uhs, const float* uls,
                                      double* __restrict__ part) {
    const int lane = threadIdx.x & 31;
    typename S::U u[MODE == 1 ? RL : 1];
    if (MODE == 1) {
#pragma unroll
      for (int i = 0; i < RL; ++i) u[i] = S::u_of(uhs[row0 + off(i)], uls[row0 + off(i)]);
    }
    for (int i0 = 0; i0 < cnt; i0 += 4) {
      std::conditional_t<MODE == 1, S, R> c[4];
#pragma unroll
      for (int v = 0; v < 4; ++v) {
        load(i0 + v + NB - 1, x[(v + NB - 1) % NB]);
        if constexpr (MODE == 1) {
#pragma unroll
          for (int e = 0; e < RL; ++e) c[v].mac(x[v % NB][e], u[e]);
        } else if constexpr (std::is_same_v<S, R>) {
#pragma unroll
          for (int e = 0; e < RL; ++e) c[v].sq(x[v % NB][e]);
        } else {
          bool plain = true;
#pragma unroll
          for (int e = 0; e < RL; ++e) plain = plain && widens(x[v % NB][e]);
          if (plain) {
#pragma unroll
            for (int e = 0; e < RL; ++e) c[v].sq(widen_normal(x[v % NB][e]));
          } else {
#pragma unroll
            for (int e = 0; e < RL; ++e) c[v].sq((double)x[v % NB][e]);
          }
        }
      }
      R r;
      total4(c, lane, r);
      const int i = i0 + (lane >> 3);
      if ((lane & 7) == 0 && i < cnt) part[warp + CW * i] = r.bits();
    }
  }
};

template <typename T, bool VEC, int RL>
__global__ void __launch_bounds__(CT, 1) coarse_coop_kernel(CoopArgs a) {
  using S = Total<T, VEC>;
  extern __shared__ __align__(16) float2 vs[];   // vs_cols x vs_rows: this CTA's rows of V
  __shared__ int sflag;
  __shared__ __align__(16) float uhs[RMAX];
  __shared__ __align__(16) float uls[RMAX];
  __shared__ float2 fp[kLMax];
  __shared__ double hs[HP], hvec[kLMax], vrow[kLMax];
  __shared__ double red[CW];
  __shared__ float2 sigw[CW];
  __shared__ unsigned long long pk[CW];
  __shared__ int pi[CW];
  __shared__ double sh_tol, sh_sigma, sh_beta, sh_tau;
  __shared__ int nrec_s;
  // 1 / (u_s - beta) of the last step, in FP64 and as an FP32 pair: formed once
  // (an FP64 division per thread costs GB300's narrow FP64 pipe)
  __shared__ double rden_sh;
  __shared__ float2 rdf_sh;

  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int G = gridDim.x, b = blockIdx.x;
  const int64_t mc = a.mc;
  const int n = a.n;
  const T* Ac = reinterpret_cast<const T*>(a.Ac);
  const int64_t gran = VEC ? 4 : 1, Q = mc / gran;   // whole row quads with VEC
  const int64_t r0 = gran * (Q * b / G);
  const int nrows = (int)(gran * (Q * (b + 1) / G) - r0);
  const int c0 = (int)((int64_t)n * b / G), c1 = (int)((int64_t)n * (b + 1) / G);
  double* const mypart = a.gpart + (int64_t)b * n;
  int epoch = 0;
  // entry (row r of the CTA, column t) of V
  auto vat = [&](int t, int r) -> float2& {
    return t < a.vs_cols ? vs[t * a.vs_rows + r] : a.V[(int64_t)t * mc + r0 + r];
  };

  if (tid == 0) {
    sflag = 0;
    rden_sh = 0.0;
    rdf_sh = make_float2(0.f, 0.f);
  }
  __syncthreads();

  // ---- column norms (pass 0) and the rank tolerance
  Pass<T, VEC, RL> pass;
  pass.init(Ac + r0, mc, n, nrows, a.keep_cols);
  pass.begin();
  pass.template run<0>(uhs, uls, mypart);
  bool ok = grid_sync(a, &sflag, epoch);
  double nsum = 0.0;
  if (ok) {
    for (int j = c0 + warp; j < c1; j += CW) {   // sum over the CTAs, fixed order
      S sm;
      for (int bb = lane; bb < G; bb += 32) sm.add(S::of_bits(a.gpart[(int64_t)bb * n + j]));
      warp_reduce(sm);
      const double s2 = sm.value();
      if (lane == 0) {
        a.nu2[j] = s2;
        a.nu20[j] = s2;
        a.colpos[j] = -1;
        nsum += s2;
      }
    }
  }
  nsum = cta_sum(nsum, red);
  if (tid == 0) reinterpret_cast<double*>(a.upart)[(int64_t)b * HP] = nsum;
  ok = ok && grid_sync(a, &sflag, epoch);
  if (ok) {
    double tot = 0.0;
    for (int bb = tid; bb < G; bb += CT)
      tot += reinterpret_cast<const double*>(a.upart)[(int64_t)bb * HP];
    tot = cta_sum(tot, red);
    if (tid == 0) {
      sh_tol = a.tol_factor * DBL_EPSILON * sqrt(tot);
      if (b == 0) {
        a.cint[CI_STOP] = 0;
        a.cint[CI_KOUT] = 0;
      }
    }
  }
  __syncthreads();

  int s = 0;
  for (; ok && s < a.kmax; ++s) {
    // ---------------------------------------------------------- phase A
    // pivot: largest residual norm, ties to the lowest index
    CC_TRACE(s, 0);
    int p = 0x7fffffff;
    {
      unsigned long long v = 0ull;
      for (int j = tid; j < n; j += CT) {
        const unsigned long long key = norm_key(a.nu2[j]);
        if (p == 0x7fffffff || key > v) {
          v = key;
          p = j;
        }
      }
      warp_top(v, p);
      if (lane == 0) {
        pk[warp] = v;
        pi[warp] = p;
      }
      __syncthreads();
      v = pk[lane & (CW - 1)];
      p = pi[lane & (CW - 1)];
      warp_top(v, p);
      const double tol = sh_tol;
      if (p == 0x7fffffff || !(v > norm_key(tol * tol))) {   // the same in every thread
        if (b == 0 && tid == 0) {
          a.cint[CI_STOP] = 1;
          a.cint[CI_KOUT] = s;
        }
        break;
      }
      if (b == 0 && tid == 0) {
        a.cint[CI_P] = p;
        a.Jc[s] = p;
        a.cint[nrec_slot(s)] = 0;
      }
    }
    CC_TRACE(s, 1);
    for (int t = tid; t < s; t += CT) fp[t] = df_of(a.F[(int64_t)t * a.ldf + p]);
    // v_{s-1} from u_{s-1}, then u = A(:, p) - V_s F(p, :)^T for this CTA's rows
    const int64_t i = r0 + tid;
    const bool in = tid < nrows;
    const T aip = in && i >= s ? Ac[i + (int64_t)p * mc] : T(0);
    float2 sig = make_float2(0.f, 0.f);
    if (in && s > 0) {
      float2& vp = vat(s - 1, tid);
      if (i == s - 1)
        vp = make_float2(1.f, 0.f);
      else if (i > s - 1)
        vp = df_mul(vp, rdf_sh);   // 1 / (u_{s-1} - beta_{s-1})
    }
    __syncthreads();
    float2 u = make_float2(0.f, 0.f);
    if (in && i >= s) {
      u = sizeof(T) == 4 ? make_float2((float)aip, 0.f) : df_of((double)aip);
      const int ns = min(s, a.vs_cols);
#pragma unroll 8
      for (int t = 0; t < ns; ++t) {
        const float2 pr = df_mul(vs[t * a.vs_rows + tid], fp[t]);
        df_add(u.x, u.y, -pr.x, -pr.y);
      }
      for (int t0 = ns; t0 < s; t0 += 16) {
        float2 vv[16];
#pragma unroll
        for (int q = 0; q < 16; ++q)
          vv[q] = t0 + q < s ? a.V[(int64_t)(t0 + q) * mc + i] : make_float2(0.f, 0.f);
#pragma unroll
        for (int q = 0; q < 16; ++q)
          if (t0 + q < s) {
            const float2 pr = df_mul(vv[q], fp[t0 + q]);
            df_add(u.x, u.y, -pr.x, -pr.y);
          }
      }
      u = df_norm(u.x, u.y);
    }
    if (in) vat(s, tid) = u;
    {
      const float2 uu = i > s ? u : make_float2(0.f, 0.f);
      uhs[tid] = uu.x;
      uls[tid] = uu.y;
      const float2 u2 = df_mul(uu, uu);
      df_add(sig.x, sig.y, u2.x, u2.y);
    }
    if (s >= r0 && s < r0 + nrows) {   // row s of V and u_s for every CTA
      if (tid < s) a.vrow[tid] = vat(tid, (int)(s - r0));
      if (in && i == s) a.vrow[kLMax] = u;
    }
    warp_pair_sum(sig.x, sig.y);
    if (lane == 0) sigw[warp] = sig;
    __syncthreads();
    CC_TRACE(s, 2);
    // partials of V_s^T u (warp w: t = w + 16 q, q < 4, together)
    auto vtu = [&]() {
      if (warp >= s) return;
      Sum<float> acc[4];
      const int nq = (s - warp + CW - 1) / CW;   // this warp's columns of V
      // NQ fixed per instantiation: a test per column and row costs as much as
      // the products; col(t, r): row r of column t
      auto dots = [&](auto nqc, auto col) {
        constexpr int NQ = decltype(nqc)::value;
#pragma unroll 2
        for (int rr = lane; rr < nrows; rr += 32) {
          const float2 uu = make_float2(uhs[rr], uls[rr]);
#pragma unroll
          for (int q = 0; q < NQ; ++q) {
            const float2 pr = df_mul(col(warp + CW * q, rr), uu);
            df_add(acc[q].h, acc[q].l, pr.x, pr.y);
          }
        }
      };
      auto in_shared = [&](int t, int rr) { return vs[t * a.vs_rows + rr]; };
      if (s > a.vs_cols) {
        auto any = [&](int t, int rr) { return t < s ? vat(t, rr) : make_float2(0.f, 0.f); };
        dots(std::integral_constant<int, 4>(), any);
      } else if (nq == 1) {
        dots(std::integral_constant<int, 1>(), in_shared);
      } else if (nq == 2) {
        dots(std::integral_constant<int, 2>(), in_shared);
      } else if (nq == 3) {
        dots(std::integral_constant<int, 3>(), in_shared);
      } else {
        dots(std::integral_constant<int, 4>(), in_shared);
      }
      const Sum<float> r = reduce4(acc, lane);
      const int q = lane >> 3;
      if ((lane & 7) == 0 && q < nq)
        a.upart[(int64_t)b * HP + warp + CW * q] = df_norm(r.h, r.l);
    };
    if (warp == CW - 1) {   // ||u||^2
      float2 x = lane < CW ? sigw[lane] : make_float2(0.f, 0.f);
      warp_pair_sum(x.x, x.y);
      if (lane == 0) a.upart[(int64_t)b * HP + kLMax] = df_norm(x.x, x.y);
    }
    // A^T u over this CTA's rows (u is zero at and above row s): it needs
    // only this CTA's u, so it runs before the barrier.  Half of the warps
    // form V_s^T u before it and half after, beside the others' loads.
    if (!(warp & 1)) vtu();
    CC_TRACE(s, 3);
    pass.begin();
    pass.template run<1>(uhs, uls, mypart);
    if (warp & 1) vtu();
    CC_TRACE(s, 4);
    if (!grid_sync(a, &sflag, epoch)) {
      ok = false;
      break;
    }
    // ---------------------------------------------------------- phase B
    CC_TRACE(s, 5);
    // Householder scalars and h = V_s^T v_s, every CTA from the partials in
    // a fixed order; the last warp takes ||u||^2, the square root and the
    // division while the others sum V_s^T u.
    // The loads that do not depend on the sums go first: u_s, v_t[s] (thread
    // t < s), and the CTAs' partials of (A^T u)_j and F(j, 0:s) for this warp's
    // first two columns of phase C
    const float2 us = a.vrow[kLMax];
    const float2 vts = tid < s ? a.vrow[tid] : make_float2(0.f, 0.f);
    struct ColIn {
      double g[8], f[2];   // G <= 256, s <= 64
    };
    auto col_in = [&](int j, ColIn& x) {
      const bool on = j < c1;
#pragma unroll
      for (int e = 0; e < 8; ++e) {
        const int bb = lane + 32 * e;
        x.g[e] = (on && bb < G) ? a.gpart[(int64_t)bb * n + j] : 0.0;
      }
#pragma unroll
      for (int e = 0; e < 2; ++e) {
        const int t = lane + 32 * e;
        x.f[e] = (on && t < s) ? a.F[(int64_t)t * a.ldf + j] : 0.0;
      }
    };
    // warp w takes the column pairs c0 + 2 w, c0 + 2 w + 32, ...; lanes 0 and
    // 16 finish the first and the second column of a pair
    const int jw = c0 + 2 * warp;
    ColIn ci[2];
    col_in(jw, ci[0]);
    col_in(jw + 1, ci[1]);
    if (warp == CW - 1) {
      // ||u||^2 and the scalars
      float2 sum = make_float2(0.f, 0.f);
      {
        float2 xv[8];
#pragma unroll
        for (int e = 0; e < 8; ++e) {
          const int bb = lane + 32 * e;
          xv[e] = bb < G ? a.upart[(int64_t)bb * HP + kLMax] : make_float2(0.f, 0.f);
        }
#pragma unroll
        for (int e = 0; e < 8; ++e) pair_add(sum, xv[e]);
      }
      warp_pair_sum(sum.x, sum.y);
      const double sigma = df_val(sum);
      const double alpha = df_val(us);
      double beta = alpha, q = 0.0;
      if (sigma != 0.0) {
        const double nrm = sqrt(alpha * alpha + sigma);
        beta = alpha >= 0.0 ? -nrm : nrm;
        // 1 / den in lane 0 and tau in lane 1: one division
        q = (lane == 1 ? beta - alpha : 1.0) / (lane == 1 ? beta : alpha - beta);
      }
      if (lane == 0) {
        sh_sigma = sigma;
        sh_beta = beta;
        rden_sh = q;
        rdf_sh = df_of(q);
      }
      if (lane == 1) sh_tau = q;
    } else {
      // V_t^T u, t < s (s < 64): the 4 threads 4 t .. 4 t + 3, thread j over
      // the CTAs b = j mod 4 (whole warps)
      const int g = tid >> 2, j = tid & 3;
      if (g < ((s + 7) & ~7)) {
        // (four running sums each, beside one another)
        float2 acc[4] = {};
        for (int e0 = 0; 4 * e0 < G; e0 += 20) {   // 20 loads in flight
          float2 xv[20];
#pragma unroll
          for (int e = 0; e < 20; ++e) {
            const int bb = j + 4 * (e0 + e);
            xv[e] = (g < s && bb < G) ? a.upart[(int64_t)bb * HP + g] : make_float2(0.f, 0.f);
          }
#pragma unroll
          for (int e = 0; e < 20; ++e) pair_add(acc[e & 3], xv[e]);
        }
        pair_add(acc[0], acc[1]);
        pair_add(acc[2], acc[3]);
        pair_add(acc[0], acc[2]);
#pragma unroll
        for (int o = 1; o < 4; o <<= 1) {
          const float oh = __shfl_xor_sync(0xffffffffu, acc[0].x, o);
          const float ol = __shfl_xor_sync(0xffffffffu, acc[0].y, o);
          pair_add(acc[0], make_float2(oh, ol));
        }
        if (j == 0 && g < s) hs[g] = df_val(acc[0]);
      }
    }
    __syncthreads();
    if (tid < s) {
      const double vst = df_val(vts);   // v_t[s], t = tid
      hvec[tid] = vst + hs[tid] * rden_sh;
      vrow[tid] = vst;
    }
    __syncthreads();
    // ---------------------------------------------------------- phase C
    CC_TRACE(s, 6);
    {
      const double tau = sh_tau, sigma = sh_sigma, rden = rden_sh;
      for (int j0 = jw; j0 < c1; j0 += 2 * CW) {
        if (j0 != jw) {
          col_in(j0, ci[0]);
          col_in(j0 + 1, ci[1]);
        }
        const int j = j0 + (lane >> 4);
        const bool fin = (lane & 15) == 0 && j < c1;
        // the column's own entries, loaded while the sums run
        const int cp = fin ? a.colpos[j] : 0;
        const double asj = fin ? (double)Ac[s + (int64_t)j * mc] : 0.0;
        const double nu2 = fin ? a.nu2[j] : 0.0, nu20 = fin ? a.nu20[j] : 0.0;
        // (A^T u)_j: the CTAs' partials in lane order, then a fixed tree whose
        // first exchange leaves column 0 to lanes 0-15 and 1 to lanes 16-31
        S g0, g1;
#pragma unroll
        for (int e = 0; e < 8; ++e) {
          g0.add(S::of_bits(ci[0].g[e]));
          g1.add(S::of_bits(ci[1].g[e]));
        }
        const S give = lane & 16 ? g0 : g1;
        S gsum = lane & 16 ? g1 : g0;
        gsum.add(give.from(16));
#pragma unroll
        for (int o = 8; o > 0; o >>= 1) gsum.add(gsum.from(o));
        // F(j, :) h and v(s, :) F(j, :)^T of both columns in one tree
        Sum<double> d[4];
#pragma unroll
        for (int e = 0; e < 2; ++e) {
          const int t = lane + 32 * e;
          if (t < s) {
            const double hv = hvec[t], vr = vrow[t];
            d[0].mac(ci[0].f[e], hv);
            d[1].mac(ci[0].f[e], vr);
            d[2].mac(ci[1].f[e], hv);
            d[3].mac(ci[1].f[e], vr);
          }
        }
        const double q = reduce4(d, lane).v;   // lanes 0, 8: column 0's; 16, 24: column 1's
        const double fh = q, rr = __shfl_xor_sync(0xffffffffu, q, 8);
        if (fin) {
          if (j == p) {
            a.colpos[j] = s;
            a.nu2[j] = -1.0;   // never a pivot again
            a.Rc[(int64_t)s * n + j] = sh_beta;
          } else if (cp >= 0) {
            a.Rc[(int64_t)s * n + j] = 0.0;
          } else {
            const double gj = sigma != 0.0 ? asj + gsum.value() * rden : asj;
            const double fjs = tau * (gj - fh);
            a.F[(int64_t)s * a.ldf + j] = fjs;
            const double r = asj - rr - fjs;   // v_s[s] = 1
            a.Rc[(int64_t)s * n + j] = r;
            const double nn = nu2 - r * r;
            a.nu2[j] = nn;
            if (nn <= kRecomputeFrac * nu20) {
              const int slot = atomicAdd(&a.cint[nrec_slot(s)], 1);
              a.rlist[slot] = j;
            }
          }
        }
      }
    }
    CC_TRACE(s, 7);
    if (!grid_sync(a, &sflag, epoch)) {
      ok = false;
      break;
    }
    CC_TRACE(s, 8);
    // norms that lost too many bits: recomputed from their definition
    // ||A^(s+1)(s+1:, j)||^2 in FP64, rows split over the CTAs
    if (tid == 0) nrec_s = *(volatile int*)&a.cint[nrec_slot(s)];
    __syncthreads();
    const int nrec = nrec_s;
    if (nrec > 0) {
      const double rden = rden_sh;
      for (int idx = 0; idx < nrec; ++idx) {
        const int j = a.rlist[idx];
        double ssum = 0.0;
        if (in && i > s) {
          double x = (double)Ac[i + (int64_t)j * mc];
          for (int t = 0; t < s; ++t) x -= df_val(vat(t, tid)) * a.F[(int64_t)t * a.ldf + j];
          x -= df_val(vat(s, tid)) * rden * a.F[(int64_t)s * a.ldf + j];
          ssum = x * x;
        }
        ssum = cta_sum(ssum, red);
        if (tid == 0) a.gpart[(int64_t)b * n + idx] = ssum;
      }
      if (!grid_sync(a, &sflag, epoch)) {
        ok = false;
        break;
      }
      for (int idx = tid; idx < nrec; idx += CT) {
        const int j = a.rlist[idx];
        if (j < c0 || j >= c1) continue;
        double ssum = 0.0;
        for (int bb = 0; bb < G; ++bb) ssum += a.gpart[(int64_t)bb * n + idx];
        a.nu2[j] = ssum;
        a.nu20[j] = ssum;
      }
      if (!grid_sync(a, &sflag, epoch)) {
        ok = false;
        break;
      }
    }
  }
  // steps done (or stopped): k_out and the unused pivot slots
  if (ok && b == 0) {
    if (tid == 0) a.cint[CI_KOUT] = s;
    for (int q = s + tid; q < a.k; q += CT) a.Jc[q] = -1;
  }
  if (!ok && tid == 0) atomicOr(a.status, 1);
}

// ------------------------------------------------------------------------
// Self-check of the bounded waits' give-up path (no fault, no hang): the
// waits of the kernels above, instantiated with a limit of ~1 ms, on a phase
// or a barrier that nothing completes, and the same waits on one that
// completes.  The status word is raised exactly as in the real kernels.
constexpr long long kCheckWaitCycles = 1ll << 21;
__device__ int g_check_words[8];   // barrier counter (CI_BAR) and, in slot 7, the status

// One CTA waits on phase 0 of an mbarrier; `complete`: thread 0 arrives
// first (the phase completes), else nobody does.
__global__ void mbar_check_kernel(int complete, int* status) {
  __shared__ __align__(8) uint64_t bar;
  __shared__ int abort_flag;
  const uint32_t b = tc::smem_u32(&bar), af = tc::smem_u32(&abort_flag);
  if (threadIdx.x == 0) {
    tc::mbar_init(b, 1);
    abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncthreads();
  if (complete && threadIdx.x == 0) tc::mbar_arrive(b);
  if (!tc::mbar_wait<kCheckWaitCycles>(b, 0, af)) atomicOr(status, 1);
}

// One warp waits as a whole, its lower half on a barrier that completes, its
// upper half on one that completes only with `complete`: the status is raised
// when every lane gave up.
__global__ void mbar_warp_check_kernel(int complete, int* status) {
  __shared__ __align__(8) uint64_t bars[2];
  __shared__ int abort_flag;
  const uint32_t b = tc::smem_u32(&bars[0]), af = tc::smem_u32(&abort_flag);
  if (threadIdx.x == 0) {
    tc::mbar_init(b, 1);
    tc::mbar_init(b + 8, 1);
    abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    tc::mbar_arrive(b);
    if (complete) tc::mbar_arrive(b + 8);
  }
  const bool ok = tc::mbar_wait_warp<kCheckWaitCycles>(b + (threadIdx.x < 16 ? 0u : 8u), 0, af);
  const unsigned gave = __ballot_sync(0xffffffffu, !ok);
  if (threadIdx.x == 0 && gave == 0xffffffffu) atomicOr(status, 1);
}

// The coarse kernel's grid barrier over a cooperative launch; `skip`: the
// last CTA returns without reaching it.
__global__ void __launch_bounds__(CT, 1) grid_check_kernel(CoopArgs a, int skip) {
  __shared__ int sflag;
  if (threadIdx.x == 0) sflag = 0;
  __syncthreads();
  if (skip && blockIdx.x == gridDim.x - 1) return;
  int epoch = 0;
  if (!grid_sync<kCheckWaitCycles>(a, &sflag, epoch) && threadIdx.x == 0) atomicOr(a.status, 1);
}

}  // namespace

#ifdef IDSK_CC_TRACE
// Profiling harness only: clock64 of CTA 0 at the phase boundaries, entry
// [s * 16 + point]: 0 step start, 1 pivot chosen, 2 u formed, 3 partials
// written, 4 pass over A_c done, 5 after the first barrier, 6 scalars done,
// 7 columns finalized, 8 after the second barrier.
extern "C" int idsk_cc_trace_read(long long* host) {
  return (int)cudaMemcpyFromSymbol(host, g_cc_trace, sizeof(g_cc_trace));
}
#endif

// Whether the cooperative form serves this handle: at most 512 rows per CTA.
bool coarse_coop_ok(const id_sketch* h) { return coarse_coop_ok_ctas(h, 0); }

// The same with at most max_ctas CTAs (0: one per SM).
bool coarse_coop_ok_ctas(const id_sketch* h, int max_ctas) {
  if (getenv("IDSKETCH_COARSE_MULTI")) return false;
  int coop = 0;
  if (cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, h->dev) != cudaSuccess ||
      !coop) {
    cudaGetLastError();
    return false;
  }
  const int64_t gran = h->cfg.dtype == ID_F32 && (h->mc & 3) == 0 ? 4 : 1, Q = h->mc / gran;
  const int cap = max_ctas > 0 ? std::min(max_ctas, h->nsm) : h->nsm;
  const int64_t G = std::min<int64_t>(cap, Q);
  return Q >= 1 && G >= 1 && G <= 256 && (Q + G - 1) / G * gran <= RMAX && h->coarse_blocks >= G;
}

// Runs one self-check of the bounded waits (modes as id_check_wait) on
// stream st; *gave_up = 1 when the wait gave up and raised the status word.
cudaError_t run_wait_check(int mode, cudaStream_t st, int* gave_up) {
  int* words = nullptr;
  cudaError_t e = cudaGetSymbolAddress((void**)&words, g_check_words);
  if (e != cudaSuccess) return e;
  if ((e = cudaMemsetAsync(words, 0, sizeof(g_check_words), st)) != cudaSuccess) return e;
  if (mode == 0 || mode == 1) {
    mbar_check_kernel<<<1, 32, 0, st>>>(mode == 1, words + 7);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
  } else if (mode >= 4) {
    mbar_warp_check_kernel<<<1, 32, 0, st>>>(mode == 5, words + 7);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
  } else {
    CoopArgs a;
    memset(&a, 0, sizeof(a));
    a.cint = words;
    a.status = words + 7;
    int skip = mode == 2;
    void* args[] = {&a, &skip};
    e = cudaLaunchCooperativeKernel((const void*)grid_check_kernel, dim3(2), dim3(CT), args, 0,
                                   st);
    if (e != cudaSuccess) return e;
  }
  count_launches(1);
  int h = 0;
  if ((e = cudaMemcpyAsync(&h, words + 7, sizeof(int), cudaMemcpyDeviceToHost, st)) !=
      cudaSuccess)
    return e;
  if ((e = cudaStreamSynchronize(st)) != cudaSuccess) return e;
  *gave_up = h != 0;
  return cudaSuccess;
}

cudaError_t launch_coarse_coop(id_sketch* h, int64_t n64, cudaStream_t st, int max_ctas) {
  const int n = (int)n64;
  const bool f64 = h->cfg.dtype == ID_F64, vec = !f64 && (h->mc & 3) == 0;
  const int64_t gran = vec ? 4 : 1, Q = h->mc / gran;
  const int cap = max_ctas > 0 ? std::min(max_ctas, h->nsm) : h->nsm;
  // every CTA owns rows: at most 512, and 16,384 entries of A_c (FP64: 4096) or
  // more where that leaves fewer CTAs than the cap
  const int64_t per = f64 ? 4096 : 16384;
  const int64_t want = std::max((Q + RMAX / gran - 1) / (RMAX / gran),
                                (h->mc * n64 + per - 1) / per);
  const int G = (int)std::min<int64_t>(std::min<int64_t>(cap, Q), want);
  CoopArgs a;
  a.Ac = h->d_Ac;
  a.mc = h->mc;
  a.n = n;
  a.k = h->k;
  a.kmax = (int)std::min<int64_t>(h->k, std::min<int64_t>(h->mc, n64));
  a.ldf = h->n_max;
  a.V = reinterpret_cast<float2*>(h->d_V);
  a.F = h->d_F;
  a.Rc = h->d_Rc;
  a.nu2 = h->d_nu2;
  a.nu20 = h->d_nu20;
  a.colpos = h->d_colposc;
  a.Jc = h->d_Jc;
  a.gpart = h->d_gvec;
  a.upart = reinterpret_cast<float2*>(h->d_upart);
  a.rlist = h->d_rlist;
  a.cint = h->d_cint;
  a.status = h->d_status;
  a.tol_factor = ID_RANK_TOL_FACTOR;
  int l2 = 0;
  if (cudaDeviceGetAttribute(&l2, cudaDevAttrL2CacheSize, h->dev) != cudaSuccess) {
    cudaGetLastError();
    l2 = 0;
  }
  // about 3/8 of L2 holds the leading columns of A_c from one step to the next
  double keep = 0.375;
  if (const char* env = getenv("IDSKETCH_COARSE_L2_KEEP")) keep = atof(env);
  a.keep_cols = (int)std::min<int64_t>(
      n, (int64_t)(std::max(0.0, std::min(1.0, keep)) * l2 / ((double)h->esz * (double)h->mc)));
  a.vrow = reinterpret_cast<float2*>(h->d_hvec);
  a.vs_rows = (int)((Q + G - 1) / G * gran);
  constexpr size_t room = kSmemMost - 8 * 1024;   // static shared memory: about 7 KB
  a.vs_cols = (int)std::min<int64_t>(a.kmax, (int64_t)(room / (sizeof(float2) * a.vs_rows)));
  const size_t sm = sizeof(float2) * (size_t)a.vs_cols * a.vs_rows;
  cudaError_t e = cudaMemsetAsync(h->d_cint, 0, 8 * sizeof(int), st);
  if (e != cudaSuccess) return e;
  // rows per lane of a pass.  FP64 data is bound by the FP64 units, where a row
  // that is not there costs as much as one that is: 25,000 x 1000, k = 20 (6 rows)
  // 3483 us with the 16-row instantiation next after 4, 1728 us with these
  // (the multi-launch form 3094 us).
  const int rl = (a.vs_rows + 31) / 32;
  const void* kern;
  if (f64)
    kern = rl <= 1    ? (const void*)coarse_coop_kernel<double, false, 1>
           : rl <= 2  ? (const void*)coarse_coop_kernel<double, false, 2>
           : rl <= 4  ? (const void*)coarse_coop_kernel<double, false, 4>
           : rl <= 6  ? (const void*)coarse_coop_kernel<double, false, 6>
           : rl <= 8  ? (const void*)coarse_coop_kernel<double, false, 8>
           : rl <= 12 ? (const void*)coarse_coop_kernel<double, false, 12>
                      : (const void*)coarse_coop_kernel<double, false, 16>;
  else if (vec)
    kern = rl <= 4    ? (const void*)coarse_coop_kernel<float, true, 4>
           : rl <= 8  ? (const void*)coarse_coop_kernel<float, true, 8>
           : rl <= 12 ? (const void*)coarse_coop_kernel<float, true, 12>
                      : (const void*)coarse_coop_kernel<float, true, 16>;
  else
    kern = rl <= 4    ? (const void*)coarse_coop_kernel<float, false, 4>
           : rl <= 8  ? (const void*)coarse_coop_kernel<float, false, 8>
           : rl <= 12 ? (const void*)coarse_coop_kernel<float, false, 12>
                      : (const void*)coarse_coop_kernel<float, false, 16>;
  e = allow_smem(kern, room);
  if (e != cudaSuccess) return e;
  void* args[] = {&a};
  e = cudaLaunchCooperativeKernel(kern, dim3(G), dim3(CT), args, sm, st);
  if (e != cudaSuccess) return e;
  count_launches(1);
  return launch_solve_p(h->d_Rc, h->d_Jc, h->d_colposc, h->d_cint + CI_KOUT, h->k, n, h->d_Pc,
                        st);
}

}  // namespace idsk
