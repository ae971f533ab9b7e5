// Fused reconstruction-error pass: one read of A gives
//   ||A - A(:,J) P||_F^2, ||A||_F^2 and max_ij |A_ij - A_hat_ij| / |A_ij|
// (Frobenius metric of Sec. 3.3; entry-wise metric of Sec. 3.1, skipping
// A_ij == 0 where the ratio is undefined).  The reconstruction
// A_hat = A(:,J) P is the ID of eq. eqn:id written for columns; the skeleton
// block A(R, J) is gathered once per row tile R.
//
// FP32 data with fewer than 128 rows (more rows: recon_tc.cu): products and the
// residual in FP32 (P rounded to FP32), every square added with Kahan
// compensation in FP32 per thread, then FP64 across threads and CTAs.
// FP64 data: FP64 throughout; the up to 8 squares of a thread's chunk of 32
// columns are summed plainly and the chunks with Kahan compensation.  Against
// 64-bit-mantissa sums ||A - A_hat|| / ||A|| is off by 6.7e-17 (98,304 x 200),
// 7.9e-17 (20,000 x 100) and 8.0e-17 (4001 x 333), rms over 8 matrices; with
// every square compensated, in more CTAs, it was off by 9.2e-16, 4.2e-16 and
// 1.1e-16.  The cross-CTA sum runs in a fixed order, so the result is
// deterministic.
#include <algorithm>

#include "idsk_internal.h"

namespace idsk {
namespace {

constexpr int TM = 64;
constexpr int TC = 32;
constexpr int NT = 256;

// Warp maximum of non-negative numbers (ordered like their bit patterns).
__device__ __forceinline__ float warp_max(float x) {
  return __int_as_float(__reduce_max_sync(0xffffffffu, __float_as_int(x)));
}
__device__ __forceinline__ double warp_max(double x) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(x);
  const unsigned hi = __reduce_max_sync(0xffffffffu, (unsigned)(b >> 32));
  const unsigned lo =
      __reduce_max_sync(0xffffffffu, (unsigned)(b >> 32) == hi ? (unsigned)b : 0u);
  return __longlong_as_double((long long)(((unsigned long long)hi << 32) | lo));
}

// Out of line: inlined, the compiler divides for every entry and selects.
template <typename T>
__device__ __noinline__ T ratio(T a, T b) {
  return a / b;
}

// |x| and x != 0 on the integer units.
__device__ __forceinline__ float magnitude(float x) { return fabsf(x); }
__device__ __forceinline__ double magnitude(double x) {
  return __longlong_as_double(__double_as_longlong(x) & 0x7fffffffffffffffll);
}
__device__ __forceinline__ bool nonzero(float x) { return (__float_as_int(x) << 1) != 0; }
__device__ __forceinline__ bool nonzero(double x) { return (__double_as_longlong(x) << 1) != 0; }

template <typename T>
struct Acc {
  T s = T(0), c = T(0);
  __device__ __forceinline__ void add(T x) {   // Kahan-Babuska step
    const T y = x - c;
    const T t = s + y;
    c = (t - s) - y;
    s = t;
  }
};

// CTA b takes the rows [16 U b / G, 16 U (b + 1) / G) of the U = ceil(m / 16)
// groups of 16 rows, in steps of 64, and every column in chunks of 32.  Thread
// (tr, tc) = (t mod 16, t / 16) forms A_hat at rows tr + 16 e (e < 4) and
// columns tc, tc + 16 of the chunk, and reads those entries of A straight from
// global memory (the next chunk's while this one is multiplied).
// Bound by the FP64 units (2 operations per clock and SM) for FP64 data, so
// the operations per entry count: k for A_hat, one difference, two squares
// added to the chunk's sums, two for the running maximum; magnitudes and the
// zero test take none, the compensated sums get one term per chunk, and groups
// of 16 rows balance the SMs.  98,304 x 200, k = 20: 2364 -> 1176 us (before:
// about 16 operations an entry beside the products and the ratio's division,
// 1216 CTAs in 2.7 waves).
template <typename T, bool RES>
__global__ void __launch_bounds__(NT, 2) recon_kernel(const T* __restrict__ A, int64_t lda,
                                                   int64_t m, int64_t n,
                                                   const int* __restrict__ J,
                                                   const double* __restrict__ P, int k,
                                                   double* __restrict__ part, InterpGeom geo) {
  extern __shared__ __align__(16) unsigned char smem[];
  T* sk = reinterpret_cast<T*>(smem);   // k x TM   : A(R, J)
  T* ps = sk + k * TM;                  // RES: k x n, all of P; else k x TC, P(:, chunk)
  __shared__ int Js[kRecKMax];
  __shared__ double red[3][NT / 32];

  const int t = threadIdx.x, tr = t & 15, tc = t >> 4;
  for (int u = t; u < k; u += NT) Js[u] = J[u];
  if (RES)
    for (int64_t e = t; e < (int64_t)k * n; e += NT) ps[e] = (T)P[e];
  const int ldp = RES ? (int)n : TC;
  Acc<T> res, tot;
  T mx = T(0);
  const int64_t units = (m + 15) / 16;
  const int64_t row1 = min(m, 16 * (units * (blockIdx.x + 1) / gridDim.x));
  for (int64_t r0 = 16 * (units * blockIdx.x / gridDim.x); r0 < row1; r0 += TM) {
    const int nrow = (int)min((int64_t)TM, row1 - r0);   // rows of this step
    __syncthreads();
    if (geo.Sc == nullptr) {
      for (int e = t; e < k * TM; e += NT) {
        const int u = e / TM, r = e % TM;
        sk[e] = r < nrow ? A[(r0 + r) + (int64_t)Js[u] * lda] : T(0);
      }
    } else {   // single-pass ID: skeleton rows interpolated from the coarse ones
      const int r = t % TM;
      int64_t idx[8];
      T w[8];
      if (r < nrow) interp_corners<T>(r0 + r, geo, idx, w);
      const T* sc = reinterpret_cast<const T*>(geo.Sc);
      for (int u = t / TM; u < k; u += NT / TM) {
        T acc = T(0);
        if (r < nrow) {
#pragma unroll
          for (int q = 0; q < 8; ++q) acc += w[q] * sc[idx[q] * kSkelLd + u];
        }
        sk[u * TM + r] = acc;
      }
    }
    T va[2][4];   // this chunk's entries of A
    auto load = [&](int64_t cc) {
#pragma unroll
      for (int h = 0; h < 2; ++h)
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          const int64_t c = cc + tc + 16 * h;
          va[h][e] = (c < n && tr + 16 * e < nrow) ? A[(r0 + tr + 16 * e) + c * lda] : T(0);
        }
    };
    load(0);
    if (RES) __syncthreads();
    for (int64_t cc = 0; cc < n; cc += TC) {
      if (!RES) {
        __syncthreads();
        for (int e = t; e < k * TC; e += NT) {
          const int u = e / TC, cl = e % TC;
          ps[e] = (cc + cl < n) ? (T)P[(int64_t)u * n + cc + cl] : T(0);
        }
      }
      T a[2][4];
#pragma unroll
      for (int h = 0; h < 2; ++h)
#pragma unroll
        for (int e = 0; e < 4; ++e) a[h][e] = va[h][e];
      if (!RES) __syncthreads();
      // columns past the last read another column's P: their A_hat is not used
      const T* pc = RES ? ps + cc + tc : ps + tc;
      const T* pc1 = RES && cc + tc + 16 >= n ? pc : pc + 16;
      if (RES && cc + tc >= n) pc = pc1 = ps;
      if (cc + TC < n) load(cc + TC);
      T ah[2][4];
#pragma unroll
      for (int h = 0; h < 2; ++h)
#pragma unroll
        for (int e = 0; e < 4; ++e) ah[h][e] = T(0);
      if (nrow == TM) {
#pragma unroll 2
        for (int u = 0; u < k; ++u) {
          const T p0 = pc[u * ldp], p1 = pc1[u * ldp];
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            const T sv = sk[u * TM + tr + 16 * e];
            ah[0][e] += sv * p0;
            ah[1][e] += sv * p1;
          }
        }
      } else {   // the range's last step: whole groups of 16 rows are skipped
        for (int u = 0; u < k; ++u) {
          const T p0 = pc[u * ldp], p1 = pc1[u * ldp];
#pragma unroll
          for (int e = 0; e < 4; ++e)
            if (16 * e < nrow) {
              const T sv = sk[u * TM + tr + 16 * e];
              ah[0][e] += sv * p0;
              ah[1][e] += sv * p1;
            }
        }
      }
      T se = T(0), sa = T(0);
#pragma unroll
      for (int h = 0; h < 2; ++h)
#pragma unroll
        for (int e = 0; e < 4; ++e)
          if (16 * e < nrow) {   // entries outside the range or the matrix: zero on both sides
            const T x = a[h][e], d = x - ah[h][e];
            if (cc + tc + 16 * h >= n || tr + 16 * e >= nrow) continue;
            if constexpr (sizeof(T) == 4) {
              res.add(d * d);
              tot.add(x * x);
            } else {
              se += d * d;
              sa += x * x;
            }
            const T ad = magnitude(d), aa = magnitude(x);
            if (nonzero(x) && ad > mx * aa) mx = ratio(ad, aa);
          }
      if constexpr (sizeof(T) == 8) {
        res.add(se);
        tot.add(sa);
      }
      // the warp's largest ratio so far, so that the division for a new one
      // stays rare
      mx = warp_max(mx);
    }
  }
  // block reduction (fixed order)
  double v0 = (double)res.s - (double)res.c, v1 = (double)tot.s - (double)tot.c, v2 = (double)mx;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    v0 += __shfl_xor_sync(0xffffffffu, v0, o);
    v1 += __shfl_xor_sync(0xffffffffu, v1, o);
    v2 = fmax(v2, __shfl_xor_sync(0xffffffffu, v2, o));
  }
  const int lane = t & 31, warp = t >> 5;
  __syncthreads();
  if (lane == 0) {
    red[0][warp] = v0;
    red[1][warp] = v1;
    red[2][warp] = v2;
  }
  __syncthreads();
  if (t == 0) {
    double a0 = 0.0, a1 = 0.0, a2 = 0.0;
    for (int w = 0; w < NT / 32; ++w) {
      a0 += red[0][w];
      a1 += red[1][w];
      a2 = fmax(a2, red[2][w]);
    }
    part[3 * blockIdx.x + 0] = a0;
    part[3 * blockIdx.x + 1] = a1;
    part[3 * blockIdx.x + 2] = a2;
  }
}

// The CTAs' partials into the three results, in a fixed order: thread t sums
// CTAs t, t + 256, ..., then warps and their sums as trees (one thread over
// all CTAs took 28 us for 152 of them and 229 us for 1216).
constexpr int FT = 256;
__global__ void __launch_bounds__(FT) recon_finalize_kernel(const double* __restrict__ part,
                                                            int nblk,
                                                            double* __restrict__ out3) {
  __shared__ double red[3][FT / 32];
  double a0 = 0.0, a1 = 0.0, a2 = 0.0;
  for (int b = threadIdx.x; b < nblk; b += FT) {
    a0 += part[3 * b];
    a1 += part[3 * b + 1];
    a2 = fmax(a2, part[3 * b + 2]);
  }
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    a0 += __shfl_xor_sync(0xffffffffu, a0, o);
    a1 += __shfl_xor_sync(0xffffffffu, a1, o);
    a2 = fmax(a2, __shfl_xor_sync(0xffffffffu, a2, o));
  }
  if (lane == 0) {
    red[0][warp] = a0;
    red[1][warp] = a1;
    red[2][warp] = a2;
  }
  __syncthreads();
  if (warp == 0) {
    a0 = lane < FT / 32 ? red[0][lane] : 0.0;
    a1 = lane < FT / 32 ? red[1][lane] : 0.0;
    a2 = lane < FT / 32 ? red[2][lane] : 0.0;
#pragma unroll
    for (int o = FT / 64; o > 0; o >>= 1) {
      a0 += __shfl_xor_sync(0xffffffffu, a0, o);
      a1 += __shfl_xor_sync(0xffffffffu, a1, o);
      a2 = fmax(a2, __shfl_xor_sync(0xffffffffu, a2, o));
    }
    if (lane == 0) {
      out3[0] = a0;
      out3[1] = a1;
      out3[2] = a2;
    }
  }
}

constexpr size_t kReconSmem = 112 * 1024;   // at most
// All of P in shared memory when two CTAs per SM hold it beside the skeleton
// rows: no barrier and no load of P per chunk.
template <typename T>
bool recon_resident(int k, int64_t n) {
  return sizeof(T) * (size_t)k * (TM + (size_t)n) <= kReconSmem;
}
template <typename T>
size_t recon_smem(int k, int64_t n) {
  return sizeof(T) * (size_t)k * (TM + (recon_resident<T>(k, n) ? (size_t)n : TC));
}

}  // namespace

cudaError_t launch_recon_error(const void* A, int64_t lda, int64_t m, int64_t n, int dtype,
                               const int* J, const double* P, int k, double* part, int nblk,
                               double* out3, int* status, cudaStream_t st, KernelTimer* timer,
                               const InterpGeom* interp) {
  const InterpGeom geo = interp ? *interp : InterpGeom{};
  int dev = 0, nsm = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
  if (e != cudaSuccess) return e;
  if (dtype == ID_F32 && m >= 128) {
    // FP32 data: tensor-core pass (products split into bf16 pieces)
    const int grid = std::min(recon_tc_grid(m, n, nsm), nblk);
    if (grid * 1 < (int)((n + 255) / 256)) return cudaErrorInvalidValue;
    e = launch_recon_tc(reinterpret_cast<const float*>(A), lda, m, n, J, P, k, part, grid,
                        status, st, timer, interp);
    if (e != cudaSuccess) return e;
    recon_finalize_kernel<<<1, FT, 0, st>>>(part, grid, out3);
    count_launches(1);
    return cudaGetLastError();
  }
  // two CTAs per SM (16 warps, 128 registers), at least a step of 64 rows each
  const int grid =
      (int)std::max<int64_t>(1, std::min<int64_t>((m + TM - 1) / TM, std::min(nblk, 2 * nsm)));
  if (timer && (e = timer->mark(st)) != cudaSuccess) return e;
  auto go = [&](auto kern, const auto* data, size_t sm) {
    const cudaError_t r = allow_smem(kern, kReconSmem);
    if (r == cudaSuccess) kern<<<grid, NT, sm, st>>>(data, lda, m, n, J, P, k, part, geo);
    return r;
  };
  if (dtype == ID_F64)
    e = go(recon_resident<double>(k, n) ? recon_kernel<double, true> : recon_kernel<double, false>,
           reinterpret_cast<const double*>(A), recon_smem<double>(k, n));
  else
    e = go(recon_resident<float>(k, n) ? recon_kernel<float, true> : recon_kernel<float, false>,
           reinterpret_cast<const float*>(A), recon_smem<float>(k, n));
  if (e != cudaSuccess) return e;
  e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  if (timer && (e = timer->mark(st)) != cudaSuccess) return e;
  recon_finalize_kernel<<<1, FT, 0, st>>>(part, grid, out3);
  count_launches(2);
  return cudaGetLastError();
}

}  // namespace idsk
