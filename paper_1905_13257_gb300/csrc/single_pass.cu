// Single-pass ID (Algorithm 6, Sec. 2.6, eq. eqn:single_ID), column
// orientation: A ~ M A_c(:, J_c) P_c.  The fine skeleton is not read from A a
// second time; the coarse skeleton A_c(:, J_c) is interpolated back to the
// fine grid by the coarse-to-fine operator M (Algorithm 6 step 4).
//
// M is trilinear interpolation on the mesh (t = 8 coarse points per fine
// point), applied as a tensor product of one-dimensional rules:
//   * coarse points are every s-th index from 0 in each direction (the direct
//     injection of Sec. 2.5);
//   * between two coarse points the weight of the upper one is the fraction
//     of the physical distance, (x_i - x_lo) / (x_hi - x_lo);
//   * past the last coarse point a periodic direction wraps to coarse point 0
//     at x_0 + period, a non-periodic one extrapolates linearly from its last
//     two coarse points.
// M is never stored: each fine row finds its 8 corners from three small
// per-direction tables (interp_corners).
#include <algorithm>
#include <cmath>

#include "idsk_internal.h"

namespace idsk {

void build_axis_weights(const double* x, int n, int stride, double period, AxisW* out) {
  const int c = (n + stride - 1) / stride;
  for (int i = 0; i < n; ++i) {
    const int a = i / stride;
    AxisW e{a, a, 0.0};
    if (i % stride != 0) {
      if (a + 1 < c) {
        e.hi = a + 1;
        e.w = (x[i] - x[a * stride]) / (x[(a + 1) * stride] - x[a * stride]);
      } else if (period > 0.0) {
        e.hi = 0;
        e.w = (x[i] - x[a * stride]) / (x[0] + period - x[a * stride]);
      } else if (c >= 2) {
        e.lo = c - 2;
        e.hi = c - 1;
        e.w = (x[i] - x[(c - 2) * stride]) / (x[(c - 1) * stride] - x[(c - 2) * stride]);
      } else {
        e.lo = e.hi = 0;
      }
    }
    out[i] = e;
  }
}

namespace {

// Sc(i, u) = A_c(i, J_c[u]) for u < k, 0 for k <= u < kSkelLd (row-major).
template <typename T>
__global__ void skeleton_compact_kernel(const T* __restrict__ Ac, int64_t mc,
                                        const int* __restrict__ Jc, int k, T* __restrict__ Sc) {
  const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= mc * kSkelLd) return;
  const int64_t i = e / kSkelLd;
  const int u = (int)(e - i * kSkelLd);
  Sc[e] = u < k ? Ac[i + (int64_t)Jc[u] * mc] : T(0);
}

// S = M A_c(:, J_c), column-major m x k, a fine row per thread: S(r, u) = sum over
// the 8 corners of w * Sc(corner, u).  For short lines and few columns, where a
// segment of lift_kernel does too little to pay for its tables and barriers.
template <typename T>
__global__ void lift_rows_kernel(InterpGeom g, int64_t m, int k, T* __restrict__ S) {
  const int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (r >= m) return;
  int64_t idx[8];
  T w[8];
  interp_corners<T>(r, g, idx, w);
  const T* Sc = reinterpret_cast<const T*>(g.Sc);
  for (int u = 0; u < k; ++u) {
    T acc = T(0);
#pragma unroll
    for (int q = 0; q < 8; ++q) acc += w[q] * Sc[idx[q] * kSkelLd + u];
    S[r + (int64_t)u * m] = acc;
  }
}

// The same by lines: a line is the nx fine rows
// of one (component, y, z), cut into segments of at most 128.  Per segment the
// CTA first interpolates in y and z at the coarse x points that the segment
// touches (lanes along the skeleton's columns: coalesced), into shared memory,
// then in x, one fine row per lane: two shared loads and one store per value
// where eight scattered loads stood before.  FP32 data interpolate in FP32
// (weights rounded), FP64 data in FP64.
// 1,824,768 x 40 FP32: 515 -> 125 us (the write of S alone takes 43 us; the
// rest is the latency of a segment's tables and coarse values).
constexpr int LF_SEG = 128, LF_THREADS = 256;
constexpr int LF_LD = LF_SEG + 5;   // coarse points of a segment, the wrapped point; odd
template <typename T>
__global__ void __launch_bounds__(LF_THREADS) lift_kernel(InterpGeom g, int64_t lines, int nseg,
                                                          int64_t m, int k, T* __restrict__ S) {
  extern __shared__ __align__(16) unsigned char smem[];
  T* L = reinterpret_cast<T*>(smem);   // k x LF_LD: the line's coarse points after y and z
  const T* Sc = reinterpret_cast<const T*>(g.Sc);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  for (int64_t w = blockIdx.x; w < lines * nseg; w += gridDim.x) {
    // 64-bit divisions cost more than a segment's other work: 32-bit ones
    // wherever the indices allow
    const bool small = lines * nseg < ((int64_t)1 << 31);
    auto quot = [&](int64_t a, int b) {
      return small ? (int64_t)((uint32_t)a / (uint32_t)b) : a / b;
    };
    const int64_t ln = quot(w, nseg);
    const int i0 = (int)(w - ln * nseg) * LF_SEG, i1 = min(i0 + LF_SEG, g.nx);
    const int64_t cj = quot(ln, g.nz);
    const int kz = (int)(ln - cj * g.nz);
    const int64_t c = quot(cj, g.ny);
    const AxisW Y = g.ay[cj - c * g.ny], Z = g.az[kz];
    // coarse x points of the segment: the neighbours rise with i, but past the
    // last coarse point they are the last two, or the last and (wrapped) 0
    const AxisW X0 = g.ax[i0], X1 = g.ax[i1 - 1];
    const int a0 = min(X0.lo, X1.lo), a1 = max(X1.lo, X1.hi);
    const bool wraps = X1.hi < X1.lo;
    const int np = max(a1, X0.lo) - a0 + 1, tot = np + (wraps ? 1 : 0);
    const T y1 = (T)Y.w, y0 = (T)1 - y1, z1 = (T)Z.w, z0 = (T)1 - z1;
    const T w00 = y0 * z0, w01 = y0 * z1, w10 = y1 * z0, w11 = y1 * z1;
    const int64_t base0 = (c * g.cy + Y.lo) * g.cz, base1 = (c * g.cy + Y.hi) * g.cz;
    const T* p00 = Sc + (base0 + Z.lo) * g.cx * kSkelLd;
    const T* p01 = Sc + (base0 + Z.hi) * g.cx * kSkelLd;
    const T* p10 = Sc + (base1 + Z.lo) * g.cx * kSkelLd;
    const T* p11 = Sc + (base1 + Z.hi) * g.cx * kSkelLd;
    __syncthreads();   // the segment before has been written out
    {
      constexpr int PER = LF_THREADS / kSkelLd;   // coarse points per round of the CTA
      const int u = threadIdx.x & (kSkelLd - 1);
      for (int q0 = threadIdx.x / kSkelLd; q0 < tot && u < k; q0 += 4 * PER) {
        T v[4][4];   // four rounds' loads in flight
#pragma unroll
        for (int h = 0; h < 4; ++h) {
          const int q = min(q0 + h * PER, tot - 1);
          const int64_t o = (int64_t)(q < np ? a0 + q : 0) * kSkelLd + u;
          v[h][0] = __ldg(p00 + o);
          v[h][1] = __ldg(p01 + o);
          v[h][2] = __ldg(p10 + o);
          v[h][3] = __ldg(p11 + o);
        }
#pragma unroll
        for (int h = 0; h < 4; ++h)
          if (q0 + h * PER < tot)
            L[u * LF_LD + q0 + h * PER] =
                w00 * v[h][0] + w01 * v[h][1] + w10 * v[h][2] + w11 * v[h][3];
      }
    }
    __syncthreads();
    // warps over (32 rows, every LF_THREADS / 32-th column)
    for (int i = i0 + lane; i - lane < i1; i += 32) {
      if (i >= i1) continue;
      const AxisW X = g.ax[i];
      const int lo = X.lo - a0, hi = X.hi < X.lo ? np : X.hi - a0;
      const T x1 = (T)X.w, x0 = (T)1 - x1;
      T* dst = S + ln * g.nx + i;
#pragma unroll 4
      for (int u = warp; u < k; u += LF_THREADS / 32)
        dst[(int64_t)u * m] = x0 * L[u * LF_LD + lo] + x1 * L[u * LF_LD + hi];
    }
  }
}

// Which form is faster depends on a line's length, its coarse points and k (the
// number of lines matters to neither), found over nx = 4 to 256, k = 2 to 64,
// strides 2 and 4 at 0.3 and 1.5 million rows; the whole call in us, by rows and
// by lines, 1.5 million rows, stride 2:
//   FP32 nx = 8, k = 24: 390, 627;  nx = 24, k = 8: 227, 257;  k = 16: 368, 265;
//        nx = 96, k = 2: 123, 150;  k = 40: 913, 228
//   FP64 nx = 8, k = 64: 1439, 3223;  nx = 32, k = 24: 626, 560;  k = 16: 464, 524;
//        nx = 128, k = 8: 296, 361;  k = 24: 626, 453
bool lift_by_rows(const InterpGeom& g, int dtype, int k) {
  const int64_t nx = g.nx, cx = g.cx;
  if (dtype == ID_F64) return k * nx < 1000 || k * nx < 28 * cx;
  return k < 4 || k * cx * cx < 110 * cx + 400;
}

}  // namespace

cudaError_t launch_skeleton_compact(const void* Ac, int64_t mc, int dtype, const int* Jc, int k,
                                    void* Sc, cudaStream_t st) {
  const int64_t tot = mc * kSkelLd;
  const int blocks = (int)((tot + 255) / 256);
  if (dtype == ID_F64)
    skeleton_compact_kernel<double><<<blocks, 256, 0, st>>>(
        reinterpret_cast<const double*>(Ac), mc, Jc, k, reinterpret_cast<double*>(Sc));
  else
    skeleton_compact_kernel<float><<<blocks, 256, 0, st>>>(
        reinterpret_cast<const float*>(Ac), mc, Jc, k, reinterpret_cast<float*>(Sc));
  count_launches(1);
  return cudaGetLastError();
}

cudaError_t launch_single_pass_lift(const InterpGeom& g, int64_t m, int dtype, int k, void* S,
                                    cudaStream_t st) {
  if (lift_by_rows(g, dtype, k)) {
    const int blocks = (int)((m + 255) / 256);
    if (dtype == ID_F64)
      lift_rows_kernel<double><<<blocks, 256, 0, st>>>(g, m, k, reinterpret_cast<double*>(S));
    else
      lift_rows_kernel<float><<<blocks, 256, 0, st>>>(g, m, k, reinterpret_cast<float*>(S));
    count_launches(1);
    return cudaGetLastError();
  }
  const int nseg = (g.nx + LF_SEG - 1) / LF_SEG;
  const int64_t lines = m / g.nx;
  const unsigned grid = (unsigned)std::min<int64_t>(lines * nseg, 1 << 14);
  auto go = [&](auto kern, auto* out) {
    const size_t sm = sizeof(*out) * (size_t)k * LF_LD;
    const cudaError_t e = allow_smem(kern, sizeof(*out) * (size_t)kSkelLd * LF_LD);
    if (e == cudaSuccess) kern<<<grid, LF_THREADS, sm, st>>>(g, lines, nseg, m, k, out);
    return e;
  };
  const cudaError_t e = dtype == ID_F64 ? go(lift_kernel<double>, reinterpret_cast<double*>(S))
                                        : go(lift_kernel<float>, reinterpret_cast<float*>(S));
  if (e != cudaSuccess) return e;
  count_launches(1);
  return cudaGetLastError();
}

}  // namespace idsk
