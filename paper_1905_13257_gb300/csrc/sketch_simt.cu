// Fused single-read sketch, CUDA-core (SIMT) form, and the Gaussian fill.
//
// One read of each tile of A forms both randomized sketches of the streamed
// columns (Algorithm 4 step 3, transposed orientation, and eq. eq:sampmatrix):
//   W(:, cols) = Psi A(:, cols)        (l x ncols; 64-row sums in the data's
//                                       type, accumulated in FP64)
//   Y         += A(:, cols) Omega(cols, :)   (m x l)
// and, when asked, gathers the coarse-grid rows A_c = A(rows_c, cols) of
// Algorithm 5 step 3 from the same tile.  Psi is never stored: each CTA draws
// Psi(:, R) for its row tile R from the counter generator.
//
// This form serves FP64 data and any shape; the tensor-core form in
// sketch_tc.cu serves FP32 data at HBM speed.
#include <cuda_bf16.h>

#include <algorithm>
#include <type_traits>

#include "df.cuh"
#include "idsk_internal.h"

namespace idsk {
namespace {

constexpr int TM = 64;    // rows per tile
constexpr int NT = 256;   // threads per CTA
// columns per chunk (multiples of 16; FP64 keeps room for the accumulators)
template <typename T>
constexpr int kTC = sizeof(T) == 4 ? 64 : 32;
// leading dimension of the Psi and A tiles: rows 16 bytes apart modulo a
// 128-byte line, so that 128-bit loads of 8 columns hit all banks
template <typename T>
constexpr int kLdt = TM + 16 / (int)sizeof(T);

__global__ void gaussian_fill_kernel(uint32_t which, uint32_t k0, uint32_t k1, int64_t first,
                                     int64_t count, int width, const float* __restrict__ table,
                                     float* __restrict__ out) {
  const int nblk = (width + 9) / 10;
  const int64_t total = count * nblk;
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < total;
       e += (int64_t)gridDim.x * blockDim.x) {
    const int64_t i = e / nblk;
    const int sb = (int)(e % nblk);
    float g[10];
    gauss10((uint64_t)(first + i), (uint32_t)sb, which, k0, k1, table, g);
#pragma unroll
    for (int f = 0; f < 10; ++f) {
      const int s = sb * 10 + f;
      if (s < width) out[i * width + s] = g[f];
    }
  }
}

__device__ __forceinline__ float to_bf16_rn(float x) {
  return __bfloat162float(__float2bfloat16_rn(x));
}

template <typename T>
__device__ __forceinline__ T maybe_bf16(T v, int on) {
  return v;
}
template <>
__device__ __forceinline__ float maybe_bf16<float>(float v, int on) {
  return on ? to_bf16_rn(v) : v;
}

template <typename I>
__device__ __forceinline__ int64_t coarse_index_of(I r, const CoarseGeom& g) {
  const I i = r % (I)g.nx, rest = r / (I)g.nx;
  const I z = rest % (I)g.nz, rest2 = rest / (I)g.nz;
  const I j = rest2 % (I)g.ny, c = rest2 / (I)g.ny;
  if (i % (I)g.sx || j % (I)g.sy || z % (I)g.sz) return -1;
  return ((int64_t)(c * (I)g.cy + j / (I)g.sy) * g.cz + z / (I)g.sz) * g.cx + i / (I)g.sx;
}
__device__ __forceinline__ int64_t coarse_index(int64_t r, const CoarseGeom& g) {
  return r < ((int64_t)1 << 31) ? coarse_index_of((uint32_t)r, g) : coarse_index_of(r, g);
}

// 16 bytes of T.
template <typename T>
struct Vec;
template <>
struct Vec<float> {
  static constexpr int N = 4;
  float4 x;
  __device__ __forceinline__ void load(const float* p) { x = *reinterpret_cast<const float4*>(p); }
  __device__ __forceinline__ float at(int e) const {
    return e == 0 ? x.x : e == 1 ? x.y : e == 2 ? x.z : x.w;
  }
};
template <>
struct Vec<double> {
  static constexpr int N = 2;
  double2 x;
  __device__ __forceinline__ void load(const double* p) {
    x = *reinterpret_cast<const double2*>(p);
  }
  __device__ __forceinline__ double at(int e) const { return e == 0 ? x.x : x.y; }
};

// Shared layout: W accumulators l x ncols | column pointers | coarse rows TM |
// quantile table | Psi tile 16 SU x kLdt | A tile kTC x kLdt | Omega tile
// kTC x 16 SU (Psi and Omega held in T, so that no product converts them).
template <typename T>
__host__ __device__ inline size_t simt_fixed_bytes(int su) {
  return sizeof(int64_t) * TM + sizeof(float) * kTableSize +
         sizeof(T) * ((size_t)(16 * su + kTC<T>) * kLdt<T> + (size_t)kTC<T> * 16 * su);
}

// SU: groups of 16 sketch rows (l <= 16 SU).  Per 64-row tile the CTA draws
// Psi(:, R), then takes the window's columns in chunks of kTC: the chunk's
// entries and its rows of Omega are loaded into registers while the chunk
// before is multiplied.  Thread (tj, ti) = (t mod 16, t / 16) forms the 4 x SU
// (FP64: 2 x SU) products of W with columns tj + 16 u and sketch rows ti + 16
// v over the tile's rows, and the 4 x SU of Y with rows 4 tj .. 4 tj + 3 and
// sketch columns ti + 16 v over the chunk's columns: SU + 4 128-bit (or
// 4 + SU smaller) shared loads per 16 SU products, where one product per two
// loads made the kernel shared-memory bound; groups of 16 columns past the
// window's last are skipped.  FP64 data: now bound by the FP64 units (2 fused
// multiply-adds per clock and SM: 1.9 ms for 98,304 x 200, l = 30 with Y);
// FP32 data: by the shared-memory bandwidth of the 4 x 4 blocks (512 bytes a
// warp for every 16 products of a lane, twice the FP32 units' time).
// Measured: 98,304 x 200 FP64, l = 30 with Y in 7 launches: 8844 -> 2598 us;
// 315,315 x 333 FP32, l = 60 with Y: 3967 -> 1394 us with W's sums as FP32
// pairs, about 100 us more with the FP64 sums they have.
template <typename T, int SU>
__global__ void __launch_bounds__(NT, 1) sketch_simt_kernel(const __grid_constant__ SketchArgs a,
                                                            const __grid_constant__ Window w) {
  using V = Vec<T>;
  constexpr int TC = kTC<T>, LD = kLdt<T>, LO = 16 * SU;
  constexpr int CU = TC / 16;            // groups of 16 columns in a chunk
  constexpr int NA = TC * TM / NT;       // entries of A per thread and chunk
  constexpr int NO = TC * LO / NT;       // entries of Omega per thread and chunk
  extern __shared__ __align__(16) unsigned char smem[];
  const int ncols = w.ncols, l = a.l;
  const int nacc = (l * ncols + 1) & ~1;   // keeps what follows 16-byte aligned
  double* wacc = reinterpret_cast<double*>(smem);   // W's sums: FP64 over the row tiles
  T* psi_s = reinterpret_cast<T*>(wacc + nacc);
  T* a_s = psi_s + LO * LD;
  T* om_s = a_s + TC * LD;
  float* tab = reinterpret_cast<float*>(om_s + TC * LO);
  int64_t* rc_s = reinterpret_cast<int64_t*>(tab + kTableSize);
  const T** cptr_s = reinterpret_cast<const T**>(rc_s + TM);

  const int t = threadIdx.x, tj = t & 15, ti = t >> 4;
  const int lr = t & (TM - 1), lc = t / TM;   // loads of A: row, first column

  for (int e = t; e < kTableSize; e += NT) tab[e] = a.table[e];
  for (int e = t; e < l * ncols; e += NT) wacc[e] = 0.0;
  for (int c = t; c < ncols; c += NT) {
    const T* p = nullptr;
    for (int q = 0; q < w.nseg; ++q) {
      const Seg& sg = w.seg[q];
      if (c >= sg.col0 && c < sg.col0 + sg.ncols)
        p = reinterpret_cast<const T*>(sg.ptr) + (int64_t)(c - sg.col0) * sg.ld;
    }
    cptr_s[c] = p;
  }
  __syncthreads();

  const int64_t ntiles = (a.m + TM - 1) / TM;
  T va[NA];
  float vo[NO];
  auto load = [&](int64_t tile, int cc) {
    const int64_t r = tile * TM + lr;
#pragma unroll
    for (int q = 0; q < NA; ++q) {
      const int c = cc + lc + q * (NT / TM);
      va[q] = (c < ncols && r < a.m) ? cptr_s[c][r] : T(0);
    }
#pragma unroll
    for (int q = 0; q < NO; ++q) {
      const int e = t + q * NT, c = cc + e / LO, sv = e % LO;
      vo[q] = (a.want_Y && c < ncols && sv < l) ? a.omega[(w.col_base + c) * l + sv] : 0.f;
    }
  };
  // W(:, chunk) += Psi(:, R) A(R, chunk) over the first CUN groups of columns
  auto products_w = [&](auto cun, int cc) {
    constexpr int CUN = decltype(cun)::value;
    T acc[SU][CUN];
#pragma unroll
    for (int v = 0; v < SU; ++v)
#pragma unroll
      for (int u = 0; u < CUN; ++u) acc[v][u] = T(0);
#pragma unroll 2
    for (int r = 0; r < TM; r += V::N) {
      V ps[SU], av[CUN];
#pragma unroll
      for (int v = 0; v < SU; ++v) ps[v].load(psi_s + (ti + 16 * v) * LD + r);
#pragma unroll
      for (int u = 0; u < CUN; ++u) av[u].load(a_s + (tj + 16 * u) * LD + r);
#pragma unroll
      for (int e = 0; e < V::N; ++e)
#pragma unroll
        for (int v = 0; v < SU; ++v)
#pragma unroll
          for (int u = 0; u < CUN; ++u) acc[v][u] += ps[v].at(e) * av[u].at(e);
    }
    auto add = [&](auto widen) {
#pragma unroll
      for (int v = 0; v < SU; ++v)
#pragma unroll
        for (int u = 0; u < CUN; ++u) {
          const int sr = ti + 16 * v, c = cc + tj + 16 * u;
          if (sr < l && c < ncols) wacc[sr * ncols + c] += widen(acc[v][u]);
        }
    };
    if constexpr (sizeof(T) == 4) {
      bool plain = true;
#pragma unroll
      for (int v = 0; v < SU; ++v)
#pragma unroll
        for (int u = 0; u < CUN; ++u) plain = plain && widens(acc[v][u]);
      if (plain)
        add([](float x) { return widen_normal(x); });
      else
        add([](float x) { return (double)x; });
    } else {
      add([](double x) { return x; });
    }
  };

  if (blockIdx.x < ntiles) load(blockIdx.x, 0);
  for (int64_t tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
    const int64_t r0 = tile * TM;
    __syncthreads();   // previous tile fully consumed
    // Psi(:, R) from the counter generator
    {
      const int64_t i = r0 + lr;
      for (int sb = lc; sb * 10 < LO; sb += NT / TM) {
        float g[10];
        if (i < a.m) {
          gauss10((uint64_t)i, (uint32_t)sb, kStreamPsi, a.k0, a.k1, tab, g);
        } else {
#pragma unroll
          for (int f = 0; f < 10; ++f) g[f] = 0.f;
        }
#pragma unroll
        for (int f = 0; f < 10; ++f) {
          const int sr = sb * 10 + f;
          if (sr < LO) psi_s[sr * LD + lr] = (sr < l) ? (T)g[f] : T(0);
        }
      }
      if (t < TM) rc_s[t] = (a.cg.on && r0 + t < a.m) ? coarse_index(r0 + t, a.cg) : -1;
    }
    T yacc[SU][4];
#pragma unroll
    for (int v = 0; v < SU; ++v)
#pragma unroll
      for (int e = 0; e < 4; ++e) yacc[v][e] = T(0);

    for (int cc = 0; cc < ncols; cc += TC) {
      __syncthreads();   // Psi and the coarse rows written; previous chunk consumed
      const int64_t rc = rc_s[lr];
#pragma unroll
      for (int q = 0; q < NA; ++q) {
        const int c = lc + q * (NT / TM);
        if (rc >= 0 && cc + c < ncols)
          reinterpret_cast<T*>(a.Ac)[rc + a.cg.mc * (w.col_base + cc + c)] = va[q];
        a_s[c * LD + lr] = maybe_bf16(va[q], a.bf16);
      }
#pragma unroll
      for (int q = 0; q < NO; ++q) om_s[t + q * NT] = (T)vo[q];
      __syncthreads();
      if (cc + TC < ncols)
        load(tile, cc + TC);
      else if (tile + gridDim.x < ntiles)
        load(tile + gridDim.x, 0);
      // Y(R, :) += A(R, chunk) Omega(chunk, :)
      if (a.want_Y) {
        const int nc = min(TC, ncols - cc);
#pragma unroll 4
        for (int c = 0; c < nc; ++c) {
          V av[4 / V::N];
#pragma unroll
          for (int h = 0; h < 4 / V::N; ++h) av[h].load(a_s + c * LD + 4 * tj + V::N * h);
#pragma unroll
          for (int v = 0; v < SU; ++v) {
            const T o = om_s[c * LO + ti + 16 * v];
#pragma unroll
            for (int e = 0; e < 4; ++e) yacc[v][e] += av[e / V::N].at(e % V::N) * o;
          }
        }
      }
      const int nu = min(CU, (ncols - cc + 15) / 16);
      if constexpr (CU == 4) {
        if (nu == 4)
          products_w(std::integral_constant<int, 4>(), cc);
        else if (nu == 3)
          products_w(std::integral_constant<int, 3>(), cc);
      }
      if (nu == 2)
        products_w(std::integral_constant<int, 2>(), cc);
      else if (nu == 1)
        products_w(std::integral_constant<int, 1>(), cc);
    }
    if (a.want_Y) {
      T* Y = reinterpret_cast<T*>(a.Y);
#pragma unroll
      for (int v = 0; v < SU; ++v) {
        const int sr = ti + 16 * v;
        if (sr >= l) continue;
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          const int64_t i = r0 + 4 * tj + e;
          if (i < a.m) {
            const int64_t o = i + sr * a.m;
            Y[o] = a.y_accumulate ? Y[o] + yacc[v][e] : yacc[v][e];
          }
        }
      }
    }
  }
  __syncthreads();
  for (int e = t; e < l * ncols; e += NT) {
    const int sr = e / ncols, c = e % ncols;
    atomicAdd(&a.W[sr * a.ldw + w.col_base + c], wacc[e]);
  }
}

template <typename T>
size_t simt_smem_bytes(int l, int ncols) {
  return sizeof(double) * (((size_t)l * ncols + 1) & ~(size_t)1) +
         simt_fixed_bytes<T>((l + 15) / 16) + sizeof(void*) * (size_t)ncols;
}

template <typename T>
cudaError_t launch_simt(const SketchArgs& a, const Window& w, int grid, cudaStream_t st) {
  const size_t sm = simt_smem_bytes<T>(a.l, w.ncols);
  auto go = [&](auto kern) {
    const cudaError_t e = allow_smem(kern, kSmemMost);
    if (e != cudaSuccess) return e;
    kern<<<grid, NT, sm, st>>>(a, w);
    return cudaGetLastError();
  };
  switch ((a.l + 15) / 16) {
    case 1: return go(sketch_simt_kernel<T, 1>);
    case 2: return go(sketch_simt_kernel<T, 2>);
    case 3: return go(sketch_simt_kernel<T, 3>);
    default: return go(sketch_simt_kernel<T, 4>);
  }
}

}  // namespace

cudaError_t launch_gaussian_fill(uint32_t which, uint32_t k0, uint32_t k1, int64_t first,
                                 int64_t count, int width, const float* table, float* out,
                                 cudaStream_t st) {
  if (count <= 0 || width <= 0) return cudaSuccess;
  const int64_t total = count * ((width + 9) / 10);
  const int blocks = (int)std::min<int64_t>((total + 255) / 256, 4096);
  gaussian_fill_kernel<<<blocks, 256, 0, st>>>(which, k0, k1, first, count, width, table, out);
  count_launches(1);
  return cudaGetLastError();
}

// Columns of one launch: what the shared memory holds, at most kSimtWindowMax.
int simt_window_cols(int l, int dtype) {
  int n = kSimtWindowMax;
  while (n > 16 && (dtype == ID_F64 ? simt_smem_bytes<double>(l, n)
                                    : simt_smem_bytes<float>(l, n)) > kSmemMost)
    n -= 16;
  return n;
}

cudaError_t launch_sketch_simt(const SketchArgs& a, const Window& w, int dtype, int nsm,
                               cudaStream_t st) {
  if (w.ncols <= 0) return cudaSuccess;
  if (a.l > kLMax) return cudaErrorInvalidValue;
  const int64_t ntiles = (a.m + TM - 1) / TM;
  const int grid = (int)std::min<int64_t>(ntiles, nsm);
  const cudaError_t e =
      dtype == ID_F64 ? launch_simt<double>(a, w, grid, st) : launch_simt<float>(a, w, grid, st);
  count_launches(1);
  return e;
}

}  // namespace idsk
