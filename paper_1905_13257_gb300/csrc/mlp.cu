// Learned skeleton proposal: the network's training and inference kernels.
// No counterpart in the paper (which motivates the ID as the selection of the
// most important snapshots, Sec. 4); the network is
//   s = w2 . gelu(x W1 + b1) + b2,  gelu(z) = z Phi(z)  (exact GELU),
// on features x of a snapshot column (its values on a coarse sub-grid),
// trained on the skeletons of the plain randomized ID with the mean binary
// cross entropy of sigmoid(s).
//
// Kernels (every sum in a fixed order, no atomics on data):
//   features_kernel  X(j, f) = scale * A(rows[f], j)
//   tc_gemm_kernel   the two dense products on the tcgen05 tensor cores,
//                    bfloat16 operands (weights and features) with FP32
//                    accumulation: forward Z = X W1 + b1 with G = gelu(Z) in
//                    the epilogue; backward dW1 = X^T dZ
//   score_kernel     s = G w2 + b2, one warp per column, shuffle tree
//   backward_kernel  ds = d loss / d s, dZ = ds w2^T .* gelu'(Z) and the column
//                    sums db1 = sum dZ, dw2 = G^T ds, db2 = sum ds
//   sgd_kernel       p -= lr g
#include <cooperative_groups.h>
#include <limits.h>
#include <math.h>

#include <atomic>

#include <algorithm>

#include "idsk_internal.h"
#include "tc_common.cuh"

namespace idsk {
extern std::atomic<int> g_last_cuda_error;
}

using namespace idsk;
namespace cg = cooperative_groups;

namespace {

__device__ __forceinline__ float gelu_f(float z) { return z * normcdff(z); }
__device__ __forceinline__ float gelu_grad_f(float z) {
  return normcdff(z) + z * (expf(-0.5f * z * z) * 0.3989422804014327f);
}

// A row index outside [0, m) gives a NaN feature (never an out-of-bounds read).
template <typename T>
__global__ void features_kernel(const T* __restrict__ A, int64_t lda, int64_t m, int64_t n,
                                const int64_t* __restrict__ rows, int64_t F, float scale,
                                float* __restrict__ X) {
  const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= n * F) return;
  const int64_t j = e / F, f = e - j * F;
  const int64_t r = rows[f];
  X[e] = (r >= 0 && r < m) ? scale * (float)A[r + j * lda] : __int_as_float(0x7fc00000);
}

// ---------------------------------------------------------------------------
// The two dense products of the network on the tcgen05 tensor cores, with
// bfloat16 operands and FP32 accumulation in TMEM:
//   forward   Z (n x H) = X (n x F) W1 (F x H)       [+ b1, G = gelu(Z)]
//   backward  gW1 (F x H) = X^T (F x n) dZ (n x H)
// C (M x N, row-major FP32, ldc = N) = A (M x K) B (K x N), where element
// (i, k) of A is A[i * a_si + k * a_sk] and element (k, j) of B is
// B[k * b_sk + j * b_sj] (FP32 in global memory; any of the two layouts of
// each operand).  Every operand value is rounded to bfloat16 as it is staged,
// so the weights and the features enter the products in bfloat16 and every
// product accumulates in FP32.
//
// A CTA of 16 warps owns a 128 x TN output tile over all of K.  All warps stage
// KC-wide K chunks of A and B as K-major 128-byte-swizzled bfloat16 tiles in
// two shared-memory stages, with the global loads of the next chunk in flight
// in registers; one thread issues the chunk's kind::f16 MMAs (M = 128, N = TN,
// K = 16) into a TN-column TMEM accumulator and commits them to the stage's
// mbarrier.  The epilogue reads the accumulator (row i = TMEM lane i)
// and adds the bias / applies the GELU.  Every output is the sum of its K
// products in ascending order in one accumulator, so the result does not
// depend on scheduling or on the tile (K split over a cluster of 8 CTAs was
// faster, 68 against 91 us for a whole training step, but its sums round
// differently).
// The products are small (512 x 4096 x 256: 1 GFLOP, 12 MB); what bounds them is
// how many SMs stage operands and the fixed cost of a chunk (two barriers, the
// proxy fence, the conversion: about 0.6 us).  Forward: TN = 32, KC = 128, 32
// CTAs for 512 x 256 outputs (TN = 64 or KC = 64 were 20% and 13% slower; two
// or three chunks of loads ahead no faster); gW1, whose M = F gives 128 CTAs:
// TN = 64, KC = 64 (TN = 32 reads X twice as often: 28 against 21 us).
// Measured (512 x 4096 x 256): forward with scores 45.1 us, backward with its
// sums 19.9 us; 8 CTAs of 128 x 128 before: 412 us for either product.
// The waits are bounded: on timeout the kernel raises g_mlp_abort, writes NaN
// to its tile and frees its TMEM.
constexpr int TG_M = 128, TG_THREADS = 512;

__device__ int g_mlp_abort;

// A tile's operand: TILE rows (r) x KC-wide K chunks of a strided FP32 matrix,
// N values per thread and chunk.  What a thread reads of a chunk lies at fixed
// 32-bit offsets from a pointer that is the same for the whole CTA and moves
// from chunk to chunk; rows past the last are clamped to it (they only feed
// outputs that nobody stores).
// ROWS_K (element (r, k) at X[r * ld + k]): pieces of 4 consecutive k of one
// row, one 128-bit load each where VEC (16-byte aligned rows).  Otherwise
// (element (r, k) at X[k * ld + r]): pieces of 8 consecutive k of one row,
// consecutive lanes take consecutive rows.
template <int TILE, int KC, bool ROWS_K, bool VEC, int THREADS>
struct Operand {
  static constexpr int PIECE = ROWS_K ? 4 : 8;
  static constexpr int NP = TILE * KC / PIECE / THREADS;   // pieces per thread
  static constexpr int N = NP * PIECE;
  static_assert(NP >= 1, "a piece per thread");
  const float* base;      // of the tile's rows
  uint32_t ld;
  uint32_t off[NP];       // of each piece in a chunk
  uint32_t dst[NP];       // its place in the staged tile

  __device__ __forceinline__ void init(const float* X, int64_t ld_, int rows, int r0, int t) {
    base = X + (ROWS_K ? (int64_t)r0 * ld_ : (int64_t)r0);
    ld = (uint32_t)ld_;
#pragma unroll
    for (int q = 0; q < NP; ++q) {
      const uint32_t c = (uint32_t)(t + q * THREADS);
      const uint32_t r = ROWS_K ? c / (KC / 4) : c & (TILE - 1);
      const uint32_t k = ROWS_K ? 4 * (c % (KC / 4)) : 8 * (c / TILE);
      const uint32_t rc = (uint32_t)min((int)r, rows - 1 - r0);
      off[q] = ROWS_K ? rc * ld + k : rc + k * ld;
      dst[q] = tc::swz(r, k, KC * 16u);
    }
  }
  __device__ __forceinline__ void load(int kc, float (&v)[N]) const {
    const float* p = base + (int64_t)kc * KC * (ROWS_K ? 1 : (int64_t)ld);
#pragma unroll
    for (int q = 0; q < NP; ++q) {
      if (ROWS_K && VEC) {
        const float4 x = *reinterpret_cast<const float4*>(p + off[q]);
        v[4 * q] = x.x, v[4 * q + 1] = x.y, v[4 * q + 2] = x.z, v[4 * q + 3] = x.w;
      } else {
#pragma unroll
        for (int e = 0; e < PIECE; ++e)
          v[PIECE * q + e] = p[off[q] + (uint32_t)e * (ROWS_K ? 1u : ld)];
      }
    }
  }
  // the last chunk when K is not a multiple of KC: zeros past it
  __device__ __forceinline__ void load_tail(int kc, int kleft, int t, float (&v)[N]) const {
    const float* p = base + (int64_t)kc * KC * (ROWS_K ? 1 : (int64_t)ld);
#pragma unroll
    for (int q = 0; q < NP; ++q) {
      const int c = t + q * THREADS, k = ROWS_K ? 4 * (c % (KC / 4)) : 8 * (c / TILE);
#pragma unroll
      for (int e = 0; e < PIECE; ++e)
        v[PIECE * q + e] =
            k + e < kleft ? p[off[q] + (uint32_t)e * (ROWS_K ? 1u : ld)] : 0.f;
    }
  }
  __device__ __forceinline__ void store(uint32_t tile, const float (&v)[N]) const {
#pragma unroll
    for (int q = 0; q < NP; ++q) {
      const float* x = v + PIECE * q;
      if (ROWS_K)
        tc::st_shared_v2(tile + dst[q], tc::pack_bf16x2(x[0], x[1]), tc::pack_bf16x2(x[2], x[3]));
      else
        asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(tile + dst[q]),
                     "r"(tc::pack_bf16x2(x[0], x[1])), "r"(tc::pack_bf16x2(x[2], x[3])),
                     "r"(tc::pack_bf16x2(x[4], x[5])), "r"(tc::pack_bf16x2(x[6], x[7]))
                     : "memory");
    }
  }
};

// FWD: C = A B + bias[j] and G = gelu(C), A K-major (a_sk == 1); otherwise
// C = A B with A's rows contiguous (a_si == 1).  B's columns are contiguous
// (element (k, j) at B[k * N + j]).  VEC: A's rows are 16-byte aligned.
template <bool FWD, bool VEC, int TN, int KC>
__global__ void __launch_bounds__(TG_THREADS, 1) tc_gemm_kernel(
    const float* __restrict__ A, int64_t lda, const float* __restrict__ B, int M, int N, int K,
    const float* __restrict__ bias, float* __restrict__ C, float* __restrict__ G) {
  constexpr uint32_t A_BYTES = TG_M * KC * 2, B_BYTES = TN * KC * 2;   // per stage
  constexpr uint32_t SBO = KC * 16;   // bytes between 8-row groups of a staged tile
  constexpr uint32_t IDESC = tc::idesc_bf16(TG_M, TN, 0);
  // B's pieces (8 k of one column): the first TN * 8 threads have one each
  constexpr int B_THREADS = TN * (KC / 8);
  static_assert(B_THREADS <= TG_THREADS && TN % 32 == 0, "one piece of B per thread");
  using OpA = Operand<TG_M, KC, FWD, VEC, TG_THREADS>;
  using OpB = Operand<TN, KC, false, false, B_THREADS>;
  extern __shared__ uint8_t smem_raw[];
  __shared__ __align__(8) uint64_t bars[3];   // two stages, all MMAs done
  __shared__ uint32_t tmem_slot;
  __shared__ int abort_flag;
  const uint32_t sa = (tc::smem_u32(smem_raw) + 1023u) & ~1023u, sb = sa + 2 * A_BYTES;
  const uint32_t bar0 = tc::smem_u32(&bars[0]);
  const uint32_t abort_a = tc::smem_u32(&abort_flag);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int i0 = blockIdx.y * TG_M, j0 = blockIdx.x * TN;
  if (tid == 0) {
    tc::mbar_init(bar0, 1);
    tc::mbar_init(bar0 + 8, 1);
    tc::mbar_init(bar0 + 16, 1);
    abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     tc::smem_u32(&tmem_slot)),
                 "n"(TN)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  const int nk = (K + KC - 1) / KC;
  const int nfull = K / KC;   // chunks before the tail
  const bool has_b = tid < B_THREADS;
  OpA opa;
  OpB opb;
  opa.init(A, lda, M, i0, tid);
  opb.init(B, N, N, j0, has_b ? tid : 0);
  float va[OpA::N], vb[OpB::N];   // the next chunk's values
  auto load = [&](int kc) {
    opa.load(kc, va);
    if (has_b) opb.load(kc, vb);
  };
  if (nfull > 0) load(0);
  tc::tc_fence_before();
  __syncthreads();
  tc::tc_fence_after();
  const uint32_t tmem = tmem_slot;
  bool ok = true;
  auto chunk = [&](int kc) {   // ok = false: a wait gave up
    const int st = kc & 1;
    // the MMAs of chunk kc - 2 have read this stage
    if (kc >= 2 && !tc::mbar_wait_spin(bar0 + 8u * st, ((kc >> 1) - 1) & 1, abort_a)) ok = false;
    if (__syncthreads_or(!ok)) {
      ok = false;
      return;
    }
    opa.store(sa + st * A_BYTES, va);
    if (has_b) opb.store(sb + st * B_BYTES, vb);
    if (kc + 1 < nfull) load(kc + 1);
    tc::fence_proxy_async();
    __syncthreads();
    if (tid == 0) {
      tc::tc_fence_after();
#pragma unroll
      for (int kk = 0; kk < KC / 16; ++kk) {
        const uint32_t ko = (uint32_t)((kk >> 2) * 1024 + (kk & 3) * 32);
        tc::mma_bf16(tmem, tc::sdesc(sa + st * A_BYTES + ko, 0u, SBO),
                     tc::sdesc(sb + st * B_BYTES + ko, 0u, SBO), IDESC, (uint32_t)(kc | kk));
      }
      tc::mma_commit(bar0 + 8u * st);
    }
  };
  for (int kc = 0; kc < nfull && ok; ++kc) chunk(kc);
  if (ok && nfull < nk) {
    opa.load_tail(nfull, K - nfull * KC, tid, va);
    if (has_b) opb.load_tail(nfull, K - nfull * KC, tid, vb);
    chunk(nfull);
  }
  // the last chunk's commit covers every MMA issued before it
  if (ok && !tc::mbar_wait(bar0 + 8u * ((nk - 1) & 1), ((nk - 1) >> 1) & 1, abort_a)) ok = false;
  ok = !__syncthreads_or(!ok);
  tc::tc_fence_after();
  {   // warp w: lane quarter w % 4 (TMEM lane = output row), TN / 4 columns
    constexpr int EC = TN / 4;
    const int i = i0 + 32 * (warp & 3) + lane, jc = (warp >> 2) * EC;
    float v[EC];
    tc::tmem_ld_cols(tmem + ((uint32_t)(32 * (warp & 3)) << 16) + (uint32_t)jc, v);
    if (i < M) {
#pragma unroll
      for (int e = 0; e < EC; ++e) {
        const int j = j0 + jc + e;
        if (j < N) {
          float z = ok ? v[e] : __int_as_float(0x7fc00000);
          if (FWD) {
            z += bias[j];
            G[(int64_t)i * N + j] = gelu_f(z);
          }
          C[(int64_t)i * N + j] = z;
        }
      }
    }
  }
  // every MMA this CTA issued has completed before its TMEM is released
  // (after a timeout as well: bounded)
  if (tid == 0) {
    tc::mma_commit(bar0 + 16);
    const long long t0 = clock64();
    while (!tc::mbar_try(bar0 + 16, 0))
      if (clock64() - t0 > tc::kWaitCycles) {
        ok = false;
        break;
      }
    if (!ok) atomicOr(&g_mlp_abort, 1);
  }
  tc::tc_fence_before();
  __syncthreads();
  tc::tc_fence_after();
  if (warp == 0)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "n"(TN)
                 : "memory");
}

template <bool FWD, int TN, int KC>
cudaError_t launch_tc_gemm(const float* A, int64_t lda, const float* B, int M, int N, int K,
                           const float* bias, float* C, float* G, cudaStream_t st) {
  const size_t sm = 1024 + 4 * (size_t)(TG_M + TN) * KC;
  const dim3 grid((unsigned)((N + TN - 1) / TN), (unsigned)((M + TG_M - 1) / TG_M));
  auto go = [&](auto kern) {
    const cudaError_t e = cudaFuncSetAttribute(
        kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
    if (e != cudaSuccess) return e;
    kern<<<grid, TG_THREADS, sm, st>>>(A, lda, B, M, N, K, bias, C, G);
    return cudaGetLastError();
  };
  if (FWD && ((uintptr_t)A & 15u) == 0 && (lda & 3) == 0) return go(tc_gemm_kernel<FWD, FWD, TN, KC>);
  return go(tc_gemm_kernel<FWD, false, TN, KC>);
}

// s[j] = sum_h G[j, h] w2[h] + b2: one warp per row, lanes stride h, then a
// fixed shuffle tree.
__global__ void score_kernel(const float* __restrict__ G, int64_t n, int H,
                             const float* __restrict__ w2, const float* __restrict__ b2,
                             float* __restrict__ s) {
  const int64_t j = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int lane = threadIdx.x & 31;
  if (j >= n) return;
  float a = 0.f;
  for (int h = lane; h < H; h += 32) a = fmaf(G[j * H + h], w2[h], a);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) a += __shfl_xor_sync(0xffffffffu, a, o);
  if (lane == 0) s[j] = a + b2[0];
}

// The backward pass up to dZ, and the gradients that are column sums, in one
// read of Z and G:
//   ds[j] = d/ds_j of mean_j [ w y softplus(-s) + (1 - y) softplus(s) ]
//   dZ = ds w2^T .* gelu'(Z),  gw2 = G^T ds,  gb1 = sum_j dZ,  gb2 = sum ds
// A cluster of 8 CTAs owns 32 columns h (one per lane); its 64 warps take rows
// w, w + 64, ... in order; each CTA adds its warps' sums in order and CTA 0 of
// the cluster the CTAs' in order, through distributed shared memory.  The
// cluster of the first columns also writes ds and gb2.  What bounds it is the
// instructions of gelu' and the sigmoid (about 150 per entry): 64 CTAs for
// H = 256.  (Before: one thread per column over all rows, 110 us for 512 x
// 256, beside two element-wise launches of 3 us.)
constexpr int BW_CTAS = 8, BW_WARPS = 8;
__global__ void __cluster_dims__(1, BW_CTAS, 1) __launch_bounds__(BW_WARPS * 32)
    backward_kernel(const float* __restrict__ s, const float* __restrict__ y, int64_t n,
                    float pos_weight, const float* __restrict__ Z, const float* __restrict__ G,
                    const float* __restrict__ w2, int H, float* __restrict__ ds,
                    float* __restrict__ dZ, float* __restrict__ gw2, float* __restrict__ gb1,
                    float* __restrict__ gb2) {
  cg::cluster_group cl = cg::this_cluster();
  __shared__ float red[3][BW_WARPS][32];
  __shared__ float cta[3][32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int h = blockIdx.x * 32 + lane;
  const bool in = h < H;
  const float wh = in ? w2[h] : 0.f;
  float a2 = 0.f, a1 = 0.f, ab = 0.f;
#pragma unroll 4
  for (int64_t j = blockIdx.y * BW_WARPS + warp; j < n; j += BW_CTAS * BW_WARPS) {
    const float v = s[j], yj = y[j];
    const float z = in ? Z[j * H + h] : 0.f, gv = in ? G[j * H + h] : 0.f;
    const float sg = v >= 0.f ? 1.f / (1.f + expf(-v)) : expf(v) / (1.f + expf(v));
    const float d = (-pos_weight * yj * (1.f - sg) + (1.f - yj) * sg) / (float)n;
    const float dz = d * wh * gelu_grad_f(z);
    if (in) dZ[j * H + h] = dz;
    if (blockIdx.x == 0 && lane == 0) ds[j] = d;
    a2 = fmaf(gv, d, a2);
    a1 += dz;
    ab += d;
  }
  red[0][warp][lane] = a2;
  red[1][warp][lane] = a1;
  red[2][warp][lane] = ab;
  __syncthreads();
  if (warp < 3) {
    float a = 0.f;
    for (int w = 0; w < BW_WARPS; ++w) a += red[warp][w][lane];
    cta[warp][lane] = a;
  }
  cl.sync();
  if (blockIdx.y == 0 && warp < 3) {
    float a = 0.f;
    for (int c = 0; c < BW_CTAS; ++c) a += *cl.map_shared_rank(&cta[warp][lane], c);
    if (warp < 2 && in) (warp ? gb1 : gw2)[h] = a;
    if (warp == 2 && blockIdx.x == 0 && lane == 0) gb2[0] = a;
  }
  cl.sync();   // no CTA leaves while another still reads its sums
}

__global__ void sgd_kernel(float* __restrict__ p, const float* __restrict__ g, int64_t count,
                           float lr) {
  const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (e < count) p[e] -= lr * g[e];
}

// The count columns of highest score, ties to the lower index, written in
// increasing column order (the learned proposal's candidates).  One CTA:
// column j is taken when fewer than count columns rank above it (score
// greater, or equal with a lower index); its output slot is the number of
// taken columns before it.  A NaN score ranks below every number.
constexpr int PR_THREADS = 1024, PR_MAX = 4096;

__device__ __forceinline__ int score_key(float v) {
  if (v != v) return INT_MIN;   // NaN lowest
  if (v == 0.f) return 0;       // -0 ties with +0
  const int b = __float_as_int(v);
  return b >= 0 ? b : (int)(0x80000000u - (unsigned)b) - 1;   // monotone in v
}

// strata > 1: the columns form `strata` consecutive ranges [q n / strata,
// (q + 1) n / strata) and column j competes only within its range for `count`
// places (the stratified proposal); strata = 1: one range.
__global__ void __launch_bounds__(PR_THREADS) propose_kernel(const float* __restrict__ s, int n,
                                                              int count, int strata,
                                                              int* __restrict__ cand,
                                                              int* __restrict__ ncand) {
  __shared__ int key[PR_MAX];
  __shared__ unsigned char take[PR_MAX];
  __shared__ int wsum[PR_THREADS / 32];
  for (int j = threadIdx.x; j < n; j += PR_THREADS) key[j] = score_key(s[j]);
  __syncthreads();
  for (int j = threadIdx.x; j < n; j += PR_THREADS) {
    const int kj = key[j];
    // the range holding j: the largest q with q n / strata <= j
    int q = (int)(((int64_t)j * strata) / n);
    while (q + 1 < strata && ((int64_t)(q + 1) * n) / strata <= j) ++q;
    while (q > 0 && ((int64_t)q * n) / strata > j) --q;
    const int lo = (int)(((int64_t)q * n) / strata), hi = (int)(((int64_t)(q + 1) * n) / strata);
    int above = 0;
    for (int i = lo; i < hi; ++i) above += (key[i] > kj) || (key[i] == kj && i < j);
    take[j] = above < count;
  }
  __syncthreads();
  // exclusive prefix count of take[] over j, in chunks of PR_THREADS
  int base = 0;
  for (int c0 = 0; c0 < n; c0 += PR_THREADS) {
    const int j = c0 + threadIdx.x;
    const int t = j < n ? take[j] : 0;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int incl = t;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int y = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += y;
    }
    if (lane == 31) wsum[warp] = incl;
    __syncthreads();
    int before = 0;
    for (int w = 0; w < warp; ++w) before += wsum[w];
    if (t) cand[base + before + incl - 1] = j;
    __syncthreads();
    int tot = 0;
    for (int w = 0; w < PR_THREADS / 32; ++w) tot += wsum[w];
    base += tot;
    __syncthreads();
  }
  if (threadIdx.x == 0 && ncand) *ncand = base;
}

id_status cuda_status(cudaError_t e) {
  if (e == cudaSuccess) return ID_OK;
  g_last_cuda_error.store((int)e);
  return ID_ERR_CUDA;
}

int blocks_for(int64_t count, int threads) { return (int)((count + threads - 1) / threads); }

bool gemm_dims_ok(int64_t M, int64_t N, int64_t K) {
  return M >= 1 && N >= 1 && K >= 1 && M <= (1 << 24) && N <= (1 << 24) && K <= (1 << 24) &&
         (M + TG_M - 1) / TG_M <= 65535;
}

// The element-wise kernels take one thread per entry of an n x H (or n x 32)
// array: their grid (blocks of 256) must stay below 2^31 blocks.
bool elementwise_grid_ok(int64_t n, int64_t H) {
  return n * std::max<int64_t>(H, 32) / 256 + 1 < ((int64_t)1 << 31);
}

}  // namespace

extern "C" {

id_status id_mlp_features(const void* d_A, int64_t lda, int64_t m, int64_t n, int32_t dtype,
                          const int64_t* d_rows, int64_t F, float scale, float* d_X,
                          void* cuda_stream) {
  if (!d_A || !d_rows || !d_X || m < 1 || n < 1 || F < 1 || lda < m ||
      (dtype != ID_F32 && dtype != ID_F64) || n * F > ((int64_t)1 << 40))
    return ID_ERR_INVALID_ARG;
  const cudaStream_t st = (cudaStream_t)cuda_stream;
  const int64_t tot = n * F;
  if (tot / 256 + 1 > ((int64_t)1 << 31) - 1) return ID_ERR_INVALID_ARG;
  if (dtype == ID_F64)
    features_kernel<double><<<blocks_for(tot, 256), 256, 0, st>>>(
        reinterpret_cast<const double*>(d_A), lda, m, n, d_rows, F, scale, d_X);
  else
    features_kernel<float><<<blocks_for(tot, 256), 256, 0, st>>>(
        reinterpret_cast<const float*>(d_A), lda, m, n, d_rows, F, scale, d_X);
  count_launches(1);
  return cuda_status(cudaGetLastError());
}

id_status id_mlp_forward(const float* d_X, int64_t n, int64_t F, int32_t H, const float* d_W1,
                         const float* d_b1, const float* d_w2, const float* d_b2, float* d_Z,
                         float* d_G, float* d_s, void* cuda_stream) {
  if (!d_X || !d_W1 || !d_b1 || !d_w2 || !d_b2 || !d_Z || !d_G || !d_s || H < 1 ||
      !gemm_dims_ok(n, H, F) || !elementwise_grid_ok(n, H))
    return ID_ERR_INVALID_ARG;
  const cudaStream_t st = (cudaStream_t)cuda_stream;
  // Z = X W1: A = X (n x F, row-major), B = W1 (F x H, row-major)
  cudaError_t e = launch_tc_gemm<true, 32, 128>(d_X, F, d_W1, (int)n, H, (int)F, d_b1, d_Z, d_G, st);
  if (e != cudaSuccess) return cuda_status(e);
  score_kernel<<<blocks_for(n * 32, 256), 256, 0, st>>>(d_G, n, H, d_w2, d_b2, d_s);
  count_launches(2);
  return cuda_status(cudaGetLastError());
}

id_status id_mlp_backward(const float* d_X, int64_t n, int64_t F, int32_t H, const float* d_Z,
                          const float* d_G, const float* d_w2, const float* d_s,
                          const float* d_y, float pos_weight, float* d_gW1, float* d_gb1,
                          float* d_gw2, float* d_gb2, float* d_ds, float* d_dZ,
                          void* cuda_stream) {
  if (!d_X || !d_Z || !d_G || !d_w2 || !d_s || !d_y || !d_gW1 || !d_gb1 || !d_gw2 || !d_gb2 ||
      !d_ds || !d_dZ || H < 1 || !gemm_dims_ok(F, H, n) || !elementwise_grid_ok(n, H) ||
      !(pos_weight >= 0.f))
    return ID_ERR_INVALID_ARG;
  const cudaStream_t st = (cudaStream_t)cuda_stream;
  backward_kernel<<<dim3(blocks_for(H, 32), BW_CTAS), BW_WARPS * 32, 0, st>>>(
      d_s, d_y, n, pos_weight, d_Z, d_G, d_w2, H, d_ds, d_dZ, d_gw2, d_gb1, d_gb2);
  // gW1 = X^T dZ: A = X^T (element (f, j) at X[j F + f]), B = dZ (n x H)
  const cudaError_t e =
      launch_tc_gemm<false, 64, 64>(d_X, F, d_dZ, (int)F, H, (int)n, nullptr, d_gW1, nullptr, st);
  if (e != cudaSuccess) return cuda_status(e);
  count_launches(2);
  return cuda_status(cudaGetLastError());
}

id_status id_mlp_propose(const float* d_s, int64_t n, int32_t count, int32_t* d_cand,
                         void* cuda_stream) {
  if (!d_s || !d_cand || n < 1 || n > PR_MAX || count < 1 || count > n)
    return ID_ERR_INVALID_ARG;
  propose_kernel<<<1, PR_THREADS, 0, (cudaStream_t)cuda_stream>>>(d_s, (int)n, count, 1, d_cand,
                                                                   nullptr);
  count_launches(1);
  return cuda_status(cudaGetLastError());
}

id_status id_mlp_propose_stratified(const float* d_s, int64_t n, int32_t strata, int32_t per,
                                    int32_t* d_cand, int32_t* d_ncand, void* cuda_stream) {
  if (!d_s || !d_cand || n < 1 || n > PR_MAX || strata < 1 || strata > n || per < 1)
    return ID_ERR_INVALID_ARG;
  propose_kernel<<<1, PR_THREADS, 0, (cudaStream_t)cuda_stream>>>(d_s, (int)n, per, strata,
                                                                   d_cand, d_ncand);
  count_launches(1);
  return cuda_status(cudaGetLastError());
}

id_status id_mlp_check(void* cuda_stream) {
  if (cudaStreamSynchronize((cudaStream_t)cuda_stream) != cudaSuccess)
    return cuda_status(cudaGetLastError());
  int flag = 0;
  const int zero = 0;
  if (cudaMemcpyFromSymbol(&flag, g_mlp_abort, sizeof(int)) != cudaSuccess ||
      (flag && cudaMemcpyToSymbol(g_mlp_abort, &zero, sizeof(int)) != cudaSuccess))
    return cuda_status(cudaGetLastError());
  return flag ? ID_ERR_TIMEOUT : ID_OK;
}

id_status id_mlp_sgd(float* d_p, const float* d_g, int64_t count, float lr, void* cuda_stream) {
  if (!d_p || !d_g || count < 1 || !isfinite(lr)) return ID_ERR_INVALID_ARG;
  if (count / 256 + 1 > ((int64_t)1 << 31) - 1) return ID_ERR_INVALID_ARG;
  sgd_kernel<<<blocks_for(count, 256), 256, 0, (cudaStream_t)cuda_stream>>>(d_p, d_g, count, lr);
  count_launches(1);
  return cuda_status(cudaGetLastError());
}

}  // extern "C"
