// SIMT kernels of the sampler: the small FP64 GEMMs with fused epilogues (the
// large ones run on the tensor cores, k_gemm64.cu), the full-KLE prior draw,
// and small elementwise helpers.
//
// GEMM convention: out = epilogue(A B^T) with A: M x K (row pitch lda) and
// B: N x K (row pitch ldb), i.e. both operands K-contiguous.
#include <algorithm>

#include "dino_internal.h"
#include "epi64.cuh"
#include "pdl.cuh"
#include "philox.cuh"

namespace dino {
namespace {

// SIMT GEMM for the products too small for the tensor cores' digits (and for
// operands without digits).  A CTA of 256 threads computes a T x T tile, kKG
// threads per output: thread q takes the columns q, q + kKG, ... in two
// alternating sums, joined by a butterfly, so that a long reduction over few
// outputs still spreads over many CTAs.  The FP64 pipe takes one warp
// instruction in 16 cycles, so operands read straight from L1 keep up with
// it; what counts is to have every SM's pipe busy.  kKG depends on K alone:
// an output's value does not depend on how many rows the product has.
// (64 x 64 tiles staged in shared memory, the layout before: 1200 us for 64 x
// 16 outputs over K = 1089 on one CTA, 117 us for 64 x 64 x 64 with a tanh;
// now 18 and 9 us.)
constexpr int kGemmThreads = 256;

template <typename T, int kT, int kKG, class Epi>
__global__ void __launch_bounds__(kGemmThreads)
    k_gemm(int M, int N, int K, const T *A, int lda, const T *B, int ldb, Epi epi) {
  static_assert(kT * kT * kKG == kGemmThreads, "one output per kKG threads");
  pdl_begin();
  A = pdl_after(A);
  B = pdl_after(B);
  __shared__ T out[kT * kT];
  const int o = threadIdx.x / kKG, q = threadIdx.x % kKG;
  const int mt = (M + kT - 1) / kT;  // tiles by columns; one dimension, the others end at 65535
  const int row0 = (int)(blockIdx.x % mt) * kT, col0 = (int)(blockIdx.x / mt) * kT;
  const T *a = A + (size_t)min(row0 + o / kT, M - 1) * lda;
  const T *b = B + (size_t)min(col0 + o % kT, N - 1) * ldb;
  T s0 = T(0), s1 = T(0);
  int k = q;
#pragma unroll 4
  for (; k + kKG < K; k += 2 * kKG) {
    s0 += __ldg(a + k) * __ldg(b + k);
    s1 += __ldg(a + k + kKG) * __ldg(b + k + kKG);
  }
  if (k < K) s0 += __ldg(a + k) * __ldg(b + k);
  s0 += s1;
#pragma unroll
  for (int w = kKG / 2; w; w >>= 1) s0 += __shfl_xor_sync(0xffffffffu, s0, w);
  if (q == 0) out[o] = s0;
  __syncthreads();
  if (threadIdx.x < kT * kT) {
    const int r = row0 + threadIdx.x / kT, c = col0 + threadIdx.x % kT;
    if (r < M && c < N) epi(r, c, out[threadIdx.x]);
  }
}

template <typename T, class Epi>
cudaError_t run_gemm(int M, int N, int K, const T *A, int lda, const T *B, int ldb, Epi epi,
                     cudaStream_t st) {
  if (M <= 0 || N <= 0) return cudaSuccess;
  if (K > 256) {  // long reductions: 16 threads per output, 4 x 4 tiles
    const long grid = (long)((M + 3) / 4) * ((N + 3) / 4);
    if (grid > 0x7fffffffL) return cudaErrorInvalidValue;
    return launch_pdl(k_gemm<T, 4, 16, Epi>, dim3((unsigned)grid), kGemmThreads, 0, st, M, N, K,
                      A, lda, B, ldb, epi);
  } else {
    const long grid = (long)((M + 7) / 8) * ((N + 7) / 8);
    if (grid > 0x7fffffffL) return cudaErrorInvalidValue;
    return launch_pdl(k_gemm<T, 8, 4, Epi>, dim3((unsigned)grid), kGemmThreads, 0, st, M, N, K, A,
                      lda, B, ldb, epi);
  }
}

// Prior draw: one CTA per chain; X = sqrt(Lambda) .* Z (spectral), Y = X S,
// M = S^T Y, all n x n in shared memory with rows padded to a multiple of 4
// (zero-filled).  The sine matrix is symmetric in its nodes, S[k][n - 1 - i] =
// (-1)^k S[k][i] (k from 0), so of each product only the first h = ceil(n / 2)
// node rows or columns are formed, the even k into U and the odd k into V:
// the node is U + V and its mirror image U - V, half the multiply-adds.  U
// and V of a 4 x 4 tile are the work of two threads (one half of the CTA
// each), V handed over through the destination; per step of the reduction a
// tile reads one float4 (or double4-as-two-loads) row segment of the right
// operand and one of the left.  FP64 is bound by its pipe (16 cycles a warp
// instruction), FP32 by shared-memory reads and the transforms' latency.
// kPriorThreads threads hold the tiles of n = 65 in one round.  (All n x n
// nodes formed, n = 65: 0.84 ms for 16384 chains in FP32, 1.53 ms for 1024 in
// FP64; 0.70 and 0.93 ms now.)
constexpr int kPriorThreads = 320;

__host__ __device__ inline int prior_ld(int n) { return (n + 3) / 4 * 4; }

// Four consecutive values of a padded shared-memory row (16-byte aligned: the
// rows are multiples of 4 values and the arrays start on 16 bytes).
template <typename T>
__device__ __forceinline__ void load4(const T *p, T v[4]) {
  if constexpr (sizeof(T) == 4) {
    const float4 x = *reinterpret_cast<const float4 *>(p);
    v[0] = x.x;
    v[1] = x.y;
    v[2] = x.z;
    v[3] = x.w;
  } else {
    const double2 x = reinterpret_cast<const double2 *>(p)[0];
    const double2 y = reinterpret_cast<const double2 *>(p)[1];
    v[0] = x.x;
    v[1] = x.y;
    v[2] = y.x;
    v[3] = y.y;
  }
}

// A 4 x 4 tile of sum_k a[k][0..3] b[k][0..3] over k = k0, k0 + 2, ... < n (rows
// of pitch ld)
template <typename T>
__device__ __forceinline__ void half_tile(const T *a, const T *b, int ld, int k0, int n,
                                          T acc[4][4]) {
#pragma unroll
  for (int p = 0; p < 4; ++p)
#pragma unroll
    for (int q = 0; q < 4; ++q) acc[p][q] = T(0);
#pragma unroll 3
  for (int k = k0; k < n; k += 2) {
    T x[4], y[4];
    load4(a + k * ld, x);
    load4(b + k * ld, y);
#pragma unroll
    for (int p = 0; p < 4; ++p)
#pragma unroll
      for (int q = 0; q < 4; ++q) acc[p][q] += x[p] * y[q];
  }
}

template <typename T>
__global__ void __launch_bounds__(kPriorThreads, sizeof(T) == 4 ? 4 : 2)
    k_prior_draw(int n, const T *__restrict__ sqrtlam, const T *__restrict__ S, uint64_t seed,
                 uint64_t id_base, uint32_t stream, uint32_t step, T *out, int ldo,
                 __nv_bfloat16 *ms, int ldms, size_t ms_plane, int ms_slices,
                 const double *__restrict__ ext_z, const int *only) {
  if (only) {  // flags of the kernel before this one: read behind the wait
    pdl_wait();
    if (!pdl_after(only)[blockIdx.x]) return;  // the whole CTA: this chain draws nothing
  }
  extern __shared__ __align__(16) unsigned char smraw[];
  const int ld = prior_ld(n), nt = ld / 4, NN = ld * ld;
  const int h = (n + 1) / 2, ht = (h + 3) / 4;  // nodes formed, and their tiles
  T *X = reinterpret_cast<T *>(smraw);
  T *Ss = X + NN;
  T *Y = Ss + NN;
  const int c = blockIdx.x, N = n * n;
  const uint32_t chain = (uint32_t)(id_base + (uint64_t)c);
  // q / d for 0 <= q < d^2 + 4d, d <= 256, from the FP32 reciprocal: (q + 1/2) / d
  // stays at least 1/(2d) away from an integer, far beyond the rounding error
  // (rounded operations, no contraction)
  const float inv_ld = 1.0f / (float)ld, inv_n = 1.0f / (float)n;
  auto quot = [](int q, float inv) {
    return (int)__fmul_rn(__fadd_rn((float)q, 0.5f), inv);
  };
  for (int e = threadIdx.x; e < NN; e += blockDim.x) {
    const int row = quot(e, inv_ld), col = e - row * ld;
    const bool in = row < n && col < n;
    X[e] = T(0);
    Ss[e] = in ? S[row * n + col] : T(0);
  }
  __syncthreads();
  for (int blk = threadIdx.x; blk < (N + 3) / 4; blk += blockDim.x) {
    T z[4];
    if (ext_z) {
      for (int q = 0; q < 4; ++q)
        z[q] = 4 * blk + q < N ? (T)ext_z[(size_t)c * N + 4 * blk + q] : T(0);
    } else {
      const uint4 w = philox_block(seed, stream, step, chain, blk);
      if constexpr (sizeof(T) == 8) {
        normals4_f64(w, z);
      } else {
        normals4_f32(w, z);
      }
    }
    for (int q = 0; q < 4; ++q) {
      const int m = 4 * blk + q;
      if (m < N) {
        const int j = quot(m, inv_n);
        X[(m - j * n) * ld + j] = sqrtlam[m] * z[q];  // stored transposed
      }
    }
  }
  __syncthreads();
  const int team = blockDim.x / 2, odd = threadIdx.x >= team ? 1 : 0,
            mate = threadIdx.x - odd * team;
  // Y[ky][i] = sum_kx X[ky][kx] S[kx][i], with X held transposed (X[kx][ky]
  // at kx * ld + ky) so that both operands are read as row segments
  for (int t0 = 0; t0 < nt * ht; t0 += team) {  // the same passes in every thread
    const int tt = t0 + mate, r0 = 4 * (tt / ht), c0 = 4 * (tt % ht);
    const bool on = tt < nt * ht;
    T acc[4][4];
    if (on) {
      half_tile(X + r0, Ss + c0, ld, odd, n, acc);
      if (odd)
#pragma unroll
        for (int p = 0; p < 4; ++p)
#pragma unroll
          for (int q = 0; q < 4; ++q)
            if (c0 + q < h) Y[(r0 + p) * ld + c0 + q] = acc[p][q];
    }
    __syncthreads();
    if (on && !odd) {
#pragma unroll
      for (int p = 0; p < 4; ++p)
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const int i = c0 + q;
          if (i < h) {
            T *row = Y + (r0 + p) * ld;
            const T v = row[i];
            row[i] = acc[p][q] + v;
            if (n - 1 - i != i) row[n - 1 - i] = acc[p][q] - v;
          }
        }
    }
  }
  __syncthreads();
  // M[j][i] = sum_ky S[ky][j] Y[ky][i]; node p = i + n j.  The tiles land in
  // shared memory (X's array, which the first product no longer reads: n^2
  // nodes in order), and the CTA then writes M and its slices with
  // consecutive threads on consecutive nodes.
  T *Mo = X;
  for (int t0 = 0; t0 < ht * nt; t0 += team) {
    const int tt = t0 + mate, r0 = 4 * (tt / nt), c0 = 4 * (tt % nt);
    const bool on = tt < ht * nt;
    T acc[4][4];
    if (on) {
      half_tile(Ss + r0, Y + c0, ld, odd, n, acc);
      if (odd)
#pragma unroll
        for (int p = 0; p < 4; ++p)
#pragma unroll
          for (int q = 0; q < 4; ++q)
            if (r0 + p < h && c0 + q < n) Mo[(r0 + p) * n + c0 + q] = acc[p][q];
    }
    __syncthreads();
    if (on && !odd) {
#pragma unroll
      for (int p = 0; p < 4; ++p)
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const int j = r0 + p, i = c0 + q;
          if (j < h && i < n) {
            const T v = Mo[j * n + i];
            Mo[j * n + i] = acc[p][q] + v;
            if (n - 1 - j != j) Mo[(n - 1 - j) * n + i] = acc[p][q] - v;
          }
        }
    }
  }
  __syncthreads();
  pdl_begin();  // the draw needs nothing of the kernels before; its outputs may be in use
  T *o = out + (size_t)c * ldo;
  for (int e = threadIdx.x; e < N; e += blockDim.x) {
    const T v = Mo[e];
    o[e] = v;
    if constexpr (sizeof(T) == 4) {
      if (ms) {
        __nv_bfloat16 *d = ms + (size_t)c * ldms + e;
        float rem = v;
        for (int sl = 0; sl < ms_slices; ++sl) {
          const __nv_bfloat16 hb = __float2bfloat16_rn(rem);
          d[sl * ms_plane] = hb;
          // exact widening: the bf16 bits in the upper half of an FP32 word
          rem -= __uint_as_float((uint32_t)__bfloat16_as_ushort(hb) << 16);
        }
      }
    }
  }
}

template <typename T>
__global__ void k_jac_init(int C, int d_y, int w, const T *__restrict__ WL, const T *der, int ldd,
                           T *__restrict__ P) {
  pdl_begin();
  der = pdl_after(der);
  const size_t total = (size_t)C * d_y * w;
  for (size_t e = blockIdx.x * (size_t)blockDim.x + threadIdx.x; e < total;
       e += (size_t)gridDim.x * blockDim.x) {
    const size_t row = e / w;
    const int k = (int)(e % w);
    const size_t c = row / d_y;
    const int i = (int)(row % d_y);
    P[e] = WL[(size_t)i * w + k] * __ldg(der + c * ldd + k);
  }
}

template <typename T>
__global__ void k_broadcast(int C, size_t n, const T *__restrict__ src, T *__restrict__ out) {
  const size_t total = (size_t)C * n;
  for (size_t e = blockIdx.x * (size_t)blockDim.x + threadIdx.x; e < total;
       e += (size_t)gridDim.x * blockDim.x)
    out[e] = src[e % n];
}

template <typename S, typename D>
__global__ void k_convert(size_t n, const S *__restrict__ src, D *__restrict__ dst) {
  for (size_t e = blockIdx.x * (size_t)blockDim.x + threadIdx.x; e < n;
       e += (size_t)gridDim.x * blockDim.x)
    dst[e] = (D)src[e];
}

inline int grid_for(size_t n) {
  size_t g = (n + 255) / 256;
  return (int)(g > 152 * 32 ? 152 * 32 : (g ? g : 1));
}

}  // namespace

template <typename T>
cudaError_t gemm_store(int M, int N, int K, const T *A, int lda, const T *B, int ldb, T *out,
                       int ldo, cudaStream_t st) {
  return run_gemm(M, N, K, A, lda, B, ldb, EpiStore<T>{out, ldo}, st);
}

template <typename T>
cudaError_t gemm_bias_act(int M, int N, int K, const T *A, int lda, const T *B, int ldb,
                          const T *bias, int act, T *out, T *der, int ldo, cudaStream_t st) {
  return run_gemm(M, N, K, A, lda, B, ldb, EpiBiasAct<T>{bias, act, out, der, ldo}, st);
}

template <typename T>
cudaError_t gemm_scale_group(int M, int N, int K, const T *A, int lda, const T *B, int ldb,
                             const T *scale, int lds, int group, T *out, int ldo,
                             cudaStream_t st) {
  return run_gemm(M, N, K, A, lda, B, ldb, EpiScaleGroup<T>{scale, lds, group, out, ldo}, st);
}

template <typename T>
cudaError_t gemm_coef(int M, int N, int K, const T *A, int lda, const T *B, int ldb,
                      const double *coef, int ldc, double c, T *out, int ldo, cudaStream_t st) {
  return run_gemm(M, N, K, A, lda, B, ldb, EpiCoef<T>{coef, ldc, c, out, ldo}, st);
}

template <typename T>
cudaError_t gemm_field(int M, int N, int K, const T *A, int lda, const T *B, int ldb,
                       const int *acc_flag, double s, double c, T *m, const T *Mf, int ldm,
                       cudaStream_t st) {
  return run_gemm(M, N, K, A, lda, B, ldb, EpiField<T>{acc_flag, s, c, m, Mf, ldm}, st);
}

cudaError_t launch_ns_poly(int d, const double *Y, double *P, unsigned long long *res,
                           cudaStream_t st) {
  return run_gemm(d, d, d, Y, d, Y, d, EpiPoly{P, d, res}, st);
}

cudaError_t launch_ns_update(int d, const double *P, const double *X, double *Y, double *X2,
                             cudaStream_t st) {
  return run_gemm(d, d, d, P, d, X, d, EpiBoth{Y, X2, d}, st);
}

// Tiles of 32 x 32 through shared memory (rows padded by one), so that reads
// and writes are both along rows: HBM-bound (4096 blocks of 128 x 200 FP32, 839
// MB: 361 us with strided reads, 168 us).
template <typename T>
__global__ void __launch_bounds__(256)
    k_batched_transpose(int a, int b, const T *src, T *__restrict__ dst) {
  pdl_begin();
  src = pdl_after(src);
  __shared__ T tile[32][33];
  const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
  const int nb = (b + 31) / 32;
  const int i0 = (blockIdx.x / nb) * 32, j0 = (blockIdx.x % nb) * 32;  // rows of a, columns of b
  const size_t off = (size_t)blockIdx.y * a * b;
#pragma unroll
  for (int k = 0; k < 32; k += 8)
    if (i0 + ty + k < a && j0 + tx < b)
      tile[ty + k][tx] = __ldg(src + off + (size_t)(i0 + ty + k) * b + j0 + tx);
  __syncthreads();
#pragma unroll
  for (int k = 0; k < 32; k += 8)
    if (j0 + ty + k < b && i0 + tx < a)
      dst[off + (size_t)(j0 + ty + k) * a + i0 + tx] = tile[tx][ty + k];
}

cudaError_t launch_batched_transpose(int C, int a, int b, const void *src, int f32, void *dst,
                                     cudaStream_t st) {
  if (C <= 0 || a <= 0 || b <= 0) return cudaSuccess;
  const size_t blk = (size_t)a * b;
  for (int c0 = 0; c0 < C; c0 += 65535) {  // the grid's second dimension ends there
    const dim3 grid(((a + 31) / 32) * ((b + 31) / 32), std::min(65535, C - c0));
    const cudaError_t e =
        f32 ? launch_pdl(k_batched_transpose<float>, grid, 256, 0, st, a, b,
                         (const float *)src + c0 * blk, (float *)dst + c0 * blk)
            : launch_pdl(k_batched_transpose<double>, grid, 256, 0, st, a, b,
                         (const double *)src + c0 * blk, (double *)dst + c0 * blk);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

// Eight independent FMA chains per thread: with 8 warps per scheduler the
// chains' latency is hidden and the FP32 pipe runs at its issue rate.
constexpr int kFmaIters = 8192;
__global__ void __launch_bounds__(256) k_fma_peak(float seed, float *out) {
  float a[8];
#pragma unroll
  for (int q = 0; q < 8; ++q) a[q] = seed * (float)(threadIdx.x + q);
  const float b = 0.999999f, c = 1e-7f;
#pragma unroll 4
  for (int it = 0; it < kFmaIters; ++it)
#pragma unroll
    for (int q = 0; q < 8; ++q) a[q] = fmaf(a[q], b, c);
  float s = 0.0f;
#pragma unroll
  for (int q = 0; q < 8; ++q) s += a[q];
  if (s == 12345.678f) out[0] = s;  // keeps the chains alive
}

cudaError_t measure_fma_peak(cudaStream_t st, float *ms, double *flops) {
  int dev = 0, sms = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (e != cudaSuccess) return e;
  const int blocks = sms * 8;  // 2048 threads per SM
  cudaEvent_t e0, e1;
  if ((e = cudaEventCreate(&e0)) != cudaSuccess) return e;
  if ((e = cudaEventCreate(&e1)) != cudaSuccess) {
    cudaEventDestroy(e0);
    return e;
  }
  float best = 0.0f;
  for (int rep = 0; rep < 4 && e == cudaSuccess; ++rep) {
    cudaEventRecord(e0, st);
    k_fma_peak<<<blocks, 256, 0, st>>>(1e-3f, nullptr);
    cudaEventRecord(e1, st);
    e = cudaEventSynchronize(e1);
    if (e == cudaSuccess) e = cudaGetLastError();
    float t = 0.0f;
    if (e == cudaSuccess) cudaEventElapsedTime(&t, e0, e1);
    if (rep > 0 && (best == 0.0f || t < best)) best = t;  // the first launch warms up
  }
  cudaEventDestroy(e0);
  cudaEventDestroy(e1);
  *ms = best;
  *flops = 2.0 * 8.0 * kFmaIters * (double)blocks * 256.0;
  return e;
}

size_t prior_draw_smem_bytes(int n, int elem) {
  return 3 * (size_t)prior_ld(n) * prior_ld(n) * elem;
}

template <typename T>
cudaError_t launch_prior_draw(int C, int n, const T *sqrtlam, const T *S, uint64_t seed,
                              uint64_t id_base, uint32_t stream, uint32_t step, T *out, int ldo,
                              cudaStream_t st, __nv_bfloat16 *ms, int ldms, size_t ms_plane,
                              int ms_slices, const double *ext_z, const int *only,
                              bool overlap) {
  if (C <= 0) return cudaSuccess;
  if (ms && (sizeof(T) != 4 || ms_slices < 1 || ldms < n * n)) return cudaErrorInvalidValue;
  const size_t smem = prior_draw_smem_bytes(n, (int)sizeof(T));
  cudaError_t e = cudaFuncSetAttribute(k_prior_draw<T>,
                                       cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  // beside the geometry kernel: 64 chains, n = 65, 19 us of 317 hidden
  if (overlap)
    return launch_pdl_n(chain_ctas(C), k_prior_draw<T>, C, kPriorThreads, smem, st, n, sqrtlam, S,
                        seed, id_base, stream, step, out, ldo, ms, ldms, ms_plane, ms_slices, ext_z,
                        only);
  k_prior_draw<T><<<C, kPriorThreads, smem, st>>>(n, sqrtlam, S, seed, id_base, stream, step, out,
                                                  ldo, ms, ldms, ms_plane, ms_slices, ext_z, only);
  return cudaGetLastError();
}

template <typename T>
cudaError_t launch_jac_init(int C, int d_y, int w, const T *WL, const T *der, int ldd, T *P,
                            cudaStream_t st) {
  return launch_pdl(k_jac_init<T>, grid_for((size_t)C * d_y * w), 256, 0, st, C, d_y, w, WL, der,
                    ldd, P);
}

template <typename T>
cudaError_t launch_broadcast(int C, size_t n, const T *src, T *out, cudaStream_t st) {
  k_broadcast<T><<<grid_for((size_t)C * n), 256, 0, st>>>(C, n, src, out);
  return cudaGetLastError();
}

cudaError_t launch_copy_f64(size_t n, const double *src, double *dst, cudaStream_t st) {
  k_convert<double, double><<<grid_for(n), 256, 0, st>>>(n, src, dst);
  return cudaGetLastError();
}

cudaError_t launch_f32_to_f64(size_t n, const float *src, double *dst, cudaStream_t st) {
  k_convert<float, double><<<grid_for(n), 256, 0, st>>>(n, src, dst);
  return cudaGetLastError();
}

cudaError_t launch_f64_to_f32(size_t n, const double *src, float *dst, cudaStream_t st) {
  k_convert<double, float><<<grid_for(n), 256, 0, st>>>(n, src, dst);
  return cudaGetLastError();
}

// The SIMT GEMMs serve the FP64 path; the prior draw both paths.
template cudaError_t gemm_store<double>(int, int, int, const double *, int, const double *, int,
                                        double *, int, cudaStream_t);
template cudaError_t gemm_bias_act<double>(int, int, int, const double *, int, const double *,
                                           int, const double *, int, double *, double *, int,
                                           cudaStream_t);
template cudaError_t gemm_scale_group<double>(int, int, int, const double *, int, const double *,
                                              int, const double *, int, int, double *, int,
                                              cudaStream_t);
template cudaError_t gemm_coef<double>(int, int, int, const double *, int, const double *, int,
                                       const double *, int, double, double *, int, cudaStream_t);
template cudaError_t gemm_field<double>(int, int, int, const double *, int, const double *, int,
                                        const int *, double, double, double *, const double *,
                                        int, cudaStream_t);
template cudaError_t launch_jac_init<double>(int, int, int, const double *, const double *, int,
                                             double *, cudaStream_t);
template cudaError_t launch_broadcast<double>(int, size_t, const double *, double *,
                                              cudaStream_t);
#define DINO_INST_DRAW(T)                                                                     \
  template cudaError_t launch_prior_draw<T>(int, int, const T *, const T *, uint64_t,         \
                                            uint64_t, uint32_t, uint32_t, T *, int,           \
                                            cudaStream_t, __nv_bfloat16 *, int, size_t, int, \
                                            const double *, const int *, bool);
DINO_INST_DRAW(double)
DINO_INST_DRAW(float)

}  // namespace dino
