// Allocation-free evaluation of the surrogate forward pass and its reduced
// Jacobian (FP64), for host code that is not allowed to allocate device memory.
//
// Such callers exist: a plugin running inside a framework that owns every
// device byte through its own pool, or a latency-critical loop in which the
// device-wide synchronisation that cudaMalloc/cudaFree may imply is not
// acceptable.  The entry point below therefore never allocates.  Inputs and
// outputs are device buffers the caller owns.  Intermediate values live in one
// file-scope device array of fixed size and in shared memory.
// Every GPU that loads this library holds that array until the process exits.
//
// Set-up: the host cannot use the array's name as a device address (in host
// code it is only a stand-in symbol).  The first call on each device looks up
// the real address with cudaGetSymbolAddress while that device is current,
// and caches it.  That first call should therefore come before any stream
// capture on the device.
//
// Sharing: every call uses the same array, and it keeps the previous call's
// contents.  The kernel writes every scratch element before reading it, so
// nothing has to start at zero.  Two calls whose kernels overlap on the GPU
// (different streams, no ordering between them) race on the array: order
// them on one stream, or wait for one before issuing the other.
#include "../../include/dino.h"

#include <cuda_runtime.h>

#include <algorithm>
#include <mutex>

namespace dino {
namespace {

constexpr int kMaxLayers = 16;
constexpr int kMaxDevices = 64;
constexpr int kThreads = 256;     // a CTA of k_jac_point
constexpr int kJacThreads = 512;  // ... of k_jac_rows

static __device__ __align__(256) double g_noalloc_scratch[DINO_NOALLOC_SCRATCH_DOUBLES];

struct Net {
  int L, act;
  int w[kMaxLayers + 1];
  const double *W[kMaxLayers];
  const double *b[kMaxLayers];
};

__device__ __forceinline__ double act_fn(int kind, double z) {
  if (kind == DINO_ACT_TANH) return tanh(z);
  if (kind == DINO_ACT_GELU) return 0.5 * z * (1.0 + erf(z * 0.70710678118654752440));
  return z;
}

__device__ __forceinline__ double act_deriv(int kind, double z) {
  if (kind == DINO_ACT_TANH) {
    const double t = tanh(z);
    return 1.0 - t * t;
  }
  if (kind == DINO_ACT_GELU)
    return 0.5 * (1.0 + erf(z * 0.70710678118654752440)) +
           z * exp(-0.5 * z * z) * 0.39894228040143267794;
  return 1.0;
}

// One CTA per point, for many points or a small network (spread_rows).  Shared
// memory holds the activations and the activation derivatives; the d_y x w
// products of the reverse sweep go to a per-point slab of the scratch array (two
// ping-pong buffers of d_y * wmax doubles).
__global__ void __launch_bounds__(kThreads)
    k_jac_point(const Net net, int wmax, const double *__restrict__ x, double *__restrict__ f,
                double *__restrict__ J, double *__restrict__ scratch) {
  extern __shared__ double sm[];
  const int p = blockIdx.x, L = net.L, r = net.w[0], dy = net.w[L];
  double *a[kMaxLayers + 1];
  double *d[kMaxLayers];
  int off = 0;
  for (int l = 0; l < L; ++l) {  // a[0..L-1]: layer inputs; d[0..L-2]: derivatives
    a[l] = sm + off;
    off += net.w[l];
  }
  for (int l = 0; l + 1 < L; ++l) {
    d[l] = sm + off;
    off += net.w[l + 1];
  }
  for (int i = threadIdx.x; i < r; i += blockDim.x) a[0][i] = x[(size_t)p * r + i];
  __syncthreads();
  for (int l = 0; l < L; ++l) {
    const int wi = net.w[l], wo = net.w[l + 1];
    const double *W = net.W[l];
    for (int o = threadIdx.x; o < wo; o += blockDim.x) {
      double z = net.b[l][o];
      for (int i = 0; i < wi; ++i) z += W[(size_t)o * wi + i] * a[l][i];
      if (l + 1 < L) {
        a[l + 1][o] = act_fn(net.act, z);
        d[l][o] = act_deriv(net.act, z);
      } else {
        f[(size_t)p * dy + o] = z;
      }
    }
    __syncthreads();
  }
  double *Jp = J + (size_t)p * dy * r;
  if (L == 1) {
    for (int e = threadIdx.x; e < dy * r; e += blockDim.x) Jp[e] = net.W[0][e];
    return;
  }
  double *P = scratch + (size_t)p * 2 * dy * wmax;
  double *Q = P + (size_t)dy * wmax;
  const int wl = net.w[L - 1];
  for (int e = threadIdx.x; e < dy * wl; e += blockDim.x)
    P[e] = net.W[L - 1][e] * d[L - 2][e % wl];
  __syncthreads();
  for (int l = L - 2; l >= 1; --l) {  // P <- (P W_l) .* d_{l-1}
    const int wi = net.w[l], wo = net.w[l + 1];
    const double *W = net.W[l];
    for (int e = threadIdx.x; e < dy * wi; e += blockDim.x) {
      const int i = e / wi, j = e % wi;
      double acc = 0.0;
      for (int k = 0; k < wo; ++k) acc += P[(size_t)i * wo + k] * W[(size_t)k * wi + j];
      Q[e] = acc * d[l - 1][j];
    }
    __syncthreads();
    double *t = P;
    P = Q;
    Q = t;
  }
  const int w1 = net.w[1];
  for (int e = threadIdx.x; e < dy * r; e += blockDim.x) {  // J = P W_0
    const int i = e / r, j = e % r;
    double acc = 0.0;
    for (int k = 0; k < w1; ++k) acc += P[(size_t)i * w1 + k] * net.W[0][(size_t)k * r + j];
    Jp[e] = acc;
  }
}

// One layer of the forward pass for every point of the chunk: a warp per
// output, lanes along the weight row.  The activations ping-pong between two
// halves of a point's slab of the scratch array; the activation derivatives of
// all hidden layers follow them (offset der_off of layer l).
__global__ void __launch_bounds__(256)
    k_layer(const Net net, int l, int wmax, int der_off, size_t slab, const double *__restrict__ x,
            double *__restrict__ f, double *__restrict__ scratch) {
  const int p = blockIdx.y, o = blockIdx.x * 8 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  const int wi = net.w[l], wo = net.w[l + 1], r = net.w[0], dy = net.w[net.L];
  if (o >= wo) return;
  double *s = scratch + (size_t)p * slab;
  const double *a = l == 0 ? x + (size_t)p * r : s + ((l - 1) & 1) * (size_t)wmax;
  const double *W = net.W[l] + (size_t)o * wi;
  double z = 0.0;
  for (int i = lane; i < wi; i += 32) z += W[i] * a[i];
#pragma unroll
  for (int q = 16; q; q >>= 1) z += __shfl_xor_sync(0xffffffffu, z, q);
  if (lane) return;
  z += net.b[l][o];
  if (l + 1 < net.L) {
    s[(l & 1) * (size_t)wmax + o] = act_fn(net.act, z);
    s[2 * (size_t)wmax + der_off + o] = act_deriv(net.act, z);
  } else {
    f[(size_t)p * dy + o] = z;
  }
}

// Reverse sweep, rows [i0, i0 + rows) of one point's Jacobian per CTA: the rows
// of P = W_{L-1} .* d_{L-2}, P <- (P W_l) .* d_{l-1}, J = P W_0 are independent, so
// they stay in the CTA's shared memory and the d_y rows of a point spread over
// as many SMs as there are.  The FP64 pipe (2 multiply-adds a cycle and SM)
// bounds it, so a thread per output with its operands from L1 and shared
// memory keeps up.  Eight points of widths 200-400-400-100: 8.0 ms with a CTA
// per point and the products in global scratch, 0.44 ms here (0.31 ms at the
// rate of 152 FP64 pipes).
__global__ void __launch_bounds__(kJacThreads)
    k_jac_rows(const Net net, int wmax, int rows, size_t slab, double *__restrict__ J,
               const double *__restrict__ scratch) {
  extern __shared__ double sm[];
  const int p = blockIdx.y, L = net.L, r = net.w[0], dy = net.w[L];
  const int i0 = blockIdx.x * rows, nr = min(rows, dy - i0);
  double *Jp = J + ((size_t)p * dy + i0) * r;
  // A single layer: spread_rows sends it to k_jac_point, but without this branch the
  // compiler's inner loop is the slower one (one point of 100-200-200-20 49.5 -> 53.7 us).
  if (L == 1) {
    for (int e = threadIdx.x; e < nr * r; e += blockDim.x)
      Jp[e] = net.W[0][(size_t)i0 * r + e];
    return;
  }
  const double *der = scratch + (size_t)p * slab + 2 * (size_t)wmax;
  int off = 0;  // of d_{l - 1} (layer widths w_1 .. w_{L - 1})
  for (int l = 1; l < L - 1; ++l) off += net.w[l];
  double *P = sm, *Q = sm + (size_t)rows * wmax;
  const int wl = net.w[L - 1];
  for (int e = threadIdx.x; e < nr * wl; e += blockDim.x)
    P[e] = net.W[L - 1][(size_t)i0 * wl + e] * der[off + e % wl];
  __syncthreads();
  for (int l = L - 2; l >= 0; --l) {
    const int wi = net.w[l], wo = net.w[l + 1];
    const double *__restrict__ W = net.W[l];
    if (l > 0) off -= wi;
    for (int e = threadIdx.x; e < nr * wi; e += blockDim.x) {
      const int i = e / wi, j = e - i * wi;
      const double *Pi = P + (size_t)i * wo, *Wj = W + j;
      double acc = 0.0;
#pragma unroll 8
      for (int k = 0; k < wo; ++k) acc += Pi[k] * Wj[(size_t)k * wi];
      if (l > 0)
        Q[e] = acc * der[off + j];
      else
        Jp[e] = acc;
    }
    __syncthreads();
    double *t = P;
    P = Q;
    Q = t;
  }
}

// Whether n points spread their outputs over all SMs (k_layer and k_jac_rows)
// instead of taking a CTA each (k_jac_point): by the times of both, in us.  A
// point's CTA runs its layers as chains of w multiply-adds (0.167 each) and the
// Jacobian's multiply-adds on the FP64 pipe of its SM (0.31 per 1000), the same for
// every point while each has an SM of its own.  Spread, a layer costs a launch, its
// values and derivatives come from one lane a warp (1.16, 3.1 and 7.1 per 1000 hidden
// units and point for the identity, tanh and GELU) and the Jacobian's multiply-adds
// run on all SMs (0.0036 per 1000).  Fitted to 450 measured calls (16 networks of 1
// to 11 layers, 4 to 3200 wide, 1 to 2000 points): the way taken is at most 9% slower
// than a CTA per point, and at most 27% slower than the other way (at 150 points
// of 200-400-400-1 with the identity, 257 against 203).  16-64-64-49, GELU, a CTA each
// and spread: 1 point 96 and 45, 24 points 95 and 78, 48 points 96 and 116, 150 points 97
// and 238; 12-30-7: 1 point 16 and 26, 1000 points 32 and 259; 200-400-400-100: 1 point
// 8164 and 113, 8 points 8160 and 444.
bool spread_rows(const Net &net, int n, int sms) {
  const int L = net.L;
  if (L < 2 || n > sms) return false;
  double hidden = 0.0, macs = 0.0;  // multiply-adds of one point's Jacobian, in thousands
  for (int l = 1; l < L; ++l) hidden += net.w[l];
  for (int l = 0; l + 1 < L; ++l) macs += 1e-3 * net.w[L] * net.w[l] * net.w[l + 1];
  const bool gelu = net.act == DINO_ACT_GELU, tanh = net.act == DINO_ACT_TANH;
  const double value = gelu ? 7.1e-3 : tanh ? 3.1e-3 : 1.16e-3;
  const double layer = gelu ? 7.7 : tanh ? 2.4 : 0.0;
  const double point = 9.8 + 0.31 * macs + 0.167 * (net.w[0] + hidden);
  const double spread = 1.7 + 7.2 * L + 0.056 * hidden + layer * (L - 1) +
                        n * (value * hidden + 0.0036 * macs);
  return spread < point;
}

std::mutex g_mu;
double *g_addr[kMaxDevices] = {nullptr};

}  // namespace
}  // namespace dino

extern "C" int dino_surrogate_jacobian_noalloc(int n, int n_layers, const int *widths,
                                               int activation, const double *const *W,
                                               const double *const *b, const double *x,
                                               double *f, double *J, void *stream) {
  using namespace dino;
  if (n < 1 || n_layers < 1 || n_layers > kMaxLayers || !widths || !W || !b || !x || !f || !J)
    return DINO_EINVAL;
  if (activation < DINO_ACT_IDENTITY || activation > DINO_ACT_GELU) return DINO_EINVAL;
  Net net{};
  net.L = n_layers;
  net.act = activation;
  int wmax = 0;
  size_t smem_doubles = 0;
  for (int l = 0; l <= n_layers; ++l) {
    if (widths[l] < 1) return DINO_EINVAL;
    net.w[l] = widths[l];
    if (l < n_layers) smem_doubles += widths[l];
    if (l >= 1 && l < n_layers) {
      wmax = widths[l] > wmax ? widths[l] : wmax;
      smem_doubles += widths[l];
    }
  }
  for (int l = 0; l < n_layers; ++l) {
    if (!W[l] || !b[l]) return DINO_EINVAL;
    net.W[l] = W[l];
    net.b[l] = b[l];
  }
  const size_t smem = smem_doubles * sizeof(double);
  if (smem > 200 * 1024) return DINO_EINVAL;
  // the fixed scratch must hold two d_y x wmax buffers per point
  const size_t need = (size_t)n * 2 * (size_t)widths[n_layers] * (size_t)wmax;
  if (need > (size_t)DINO_NOALLOC_SCRATCH_DOUBLES) return DINO_ENOMEM;

  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) return DINO_ECUDA;
  // Held to the last launch: the kernels of calls that host threads make on one
  // stream must not alternate on the scratch, nor one call lower the
  // shared-memory limit that another has just set.
  std::lock_guard<std::mutex> lk(g_mu);
  if (!g_addr[dev]) {
    void *p = nullptr;
    if (cudaGetSymbolAddress(&p, g_noalloc_scratch) != cudaSuccess || !p) {
      cudaGetLastError();
      return DINO_ECUDA;
    }
    g_addr[dev] = (double *)p;
  }
  double *scratch = g_addr[dev];
  const cudaStream_t st = (cudaStream_t)stream;
  int sms = 0;
  if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || sms < 1)
    return DINO_ECUDA;
  if (!spread_rows(net, n, sms)) {
    if (smem > 48 * 1024 &&
        cudaFuncSetAttribute(k_jac_point, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)smem) != cudaSuccess)
      return DINO_ECUDA;
    k_jac_point<<<n, kThreads, smem, st>>>(net, wmax, x, f, J, scratch);
    return cudaGetLastError() == cudaSuccess ? DINO_OK : DINO_ECUDA;
  }
  // a point's slab: two activation buffers and every hidden layer's derivatives
  size_t hidden = 0;
  for (int l = 1; l < n_layers; ++l) hidden += widths[l];
  const int r = widths[0], dy = widths[n_layers];
  const size_t slab = 2 * (size_t)wmax + hidden;
  // blockIdx.y runs over the points of a chunk
  const int chunk = (int)std::min((size_t)DINO_NOALLOC_SCRATCH_DOUBLES / slab, (size_t)n);
  // rows per CTA: one CTA on every SM, within the shared memory of one CTA
  // (two buffers of rows x wmax; one row always fits, since the widths' sums do)
  const size_t row_bytes = 2 * (size_t)wmax * sizeof(double);
  size_t rows = ((size_t)std::min(n, chunk) * dy + sms - 1) / sms;
  rows = std::min(rows, (size_t)(200 * 1024) / row_bytes);
  rows = std::max<size_t>(1, std::min(rows, (size_t)dy));
  const size_t jsm = rows * row_bytes;
  if (jsm > 48 * 1024 &&
      cudaFuncSetAttribute(k_jac_rows, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)jsm) !=
          cudaSuccess)
    return DINO_ECUDA;
  for (int p0 = 0; p0 < n; p0 += chunk) {
    const int np = std::min(chunk, n - p0);
    int off = 0;
    for (int l = 0; l < n_layers; ++l) {
      dim3 grid((widths[l + 1] + 7) / 8, np);
      k_layer<<<grid, 256, 0, st>>>(net, l, wmax, off, slab, x + (size_t)p0 * r,
                                    f + (size_t)p0 * dy, scratch);
      if (l + 1 < n_layers) off += widths[l + 1];
    }
    dim3 grid((unsigned)((dy + rows - 1) / rows), np);
    k_jac_rows<<<grid, kJacThreads, jsm, st>>>(net, wmax, (int)rows, slab,
                                               J + (size_t)p0 * dy * r, scratch);
    if (cudaGetLastError() != cudaSuccess) return DINO_ECUDA;
  }
  return DINO_OK;
}
