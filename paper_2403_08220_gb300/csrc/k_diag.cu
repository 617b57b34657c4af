// Markov-chain diagnostics on the device (Sec. 6.2): a recorded trajectory of
// n_c chains x n_s samples x d degrees of freedom, stored per degree of
// freedom and chain so that each series is contiguous:
//   traj[(i n_c + k) max_s + j] = x_{j,k}(i).
//
//   k_diag_record   appends one sample of every chain (from a pool's state or
//                   a caller buffer);
//   k_diag_ess      a cluster of 1 to 8 CTAs per degree of freedom: chain means and variances,
//                   w and v (the 1D covariance estimators), the multi-chain
//                   autocorrelation MACT(t) = 1 - (w - mean_k AC(t,k)) / v in
//                   passes of kLags lags until a pair sum is no longer positive
//                   (the initial positive sequence), ESS% = 1 / (1 + 2 sum_t
//                   MACT(t)) (eq:ess), and the squared jumps of the MSJ;
//   k_diag_center   centred samples and centred chain means (d x n_c n_s and
//                   d x n_c) whose Gram products give W and V
//                   (eq:covariance_estimator);
//   k_psd_chol      W = F F^T and V = C C^T (lower triangular, one CTA each);
//                   the eigenvalues of W^1/2 V W^1/2 are those of F^T V F, the
//                   squared singular values of C^T F, so the Wasserstein MPSRF
//                   Tr(W + V - 2 (W^1/2 V W^1/2)^1/2) is Tr W + Tr V - 2 |C^T F|_*
//                   without a square root of W;
//   k_ct_f          C^T F by columns;
//   k_ns_start, k_row_dots  the nuclear norm |A|_* = tr(U^T A) of A = C^T F from its
//                   polar factor U, the limit of the Newton-Schulz iteration
//                   X <- X (3 I - X^T X) / 2 from A / |A|_F (two d x d products a
//                   step, k_simt.cu).  Every singular value of X grows by up to
//                   1.5 a step until it reaches 1, so about log_1.5(|A|_F /
//                   sigma_min) + 5 steps do; where A is singular or nearly so
//                   they do not, and the one-sided Jacobi below takes over;
//   k_jacobi_round  one-sided Jacobi (Hestenes) on a d x d matrix held by
//                   columns: column pairs are rotated until orthogonal; a
//                   launch is one round of a round-robin over blocks of
//                   columns, whose pairs are disjoint and run on separate CTAs
//                   (the host loops over rounds and sweeps).  The final column
//                   norms are the singular values; for a symmetric positive
//                   semidefinite matrix they are its eigenvalues and the
//                   accumulated rotations its eigenvectors;
//   k_normals, k_transpose  the encoded prior draws and the stacked transposed
//                   Jacobian of the surrogate-driven DIS basis (eq:mc_ppgnh),
//                   whose eigenproblem the same Jacobi kernel solves.
// Every loop is bounded by the sizes (lags by n_s, Jacobi sweeps by
// kMaxJacobiSweeps); CTAs wait on one another only at the barriers of a cluster,
// which all of its CTAs reach the same number of times (every CTA walks the same
// MACT values).
#include <cooperative_groups.h>

#include <algorithm>

#include "chol.cuh"

namespace dino {
namespace {

namespace cg = cooperative_groups;

constexpr int kEssThreads = 256;

template <typename T>
__global__ void k_diag_record(int n_c, int d, const T *__restrict__ src, int ld_src,
                              double *__restrict__ traj, int max_s, int j) {
  const size_t n = (size_t)n_c * d;
  for (size_t e = blockIdx.x * (size_t)blockDim.x + threadIdx.x; e < n;
       e += (size_t)gridDim.x * blockDim.x) {
    const size_t k = e / d, i = e - k * d;  // source row k (chain), column i (dof)
    traj[(i * n_c + k) * max_s + j] = (double)src[k * ld_src + i];
  }
}

// Sum over the CTA of two values (every thread gets both); red >= 66 doubles.
__device__ void block_sum2(double &x, double &y, double *red) {
  for (int o = 16; o; o >>= 1) {
    x += __shfl_xor_sync(kFull, x, o);
    y += __shfl_xor_sync(kFull, y, o);
  }
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  __syncthreads();
  if (lane == 0) {
    red[warp] = x;
    red[32 + warp] = y;
  }
  __syncthreads();
  if (warp == 0) {
    double a = lane < nw ? red[lane] : 0.0, b = lane < nw ? red[32 + lane] : 0.0;
    for (int o = 16; o; o >>= 1) {
      a += __shfl_xor_sync(kFull, a, o);
      b += __shfl_xor_sync(kFull, b, o);
    }
    if (lane == 0) {
      red[64] = a;
      red[65] = b;
    }
  }
  __syncthreads();
  x = red[64];
  y = red[65];
}

// Sums over the warp of eight values at once: three steps that halve the
// values a lane carries (4 + 2 + 1 additions) and two that add what is left;
// lane l returns the sum of v[l & 7] (9 additions for 40).
__device__ __forceinline__ double warp_sum8(const double v[8]) {
  const int lane = threadIdx.x & 31;
  double a[4], b[2], c;
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const double keep = (lane & 1) ? v[2 * q + 1] : v[2 * q];
    const double give = (lane & 1) ? v[2 * q] : v[2 * q + 1];
    a[q] = keep + __shfl_xor_sync(kFull, give, 1);  // value 2 q + (lane & 1)
  }
#pragma unroll
  for (int q = 0; q < 2; ++q) {
    const double keep = (lane & 2) ? a[2 * q + 1] : a[2 * q];
    const double give = (lane & 2) ? a[2 * q] : a[2 * q + 1];
    b[q] = keep + __shfl_xor_sync(kFull, give, 2);  // value 4 q + (lane & 3)
  }
  const double keep = (lane & 4) ? b[1] : b[0], give = (lane & 4) ? b[0] : b[1];
  c = keep + __shfl_xor_sync(kFull, give, 4);  // value lane & 7
  c += __shfl_xor_sync(kFull, c, 8);
  return c + __shfl_xor_sync(kFull, c, 16);
}

constexpr int kLags = 8;     // lags per pass over the samples
constexpr int kEssMaxCluster = 8;  // CTAs that share a degree of freedom's lags
constexpr int kSegment = 128;  // samples of one chain that a warp takes at a time

// Dynamic shared memory: n_c chain means, then with kStaged the centred samples
// (n_c x n_s).  A pass forms kLags lags in each CTA of the cluster: per sample
// one multiply-add for each from consecutive shared-memory words, and one
// reduction per pass.  The CTAs exchange MACT through each other's shared memory
// and each walks the pairs in order.  Bound by the FP64 pipes; degrees of
// freedom differ in their lags, up to all n_s.  (One pass per lag pair over
// global memory, with a division per sample to find its chain, took 17.4 ms for
// 200 degrees of freedom, 10 chains of 1000 samples, of which some run all 1000
// lags; a CTA each 3.3 ms; clusters of four 1.84 ms.)
// Lags past the first non-positive pair are formed and not used.
template <bool kStaged>
__global__ void __launch_bounds__(kEssThreads)
    k_diag_ess(int n_c, int n_s, const double *__restrict__ traj, int max_s,
               double *__restrict__ means, double *__restrict__ ess, double *__restrict__ sqjump) {
  extern __shared__ double mk[];
  __shared__ double red[72], lagsum[kEssThreads / 32][kLags];
  __shared__ double mact[2][kEssMaxCluster * kLags];  // a pass's MACT, by its parity
  __shared__ bool more_s;
  double *xs = mk + n_c;
  const cg::cluster_group cluster = cg::this_cluster();
  const int cs = (int)cluster.num_blocks(), rank = (int)cluster.block_rank();
  const int i = blockIdx.x / cs;
  const double *X = traj + (size_t)i * n_c * max_s;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  // chain means, within-chain sums of squares and squared jumps (warp per chain)
  double ss = 0.0, jj = 0.0;
  for (int k = warp; k < n_c; k += nw) {
    const double *xk = X + (size_t)k * max_s;
    double s = 0.0;
    for (int j = lane; j < n_s; j += 32) s += xk[j];
    const double m = warp_sum(s) / n_s;
    if (lane == 0) mk[k] = m;
    for (int j = lane; j < n_s; j += 32) {
      const double v = xk[j], x = v - m;
      ss += x * x;
      if (kStaged) xs[(size_t)k * n_s + j] = x;
      if (j + 1 < n_s) {
        const double dx = xk[j + 1] - v;
        jj += dx * dx;
      }
    }
  }
  block_sum2(ss, jj, red);  // includes barriers
  double gm = 0.0;
  for (int k = 0; k < n_c; ++k) gm += mk[k];
  gm /= n_c;
  double bs = 0.0;
  for (int k = 0; k < n_c; ++k) bs += (mk[k] - gm) * (mk[k] - gm);
  const double w = ss / ((double)n_c * (n_s - 1));
  const double v = (double)(n_s - 1) / n_s * w + (double)(n_c + 1) / ((double)n_c * (n_c - 1)) * bs;
  // MACT(t) for lag pairs (2m, 2m + 1), MACT(0) = 1, while the pair sum is positive
  const double inv_n = 1.0 / ((double)n_s * n_c), inv_v = 1.0 / v;
  const int segs = (n_s + kSegment - 1) / kSegment;
  double total = 0.0;
  int pairs = 0;
  bool more = true;
  cluster.sync();  // every CTA runs before one writes into another's mact
  for (int base = 0, buf = 0; more && base + 1 < n_s; base += cs * kLags, buf ^= 1) {
    const int t0 = base + rank * kLags;
    double acc[kLags] = {};
    for (int it = warp; it < n_c * segs; it += nw) {
      const int k = it / segs, j0 = (it - k * segs) * kSegment;
      const double m = mk[k];
      const double *xk = kStaged ? xs + (size_t)k * n_s : X + (size_t)k * max_s;
      const int j1 = min(n_s - t0, j0 + kSegment);  // later samples have no partner
      if (j1 + t0 + kLags - 1 <= n_s) {
        for (int j = j0 + lane; j < j1; j += 32) {
          const double x = kStaged ? xk[j] : xk[j] - m;
#pragma unroll
          for (int q = 0; q < kLags; ++q)
            acc[q] += x * (kStaged ? xk[j + t0 + q] : xk[j + t0 + q] - m);
        }
      } else {
        for (int j = j0 + lane; j < j1; j += 32) {
          const double x = kStaged ? xk[j] : xk[j] - m;
#pragma unroll
          for (int q = 0; q < kLags; ++q)
            if (j + t0 + q < n_s) acc[q] += x * (kStaged ? xk[j + t0 + q] : xk[j + t0 + q] - m);
        }
      }
    }
    const double s = warp_sum8(acc);
    if (lane < kLags) lagsum[warp][lane] = s;
    __syncthreads();
    if (warp == 0 && lane < kLags) {  // MACT(t0 + lane), to every CTA
      double r = 0.0;
      for (int u = 0; u < nw; ++u) r += lagsum[u][lane];
      r = t0 + lane == 0 ? 1.0 : 1.0 - (w - r * inv_n) * inv_v;
      for (int p = 0; p < cs; ++p)
        *cluster.map_shared_rank(&mact[buf][rank * kLags + lane], p) = r;
    }
    cluster.sync();  // the other buffer is written until the next one
    if (warp == 0) {  // the pairs in order
      bool on = true;
      for (int q = 0; on && q < cs * kLags; q += 2) {
        const double pq = mact[buf][q] + mact[buf][q + 1];
        on = base + q + 1 < n_s && pq > 0.0;
        if (on) {
          total += pq;
          ++pairs;
        }
      }
      if (lane == 0) more_s = on;
    }
    __syncthreads();
    more = more_s;
  }
  if (rank) return;  // the last write into another CTA's memory came before a barrier
  if (threadIdx.x == 0) {
    ess[i] = pairs > 0 ? 1.0 / (2.0 * total - 1.0) : 1.0;
    sqjump[i] = jj;
  }
  for (int k = threadIdx.x; k < n_c; k += blockDim.x) means[(size_t)i * n_c + k] = mk[k];
}

__global__ void k_diag_center(int d, int n_c, int n_s, const double *__restrict__ traj, int max_s,
                              const double *__restrict__ means, double *__restrict__ Xc,
                              double *__restrict__ Mc) {
  const size_t K = (size_t)n_c * n_s, n = (size_t)d * K;
  for (size_t e = blockIdx.x * (size_t)blockDim.x + threadIdx.x; e < n;
       e += (size_t)gridDim.x * blockDim.x) {
    const size_t i = e / K, rem = e - i * K, k = rem / n_s, j = rem - k * n_s;
    Xc[e] = traj[(i * n_c + k) * max_s + j] - means[i * n_c + k];
  }
  for (size_t e = blockIdx.x * (size_t)blockDim.x + threadIdx.x; e < (size_t)d * n_c;
       e += (size_t)gridDim.x * blockDim.x) {
    const size_t i = e / n_c;
    double g = 0.0;
    for (int k = 0; k < n_c; ++k) g += means[i * n_c + k];
    Mc[e] = means[e] - g / n_c;
  }
}

// W = Wr / (n_c (n_s - 1)), V = (n_s - 1)/n_s W + (n_c + 1)/(n_c (n_c - 1)) Br
__global__ void k_diag_wv(int d, int n_c, int n_s, const double *__restrict__ Wr,
                          const double *__restrict__ Br, double *__restrict__ W,
                          double *__restrict__ V) {
  for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < d * d; e += gridDim.x * blockDim.x) {
    const double w = Wr[e] / ((double)n_c * (n_s - 1));
    W[e] = w;
    V[e] = (double)(n_s - 1) / n_s * w + (double)(n_c + 1) / ((double)n_c * (n_c - 1)) * Br[e];
  }
}

constexpr int kPairThreads = 128;  // threads of a column pair

// One round of a sweep: CTA pi takes the pair (p, q) of blocks of kB columns of
// the round-robin over nb blocks, holds them (and their columns of Q) in
// shared memory and rotates the kB x kB column pairs across the blocks, kB
// disjoint ones at a time, each by kPairThreads threads; in the first round
// of a sweep also the pairs inside the blocks.  With Q the rotations are
// applied to Q as well.  *rotated is set when any pair was.  What bounds it is
// the chain of dependent FP64 operations of one rotation (about 5 us with the
// launch): d = 200, 9 sweeps of 199 rounds, 12.7 ms, against 465 ms for two
// solves (W's square root, then W^1/2 V W^1/2) by one CTA that looped over all
// pairs; blocks of 2 and of 4 columns take the same time at d = 200.
template <int kB>
__global__ void __launch_bounds__(kB *kPairThreads)
    k_jacobi_round(int d, int nb, int rnd, double *__restrict__ G, double *__restrict__ Q,
                   int *__restrict__ rotated) {
  extern __shared__ double sm[];  // columns 0 .. kB - 1 of block p, kB .. 2 kB - 1 of block q
  __shared__ double part[kB][kPairThreads / 32][4];
  const int n = nb + (nb & 1);  // players, one dummy if nb is odd
  const int pi = blockIdx.x;
  const int p = pi == 0 ? n - 1 : (rnd + pi) % (n - 1);
  const int q = (rnd - pi + n - 1) % (n - 1);
  const bool inside = kB > 1 && rnd == 0;
  if ((p >= nb || q >= nb) && !inside) return;
  const int lane = threadIdx.x & 31, grp = threadIdx.x / kPairThreads,
            gt = threadIdx.x % kPairThreads, gw = gt >> 5;
  auto column = [&](int u) { return u < kB ? p * kB + u : q * kB + u - kB; };
  double *sq = sm + (size_t)2 * kB * d;
  for (int u = grp; u < 2 * kB; u += kB) {
    const int col = column(u);
    for (int k = gt; k < d; k += kPairThreads) {
      sm[(size_t)u * d + k] = col < d ? G[(size_t)col * d + k] : 0.0;
      if (Q) sq[(size_t)u * d + k] = col < d ? Q[(size_t)col * d + k] : 0.0;
    }
  }
  __syncthreads();
  bool any = false;
  // rotates columns u and v of this group's pair; every thread of the CTA calls it
  auto rotate = [&](int u, int v) {
    double *x = sm + (size_t)u * d, *y = sm + (size_t)v * d;
    double al = 0.0, be = 0.0, ga = 0.0;
    for (int k = gt; k < d; k += kPairThreads) {
      al += x[k] * x[k];
      be += y[k] * y[k];
      ga += x[k] * y[k];
    }
    // three sums over the warp in six additions: lane l ends with value l & 3
    const double k0 = (lane & 1) ? be : al, g0 = (lane & 1) ? al : be;
    const double a0 = k0 + __shfl_xor_sync(kFull, g0, 1);
    const double k1 = (lane & 1) ? 0.0 : ga, g1 = (lane & 1) ? ga : 0.0;
    const double a1 = k1 + __shfl_xor_sync(kFull, g1, 1);
    double z = ((lane & 2) ? a1 : a0) + __shfl_xor_sync(kFull, (lane & 2) ? a0 : a1, 2);
    z += __shfl_xor_sync(kFull, z, 4);
    z += __shfl_xor_sync(kFull, z, 8);
    z += __shfl_xor_sync(kFull, z, 16);
    if (lane < 4) part[grp][gw][lane] = z;
    __syncthreads();
    al = be = ga = 0.0;
#pragma unroll
    for (int w = 0; w < kPairThreads / 32; ++w) {
      al += part[grp][w][0];
      be += part[grp][w][1];
      ga += part[grp][w][2];
    }
    // |ga| > 1e-15 sqrt(al be), by squares where those stay in range
    const double ab = al * be;
    const bool turn = al != 0.0 && be != 0.0 &&
                      (ab > 1e-250 && ab < 1e250 ? ga * ga > 1e-30 * ab
                                                 : fabs(ga) > 1e-15 * sqrt(al) * sqrt(be));
    if (turn) {
      double c, s, t;
      jacobi_rotation(al, be, ga, c, s, t);
      for (int k = gt; k < d; k += kPairThreads) {
        const double a = x[k], b = y[k];
        x[k] = c * a - s * b;
        y[k] = s * a + c * b;
      }
      if (Q) {
        double *xq = sq + (size_t)u * d, *yq = sq + (size_t)v * d;
        for (int k = gt; k < d; k += kPairThreads) {
          const double a = xq[k], b = yq[k];
          xq[k] = c * a - s * b;
          yq[k] = s * a + c * b;
        }
      }
      any = true;
    }
    __syncthreads();
  };
  if constexpr (kB > 1) {
    if (inside) {  // round-robin inside each block: kB / 2 disjoint pairs each
      const int blk = grp / (kB / 2), g = grp % (kB / 2);
      for (int t = 0; t < kB - 1; ++t) {
        const int u = g == 0 ? kB - 1 : (t + g) % (kB - 1), v = (t - g + kB - 1) % (kB - 1);
        rotate(blk * kB + u, blk * kB + v);
      }
    }
  }
  for (int t = 0; t < kB; ++t) rotate(grp, kB + (grp + t) % kB);
  for (int u = grp; u < 2 * kB; u += kB) {
    const int col = column(u);
    if (col >= d) continue;
    for (int k = gt; k < d; k += kPairThreads) {
      G[(size_t)col * d + k] = sm[(size_t)u * d + k];
      if (Q) Q[(size_t)col * d + k] = sq[(size_t)u * d + k];
    }
  }
  if (any && gt == 0) *rotated = 1;
}

// sig[i] = |column i|: a warp per column
__global__ void k_col_norms(int d, const double *__restrict__ G, double *__restrict__ sig) {
  const int i = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
  if (i >= d) return;
  double s = 0.0;
  for (int k = lane; k < d; k += 32) s += G[(size_t)i * d + k] * G[(size_t)i * d + k];
  s = warp_sum(s);
  if (lane == 0) sig[i] = sqrt(s);
}

// Cholesky factors of symmetric positive semidefinite matrices, one CTA each
// (blockIdx 0: W -> F, 1: V -> C, d x d row-major, the lower triangle; above
// it zeros).  Right-looking in panels of kCholPanel columns held in shared
// memory.  A pivot at or below the rounding level of its diagonal entry (4
// eps) is a direction the matrix does not have: its column is zero.
constexpr int kCholPanel = 8;
constexpr int kCholThreads = 1024;

__global__ void __launch_bounds__(kCholThreads)
    k_psd_chol(int d, const double *__restrict__ W, const double *__restrict__ V,
               double *__restrict__ F, double *__restrict__ C) {
  extern __shared__ double sm[];
  double *P = sm, *diag = sm + (size_t)d * (kCholPanel + 1);  // panel rows padded by one
  constexpr int ldp = kCholPanel + 1;
  const double *A = blockIdx.x ? V : W;
  double *L = blockIdx.x ? C : F;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nw = blockDim.x >> 5;
  for (int e = tid; e < d * d; e += blockDim.x) {
    const int i = e / d, j = e - i * d;
    L[e] = j <= i ? A[e] : 0.0;
    if (i == j) diag[i] = A[e];
  }
  __syncthreads();
  for (int kb = 0; kb < d; kb += kCholPanel) {
    const int nb = min(kCholPanel, d - kb);
    for (int e = tid; e < (d - kb) * nb; e += blockDim.x) {
      const int i = e / nb, q = e - i * nb;
      P[i * ldp + q] = L[(size_t)(kb + i) * d + kb + q];
    }
    __syncthreads();
    for (int q = 0; q < nb; ++q) {
      const double piv = P[q * ldp + q];
      const bool has = piv > 4.4e-16 * diag[kb + q];
      const double root = has ? sqrt(piv) : 0.0, inv = has ? 1.0 / root : 0.0;
      __syncthreads();  // everyone has read the pivot
      for (int i = q + tid; i < d - kb; i += blockDim.x)
        P[i * ldp + q] = i == q ? root : P[i * ldp + q] * inv;
      __syncthreads();
      for (int i = q + 1 + tid; i < d - kb; i += blockDim.x) {
        const double l = P[i * ldp + q];
        for (int c = q + 1; c < nb && c <= i; ++c) P[i * ldp + c] -= l * P[c * ldp + q];
      }
      __syncthreads();
    }
    for (int e = tid; e < (d - kb) * nb; e += blockDim.x) {
      const int i = e / nb, q = e - i * nb;
      if (q <= i) L[(size_t)(kb + i) * d + kb + q] = P[i * ldp + q];
    }
    const int j1 = nb;  // trailing rows and columns, relative to kb
    for (int i = j1 + warp; i < d - kb; i += nw) {
      double *row = L + (size_t)(kb + i) * d + kb;
      for (int j = j1 + lane; j <= i; j += 32) {
        double s = row[j];
        for (int q = 0; q < nb; ++q) s -= P[i * ldp + q] * P[j * ldp + q];
        row[j] = s;
      }
    }
    __syncthreads();
  }
}

// Column j of C^T F at G + j d: (C^T F)(i, j) = sum_{k >= max(i, j)} C(k, i) F(k, j)
__global__ void k_ct_f(int d, const double *__restrict__ C, const double *__restrict__ F,
                       double *__restrict__ G) {
  for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < d * d; e += gridDim.x * blockDim.x) {
    const int j = e / d, i = e - j * d;
    double s = 0.0;
#pragma unroll 4
    for (int k = max(i, j); k < d; ++k) s += C[(size_t)k * d + i] * F[(size_t)k * d + j];
    G[e] = s;
  }
}

__global__ void k_eye(int d, double *__restrict__ Q) {
  for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < d * d; e += gridDim.x * blockDim.x)
    Q[e] = (e / d == e % d) ? 1.0 : 0.0;
}

// R_w = Tr W + Tr V - 2 sum_i sig_i; out = {R_w, Tr W, Tr V}
__global__ void k_mpsrf_final(int d, const double *__restrict__ W, const double *__restrict__ V,
                              const double *__restrict__ sig, double *__restrict__ out) {
  __shared__ double red[40];
  double tw = 0.0, tv = 0.0, sq = 0.0;
  for (int i = threadIdx.x; i < d; i += blockDim.x) {
    tw += W[(size_t)i * d + i];
    tv += V[(size_t)i * d + i];
    sq += sig[i];
  }
  tw = block_sum(tw, red);
  tv = block_sum(tv, red);
  sq = block_sum(sq, red);
  if (threadIdx.x == 0) {
    out[0] = tw + tv - 2.0 * sq;
    out[1] = tw;
    out[2] = tv;
  }
}

// Limits of the kernels' dynamic shared memory are set to the same value whatever
// the call's size, so that contexts of several host threads cannot lower one
// another's between the setting and the launch.
constexpr int kStagedSmem = 200 * 1024;  // also the two blocks of columns of a Jacobi CTA

int grid_for(size_t n) { return (int)std::min<size_t>((n + 255) / 256, 152 * 8) + 0; }

// out[i r + q] = normal q of Philox (seed, stream, step 0, "chain" i), i < n
__global__ void k_normals(uint64_t seed, uint32_t stream, int n, int r, double *__restrict__ out) {
  const int nb = (r + 3) / 4;
  for (size_t e = blockIdx.x * (size_t)blockDim.x + threadIdx.x; e < (size_t)n * nb;
       e += (size_t)gridDim.x * blockDim.x) {
    const int i = (int)(e / nb), blk = (int)(e - (size_t)i * nb);
    double z[4];
    normals4_f64(philox_block(seed, stream, 0, (uint32_t)i, blk), z);
    for (int q = 0; q < 4; ++q)
      if (4 * blk + q < r) out[(size_t)i * r + 4 * blk + q] = z[q];
  }
}

// dst[c rows + i] = scale * src[i ld + c]  (rows x cols -> cols x rows, FP64)
template <typename T>
__global__ void k_transpose(int rows, int cols, const T *__restrict__ src, int ld, double scale,
                            double *__restrict__ dst) {
  for (size_t e = blockIdx.x * (size_t)blockDim.x + threadIdx.x; e < (size_t)rows * cols;
       e += (size_t)gridDim.x * blockDim.x) {
    const size_t c = e / rows, i = e - c * rows;
    dst[e] = scale * (double)src[i * ld + c];
  }
}

}  // namespace

cudaError_t launch_diag_record(int n_c, int d, const void *src, int src_f32, int ld_src,
                               double *traj, int max_s, int j, cudaStream_t st) {
  const size_t n = (size_t)n_c * d;
  if (n == 0) return cudaSuccess;
  if (src_f32)
    k_diag_record<float><<<grid_for(n), 256, 0, st>>>(n_c, d, (const float *)src, ld_src, traj,
                                                      max_s, j);
  else
    k_diag_record<double><<<grid_for(n), 256, 0, st>>>(n_c, d, (const double *)src, ld_src,
                                                       traj, max_s, j);
  return cudaGetLastError();
}

cudaError_t launch_diag_ess(int d, int n_c, int n_s, const double *traj, int max_s, double *means,
                            double *ess, double *sqjump, cudaStream_t st) {
  if (d <= 0) return cudaSuccess;
  if (n_c < 2 || n_s < 2 || (size_t)n_c * 8 > 48 * 1024) return cudaErrorInvalidValue;
  // the centred samples in shared memory where they fit (two CTAs an SM up to 14000)
  const size_t staged = ((size_t)n_c * n_s + n_c) * 8;
  const bool fits = staged <= kStagedSmem;
  auto kernel = fits ? k_diag_ess<true> : k_diag_ess<false>;
  // More CTAs for a degree of freedom: the slowest one, which may run all n_s lags,
  // sets the time, but each CTA of a cluster reads all samples and a pass forms 8 lags
  // in each, which costs where few lags are needed and the CTAs take several
  // rounds of the chip (two an SM, 304).  Eight in one round, four in up to three, two in
  // up to seven.  Clusters of 1 / 2 / 4 / 8, us, 10 chains of 1000 samples, correlation 0.5,
  // 0.9, 0.99: d = 38 137 92 110 171, 466 266 180 190, 2413 1309 1016 798; d = 100 158 173 212
  // 316, 606 493 366 413, 2414 1778 1477 1606; d = 200 241 219 333 616, 862 562 558 720, 3358 2632
  // 2585 2956; d = 400 338 358 620 1151, 1192 832 961 1403, 4949 4496 4761 5737; d = 1000 576 762
  // 1436 2821, 3428 2599 2690 3486, 10259 10043 11194 13907; d = 2000 1047 1502, 3630 3523, 18545
  // 18952.
  constexpr int kRound = 304;
  int cs = d * 8 <= kRound ? kEssMaxCluster : d * 4 <= 3 * kRound ? 4 : d * 2 <= 7 * kRound ? 2 : 1;
  while (cs > 1 && n_s < 64 * cs) cs /= 2;
  cudaLaunchAttribute attr = {};
  attr.id = cudaLaunchAttributeClusterDimension;
  attr.val.clusterDim.x = cs;
  attr.val.clusterDim.y = attr.val.clusterDim.z = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(d * cs);
  cfg.blockDim = dim3(kEssThreads);
  cfg.dynamicSmemBytes = fits ? staged : (size_t)n_c * 8;
  cfg.stream = st;
  cfg.attrs = &attr;
  cfg.numAttrs = 1;
  cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       fits ? kStagedSmem : 48 * 1024);
  if (e != cudaSuccess) return e;
  return cudaLaunchKernelEx(&cfg, kernel, n_c, n_s, traj, max_s, means, ess, sqjump);
}

cudaError_t launch_diag_center(int d, int n_c, int n_s, const double *traj, int max_s,
                               const double *means, double *Xc, double *Mc, cudaStream_t st) {
  k_diag_center<<<grid_for((size_t)d * n_c * n_s), 256, 0, st>>>(d, n_c, n_s, traj, max_s, means,
                                                                 Xc, Mc);
  return cudaGetLastError();
}

cudaError_t launch_diag_wv(int d, int n_c, int n_s, const double *Wr, const double *Br, double *W,
                           double *V, cudaStream_t st) {
  k_diag_wv<<<grid_for((size_t)d * d), 256, 0, st>>>(d, n_c, n_s, Wr, Br, W, V);
  return cudaGetLastError();
}

// Y = A^T / |A|_F and X = Y^T, At = A^T row-major (one CTA: |A|_F first)
__global__ void __launch_bounds__(1024)
    k_ns_start(int d, const double *__restrict__ At, double *__restrict__ Y,
               double *__restrict__ X) {
  __shared__ double red[40];
  double s = 0.0;
  for (int e = threadIdx.x; e < d * d; e += blockDim.x) s += At[e] * At[e];
  s = block_sum(s, red);
  const double scale = 1.0 / sqrt(s);
  for (int e = threadIdx.x; e < d * d; e += blockDim.x) {
    const int i = e / d, j = e - i * d;
    const double v = At[e] * scale;
    Y[e] = v;
    X[(size_t)j * d + i] = v;
  }
}

// out[i] = sum_k Y[i][k] At[i][k]: a warp per row
__global__ void k_row_dots(int d, const double *__restrict__ Y, const double *__restrict__ At,
                           double *__restrict__ out) {
  const int i = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
  if (i >= d) return;
  double s = 0.0;
  for (int k = lane; k < d; k += 32) s += Y[(size_t)i * d + k] * At[(size_t)i * d + k];
  s = warp_sum(s);
  if (lane == 0) out[i] = s;
}

cudaError_t launch_ns_start(int d, const double *At, double *Y, double *X, cudaStream_t st) {
  k_ns_start<<<1, 1024, 0, st>>>(d, At, Y, X);
  return cudaGetLastError();
}

cudaError_t launch_row_dots(int d, const double *Y, const double *At, double *out,
                            cudaStream_t st) {
  k_row_dots<<<(d + 7) / 8, 256, 0, st>>>(d, Y, At, out);
  return cudaGetLastError();
}

cudaError_t launch_eye(int d, double *Q, cudaStream_t st) {
  k_eye<<<grid_for((size_t)d * d), 256, 0, st>>>(d, Q);
  return cudaGetLastError();
}

// Blocks of 1, 2 or 4 columns: the fewest that leave at most 152 block pairs, so
// that a round is one wave of CTAs.
static int jacobi_block(int d) { return d <= 304 ? 1 : d <= 608 ? 2 : 4; }

int jacobi_rounds(int d) {
  const int nb = (d + jacobi_block(d) - 1) / jacobi_block(d);
  return std::max(1, nb + (nb & 1) - 1);
}

template <int kB>
static cudaError_t jacobi_round(int d, int rnd, double *G, double *Q, int *rotated,
                                cudaStream_t st) {
  const int nb = (d + kB - 1) / kB, n = nb + (nb & 1);
  const size_t smem = (size_t)2 * kB * d * sizeof(double) * (Q ? 2 : 1);
  if (smem > 48 * 1024) {
    cudaError_t e = cudaFuncSetAttribute(k_jacobi_round<kB>,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize, kStagedSmem);
    if (e != cudaSuccess) return e;
  }
  k_jacobi_round<kB><<<n / 2, kB * kPairThreads, smem, st>>>(d, nb, rnd, G, Q, rotated);
  return cudaGetLastError();
}

cudaError_t launch_jacobi_round(int d, int rnd, double *G, double *Q, int *rotated,
                                cudaStream_t st) {
  if (d <= 1) return cudaSuccess;
  switch (jacobi_block(d)) {
    case 1: return jacobi_round<1>(d, rnd, G, Q, rotated, st);
    case 2: return jacobi_round<2>(d, rnd, G, Q, rotated, st);
    default: return jacobi_round<4>(d, rnd, G, Q, rotated, st);
  }
}

cudaError_t launch_col_norms(int d, const double *G, double *sig, cudaStream_t st) {
  k_col_norms<<<(d + 7) / 8, 256, 0, st>>>(d, G, sig);
  return cudaGetLastError();
}

cudaError_t launch_psd_chol(int d, const double *W, const double *V, double *F, double *C,
                            cudaStream_t st) {
  const size_t smem = (size_t)d * (kCholPanel + 2) * sizeof(double);
  cudaError_t e = cudaFuncSetAttribute(k_psd_chol, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       kStagedSmem);
  if (e != cudaSuccess) return e;
  k_psd_chol<<<2, kCholThreads, smem, st>>>(d, W, V, F, C);
  return cudaGetLastError();
}

cudaError_t launch_ct_f(int d, const double *C, const double *F, double *G, cudaStream_t st) {
  k_ct_f<<<grid_for((size_t)d * d), 256, 0, st>>>(d, C, F, G);
  return cudaGetLastError();
}

cudaError_t launch_normals(uint64_t seed, uint32_t stream, int n, int r, double *out,
                           cudaStream_t st) {
  if (n <= 0 || r <= 0) return cudaSuccess;
  k_normals<<<grid_for((size_t)n * ((r + 3) / 4)), 256, 0, st>>>(seed, stream, n, r, out);
  return cudaGetLastError();
}

cudaError_t launch_transpose(int rows, int cols, const void *src, int src_f32, int ld,
                             double scale, double *dst, cudaStream_t st) {
  const size_t n = (size_t)rows * cols;
  if (n == 0) return cudaSuccess;
  if (src_f32)
    k_transpose<float><<<grid_for(n), 256, 0, st>>>(rows, cols, (const float *)src, ld, scale, dst);
  else
    k_transpose<double><<<grid_for(n), 256, 0, st>>>(rows, cols, (const double *)src, ld, scale,
                                                     dst);
  return cudaGetLastError();
}

cudaError_t launch_mpsrf_final(int d, const double *W, const double *V, const double *sig,
                               double *out, cudaStream_t st) {
  k_mpsrf_final<<<1, 256, 0, st>>>(d, W, V, sig, out);
  return cudaGetLastError();
}

}  // namespace dino
