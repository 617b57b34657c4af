// Per-chain reduced-space kernels of the surrogate mMALA step, in FP64.
//
// Besides m_r, g, Phi and half log det(I + H), each chain keeps one factor
// slot: the packed lower Cholesky factor (row-major, entry (i, j), j <= i, at
// i (i+1)/2 + j) of I + H bordered below by the row (m_r + g)^T, so that its
// row r holds t = L^-1 (m_r + g); then p = L^T m_r.
//
//   k_propose_warp / k_propose
//               reduced proposal (eq:reduced_space_sampling in Cholesky form)
//               m_r^dag = mu + sqrt(1-s^2) L^-T xi,
//               mu = m_r - (1-s) (I+H)^-1 (m_r + g) = m_r - (1-s) L^-T t,
//               both from one two-column back substitution, and
//               log rho_{0,r}(m_r, m_r^dag) with the geometry at m_r (Sec. 5.4).
//   k_geometry  misfit, gradient, H = J^T J / noise_var + I and the bordered
//               factor at m_r^dag (Algorithm 1), log rho_{0,r}(m_r^dag, m_r),
//               log rho_r^(1) (eq:da_dino_trr_1), the accept test and the
//               state update.
//
// With L L^T = I + H, w = H x - g, mhat = (z - s x) / sqrt(1-s^2) for a move
// x -> z, t = L^-1 (x + g) and p = L^T x (exact in real arithmetic):
//   w^T (I+H)^-1 w = |p - t|^2,
//   mhat^T w = (L^T mhat)^T p - mhat^T (x + g),
//   mhat^T H mhat = |L^T mhat|^2 - |mhat|^2,
// so log rho_0 needs no pass over the factor beyond L^T mhat, and that one
// is known in closed form on both sides: on the forward side
// L^T mhat = ((1-s)(p - t) + sqrt(1-s^2) xi) / sqrt(1-s^2); on the reverse
// side the geometry kernel forms L^T z and L^T x from the factor it holds.
//
//   k_gram_f32  on the tensor-core path, I + J^T J / noise_var in double-float
//               from the FP32 Jacobian, into the slot that k_geometry factors.
//
// The FP64 pipe bounds the FP64 instantiations (1/64 of the FP32 rate on
// GB300), so the Cholesky is blocked (8-column panels with lookahead) to keep
// the FP64 units fed from shared memory; the tensor-core path factors in
// double-float on the FP32 pipe.
#include <algorithm>

#include "chol_mma.cuh"
#include "pdl.cuh"

namespace dino {
namespace {

constexpr int kThreads = 512;

// [x, z] <- L^-T [x, z] (back substitution on the upper factor L^T, read from
// global memory): per 32-row diagonal block, staged in shared memory (blk, 32 x
// 33) with the block's rows of the update loads in flight, warp 0 solves for x
// and warp 1 for z; then both take the update from one read of the rows.  (One
// right-hand side after the other, the block's entries read by the solving
// warp: 1.10 ms for 512 chains at r = 400; 0.37 ms here.)
__device__ void cta_upper_solve2(const double *Ls, const double *inv, int r, double *x, double *z,
                                 double *blk) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  for (int jb = ((r - 1) / 32) * 32; jb >= 0; jb -= 32) {
    const int nb = min(32, r - jb);
    for (int e = threadIdx.x; e < 32 * 32; e += blockDim.x) {
      const int k = e >> 5, i = e & 31;
      if (k < nb && i <= k) blk[k * 33 + i] = Ls[tri(jb + k) + jb + i];
    }
    __syncthreads();
    if (warp < 2) {
      double *v = warp == 0 ? x : z;
      double xl = lane < nb ? v[jb + lane] : 0.0;
      for (int k = nb - 1; k >= 0; --k) {
        const double yk = __shfl_sync(kFull, xl, k) * inv[jb + k];
        if (lane == k)
          xl = yk;
        else if (lane < k)
          xl -= blk[k * 33 + lane] * yk;
      }
      if (lane < nb) v[jb + lane] = xl;
    }
    __syncthreads();
    for (int i = threadIdx.x; i < jb; i += blockDim.x) {
      double ax = x[i], az = z[i];
#pragma unroll 8
      for (int k = 0; k < nb; ++k) {
        const double l = Ls[tri(jb + k) + i];
        ax -= l * x[jb + k];
        az -= l * z[jb + k];
      }
      x[i] = ax;
      z[i] = az;
    }
    __syncthreads();
  }
}

// y1 = L^T x1 and, when `two`, y2 = L^T x2 over the leading r rows of L
// (y_j = sum_{j <= i < r} L_ij x_i): column j by thread j, rows in order.
template <class A>
__device__ void cta_upper_matvec2(const typename A::T *Ls, int r, const typename A::T *x1,
                                  const typename A::T *x2, double *y1, double *y2, bool two) {
  using E = typename A::T;
  for (int j = threadIdx.x; j < r; j += blockDim.x) {
    typename A::Acc a1 = A::begin(E{}), a2 = A::begin(E{});
#pragma unroll 4
    for (int i = j; i < r; ++i) {
      const E l = Ls[tri(i) + j];
      A::sub(a1, l, A::neg(x1[i]));
      if (two) A::sub(a2, l, A::neg(x2[i]));
    }
    y1[j] = A::to(A::end(a1));
    if (two) y2[j] = A::to(A::end(a2));
  }
  __syncthreads();
}

// Shared-memory layout in doubles:
//   Ls[slot_stride(r)] inv[r+1] seven work vectors[r] res[dy] red[kRed] flag[1] | J chunk
// (red[100..102] hold the Cholesky's six work counters)
// (one double, or one double-float pair, per element).  With `global` the
// factor lives in its global slot and takes no shared memory.
struct Layout {
  size_t Ls, inv, v0, res, red, flag, tail;
  // lean: without the last four vectors (vp, vq, be, ae)
  __host__ __device__ Layout(int r, int dy, bool global, bool lean = false) {
    Ls = 0;
    inv = global ? 0 : slot_stride(r);
    v0 = inv + r + 1;
    res = v0 + (lean ? 3 : 7) * (size_t)r;
    red = res + dy;
    flag = red + kRed;
    tail = (flag + 1 + 1) & ~(size_t)1;  // 16-byte aligned start of the J chunk
  }
};

// One CTA per chain, for r beyond the register-resident warp kernel: the
// factor is read from its global slot (L2-resident while the chain is
// processed), the vectors live in shared memory.
__global__ void __launch_bounds__(kThreads) k_propose(ReducedArgs a) {
  pdl_begin();
  extern __shared__ __align__(16) double sm[];
  __shared__ double blk[32 * 33];
  const int c = blockIdx.x, r = a.r;
  const Layout lay(r, 0, true);
  const double *Ls = a.L + (size_t)a.cur[c] * a.L_slot + (size_t)c * slot_stride(r);
  const double *tv = Ls + tri(r), *pv = Ls + tri(r + 1);
  double *inv = sm + lay.inv;
  double *va = sm + lay.v0, *vg = va + r, *vx = vg + r, *z1 = vx + r, *z2 = z1 + r;
  double *red = sm + lay.red;
  for (int i = threadIdx.x; i < r; i += blockDim.x) {
    va[i] = a.mr[(size_t)c * r + i];
    vg[i] = a.g[(size_t)c * r + i];
    z1[i] = tv[i];
    inv[i] = 1.0 / Ls[tri(i) + i];
  }
  const uint32_t chain = (uint32_t)(a.id_base + (uint64_t)c);
  for (int blk = threadIdx.x; blk < (r + 3) / 4; blk += blockDim.x) {
    double n4[4];
    if (a.ext_xi) {
      for (int q = 0; q < 4; ++q)
        n4[q] = 4 * blk + q < r ? a.ext_xi[(size_t)c * r + 4 * blk + q] : 0.0;
    } else {
      normals4_f64(philox_block(a.seed, STREAM_XI, a.step, chain, blk), n4);
    }
    for (int q = 0; q < 4; ++q)
      if (4 * blk + q < r) vx[4 * blk + q] = z2[4 * blk + q] = n4[q];
  }
  __syncthreads();
  // z1 = L^-T t = (I+H)^-1 (a + g), z2 = L^-T xi
  cta_upper_solve2(Ls, inv, r, z1, z2, blk);
  const double s = a.s, cs = sqrt(1.0 - s * s);
  double t1 = 0.0, t2 = 0.0, t3 = 0.0;
  for (int i = threadIdx.x; i < r; i += blockDim.x) {
    const double mu = va[i] - (1.0 - s) * z1[i];
    const double b = mu + cs * z2[i];
    a.mu[(size_t)c * r + i] = mu;
    a.b[(size_t)c * r + i] = b;
    if (a.b_bf16)
      split_bf16_store(b, a.b_bf16 + (size_t)c * a.b_ld + i, a.b_plane, a.b_slices);
    const double p = pv[i], d = p - tv[i];               // d = L^-1 w
    const double mh = (b - s * va[i]) / cs;               // mhat
    const double u = ((1.0 - s) * d + cs * vx[i]) / cs;   // L^T mhat
    t1 += d * d;
    t2 += u * p - mh * (va[i] + vg[i]);
    t3 += u * u - mh * mh;
  }
  block_sum3(t1, t2, t3, red);
  if (threadIdx.x == 0)
    a.lq_fwd[c] = -a.dt / 8.0 * t1 + sqrt(a.dt) / 2.0 * t2 + a.hld[c] - 0.5 * t3;
}

// ---------------------------------------------------------------------------
// Warp-per-chain reduced proposal.  Each warp owns one chain; vectors live in
// registers distributed over lanes (element i in lane i % 32, slot i / 32) and
// L is read from global memory (L1/L2), so an SM keeps 16 chains in flight
// and the serial parts of the back substitution of one chain overlap with the
// FP64 work of the others.

constexpr int kPropWarps = 4;  // chains per CTA

// [x, z] <- L^-T [x, z]: back substitution with two right-hand sides, so the
// factor is read once for both.  Column k of a 32-row diagonal block is
// broadcast by shuffles; the blocks above it take the update with lanes
// reading contiguous parts of row k.
template <int S>
__device__ __forceinline__ void warp_upper_solve2(const double *__restrict__ L, int r,
                                                  const double (&invd)[S], double (&x)[S],
                                                  double (&z)[S]) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int b = S - 1; b >= 0; --b) {
    if (32 * b >= r) continue;
    const int jb = 32 * b, nb = min(32, r - jb);
    double xb = x[b], zb = z[b];
    const double ib = invd[b];
    for (int k = nb - 1; k >= 0; --k) {
      const double d = __shfl_sync(kFull, ib, k);
      const double xk = __shfl_sync(kFull, xb, k) * d;
      const double zk = __shfl_sync(kFull, zb, k) * d;
      if (lane == k) {
        xb = xk;
        zb = zk;
      } else if (lane < k) {
        const double l = L[tri(jb + k) + jb + lane];
        xb -= l * xk;
        zb -= l * zk;
      }
    }
    x[b] = xb;
    z[b] = zb;
    if (b == 0) continue;
    for (int k = 0; k < nb; ++k) {
      const double xk = __shfl_sync(kFull, xb, k);
      const double zk = __shfl_sync(kFull, zb, k);
      const double *row = L + tri(jb + k);
#pragma unroll
      for (int b2 = 0; b2 < S; ++b2) {
        if (b2 < b) {
          const double l = row[32 * b2 + lane];
          x[b2] -= l * xk;
          z[b2] -= l * zk;
        }
      }
    }
  }
}

template <int S>
__global__ void __launch_bounds__(32 * kPropWarps) k_propose_warp(ReducedArgs a) {
  pdl_begin();
  __shared__ double xi_s[kPropWarps][32 * S];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int c = blockIdx.x * kPropWarps + w;
  if (c >= a.C) return;  // whole warp
  const int r = a.r;
  const double *L = a.L + (size_t)a.cur[c] * a.L_slot + (size_t)c * slot_stride(r);
  const double *tv = L + tri(r), *pv = L + tri(r + 1);
  const uint32_t chain = (uint32_t)(a.id_base + (uint64_t)c);
  for (int blk = lane; blk < (r + 3) / 4; blk += 32) {
    double n4[4];
    if (a.ext_xi) {
      for (int q = 0; q < 4; ++q)
        n4[q] = 4 * blk + q < r ? a.ext_xi[(size_t)c * r + 4 * blk + q] : 0.0;
    } else {
      normals4_f64(philox_block(a.seed, STREAM_XI, a.step, chain, blk), n4);
    }
    for (int q = 0; q < 4; ++q)
      if (4 * blk + q < r) xi_s[w][4 * blk + q] = n4[q];
  }
  __syncwarp();
  double va[S], vg[S], vt[S], vx[S], z1[S], z2[S], invd[S];
#pragma unroll
  for (int s = 0; s < S; ++s) {
    const int i = 32 * s + lane;
    const bool in = i < r;
    va[s] = in ? a.mr[(size_t)c * r + i] : 0.0;
    vg[s] = in ? a.g[(size_t)c * r + i] : 0.0;
    vt[s] = in ? tv[i] : 0.0;
    vx[s] = in ? xi_s[w][i] : 0.0;
    invd[s] = in ? 1.0 / L[tri(i) + i] : 0.0;
    z1[s] = vt[s];
    z2[s] = vx[s];
  }
  warp_upper_solve2<S>(L, r, invd, z1, z2);  // z1 = (I+H)^-1 (a + g), z2 = L^-T xi
  const double s_ = a.s, cs = sqrt(1.0 - s_ * s_);
  double t1 = 0.0, t2 = 0.0, t3 = 0.0;
#pragma unroll
  for (int s = 0; s < S; ++s) {
    const int i = 32 * s + lane;
    if (i < r) {
      const double mu = va[s] - (1.0 - s_) * z1[s];
      const double b = mu + cs * z2[s];
      a.mu[(size_t)c * r + i] = mu;
      a.b[(size_t)c * r + i] = b;
      if (a.b_bf16)
        split_bf16_store(b, a.b_bf16 + (size_t)c * a.b_ld + i, a.b_plane, a.b_slices);
      const double p = pv[i], d = p - vt[s];                 // d = L^-1 w
      const double mh = (b - s_ * va[s]) / cs;                // mhat
      const double u = ((1.0 - s_) * d + cs * vx[s]) / cs;    // L^T mhat
      t1 += d * d;
      t2 += u * p - mh * (va[s] + vg[s]);
      t3 += u * u - mh * mh;
    }
  }
  t1 = warp_sum(t1);
  t2 = warp_sum(t2);
  t3 = warp_sum(t3);
  if (lane == 0)
    a.lq_fwd[c] = -a.dt / 8.0 * t1 + sqrt(a.dt) / 2.0 * t2 + a.hld[c] - 0.5 * t3;
}

// I + J^T J / noise_var of every chain in double-float, packed (tri(r) entries)
// at the start of the slot that k_geometry factors (the spare one in mode 1).
//
// A CTA of 128 threads takes a 64 x 64 block of one chain's lower triangle,
// 8 x 4 entries a thread; J (d_y x r, FP32) streams through two buffers of 32
// rows x (64 + 64) columns by asynchronous copies.  The sums are FP32
// multiply-adds over kGramFlush rows, added into double-float sums in
// registers, so that the FP32 rounding error grows with kGramFlush rather
// than with d_y.  What bounds it: FP32 multiply-adds, 32 for three 16-byte
// shared-memory loads.  Inside k_geometry (one CTA per chain, 4 x 4 tiles in
// several rounds over J, the sums flushed to the factor in shared or global
// memory, and the registers of the tiles halving the warps of the
// factorisation) both together took 9.85 ms for 512 chains at r = d_y = 400 and
// 2.95 ms for 4096 at r = 128, d_y = 200; apart, 1.40 + 5.70 ms and 0.65 + 2.02 ms
// (the factorisation 3.40 and 1.52 ms since its updates run on the tensor cores).
constexpr int kGramB = 64, kGramK = 32, kGramThreads = 128;
constexpr int kGramFlush = 64;  // rows per FP32 partial sum

__global__ void __launch_bounds__(kGramThreads, 4) k_gram_f32(ReducedArgs a, int mode) {
  pdl_begin();
  __shared__ __align__(16) float stage[2][kGramK][2 * kGramB];
  const int c = blockIdx.y, r = a.r, dy = a.d_y;
  int bi, bj;  // block row and column, bj <= bi
  tri_pos(blockIdx.x, bi, bj);
  const float *J = reinterpret_cast<const float *>(a.J) + (size_t)c * dy * r;
  const int slot = mode == 0 ? a.cur[c] : 1 - a.cur[c];
  float2 *M = reinterpret_cast<float2 *>(a.L + (size_t)slot * a.L_slot +
                                         (size_t)c * slot_stride(r));
  const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
  const bool vec = (r & 3) == 0;  // rows of J start on 16 bytes
  const int nch = (dy + kGramK - 1) / kGramK;
  auto issue = [&](int ch) {
    float(*dst)[2 * kGramB] = stage[ch & 1];
    const int k0 = ch * kGramK;
    if (vec) {
      for (int e = tid; e < kGramK * (2 * kGramB / 4); e += kGramThreads) {
        const int k = e / (2 * kGramB / 4), q = 4 * (e % (2 * kGramB / 4));
        const int col = q < kGramB ? bi * kGramB + q : bj * kGramB + q - kGramB;
        const bool in = k0 + k < dy && col < r;
        cp_async16(&dst[k][q], J + (in ? (size_t)(k0 + k) * r + col : 0), in ? 16 : 0);
      }
    } else {
      for (int e = tid; e < kGramK * 2 * kGramB; e += kGramThreads) {
        const int k = e / (2 * kGramB), q = e % (2 * kGramB);
        const int col = q < kGramB ? bi * kGramB + q : bj * kGramB + q - kGramB;
        const bool in = k0 + k < dy && col < r;
        cp_async4(&dst[k][q], J + (in ? (size_t)(k0 + k) * r + col : 0), in ? 4 : 0);
      }
    }
    cp_async_commit();
  };
  float acc[8][4];
  float2 sum[8][4];
#pragma unroll
  for (int p = 0; p < 8; ++p)
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      acc[p][q] = 0.0f;
      sum[p][q] = make_float2(0.0f, 0.0f);
    }
  issue(0);
  for (int ch = 0; ch < nch; ++ch) {
    if (ch + 1 < nch)
      issue(ch + 1);
    else
      cp_async_commit();
    cp_async_wait<1>();
    __syncthreads();
    const float(*x)[2 * kGramB] = stage[ch & 1];
    const int nr = min(kGramK, dy - ch * kGramK);
#pragma unroll 4
    for (int k = 0; k < nr; ++k) {
      const float4 x0 = *reinterpret_cast<const float4 *>(&x[k][8 * ty]);
      const float4 x1 = *reinterpret_cast<const float4 *>(&x[k][8 * ty + 4]);
      const float4 y = *reinterpret_cast<const float4 *>(&x[k][kGramB + 4 * tx]);
      const float xa[8] = {x0.x, x0.y, x0.z, x0.w, x1.x, x1.y, x1.z, x1.w};
      const float ya[4] = {y.x, y.y, y.z, y.w};
#pragma unroll
      for (int p = 0; p < 8; ++p)
#pragma unroll
        for (int q = 0; q < 4; ++q) acc[p][q] = fmaf(xa[p], ya[q], acc[p][q]);
    }
    __syncthreads();
    const int done = ch * kGramK + nr;
    if (done % kGramFlush == 0 || done >= dy) {
#pragma unroll
      for (int p = 0; p < 8; ++p)
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const float2 v = make_float2(acc[p][q], 0.0f);
          sum[p][q] = done <= kGramFlush ? v : DF::add(sum[p][q], v);
          acc[p][q] = 0.0f;
        }
    }
  }
  const double inv_nv = 1.0 / a.noise_var;
  const float nh = __double2float_rn(inv_nv), nl = __double2float_rn(inv_nv - (double)nh);
#pragma unroll
  for (int p = 0; p < 8; ++p) {
    const int i = bi * kGramB + 8 * ty + p;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int j = bj * kGramB + 4 * tx + q;
      if (i < r && j <= i) {
        float2 v = DF::mul(sum[p][q], make_float2(nh, nl));
        if (i == j) v = DF::add(make_float2(1.0f, 0.0f), v);
        M[tri(i) + j] = v;
      }
    }
  }
}

// One CTA per chain at the point b.  G = false: the factor is built in shared
// memory; G = true (large r): directly in the other global slot.
//
// The matrix factored is I + H bordered by the row v^T = (b + g_b)^T with
// pivot 1 + |v|^2.  Its factor's leading block is L_b and its last row is
// t_b^T = (L_b^-1 v)^T; the last pivot stays >= 1 since |L_b^-1 v| <= |v|
// when I + H >= I.  With p_b = L_b^T b and q_b = L_b^T a the reverse density
// takes L_b^T mhat = (q_b - s p_b) / sqrt(1-s^2) for mhat = (a - s b) / sqrt(1-s^2).
//
// Mode 0 makes b the chain state (slot cur[c]).  Mode 1 evaluates
// log rho_r^(1) against the current state a, takes the accept test and moves
// an accepted chain to b: its factor (stored only then, into the other slot,
// which becomes current; factors in global memory and k_gram_f32 work in that
// slot every time) and its state vectors.  The complement
// coefficient b - s a is written for every chain.
// The FP32-Jacobian instantiations find I + H in the slot (k_gram_f32).  kFac: the
// factorisation.  The blocked ones (FP32 Jacobian) keep their digits or panel at sm +
// panel; the plain one has 64 registers a thread with an FP32 Jacobian, 32 warps an
// SM where shared memory allows.
enum Factor { kPlain, kMma, kPanels };  // 8-column panels; chol_mma.cuh; cta_cholesky_global
template <typename TJ, bool G, int NT, Factor kFac>
__global__ void __launch_bounds__(NT, sizeof(TJ) == 4 && kFac == kPlain
                                          ? 1024 / NT
                                          : (NT <= 128 ? 4 : (NT <= 256 ? 2 : 1)))
    k_geometry(ReducedArgs a, int mode, int panel) {
  pdl_begin();
  // FP32 Jacobian (tensor-core path): double-float Cholesky; FP64 Jacobian: FP64
  using A = std::conditional_t<sizeof(TJ) == 4, DF, F64>;
  using E = typename A::T;
  static_assert(sizeof(E) == sizeof(double), "one factor element per double of the slot");
  extern __shared__ __align__(16) double sm[];
  const int c = blockIdx.x, r = a.r, dy = a.d_y;
  const size_t ldL = slot_stride(r), lsz = tri_size(r + 1);
  static_assert(kFac == kPlain || sizeof(TJ) == 4, "FP64 factors are plain");
  constexpr bool kLean = G && kFac != kPlain;
  const Layout lay(r, dy, G, kLean);
  const int slot = mode == 0 ? a.cur[c] : 1 - a.cur[c];
  double *Lg = a.L + (size_t)slot * a.L_slot + (size_t)c * ldL;
  E *Ls = reinterpret_cast<E *>(G ? Lg : sm + lay.Ls);
  E *inv = reinterpret_cast<E *>(sm + lay.inv);
  double *vb = sm + lay.v0, *vg = vb + r, *va = vg + r, *vp = va + r, *vq = vp + r;
  E *be = reinterpret_cast<E *>(vq + r), *ae = be + r;  // b and a as factor elements
  E *res = reinterpret_cast<E *>(sm + lay.res);  // f - y as factor elements
  double *red = sm + lay.red;
  int *flag = reinterpret_cast<int *>(sm + lay.flag);
  const TJ *J = reinterpret_cast<const TJ *>(a.J) + (size_t)c * dy * r;
  const TJ *f = reinterpret_cast<const TJ *>(a.f) + (size_t)c * dy;
  const double inv_nv = a.inv_nv;
  // The thread that takes the accept test; in FP64 it draws log u ahead, a chain of
  // FP64 operations that would otherwise follow the last sums (64 chains, r = 16,
  // d_y = 49, with the two changes beside the Gram matrix and the pivots: 47 -> 45 us).
  const bool decider = threadIdx.x == blockDim.x - 1;
  double log_u = 0.0;
  if constexpr (sizeof(TJ) == 8)
    if (mode == 1 && decider) log_u = draw_log_u(a, c);
  if constexpr (sizeof(TJ) == 4 && !G) {  // the packed I + H by 16-byte copies, all in flight
    const size_t ne = tri_size(r);
    const E *src = reinterpret_cast<const E *>(Lg);
    for (size_t q = threadIdx.x; q < ne / 2; q += blockDim.x)
      cp_async16(Ls + 2 * q, src + 2 * q, 16);
    cp_async_commit();
    if (threadIdx.x == 0 && (ne & 1)) Ls[ne - 1] = src[ne - 1];
  }

  for (int i = threadIdx.x; i < r; i += blockDim.x) {
    vb[i] = a.b[(size_t)c * r + i];
    va[i] = mode == 1 ? a.mr[(size_t)c * r + i] : 0.0;
    if constexpr (!kLean) {
      be[i] = A::from(vb[i]);
      ae[i] = A::from(va[i]);
    }
  }
  double ph = 0.0;
  for (int i = threadIdx.x; i < dy; i += blockDim.x) {
    const double rs = (double)f[i] - a.y[i];
    res[i] = A::neg(A::from(rs));
    ph += rs * rs;
  }
  const double phi_b = 0.5 * block_sum(ph, red) * inv_nv;  // includes a barrier
  // g = J^T (f - y) / noise_var: thread per column (coalesced), and where there
  // are threads for it two per column, each half of the rows
  const int half = blockDim.x / 2;
  const bool two = r <= half;
  // the second halves' sums (the lean layout has no vp yet: the panel's place)
  E *ge = reinterpret_cast<E *>(kLean ? sm + panel : vp);
  if (two) {
    const int h = threadIdx.x >= half ? 1 : 0, j = threadIdx.x - h * half;
    typename A::Acc acc = A::begin(E{});
    if (j < r) {
      const int i1 = h ? dy : dy / 2;
      for (int i = h ? dy / 2 : 0; i < i1; ++i)
        A::sub(acc, A::from_j(J[(size_t)i * r + j]), res[i]);
      if (h) ge[j] = A::end(acc);
    }
    __syncthreads();
    if (!h && j < r) vg[j] = A::to(A::add(A::end(acc), ge[j])) * inv_nv;
  } else {
    for (int j = threadIdx.x; j < r; j += blockDim.x) {
      typename A::Acc acc = A::begin(E{});
      for (int i = 0; i < dy; ++i) A::sub(acc, A::from_j(J[(size_t)i * r + j]), res[i]);
      vg[j] = A::to(A::end(acc)) * inv_nv;
    }
  }
  if constexpr (sizeof(TJ) == 4) {
    if constexpr (!G) cp_async_wait<0>();
    __syncthreads();
  } else {
    double *Ld = reinterpret_cast<double *>(Ls);
    form_gram_f64<false>(reinterpret_cast<const double *>(J), dy, r, r, inv_nv, Ld, sm + lay.tail);
    if (dy == 0) {
      for (int e = threadIdx.x; e < tri(r); e += blockDim.x) Ld[e] = 0.0;
      __syncthreads();
      for (int i = threadIdx.x; i < r; i += blockDim.x) Ld[tri(i) + i] = 1.0;
      __syncthreads();
    }
  }
  double vv = 0.0;  // bordered row v = b + g_b (each thread its own j, as for g)
  for (int j = threadIdx.x; j < r; j += blockDim.x) {
    const double v = vb[j] + vg[j];
    Ls[tri(r) + j] = A::from(v);
    vv += v * v;
  }
  vv = block_sum(vv, red);
  if (threadIdx.x == 0) Ls[tri(r) + r] = A::from(1.0 + vv);
  __syncthreads();
  if constexpr (kFac == kPlain)
    cta_cholesky_panels<A>(Ls, inv, r + 1);
  else if constexpr (kFac == kPanels)
    cta_cholesky_global<A>(Ls, inv, r + 1, reinterpret_cast<E *>(sm + panel));
  else if constexpr (G)
    cta_cholesky_global_mma(Ls, inv, r + 1, reinterpret_cast<char *>(sm + panel));
  else
    cta_cholesky_mma(Ls, inv, r + 1, reinterpret_cast<char *>(sm + panel));
  if constexpr (kLean) {  // vp, vq, and b, a as factor elements, over the panel
    __syncthreads();
    vp = sm + panel;
    vq = vp + r;
    be = reinterpret_cast<E *>(vq + r);
    ae = be + r;
    for (int i = threadIdx.x; i < r; i += blockDim.x) {
      be[i] = A::from(vb[i]);
      ae[i] = A::from(va[i]);
    }
  }
  double ld = 0.0;
  for (int i = threadIdx.x; i < r; i += blockDim.x) ld += log(A::to(Ls[tri(i) + i]));
  const double hld_b = block_sum(ld, red);
  cta_upper_matvec2<A>(Ls, r, be, ae, vp, vq, mode == 1);  // p_b = L^T b, q_b = L^T a

  // the slot holds FP64: copied from shared memory, or converted in place
  // (each thread its own elements) when the factor was built in the slot
  auto store_factor = [&]() {
    for (size_t e = threadIdx.x; e < lsz; e += blockDim.x) {
      const double x = A::to(Ls[e]);
      Lg[e] = x;
    }
  };
  if (mode == 0) {
    store_factor();
    for (int i = threadIdx.x; i < r; i += blockDim.x) {
      Lg[lsz + i] = vp[i];
      a.g[(size_t)c * r + i] = vg[i];
      a.mr[(size_t)c * r + i] = vb[i];
    }
    if (threadIdx.x == 0) {
      a.phi[c] = phi_b;
      a.hld[c] = hld_b;
    }
    return;
  }
  const E *tb = Ls + tri(r);
  const double s = a.s, inv_cs = a.inv_cs;
  double t1 = 0.0, t2 = 0.0, t3 = 0.0;
  for (int i = threadIdx.x; i < r; i += blockDim.x) {
    const double d = vp[i] - A::to(tb[i]);         // L_b^-1 w, w = H_b b - g_b
    const double mh = (va[i] - s * vb[i]) * inv_cs;  // mhat for b -> a
    const double u = (vq[i] - s * vp[i]) * inv_cs;   // L_b^T mhat
    t1 += d * d;
    t2 += u * vp[i] - mh * (vb[i] + vg[i]);
    t3 += u * u - mh * mh;
  }
  block_sum3(t1, t2, t3, red);
  double lr = 0.0;
  if (decider) {
    if constexpr (sizeof(TJ) == 4) log_u = draw_log_u(a, c);
    const double lq_rev = -a.dt / 8.0 * t1 + a.sqrt_dt / 2.0 * t2 + hld_b - 0.5 * t3;
    lr = a.phi[c] - phi_b + lq_rev - a.lq_fwd[c];
    *flag = accept_decide(lr, log_u) ? 1 : 0;
  }
  __syncthreads();
  const bool accept = *flag != 0;
  if (decider) accept_record(a, c, lr, log_u, accept, phi_b, hld_b);
  for (int i = threadIdx.x; i < r; i += blockDim.x) {
    a.coef[(size_t)c * r + i] = vb[i] - s * va[i];
    if (accept) {
      if (a.da) {
        a.g_st[(size_t)c * r + i] = vg[i];
      } else {
        a.mr[(size_t)c * r + i] = vb[i];
        a.g[(size_t)c * r + i] = vg[i];
      }
      Lg[lsz + i] = vp[i];
    }
  }
  if (accept) store_factor();
}

}  // namespace

// What k_geometry may take of dynamic shared memory beside its static variables
// (304 bytes).
constexpr size_t kGeoSmem = kSmemLimit - 512;

bool uses_global_factor(int r, int d_y) {
  const Layout lay(r, d_y, false);
  const size_t jc = (size_t)kJChunk * r * sizeof(double);
  return r > kMaxRSmem || lay.tail * sizeof(double) + jc > kGeoSmem;
}

size_t propose_smem_bytes(int r) {
  const Layout lay(r, 0, true);
  return lay.tail * sizeof(double);
}

size_t geometry_smem_bytes(int r, int d_y, int jf_f32) {
  const bool G = uses_global_factor(r, d_y);
  const Layout lay(r, d_y, G);
  const size_t jc = jf_f32 ? 0 : (size_t)kJChunk * r * sizeof(double);
  return lay.tail * sizeof(double) + jc;
}

cudaError_t launch_propose(const ReducedArgs &a, cudaStream_t st) {
  if (a.r <= 32 * 7) {
    const int grid = (a.C + kPropWarps - 1) / kPropWarps;
    auto k = a.r <= 32 * 2   ? k_propose_warp<2>
             : a.r <= 32 * 4 ? k_propose_warp<4>
                             : k_propose_warp<7>;
    return launch_pdl(k, grid, 32 * kPropWarps, 0, st, a);
  }
  const size_t smem = propose_smem_bytes(a.r);
  cudaError_t e =
      cudaFuncSetAttribute(k_propose, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  return launch_pdl_n(chain_ctas(a.C), k_propose, a.C, kThreads, smem, st, a);
}

// Whether the smem-resident factor of an FP32 Jacobian takes the blocked
// factorisation, by the CTAs an SM that either leaves room for (plain, blk).  The
// plain one's chains of dependent operations need company: four CTAs of 256
// threads, or two of 512, are the faster against fewer blocked ones; otherwise the
// blocked one is.  2048 chains, d_y = r + 20, geometry in us, plain and blocked:
// r = 106 (4, 2 CTAs) 522 653, 108 (3, 2) 727 649, 134 (2, 2) 999 875, 136 (2, 1)
// 1045 1391, 156 (2, 1) 1323 1614, 160 (1, 1) 2062 1732, 200 (1, 1) 3079 2349.
static bool takes_blocked(size_t plain, size_t blk) { return blk >= 2 ? plain < 4 : plain < 2; }
static size_t ctas_an_sm(size_t smem) { return kSmemLimit / (smem + 1024); }

// The factorisation of an FP32 Jacobian's I + H, and where its digits or panel lie
// (elements from the start of shared memory), with smem raised to hold them.
// Digits behind the layout for a factor in shared memory; for one in global
// memory the panel, in whose place the vectors vp, vq, be, ae are formed afterwards:
// of 224 bytes a row with the digits, or where that does not fit (r from about 890)
// of 136 without them (152 chains, d_y = 60, plain and in panels: r = 890 24.0 and 11.3
// ms, 1024 36.9 and 16.7).
//
// FP64 factors take the plain one wherever they lie.  (r = 209 to 900 in global
// memory, blocked in panels with 256 threads: 1.05 to 1.23 times the time, with 512 1.02
// to 1.15; the FP64 pipe bounds both.)
static Factor geometry_factor(int r, int d_y, size_t &smem, int &panel) {
  const bool G = uses_global_factor(r, d_y);
  const size_t at = Layout(r, d_y, G, G).tail, n = r + 1, after = 32 * (size_t)r;
  panel = (int)at;
  if (!G) {
    const size_t need = std::max(smem, at * sizeof(double) + mma_digit_bytes((int)n));
    if (need > kGeoSmem || !takes_blocked(ctas_an_sm(smem), ctas_an_sm(need))) return kPlain;
    smem = need;
    return kMma;
  }
  const size_t mma = at * sizeof(double) + std::max(mma_panel_bytes((int)n), after);
  const size_t plain = at * sizeof(double) + std::max(n * kPanelLd * sizeof(double), after);
  if (std::min(mma, plain) > kGeoSmem) return kPlain;
  smem = mma <= kGeoSmem ? mma : plain;
  return mma <= kGeoSmem ? kMma : kPanels;
}

template <typename TJ, bool G, int NT, Factor kFac>
static cudaError_t launch_geometry_nt(const ReducedArgs &a, int mode, size_t smem, int panel,
                                      cudaStream_t st) {
  auto k = k_geometry<TJ, G, NT, kFac>;
  cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  ReducedArgs b = a;
  b.derive();
  return launch_pdl_n(chain_ctas(a.C), k, a.C, NT, smem, st, b, mode, panel);
}

// CTA size: smaller CTAs let more chains share an SM (the kernel's loops stride
// over blockDim).  FP64: 128 threads up to r = 64 and 256 up to r = 128, held to 128
// registers so that four and two CTAs fit an SM.  FP32 Jacobian, plain: the size
// that fills 32 warps with as many CTAs as the shared memory of the factor lets
// in (r = 100: four of 256 threads).  Blocked: 256 threads at 128 registers while
// two CTAs fit an SM (r = 128; factors in global memory up to r = 400), else 512.
template <typename TJ, bool G>
static cudaError_t launch_geometry_t(const ReducedArgs &a, int mode, size_t smem,
                                     cudaStream_t st) {
  if constexpr (sizeof(TJ) == 8) {
    if (!G && a.r <= 64) return launch_geometry_nt<TJ, G, 128, kPlain>(a, mode, smem, 0, st);
    if (!G && a.r <= 128) return launch_geometry_nt<TJ, G, 256, kPlain>(a, mode, smem, 0, st);
    return launch_geometry_nt<TJ, G, kThreads, kPlain>(a, mode, smem, 0, st);
  } else {
    int panel;
    const Factor fac = geometry_factor(a.r, a.d_y, smem, panel);
    const size_t ctas = ctas_an_sm(smem);
    if constexpr (G) {
      if (fac == kMma) return launch_geometry_nt<TJ, G, 256, kMma>(a, mode, smem, panel, st);
      if (fac == kPanels)
        return launch_geometry_nt<TJ, G, kThreads, kPanels>(a, mode, smem, panel, st);
    } else {
      if (fac == kMma)
        return ctas >= 2 ? launch_geometry_nt<TJ, G, 256, kMma>(a, mode, smem, panel, st)
                         : launch_geometry_nt<TJ, G, kThreads, kMma>(a, mode, smem, panel, st);
      if (a.r <= 64) return launch_geometry_nt<TJ, G, 128, kPlain>(a, mode, smem, 0, st);
      if (ctas >= 4) return launch_geometry_nt<TJ, G, 256, kPlain>(a, mode, smem, 0, st);
    }
    return launch_geometry_nt<TJ, G, kThreads, kPlain>(a, mode, smem, 0, st);
  }
}

cudaError_t launch_gram_f32(const ReducedArgs &a, int mode, cudaStream_t st) {
  const int nb = (a.r + kGramB - 1) / kGramB;
  for (int c0 = 0; c0 < a.C; c0 += 65535) {  // the grid's second dimension ends there
    ReducedArgs b = a;
    const size_t o = c0;
    b.C = std::min(65535, a.C - c0);
    b.cur = a.cur + o;
    b.L = a.L + o * slot_stride(a.r);
    b.J = reinterpret_cast<const float *>(a.J) + o * a.d_y * a.r;
    const cudaError_t e = launch_pdl(k_gram_f32, dim3(nb * (nb + 1) / 2, b.C), kGramThreads, 0, st,
                                     b, mode);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

cudaError_t launch_geometry(const ReducedArgs &a, int mode, cudaStream_t st) {
  const size_t smem = geometry_smem_bytes(a.r, a.d_y, a.jf_f32);
  const bool G = uses_global_factor(a.r, a.d_y);
  if (a.jf_f32)
    return G ? launch_geometry_t<float, true>(a, mode, smem, st)
             : launch_geometry_t<float, false>(a, mode, smem, st);
  return G ? launch_geometry_t<double, true>(a, mode, smem, st)
           : launch_geometry_t<double, false>(a, mode, smem, st);
}

}  // namespace dino
