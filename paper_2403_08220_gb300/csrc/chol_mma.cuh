// Blocked double-float Cholesky whose rank-16 trailing updates run on the tensor
// cores (mma.sync), for the r-sized factors of the tensor-core path.
//
// The panel's columns are factored in double-float as before (8-column steps);
// its rows below are then written as kDig signed base-256 digits, L_ik = 2^e_i
// sum_s d_s 2^(-7 - 8 s), with 2^e_i > sqrt(M_ii) >= |L_ik| fixed from the
// matrix's diagonal: 55 bits below 2^e_i.  Digits are integers of at most 128,
// exact in bf16; their products summed over the panel's 16 columns stay below
// 2^21, exact in FP32.  The digit products s + t = l for l < kLev = 7 (28 of them)
// make the seven level sums of an entry's update, which are joined by error-free
// sums into a double-float and subtracted from the entry.  What is left out is
// below 2^-52 sqrt(M_ii M_jj); the rounding of the double-float entries once per
// 16 columns remains.  (The direct sums round once per column: L L^T against the
// matrix, relative to sqrt(M_ii M_jj), r from 33 to 400: rms 2^-49.2 to 2^-49.5
// with them, 2^-49.5 to 2^-50.8 here; the largest entry 2^-44.8 to 2^-46.8 in both.)
//
// A rank-16 update of an entry takes 16 x 12 FP32 instructions and their
// operands' loads when summed directly, 6.7 issue cycles per entry and
// scheduler; here 28 mma.sync.m16n8k16 per 128 entries (8 cycles each on
// GB300) run beside about 42 instructions per entry that join the levels.
// Geometry of 512 chains at r = 400 (factor in global memory): 4.61 -> 3.44 ms;
// of 4096 chains at r = 128: 2.02 -> 1.60 ms (3.38 and 1.50 since the diagonal
// blocks take less).  The d_y-sized factors of the Woodbury path (101 rows, four
// chains an SM) gain nothing: 3.32 against 3.20 ms for 16384 chains, their time is
// in the panels and barriers.
#pragma once
#include "chol.cuh"

namespace dino {
namespace {

constexpr int kDig = 7, kLev = 7;  // digits, levels
// Bytes of a digit row, 7 planes of 16 bf16: padded so that the eight rows of an
// ldmatrix fall on distinct banks, or unpadded (pairs of them meet) where two
// CTAs an SM depend on it.
constexpr int kDigPitch = 240, kDigTight = 224;
constexpr int kMmaW = 16;          // panel width

// 2^e > sqrt(x), x > 0: e = floor(exponent / 2) + 1
__device__ __forceinline__ float row_scale(float x) {
  const int ex = (int)((__float_as_uint(x) >> 23) & 0xff) - 127;
  return __uint_as_float((uint32_t)(127 + (ex >> 1) + 1) << 23);
}

// The digits of two neighbouring columns' entries x0, x1 (columns 2 q, 2 q + 1 of
// the panel) into the row at `row`; inv_scale = 2^-e.
__device__ __forceinline__ void put_digits(char *row, int q, float2 x0, float2 x1,
                                           float inv_scale) {
  const float f = inv_scale * 36028797018963968.0f;  // 2^55
  const long long bias = 0x808080808080ll;            // 128 per digit below the first
  const long long t0 = __float2ll_rn(x0.x * f) + __float2ll_rn(x0.y * f) + bias;
  const long long t1 = __float2ll_rn(x1.x * f) + __float2ll_rn(x1.y * f) + bias;
  const uint32_t l0 = (uint32_t)t0, l1 = (uint32_t)t1;
  const int h0 = (int)(t0 >> 32), h1 = (int)(t1 >> 32);
  auto put = [&](int s, float d0, float d1) {
    *reinterpret_cast<uint32_t *>(row + 32 * s + 4 * q) =
        __byte_perm(__float_as_uint(d0), __float_as_uint(d1), 0x7632);
  };
  auto digit = [](uint32_t b) { return __uint_as_float(0x4b000000u | b) - 8388736.0f; };
#pragma unroll
  for (int i = 0; i < 4; ++i)  // byte i: weight 256^i, digit 6 - i
    put(6 - i, digit((l0 >> (8 * i)) & 255u), digit((l1 >> (8 * i)) & 255u));
  put(2, digit((uint32_t)h0 & 255u), digit((uint32_t)h1 & 255u));
  put(1, digit(((uint32_t)h0 >> 8) & 255u), digit(((uint32_t)h1 >> 8) & 255u));
  put(0, (float)(h0 >> 16), (float)(h1 >> 16));
}

__device__ __forceinline__ void ldmatrix4(uint32_t addr, uint32_t r[4]) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(addr));
}
__device__ __forceinline__ void ldmatrix2(uint32_t addr, uint32_t r[2]) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x2.shared.b16 {%0,%1}, [%2];"
               : "=r"(r[0]), "=r"(r[1])
               : "r"(addr));
}
__device__ __forceinline__ void mma16816(float c[4], const uint32_t a[4], uint32_t b0,
                                         uint32_t b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, "
      "{%8,%9}, {%0,%1,%2,%3};"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// entry - scale * sum_l a_l 2^(-8 l)
__device__ __forceinline__ float2 sub_levels(float2 c, const float a[kLev], float scale) {
  float h, e1, e2, e3;
  two_sum(a[0], a[1] * 0x1p-8f, h, e1);
  two_sum(h, a[2] * 0x1p-16f, h, e2);
  two_sum(h, a[3] * 0x1p-24f, h, e3);
  float low = __fmaf_rn(a[6], 0x1p-8f, a[5]);
  low = __fmaf_rn(low, 0x1p-8f, a[4]);
  const float l = __fmaf_rn(low, 0x1p-32f, __fadd_rn(__fadd_rn(e1, e2), e3));
  float s, q;
  two_sum(c.x, -(h * scale), s, q);
  float2 r;
  fast_two_sum(s, __fadd_rn(q, __fadd_rn(c.y, -(l * scale))), r.x, r.y);
  return r;
}

// Entries (i, j), j0 <= j <= i < n, of the packed matrix Ls (shared or global
// memory) take the panel's rank-16 update.  dig: digit rows, row i at (i - d0)
// kPitch; scl[i] = 2^e_i.  A work item, taken from *next, is a block of 16
// rows and up to four 8-column tiles, a multiple of 16 columns from j0; the
// first item is the 16 x 16 diagonal block, and `first()` runs on the warp that
// took it when the block is final.
template <int kPitch, class First>
__device__ void trailing_mma(float2 *Ls, const char *dig, int d0, const float *scl, int n, int j0,
                             int *next, First first) {
  const int lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
  const uint32_t base = smem_addr(dig);
  const int nrb = (n - j0 + 15) / 16;
  for (;;) {
    int item = 0;
    if (lane == 0) item = atomicAdd(next, 1);
    item = __shfl_sync(kFull, item, 0);
    int rb = 0, q = item;
    for (; rb < nrb; ++rb) {  // row block rb: 2 (rb + 1) column tiles, four an item
      const int items = (rb + 2) / 2;
      if (q < items) break;
      q -= items;
    }
    if (rb == nrb) return;
    const int i0 = j0 + 16 * rb;
    uint32_t a[kDig][4];
    {
      const int m = lane >> 3, row = min(i0 + (lane & 7) + 8 * (m & 1), n - 1);
      const uint32_t addr = base + (row - d0) * kPitch + (m >> 1) * 16;
#pragma unroll
      for (int s = 0; s < kDig; ++s) ldmatrix4(addr + 32 * s, a[s]);
    }
    const int ra = i0 + g, rb8 = ra + 8;
    const float sa = (ra < n ? scl[ra] : 0.0f) * 0x1p-14f,
                sb = (rb8 < n ? scl[rb8] : 0.0f) * 0x1p-14f;
    const int t1 = min(4 * q + 4, 2 * (rb + 1));
    for (int ct = 4 * q; ct < t1; ++ct) {
      const int jt = j0 + 8 * ct;
      if (jt >= n) break;
      const int j = jt + 2 * t;  // this lane's columns j, j + 1; rows ra and rb8
      float2 *pa = Ls + tri(ra) + j, *pb = Ls + tri(rb8) + j;
      float2 c0{}, c1{}, c2{}, c3{};
      const bool v0 = ra < n && j <= ra, v1 = ra < n && j + 1 <= ra;
      const bool v2 = rb8 < n && j <= rb8, v3 = rb8 < n && j + 1 <= rb8;
      if (v0) c0 = pa[0];
      if (v1) c1 = pa[1];
      if (v2) c2 = pb[0];
      if (v3) c3 = pb[1];
      float acc[kLev][4];
#pragma unroll
      for (int l = 0; l < kLev; ++l) acc[l][0] = acc[l][1] = acc[l][2] = acc[l][3] = 0.0f;
      const int m = lane >> 3, brow = min(jt + (lane & 7), n - 1);
      const uint32_t baddr = base + (brow - d0) * kPitch + (m >> 1) * 32 + (m & 1) * 16;
#pragma unroll
      for (int u = 0; u + 1 < kDig; u += 2) {  // digits u and u + 1 of the columns' rows
        uint32_t b[4];
        ldmatrix4(baddr + 32 * u, b);
#pragma unroll
        for (int s = 0; s < kDig; ++s) {
          if (s + u < kLev) mma16816(acc[s + u], a[s], b[0], b[1]);
          if (s + u + 1 < kLev) mma16816(acc[s + u + 1], a[s], b[2], b[3]);
        }
      }
      {  // the last digit meets the first alone (lanes 0 .. 15 give the addresses)
        uint32_t b[2];
        ldmatrix2(base + (brow - d0) * kPitch + 32 * (kDig - 1) + (m & 1) * 16, b);
        mma16816(acc[kDig - 1], a[0], b[0], b[1]);
      }
      const float s0 = j < n ? scl[j] : 0.0f, s1 = j + 1 < n ? scl[j + 1] : 0.0f;
      auto lev = [&](int e, float v[kLev]) {
#pragma unroll
        for (int l = 0; l < kLev; ++l) v[l] = acc[l][e];
      };
      float v[kLev];
      lev(0, v);
      if (v0) pa[0] = sub_levels(c0, v, sa * s0);
      lev(1, v);
      if (v1) pa[1] = sub_levels(c1, v, sa * s1);
      lev(2, v);
      if (v2) pb[0] = sub_levels(c2, v, sb * s0);
      lev(3, v);
      if (v3) pb[1] = sub_levels(c3, v, sb * s1);
    }
    if (item == 0) {
      __syncwarp();
      first();
    }
  }
}

// Shared memory of the digits of rows 16 .. n - 1 and the scales of all rows.
__host__ __device__ inline size_t mma_digit_bytes(int n) {
  return (size_t)(n > kMmaW ? n - kMmaW : 0) * kDigPitch + (((size_t)n * 4 + 15) & ~(size_t)15);
}

// In-place Cholesky of the packed n x n matrix in shared memory; dig:
// mma_digit_bytes(n), 16-byte aligned.  Per 16-column panel, a CTA barrier
// after each step: the rows below the first 8 x 8 block (factored ahead) are
// solved; the second block is updated and factored by one warp while the others
// update the rows below it; those rows are solved; their digits are written;
// the trailing entries are updated, and the warp that gets the next diagonal
// block goes on to factor its first 8 x 8 block.
__device__ void cta_cholesky_mma(float2 *Ls, float2 *inv, int n, char *dig) {
  using A = DF;
  __shared__ int next_item;
  __shared__ float2 lsc[kNB * (kNB + 1) / 2];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nw = blockDim.x >> 5;
  const PackedAt<float2> at{Ls};
  float *scl = reinterpret_cast<float *>(dig + (size_t)max(0, n - kMmaW) * kDigPitch);
  for (int i = tid; i < n; i += blockDim.x) scl[i] = row_scale(Ls[tri(i) + i].x);
  __syncthreads();  // the scales are taken before the first block is factored
  if (warp == blockIdx.x % nw) warp_factor_diag<A, false>(at, inv, 0, min(kNB, n), lane, lsc);
  __syncthreads();
  for (int kb = 0; kb < n; kb += kMmaW) {
    const int rot = (kb / kMmaW + blockIdx.x) % nw, t = (tid + 32 * rot) % blockDim.x;
    const int nb1 = min(kNB, n - kb), k2 = kb + nb1, nb2 = min(kNB, n - k2), j0 = k2 + nb2;
    if (tid == 0) next_item = 0;
    for (int i = k2 + t; i < n; i += blockDim.x) panel_row<A>(at, inv, lsc, kb, i);
    __syncthreads();
    if (nb2 <= 0) return;
    auto update = [&](int i, int c) {  // entry (i, c) of the second eight columns
      A::Acc acc = A::begin(at(i, c));
#pragma unroll
      for (int k = 0; k < kNB; ++k) A::sub(acc, at(i, kb + k), at(c, kb + k));
      at(i, c) = A::end(acc);
    };
    if (warp == rot) {
      warp_factor_diag<A, true>(at, inv, k2, nb2, lane, lsc, kb);
    } else {
      const int w = (warp - rot + nw) % nw - 1;  // 0 .. nw - 2
      for (int e = 32 * w + lane; e < (n - j0) * kNB; e += 32 * (nw - 1))
        update(j0 + e / kNB, k2 + e % kNB);
    }
    __syncthreads();
    if (j0 >= n) return;
    for (int i = j0 + t; i < n; i += blockDim.x) panel_row<A>(at, inv, lsc, k2, i);
    __syncthreads();
    for (int e = tid; e < (n - j0) * (kMmaW / 2); e += blockDim.x) {
      const int i = j0 + e / (kMmaW / 2), q = e % (kMmaW / 2);
      const float2 *x = Ls + tri(i) + kb + 2 * q;
      put_digits(dig + (size_t)(i - kMmaW) * kDigPitch, q, x[0], x[1], 1.0f / scl[i]);
    }
    __syncthreads();
    trailing_mma<kDigPitch>(Ls, dig, kMmaW, scl, n, j0, &next_item, [&]() {
      warp_factor_diag<A, false>(at, inv, j0, min(kNB, n - j0), lane, lsc);
    });
    __syncthreads();
  }
}

// The same for a packed matrix in global memory (cta_cholesky_global is for those whose
// panel of digits does not fit): the panel's rows live in shared
// memory at a pitch of kDigTight bytes, are written back when solved, and their
// digits take their place.  dig: n kDigTight bytes and the scales.
__host__ __device__ inline size_t mma_panel_bytes(int n) {
  return (size_t)n * kDigTight + (((size_t)n * 4 + 15) & ~(size_t)15);
}

__device__ void cta_cholesky_global_mma(float2 *Lg, float2 *inv, int n, char *dig) {
  using A = DF;
  constexpr int kLd = kDigTight / 8;
  __shared__ int next_item;
  __shared__ float2 lsc[kNB * (kNB + 1) / 2];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nw = blockDim.x >> 5;
  float2 *P = reinterpret_cast<float2 *>(dig);
  const PanelAt<float2, kLd> at{P};
  float *scl = reinterpret_cast<float *>(dig + (size_t)n * kDigTight);
  for (int i = tid; i < n; i += blockDim.x) scl[i] = row_scale(Lg[tri(i) + i].x);
  __syncthreads();
  for (int kb = 0; kb < n; kb += kMmaW) {
    const int w = min(kMmaW, n - kb), m = n - kb;
    for (int e = tid; e < m * kMmaW; e += blockDim.x) {
      const int i = e / kMmaW, q = e % kMmaW;
      if (q < w && q <= i) at(i, q) = Lg[tri(kb + i) + kb + q];
    }
    if (tid == 0) next_item = 0;
    __syncthreads();
    for (int kk = 0; kk < w; kk += kNB) {
      const int nb = min(kNB, w - kk), c0 = kk + nb;
      if (warp == (kb / kNB + kk / kNB) % nw)
        warp_factor_diag<A, false>(at, inv + kb, kk, nb, lane, lsc);
      __syncthreads();
      for (int i = c0 + tid; i < m; i += blockDim.x) panel_row<A>(at, inv + kb, lsc, kk, i);
      __syncthreads();
      if (w > c0) {
        for (int e = tid; e < (m - c0) * kNB; e += blockDim.x) {
          const int i = c0 + e / kNB, c = c0 + e % kNB;
          if (c < w && c <= i) {
            A::Acc acc = A::begin(at(i, c));
#pragma unroll
            for (int k = 0; k < kNB; ++k) A::sub(acc, at(i, kk + k), at(c, kk + k));
            at(i, c) = A::end(acc);
          }
        }
        __syncthreads();
      }
    }
    for (int e = tid; e < m * kMmaW; e += blockDim.x) {
      const int i = e / kMmaW, q = e % kMmaW;
      if (q < w && q <= i) Lg[tri(kb + i) + kb + q] = at(i, q);
    }
    const int j0 = kb + w;
    if (j0 >= n) return;  // a narrower panel is the last
    __syncthreads();
    for (int i = j0 + tid; i < n; i += blockDim.x) {  // a row's digits in its own place
      float2 x[kMmaW];
#pragma unroll
      for (int k = 0; k < kMmaW; ++k) x[k] = at(i - kb, k);
      char *row = dig + (size_t)(i - kb) * kDigTight;
      const float is = 1.0f / scl[i];
#pragma unroll
      for (int q = 0; q < kMmaW / 2; ++q) put_digits(row, q, x[2 * q], x[2 * q + 1], is);
    }
    __syncthreads();
    trailing_mma<kDigTight>(Lg, dig, kb, scl, n, j0, &next_item, []() {});
    __syncthreads();
  }
}

}  // namespace
}  // namespace dino
