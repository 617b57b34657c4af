// FP64 matrix products on the bf16 tensor cores (tcgen05), by error-free
// splitting of the operands (Ozaki, Ogita, Oishi and Rump, "Error-free
// transformations of matrix multiplication by using fast routines of matrix
// multiplication and its applications", Numer. Algorithms 59 (2012)).
//
//   D[M x N] = A B^T, A: M x K, B: N x K, epilogue in FP64.
//
// GB300's FP64 pipe runs at about 1.2 TFLOP/s, so the FP64 path's products
// (Jacobian, encoder, complement projections) are bound by it.  Here every
// row i of A is scaled by a power of two 2^ea_i above its largest entry and
// written as kDigits signed base-128 digits, a = 2^(ea_i - 7) sum_s d_s 128^-s
// with |d_0| <= 128, |d_s| <= 64 (56 bits below the row's maximum: the residue
// is at most 2^-57 of it); B likewise.  A digit is an integer that bf16 holds
// exactly, a product of two an integer of at most 14 bits.  Of the digit
// products d_s d'_t only s + t = l < kDigits are formed (36 of 64; the rest
// lies below 2^-56), summed per level l over a chunk of kChunkK = 512 columns
// in FP32 in TMEM: at most (l + 3) 2^21, so levels 0 to 5 are exact integers
// (2^24), and levels 6 and 7, which weigh 2^-42 and 2^-49, can round only when
// nearly all digits align.  The eight level sums are combined in 64-bit
// integers and rounded to FP64 once, so the result carries no accumulated
// rounding (2-norm error against extended precision: the Jacobian of widths
// 200-400-400-100 2.2e-16 against 1.05e-15 of the multiply-add chain, its f
// 1.7e-16 against 9.2e-16, m_r = E m of 4225 nodes with |E| |m| / |E m| = 500
// 1.0e-15 against 2.6e-15).
//
// Accuracy entry by entry: with a' = a 2^-ea and b' = b 2^-eb the digits leave
// at most K 11 2^-58 (entries rounded at 2^-57, 7 digit products of s + t = 8),
// whatever the sum: where A's large entries meet B's small ones that is more
// than the K 2^-53 sum |a' b'| of the chain.  So a further product is formed,
// of the entries' magnitudes in bf16 (rounded down, a plane of their own): a
// lower bound of sum |a' b'|.  An output whose bound is below kLeast = 1/8 is a
// plain dot product instead; the others are within 2.75 K 2^-53 sum |a b| at
// most.  With a dense B four neighbouring columns count as one, the sum of A's
// four magnitudes times the least of B's (Magnitudes): the Jacobian's products
// of 1024 chains, widths 200-400-400-100, take 2.02 ms, 2.09 with every column on
// its own, 1.88 without the bound.  The Gram matrices J J^T that are factored
// next (gram64_slots) go without: their error counts beside |J_i| |J_j|, as the
// factorisation's own rounding does.
//
// Column equilibration: B (weights, laid out once) may carry powers of two
// f_k with max_j |B_jk| 2^-f_k in [1, 2); A's column k is then scaled by
// 2^f_k, so that an input that B weighs down cannot push the others' digits
// out of range, and an input in a column that is zero in B (kZeroCol) takes no
// part.  Outputs whose row of A or of B holds an infinity or a NaN, or a
// subnormal number that counts beside the row's largest, are plain dot products
// too.
//
// Layout: digit planes [kDigits][rows][ldp] of bf16, then the magnitudes [rows]
// [check_pitch]; TMA boxes of 32 columns x (128 rows of A | BN rows of B) x
// all eight planes (64-byte swizzle), two stages; a stage of magnitudes is
// eight blocks of 32 columns in the place of the eight planes.  The BN rows of
// consecutive B planes are contiguous in the stage, so one tcgen05.mma
// multiplies A's plane s with up to 256 / BN planes of B at once and adds into as
// many neighbouring level accumulators: 12 instructions of mostly N = 256 per 16
// columns instead of 36 of N = 64.  The eight accumulators of BN columns fill
// TMEM at BN = 64; the sums of magnitudes take the first one's place when the
// last chunk has been read.  At BN = 32 they have columns of their own and come with
// the last chunk, without a second round between the MMAs and the epilogue.
//
// What bounds it: the chain from tile to tile.  One set of accumulators means that
// the next tile's MMAs wait for the epilogue's reads, and two stages (96 KB per 32
// columns and tile) do not cover their loads' latency: tensor pipe 53% active, L2
// at 29%, 6.5 TB/s (12800 x 400 x 400).  The launcher's callers cut M into chunks
// whose planes stay in L2.
// 102400 x 400 x 400 and x 200 (the Jacobian of 1024 chains, 98 GFLOP): 46.6 ms
// on the FP64 pipe, 2.02 ms here and 0.6 ms for the digits of A.
#include <cuda_bf16.h>
#include <cudaTypedefs.h>

#include <algorithm>

#include "dino_internal.h"
#include "epi64.cuh"
#include "pdl.cuh"
#include "tcgen05.cuh"

namespace dino {
namespace {

constexpr int kDigits = kDigits64;
constexpr int kBM = 128, kKB = 32;             // tile rows, columns per stage
constexpr int kChunkK = 512;                   // columns per exact accumulation
constexpr int kStages = 2;
constexpr int kTmemCols = 512;
constexpr int kEpiWarps = 8;
constexpr int kGemm64Threads = 32 * (2 + kEpiWarps);
constexpr int kABytes = kDigits * kBM * kKB * 2;
constexpr int kStgBytes = kEpiWarps * 32 * 16 * 8;  // 32 rows x 16 doubles per warp
constexpr float kLeast = 0.125f;               // sum |a' b'| below which digits do not do
constexpr int kBadRow = INT32_MIN;             // row exponent: plain dot products
constexpr int kZeroRow = INT32_MIN + 1;        // row exponent of a row of zeros
constexpr int kZeroCol = INT32_MIN;            // column exponent of a zero column of B

// Row pitch of the magnitudes of K columns, `group` to a value: whole blocks of 32.
__host__ __device__ inline int check_pitch(int K, int group) {
  return ((K + group - 1) / group + kKB - 1) / kKB * kKB;
}

// ---- digits -----------------------------------------------------------------

struct SplitArgs {
  int rows, K, ldp;
  size_t plane;
  const double *src;  // rows x K (pitch ld), or nullptr: W[row % g] .* der[row / g]
  int ld;
  const double *W, *der;
  int g, ldd, row0;   // row0: first row of the product form
  const int *fk;      // column exponents (nullptr: 0), added (A) or subtracted (B)
  int fsign;
  Magnitudes mags;
  __nv_bfloat16 *dst;
  int *ex;
};

__device__ __forceinline__ int exp_field(double x) {
  return (__double2hiint(x) >> 20) & 0x7ff;
}

// One warp per row.  Lane l holds the columns 4 (l + 32 q) .. + 3, q < kQ, of
// the row in registers (kQ = 0: any K, the row is read twice), so that loads
// and the 8-byte digit stores of a warp are contiguous.  The digits come out
// of the 56-bit integer t + sum_s 64 128^s as unsigned 7-bit fields f, d = f -
// 64, by 32-bit operations, and turn into bf16 through the mantissa of 2^23 + f
// (64-bit shifts and integer conversions per digit took 1.6 times as long:
// 60 us against 37 us for 19456 rows of 400).
template <int kQ>
__global__ void __launch_bounds__(256, 4) k_split64(const SplitArgs a) {
  pdl_begin();
  const int lane = threadIdx.x & 31;
  const int row = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  if (row >= a.rows) return;
  const double *s1, *s2 = nullptr;
  if (a.src) {
    s1 = a.src + (size_t)row * a.ld;
  } else {
    const int gr = a.row0 + row, c = gr / a.g;
    s1 = a.W + (size_t)(gr - c * a.g) * a.K;
    s2 = a.der + (size_t)c * a.ldd;
  }
  const bool vec = ((uintptr_t)s1 & 15) == 0 && ((uintptr_t)s2 & 15) == 0;
  auto load4 = [&](int k, double v[4]) {
    if (vec && k + 4 <= a.K) {
      const double2 x = *reinterpret_cast<const double2 *>(s1 + k);
      const double2 y = *reinterpret_cast<const double2 *>(s1 + k + 2);
      v[0] = x.x;
      v[1] = x.y;
      v[2] = y.x;
      v[3] = y.y;
      if (s2) {
        const double2 dx = *reinterpret_cast<const double2 *>(s2 + k);
        const double2 dy = *reinterpret_cast<const double2 *>(s2 + k + 2);
        v[0] *= dx.x;
        v[1] *= dx.y;
        v[2] *= dy.x;
        v[3] *= dy.y;
      }
    } else {
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        v[e] = k + e < a.K ? s1[k + e] : 0.0;
        if (s2 && k + e < a.K) v[e] *= s2[k + e];
      }
    }
  };
  const bool four = a.mags == Magnitudes::kSum4 || a.mags == Magnitudes::kMin4;
  const int ngroups = a.ldp / 4;
  const int ldc = a.mags == Magnitudes::kNone ? 0 : check_pitch(a.K, four ? 4 : 1);
  uint16_t *chk = reinterpret_cast<uint16_t *>(a.dst + kDigits * a.plane) + (size_t)row * ldc;
  double x[kQ > 0 ? kQ : 1][4];
  int emax = 0;        // largest exponent field
  int tiny = INT32_MIN;  // largest one that an entry left out can have
  bool bad = false;
  // Entries k .. k + 3: column exponents into the exponent fields (entries of zero
  // columns become 0), which leaves out what is subnormal before or after.
  auto scale = [&](int k, double v[4]) {
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      const int ef = exp_field(v[e]), f = a.fk && k + e < a.K ? a.fk[k + e] : 0;
      const int es = ef + a.fsign * f, hi = __double2hiint(v[e]), lo = __double2loint(v[e]);
      bad |= ef == 0x7ff || (es >= 0x7ff && f != kZeroCol);
      const bool keep = ef > 0 && f != kZeroCol && es > 0;
      if (!keep && f != kZeroCol && ((hi & 0x7fffffff) | lo))
        tiny = max(tiny, max(es, 1 + a.fsign * f));
      emax = max(emax, keep ? es : 0);
      v[e] = keep ? __hiloint2double(hi + ((es - ef) << 20), lo) : 0.0;
    }
  };
  if constexpr (kQ > 0) {
#pragma unroll
    for (int q = 0; q < kQ; ++q) {
      const int k = 4 * (lane + 32 * q);
      load4(k, x[q]);
      scale(k, x[q]);
    }
  } else {
    for (int grp = lane; grp < ngroups; grp += 32) {
      load4(4 * grp, x[0]);
      scale(4 * grp, x[0]);
    }
  }
#pragma unroll
  for (int o = 16; o; o >>= 1) emax = max(emax, __shfl_xor_sync(0xffffffffu, emax, o));
  // what was left out is below 2^-57 of 2^ea, or the row is bad, as is one at the
  // bottom of the range (fields below 200)
  bad = __any_sync(0xffffffffu, bad || tiny > (emax ? emax - 58 : INT32_MIN) ||
                                    (emax > 0 && emax < 200));
  if (lane == 0) a.ex[row] = bad ? kBadRow : (emax ? emax - 1022 : kZeroRow);
  const int mbase = (emax - 126) << 7;
  auto emit = [&](int grp, const double v[4]) {
    uint32_t w[kDigits][2], mag[4];
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      const int ef = exp_field(v[e]);
      // |entry| 2^-ea in bf16, rounded down
      mag[e] = (uint32_t)max(0, (__double2hiint(v[e]) >> 13 & 0x3ffff) - mbase);
      long long t = 0;  // the entry in units of 2^(ea - 56), rounded
      if (ef) {
        const long long bits = __double_as_longlong(v[e]);
        const long long m = (bits & 0xfffffffffffffll) | 0x10000000000000ll;
        const int s = ef - emax + 3;
        t = s >= 0 ? m << s : (s > -60 ? (m + (1ll << (-s - 1))) >> -s : 0);
        if (bits < 0) t = -t;
      }
      // seven biased fields of 7 bits below the signed leading digit
      t += 0x1020408102040ll;
      const uint32_t lo = (uint32_t)t & 0xfffffffu, hi = (uint32_t)(t >> 28);
      auto put = [&](int d, float f) {
        const uint32_t b = __float_as_uint(f);
        w[d][e >> 1] = (e & 1) ? __byte_perm(w[d][e >> 1], b, 0x7610) : b >> 16;
      };
#pragma unroll
      for (int i = 0; i < 7; ++i) {  // field i, weight 128^i: digit kDigits - 1 - i
        const uint32_t f = (i < 4 ? lo >> (7 * i) : hi >> (7 * (i - 4))) & 127u;
        put(kDigits - 1 - i, __uint_as_float(0x4b000000u | f) - 8388672.0f);
      }
      put(0, (float)((int)hi >> 21));
    }
    __nv_bfloat16 *o = a.dst + (size_t)row * a.ldp + 4 * grp;
#pragma unroll
    for (int d = 0; d < kDigits; ++d)
      *reinterpret_cast<uint2 *>(o + d * a.plane) = make_uint2(w[d][0], w[d][1]);
    if (a.mags == Magnitudes::kEach) {
      *reinterpret_cast<uint2 *>(chk + 4 * grp) =
          make_uint2(mag[0] | mag[1] << 16, mag[2] | mag[3] << 16);
    } else if (a.mags == Magnitudes::kSum4) {
      auto f = [&](int e) { return __uint_as_float(mag[e] << 16); };
      chk[grp] = (uint16_t)(__float_as_uint((f(0) + f(1)) + (f(2) + f(3))) >> 16);
    } else if (a.mags == Magnitudes::kMin4) {
      chk[grp] = (uint16_t)min(min(mag[0], mag[1]), min(mag[2], mag[3]));
    }
  };
  if constexpr (kQ > 0) {
#pragma unroll
    for (int q = 0; q < kQ; ++q)
      if (lane + 32 * q < ngroups) emit(lane + 32 * q, x[q]);
  } else {
    for (int grp = lane; grp < ngroups; grp += 32) {
      load4(4 * grp, x[0]);
      scale(4 * grp, x[0]);
      emit(grp, x[0]);
    }
  }
  for (int k = (four ? ngroups : a.ldp) + lane; k < ldc; k += 32) chk[k] = 0;
}

// Column exponents: fk[k] with 2^fk <= max_j |B_jk| < 2^(fk + 1) over the finite
// entries (-1023 for subnormal ones, kZeroCol for a zero column).
__global__ void k_col_exp(int rows, int K, const double *__restrict__ B, int ld,
                          int *__restrict__ fk) {
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= K) return;
  int m = -1;
  for (int j = 0; j < rows; ++j) {
    const double v = B[(size_t)j * ld + k];
    const int ef = exp_field(v);
    if (v != 0.0 && ef < 0x7ff) m = max(m, ef);
  }
  fk[k] = m < 0 ? kZeroCol : m - 1023;
}

// *sparse += the nonzero rows whose least magnitudes of four columns (Magnitudes::kEach
// planes) sum to less than 2: a warp per row
__global__ void __launch_bounds__(256) k_count_sparse(int rows, int K, const uint16_t *chk,
                                                      const int *ex, int *sparse) {
  const int row = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
  if (row >= rows || ex[row] == kZeroRow) return;
  const uint16_t *c = chk + (size_t)row * check_pitch(K, 1);
  float s = 0.0f;
  for (int k = 4 * lane; k < K; k += 128)  // the pitch is a multiple of 32
    s += __uint_as_float((uint32_t)min(min(c[k], c[k + 1]), min(c[k + 2], c[k + 3])) << 16);
#pragma unroll
  for (int o = 16; o; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  if (lane == 0 && s < 2.0f) atomicAdd(sparse, 1);
}

// ---- product ------------------------------------------------------------------

struct Gemm64Params {
  int M, N, K, row0, nkb, ncb;  // nkb: 32-column blocks; ncb: of the magnitudes
  int grp;  // Gram products: rows of a group (0: one plain product)
  const int *ea, *eb;
  const double *A, *W, *der, *B;  // the FP64 operands, for plain dot products
  int lda, g, ldd, ldb;
  uint32_t tmem_cols;
  int *err;
};

// (hi + lo 2^-28) 2^ex rounded to FP64 (0 <= lo < 2^28), by integer
// operations (the FP64 pipe is the scarce one)
__device__ __forceinline__ double scaled_to_f64(long long hi, uint32_t lo, int ex) {
  const bool neg = hi < 0;
  unsigned long long u = (unsigned long long)hi;
  if (neg) {
    u = ~u + (lo == 0);
    lo = (0x10000000u - lo) & 0xfffffffu;
  }
  if (u == 0) {  // at most 28 bits: exact
    const double v = ldexp((double)lo, ex - 28);
    return neg ? -v : v;
  }
  const int lz = __clzll((long long)u);
  const unsigned long long l = (unsigned long long)lo << 36;
  u = lz ? (u << lz) | (l >> (64 - lz)) : u;
  const bool sticky = lz < 28 && (lo << (4 + lz)) != 0;
  const int e = 1023 + 63 - lz + ex;
  if (e < 1 || e > 2045) {
    const double v = ldexp((double)u, ex - lz);
    return neg ? -v : v;
  }
  const unsigned long long m = (u >> 11) + ((unsigned long long)e << 52) - 0x10000000000000ull;
  const unsigned rest = ((unsigned)u & 0x7ffu) << 1 | sticky;
  const unsigned long long up = rest > 0x800u || (rest == 0x800u && (m & 1)) ? 1 : 0;
  return __longlong_as_double(
      (long long)((m + up) | (neg ? 0x8000000000000000ull : 0ull)));
}

__device__ __forceinline__ void tmem_ld8(uint32_t taddr, int v[8]) {
  uint32_t r[8];
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]),
                 "=r"(r[6]), "=r"(r[7])
               : "r"(taddr));
#pragma unroll
  for (int i = 0; i < 8; ++i) v[i] = (int)r[i];
}
__device__ __forceinline__ void tmem_wait_ld() {
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
}

// The plain FP64 dot products of the lanes in `redo` (a warp's outputs, lane l at
// (row, col) of its own arguments), each by the whole warp: a lone lane's chain of K
// multiply-adds takes the FP64 pipe as long as 32 of them.  Every lane returns v or
// its own product.
__device__ __noinline__ double plain_dots(const Gemm64Params &p, int g0, int row, int col,
                                          unsigned redo, double v) {
  const int lane = threadIdx.x & 31;
  for (; redo; redo &= redo - 1) {
    const int l = __ffs(redo) - 1;
    const int r = __shfl_sync(0xffffffffu, row, l), c = __shfl_sync(0xffffffffu, col, l);
    const double *y = p.B + (size_t)(g0 + c) * p.ldb;
    const int gr = p.row0 + r;
    const double *x = p.A ? p.A + (size_t)(g0 + r) * p.lda : p.W + (size_t)(gr % p.g) * p.K;
    const double *d = p.A ? nullptr : p.der + (size_t)(gr / p.g) * p.ldd;
    double s = 0.0;
    for (int k = lane; k < p.K; k += 32) s += (d ? x[k] * d[k] : x[k]) * y[k];
#pragma unroll
    for (int o = 16; o; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (lane == l) v = s;
  }
  return v;
}

__device__ __forceinline__ uint64_t smem_desc_sw64(uint32_t addr) {
  return (uint64_t)((addr & 0x3FFFFu) >> 4) | ((uint64_t)1 << 16) | ((uint64_t)(512 >> 4) << 32) |
         ((uint64_t)1 << 46) | ((uint64_t)4 << 61);
}

// Warp roles as in the bf16 GEMM: warp 0 the TMA producer, warp 1 TMEM and
// the MMA issue, warps 2-9 the epilogue (four lane quarters x two halves of
// the tile's columns).  One set of accumulators: the MMAs of the next chunk or
// tile start once the epilogue has read the previous one out of TMEM.
//
// kGram: the Gram matrices of the groups of p.grp consecutive rows of A (both
// operands are A's digits, N = grp): tile t is a block of one group, and blocks
// above the diagonal are left out.
template <int BN, bool kGram, class Epi>
__global__ void __launch_bounds__(kGemm64Threads, 1)
    k_gemm64(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB,
             const __grid_constant__ CUtensorMap tmAc, const __grid_constant__ CUtensorMap tmBc,
             const Gemm64Params p, const Epi epi) {
  constexpr int NC = BN / 2;                       // columns of an epilogue warp
  // the sums of magnitudes beside the levels (TMEM column kMagCol), in the last chunk's round
  constexpr bool kBeside = !kGram && (kDigits + 1) * BN <= kTmemCols;
  constexpr int kMagCol = kBeside ? kDigits * BN : 0;
  constexpr uint32_t kBBytes = kDigits * BN * kKB * 2;
  constexpr uint32_t kStage = kABytes + kBBytes;
  extern __shared__ __align__(1024) unsigned char smraw[];
  const uint32_t raw = smem_u32(smraw);
  const uint32_t base = (raw + 1023u) & ~1023u;
  unsigned char *gbase = smraw + (base - raw);
  double *stg_all = reinterpret_cast<double *>(gbase + kStages * kStage);
  uint64_t *bars = reinterpret_cast<uint64_t *>(gbase + kStages * kStage + kStgBytes);
  // bars: full[2], empty[2], acc_full, acc_empty, drain
  volatile int *abort_flag = reinterpret_cast<volatile int *>(bars + 2 * kStages + 3);
  volatile int *consumed = abort_flag + 1;
  uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(bars + 2 * kStages + 4);
  const uint32_t acc_full = smem_u32(&bars[2 * kStages]), acc_empty = acc_full + 8,
                 drain = acc_full + 16;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int ntn = (p.N + BN - 1) / BN;
  const int mpg = kGram ? (p.grp + kBM - 1) / kBM : 0;  // row tiles of a group
  const int ntiles = kGram ? p.M / p.grp * mpg * ntn : ((p.M + kBM - 1) / kBM) * ntn;
  // tile t: first row (of A) and first column, both within the group g0 .. for kGram
  auto tile = [&](int t, int &g0, int &m0, int &n0) {
    n0 = (t % ntn) * BN;
    t /= ntn;
    g0 = kGram ? (t / mpg) * p.grp : 0;
    m0 = (kGram ? t % mpg : t) * kBM;
    return !kGram || n0 < m0 + kBM;  // false: above the diagonal
  };
  constexpr int kChunkB = kChunkK / kKB;           // stages per exact accumulation
  const int nck = kGram ? 0 : (p.ncb + kDigits - 1) / kDigits;  // stages of the magnitudes

  if (threadIdx.x == 0) {
    for (int s = 0; s < kStages; ++s) {
      mbar_init(smem_u32(&bars[s]), 1);
      mbar_init(smem_u32(&bars[kStages + s]), 1);
    }
    mbar_init(acc_full, 1);
    mbar_init(acc_empty, kEpiWarps);
    mbar_init(drain, 1);
    *abort_flag = 0;
    *consumed = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     smem_u32(tmem_slot)),
                 "r"(p.tmem_cols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  fence_before();
  __syncthreads();
  fence_after();
  const uint32_t tmem = *tmem_slot;
  pdl_begin();

  if (warp == 0) {
    if (lane == 0) {
      int g = 0;
      bool ok = true;
      for (int t = blockIdx.x; t < ntiles && ok; t += gridDim.x) {
        int g0, m0, n0;
        if (!tile(t, g0, m0, n0)) continue;
        for (int kb = 0; kb < p.nkb + nck; ++kb, ++g) {
          const int s = g % kStages;
          if (!mbar_wait(smem_u32(&bars[kStages + s]), ((uint32_t)(g / kStages) & 1u) ^ 1u,
                         abort_flag)) {
            *abort_flag = 1;
            atomicOr(p.err, 8);
            ok = false;
            break;
          }
          const uint32_t full = smem_u32(&bars[s]), sa = base + s * kStage;
          mbar_expect_tx(full, kStage);
          if (kb < p.nkb) {
            tma_load_3d(sa, &tmA, kb * kKB, g0 + m0, 0, full);
            tma_load_3d(sa + kABytes, &tmB, kb * kKB, g0 + n0, 0, full);
          } else {
            tma_load_3d(sa, &tmAc, 0, g0 + m0, (kb - p.nkb) * kDigits, full);
            tma_load_3d(sa + kABytes, &tmBc, 0, g0 + n0, (kb - p.nkb) * kDigits, full);
          }
        }
      }
      if (*abort_flag)  // let the copies already issued land
        for (int i = *consumed; i < g; ++i)
          mbar_wait(smem_u32(&bars[i % kStages]), (uint32_t)(i / kStages) & 1u, nullptr);
    }
  } else if (warp == 1) {
    if (lane == 0) {
      bool ok = true;
      int g = 0, j = 0;  // stages consumed, accumulations started
      for (int t = blockIdx.x; t < ntiles && ok; t += gridDim.x) {
        int g0, m0, n0;
        if (!tile(t, g0, m0, n0)) continue;
        // the chunks, then the magnitudes' stages [nkb, nkb + nck)
        for (int kb0 = 0; kb0 < p.nkb + nck && ok; ++j) {
          if (!mbar_wait(acc_empty, ((uint32_t)j & 1u) ^ 1u, abort_flag)) {
            *abort_flag = 1;
            atomicOr(p.err, 8);
            ok = false;
            break;
          }
          fence_after();
          int kb1 = kb0 >= p.nkb ? p.nkb + nck : min(p.nkb, kb0 + kChunkB);
          if (kBeside && kb1 == p.nkb) kb1 += nck;
          for (int kb = kb0; kb < kb1; ++kb, ++g) {
            const int s = g % kStages;
            if (!mbar_wait(smem_u32(&bars[s]), (uint32_t)(g / kStages) & 1u, abort_flag)) {
              *abort_flag = 1;
              atomicOr(p.err, 8);
              ok = false;
              break;
            }
            *consumed = g + 1;
            fence_after();
            const uint32_t sa = base + s * kStage;
            const uint64_t ad = smem_desc_sw64(sa), bd = smem_desc_sw64(sa + kABytes);
            if (!kGram && kb >= p.nkb) {
              const int nblk = min(kDigits, p.ncb - (kb - p.nkb) * kDigits);
              for (int i = 0; i < nblk; ++i)
#pragma unroll
                for (int kk = 0; kk < kKB / 16; ++kk)
                  mma_bf16(tmem + kMagCol, ad + (uint64_t)(i * kBM * kKB * 2 / 16 + 2 * kk),
                           bd + (uint64_t)(i * BN * kKB * 2 / 16 + 2 * kk), idesc_bf16(kBM, BN),
                           (kb > p.nkb || i > 0 || kk > 0) ? 1u : 0u);
              mma_commit(smem_u32(&bars[kStages + s]));
              continue;
            }
#pragma unroll
            for (int kk = 0; kk < kKB / 16; ++kk) {
#pragma unroll
              for (int i = 0; i < kDigits; ++i) {
                constexpr int kPer = 256 / BN < kDigits ? 256 / BN : kDigits;
#pragma unroll
                for (int jj = 0; jj < kDigits - i; jj += kPer) {
                  const int c = kDigits - i - jj < kPer ? kDigits - i - jj : kPer;
                  mma_bf16(tmem + (uint32_t)((i + jj) * BN),
                           ad + (uint64_t)(i * kBM * kKB * 2 / 16 + 2 * kk),
                           bd + (uint64_t)(jj * BN * kKB * 2 / 16 + 2 * kk),
                           idesc_bf16(kBM, c * BN), (kb > kb0 || kk > 0 || i > 0) ? 1u : 0u);
                }
              }
            }
            mma_commit(smem_u32(&bars[kStages + s]));
          }
          if (ok) mma_commit(acc_full);
          kb0 = kb1;
        }
      }
      if (!ok) {  // drain the MMAs already issued
        mma_commit(drain);
        mbar_wait(drain, 0, nullptr);
      }
    }
  } else {
    const int quarter = warp & 3, half = (warp - 2) >> 2;
    double *stg = stg_all + (warp - 2) * 32 * 16;
    int j = 0;
    bool ok = true;
    for (int t = blockIdx.x; t < ntiles && ok; t += gridDim.x) {
      int g0, m0, n0;
      if (!tile(t, g0, m0, n0)) continue;
      n0 += half * NC;
      const int rows = kGram ? p.grp : p.M;  // rows and columns are the group's
      const int row0 = m0 + quarter * 32, row = row0 + lane;
      long long acc[NC];  // the sum in units of level 3, and 28 bits below
      uint32_t low[NC];
#pragma unroll
      for (int c = 0; c < NC; ++c) {
        acc[c] = 0;
        low[c] = 0;
      }
      auto wait_acc = [&]() {
        int okl = 0;
        if (lane == 0) okl = mbar_wait(acc_full, (uint32_t)j & 1u, abort_flag) ? 1 : 0;
        if (__shfl_sync(0xffffffffu, okl, 0) == 0) {
          if (lane == 0) {
            *abort_flag = 1;
            atomicOr(p.err, 8);
          }
          ok = false;
        }
        fence_after();
      };
      auto free_acc = [&]() {
        fence_before();
        __syncwarp();
        if (lane == 0)
          asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(acc_empty) : "memory");
      };
      const uint32_t tacc = tmem + ((uint32_t)(quarter * 32) << 16) + (uint32_t)(half * NC);
      uint32_t redo = 0;  // bit c: this row's output in column n0 + c is a plain dot product
      auto read_magnitudes = [&]() {
#pragma unroll
        for (int c0 = 0; c0 < NC; c0 += 8) {
          int v[8];
          tmem_ld8(tacc + (uint32_t)(kMagCol + c0), v);
          tmem_wait_ld();
#pragma unroll
          for (int e = 0; e < 8; ++e)
            redo |= (__int_as_float(v[e]) >= kLeast ? 0u : 1u) << (c0 + e);
        }
      };
      for (int kb0 = 0; kb0 < p.nkb; kb0 += kChunkB, ++j) {
        wait_acc();
        if (!ok) break;
#pragma unroll
        for (int c0 = 0; c0 < NC; c0 += 8) {
          int v[kDigits][8];
#pragma unroll
          for (int l = 0; l < kDigits; ++l) tmem_ld8(tacc + (uint32_t)(l * BN + c0), v[l]);
          tmem_wait_ld();
#pragma unroll
          for (int e = 0; e < 8; ++e) {
            // the level sums are integers in FP32
            auto lv = [&](int l) { return (long long)__float2int_rn(__int_as_float(v[l][e])); };
            const long long hi = ((((lv(0) << 7) + lv(1)) << 7) + lv(2) << 7) + lv(3);
            const long long lo = ((((lv(4) << 7) + lv(5)) << 7) + lv(6) << 7) + lv(7);
            low[c0 + e] += (uint32_t)lo & 0xfffffffu;
            acc[c0 + e] += hi + (lo >> 28) + (low[c0 + e] >> 28);
            low[c0 + e] &= 0xfffffffu;
          }
        }
        if (kBeside && kb0 + kChunkB >= p.nkb) read_magnitudes();
        free_acc();
      }
      if (!ok) break;
      if constexpr (!kGram && !kBeside) {
        wait_acc();
        if (!ok) break;
        read_magnitudes();
        free_acc();
        ++j;
      }
      int ea = row < rows ? p.ea[g0 + row] : kZeroRow;
      if (ea == kZeroRow) redo = ea = 0;
      const bool bad = ea == kBadRow;
      if (bad) ea = 0;
      constexpr int kS = NC < 16 ? NC : 16;  // columns staged at a time
#pragma unroll
      for (int c0 = 0; c0 < NC; c0 += kS) {
        if (n0 + c0 >= p.N) break;
#pragma unroll
        for (int c = 0; c < kS; ++c) {
          int eb = n0 + c0 + c < p.N ? p.eb[g0 + n0 + c0 + c] : 0;
          if (eb == kZeroRow) {
            redo &= ~(1u << (c0 + c));
            eb = 0;
          }
          if (bad || eb == kBadRow) {
            redo |= 1u << (c0 + c);
            eb = 0;
          }
          stg[lane * 16 + ((((c >> 1) ^ (lane & 7)) << 1) | (c & 1))] =
              scaled_to_f64(acc[c0 + c], low[c0 + c], ea + eb - 35);
        }
        const bool some = __any_sync(0xffffffffu, redo >> c0 & ((1u << kS) - 1u));
        __syncwarp();
        for (int q = lane; q < 32 * kS; q += 32) {
          const int r = q / kS, c = q % kS, col = n0 + c0 + c;
          const bool in = row0 + r < rows && col < p.N && (!kGram || col <= row0 + r);
          double v = stg[r * 16 + ((((c >> 1) ^ (r & 7)) << 1) | (c & 1))];
          if (some) {
            const uint32_t of_row = __shfl_sync(0xffffffffu, redo, r);
            const unsigned lanes = __ballot_sync(0xffffffffu, in && (of_row >> (c0 + c) & 1u));
            if (lanes) v = plain_dots(p, g0, row0 + r, col, lanes, v);
          }
          if (in) epi(p.row0 + g0 + row0 + r, col, v);
        }
        __syncwarp();
      }
    }
  }
  fence_before();
  __syncthreads();
  if (warp == 1) {
    fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem),
                 "r"(p.tmem_cols)
                 : "memory");
  }
}

// Entry (row of all groups, column <= row within the group) of a packed triangle
// in the chain's factor slot.
struct EpiSlot {
  double *L;
  size_t slot, stride;
  const int *cur;
  int mode, g;
  __device__ void operator()(int r, int c, double v) const {
    const int chain = r / g, i = r - chain * g;
    const int s = mode == 0 ? cur[chain] : 1 - cur[chain];
    L[(size_t)s * slot + (size_t)chain * stride + (size_t)i * (i + 1) / 2 + c] = v;
  }
};

// 3D map with boxes of 32 columns x box_rows x eight
bool make_map3(CUtensorMap *tm, const __nv_bfloat16 *ptr, const cuuint64_t dims[3],
               const cuuint64_t strides[2], int box_rows) {
  static PFN_cuTensorMapEncodeTiled_v12000 fn = [] {
    void *f = nullptr;
    cudaDriverEntryPointQueryResult q;
    return cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &f, 12000,
                                            cudaEnableDefault, &q) == cudaSuccess &&
                   q == cudaDriverEntryPointSuccess
               ? (PFN_cuTensorMapEncodeTiled_v12000)f
               : nullptr;
  }();
  if (!fn) return false;
  cuuint32_t box[3] = {(cuuint32_t)kKB, (cuuint32_t)box_rows, (cuuint32_t)kDigits};
  cuuint32_t es[3] = {1, 1, 1};
  return fn(tm, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, (void *)ptr, dims, strides, box, es,
            CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_64B,
            CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// ... over digit planes: dims (K, rows, planes)
bool make_digit_map(CUtensorMap *tm, const __nv_bfloat16 *ptr, int K, int rows, int ldp,
                    size_t plane, int box_rows) {
  const cuuint64_t dims[3] = {(cuuint64_t)K, (cuuint64_t)rows, (cuuint64_t)kDigits};
  const cuuint64_t strides[2] = {(cuuint64_t)ldp * 2, (cuuint64_t)plane * 2};
  return make_map3(tm, ptr, dims, strides, box_rows);
}


// ... and over the magnitudes behind them, 32 columns to a block: dims (32, rows, blocks)
// (their rows are whole blocks, padded with zeros), box (32, box_rows, eight blocks).
bool make_check_map(CUtensorMap *tm, const __nv_bfloat16 *ptr, int ldc, int rows, size_t plane,
                    int box_rows) {
  const cuuint64_t dims[3] = {(cuuint64_t)kKB, (cuuint64_t)rows, (cuuint64_t)(ldc / kKB)};
  const cuuint64_t strides[2] = {(cuuint64_t)ldc * 2, (cuuint64_t)kKB * 2};
  return make_map3(tm, ptr + kDigits * plane, dims, strides, box_rows);
}

template <int BN, bool kGram, class Epi>
cudaError_t run_gemm64_t(const Gemm64Args &a, const Epi &epi, cudaStream_t st) {
  Gemm64Params p{};
  p.grp = kGram ? a.N : 0;
  p.M = a.M;
  p.N = a.N;
  p.K = a.K;
  p.row0 = a.row0;
  p.nkb = (a.K + kKB - 1) / kKB;
  const int ldc = check_pitch(a.K, a.B.group);
  p.ncb = ldc / kKB;
  p.ea = a.ea;
  p.eb = a.B.ex;
  p.A = a.Asrc;
  p.lda = a.lda;
  p.W = a.W;
  p.der = a.der;
  p.g = a.g;
  p.ldd = a.ldd;
  p.B = a.B.src;
  p.ldb = a.B.ld;
  p.err = a.err;
  p.tmem_cols = kGram ? kDigits * BN : kTmemCols;
  CUtensorMap tmA, tmB, tmAc, tmBc;
  const int rows_b = kGram ? a.M : a.N;
  if (!make_digit_map(&tmA, a.A, a.K, a.M, a.ldp, a.plane, kBM) ||
      !make_digit_map(&tmB, a.B.d, a.K, rows_b, a.B.ldp, a.B.plane, BN))
    return cudaErrorInvalidValue;
  if (kGram) {  // never used
    tmAc = tmA;
    tmBc = tmB;
  } else if (!make_check_map(&tmAc, a.A, ldc, a.M, a.plane, kBM) ||
             !make_check_map(&tmBc, a.B.d, ldc, rows_b, a.B.plane, BN)) {
    return cudaErrorInvalidValue;
  }
  int dev = 0, sms = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (e != cudaSuccess) return e;
  const size_t smem = 1024 + kStages * (kABytes + (size_t)kDigits * BN * kKB * 2) + kStgBytes +
                      (2 * kStages + 5) * 8;
  auto k = k_gemm64<BN, kGram, Epi>;
  e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  const int ntn = (a.N + BN - 1) / BN;
  const int tiles = kGram ? a.M / a.N * ((a.N + kBM - 1) / kBM) * ntn
                          : ((a.M + kBM - 1) / kBM) * ntn;
  return launch_pdl_n(tiles, k, std::min(tiles, sms), kGemm64Threads, smem, st, tmA, tmB, tmAc,
                      tmBc, p, epi);
}

template <class Epi>
cudaError_t run_gemm64(const Gemm64Args &a, const Epi &epi, cudaStream_t st) {
  if (a.M <= 0 || a.N <= 0) return cudaSuccess;
  if (a.K <= 0 || a.K > (1 << 28) || (a.ldp & 7) || (a.plane & 7) || (a.B.ldp & 7) ||
      (a.B.plane & 7) || ((uintptr_t)a.A & 15) || ((uintptr_t)a.B.d & 15) || !a.err)
    return cudaErrorInvalidValue;
  // 64 columns a tile; 32 where those tiles would leave SMs idle (M x 200 x 1089, 64 and
  // 32 columns: 32 tiles of 64 228 and 194 us, 64 236 and 223, 96 281 and 296, 256 576 and 606;
  // a layer with GELU, whose FP64 epilogue gains from more CTAs at any size: three of 400,
  // 56 tiles 514 and 340, 112 644 and 614, 448 2013 and 1977)
  const long t64 = (long)((a.M + kBM - 1) / kBM) * ((a.N + 63) / 64);
  if (a.N <= 32 || t64 < 100) return run_gemm64_t<32, false>(a, epi, st);
  return run_gemm64_t<64, false>(a, epi, st);
}

}  // namespace

int digit_pitch(int K) { return (K + 7) & ~7; }
size_t digit_bytes(size_t rows, int K, int group) {
  return rows * (2 * ((size_t)kDigits * digit_pitch(K) + check_pitch(K, group)));
}

cudaError_t launch_split64(int rows, int K, const double *src, int ld, const double *W,
                           const double *der, int g, int ldd, int row0, const int *fk, int fsign,
                           __nv_bfloat16 *dst, int ldp, size_t plane,
                           int *ex, cudaStream_t st, Magnitudes mags) {
  if (rows <= 0) return cudaSuccess;
  if (K <= 0 || ldp < K || (ldp & 7) || (plane & 7)) return cudaErrorInvalidValue;
  SplitArgs a{rows, K, ldp, plane, src, ld, W, der, g, ldd, row0, fk, fsign, mags, dst, ex};
  const int grid = (rows + 7) / 8;
  auto k = ldp <= 128 ? k_split64<1> : ldp <= 256 ? k_split64<2> : ldp <= 512 ? k_split64<4>
                                                                              : k_split64<0>;
  return launch_pdl(k, grid, 256, 0, st, a);
}

cudaError_t launch_col_exp(int rows, int K, const double *B, int ld, int *fk, cudaStream_t st) {
  k_col_exp<<<(K + 127) / 128, 128, 0, st>>>(rows, K, B, ld, fk);
  return cudaGetLastError();
}

cudaError_t launch_count_sparse(int rows, int K, const __nv_bfloat16 *digits, size_t plane,
                                const int *ex, int *sparse, cudaStream_t st) {
  k_count_sparse<<<(rows + 7) / 8, 256, 0, st>>>(
      rows, K, reinterpret_cast<const uint16_t *>(digits + kDigits * plane), ex, sparse);
  return cudaGetLastError();
}

cudaError_t gram64_slots(int groups, int g, int K, const double *J, int ldj,
                         const __nv_bfloat16 *digits, const int *ex, int ldp, size_t plane,
                         double *L, size_t slot, size_t stride, const int *cur, int mode, int *err,
                         cudaStream_t st) {
  if (groups <= 0) return cudaSuccess;
  if (g < 1 || K <= 0 || (long long)groups * g > 0x7fffffffLL || (ldp & 7) || (plane & 7) ||
      ((uintptr_t)digits & 15) || !err)
    return cudaErrorInvalidValue;
  Gemm64Args a;
  a.M = groups * g;
  a.N = g;
  a.K = K;
  a.A = digits;
  a.ea = ex;
  a.ldp = ldp;
  a.plane = plane;
  a.Asrc = J;
  a.lda = ldj;
  a.B.d = digits;
  a.B.ex = ex;
  a.B.ldp = ldp;
  a.B.plane = plane;
  a.B.src = J;
  a.B.ld = ldj;
  a.err = err;
  const EpiSlot epi{L, slot, stride, cur, mode, g};
  return g <= 32 ? run_gemm64_t<32, true>(a, epi, st) : run_gemm64_t<64, true>(a, epi, st);
}

cudaError_t gemm64_store(const Gemm64Args &a, double *out, int ldo, cudaStream_t st) {
  return run_gemm64(a, EpiStore<double>{out, ldo}, st);
}
cudaError_t gemm64_bias_act(const Gemm64Args &a, const double *bias, int act, double *out,
                            double *der, int ldo, cudaStream_t st) {
  return run_gemm64(a, EpiBiasAct<double>{bias, act, out, der, ldo}, st);
}
cudaError_t gemm64_scale_group(const Gemm64Args &a, const double *scale, int lds, int group,
                               double *out, int ldo, cudaStream_t st) {
  return run_gemm64(a, EpiScaleGroup<double>{scale, lds, group, out, ldo}, st);
}
cudaError_t gemm64_coef(const Gemm64Args &a, const double *coef, int ldc, double c, double *out,
                        int ldo, cudaStream_t st) {
  return run_gemm64(a, EpiCoef<double>{coef, ldc, c, out, ldo}, st);
}
cudaError_t gemm64_field(const Gemm64Args &a, const int *acc_flag, double s, double c, double *m,
                         const double *Mf, int ldm, cudaStream_t st) {
  return run_gemm64(a, EpiField<double>{acc_flag, s, c, m, Mf, ldm}, st);
}

}  // namespace dino
