// POTRS by block inverses: L Y = B, then L^T X = Y, in blocks of up to 512 rows.
//
// The wavefront sweeps of k_potrs.cu hand 64-row blocks from CTA to CTA; a link costs 2.5 us with one
// right-hand side (the handoff through L2) and 15 us with 16 (the link's products on one SM), n / 64
// of them in a row.  Here the diagonal blocks of `blk` rows are inverted first, all at once: blocks of
// 64 by substitution, then doubled to 128, 256 and 512 rows, W21 = -W22 (L21 W11) by digit products
// (k_gemm_f64.cu).  A sweep is then n / blk steps of two launches that fill the
// chip,
//   y_r = W_r b_r,   b_i -= L_ir y_r for the rows i still to come,
// and the same with the transposes on the way back.  The inverses serve every solve with the
// factor (the corrections of a refinement, further groups of 16 right-hand sides).
//
// Both products take 16 rows at a time and up to 512 inner terms, a warp 16 (few rows,
// solve_step_kernel) or 64 of them (many, solve_wide_kernel).  The entries go from memory to registers
// in the order the mma fragments want them, are cut into 8-bit digits there and multiplied exactly by
// 36 (few rows) or 28 mma per 16 terms (digits.cuh).  Scales: term k by its largest right-hand side, then a
// row of P and a column of Y by the largest entry among the terms (of the warp, whose sums are then
// added in FP64 in a fixed order; in the wide kernel of all, whose sums stay integers until the end),
// so that powers of two that scale the unknowns change nothing.
//
// Several right-hand sides share the terms' scales, and where one is large in a term that the others
// hardly see, the others' digits are too few.  One more mma per 16 terms, of the digits' magnitudes, therefore
// estimates every output's sum |a| |y| against its scales, and outputs below a line are computed by
// FP64 FMAs (a term per lane; by all lanes for the warp's outputs where there are many).  Per term the
// scales' product is held to 2^-61.5 with eight digits and 2^-54.3 with seven, ordinary digits taken
// (2^-58.9 and 2^-51.4 at worst), so that the lines at 2^-13 of a warp's 16 terms and 2^-4 of a wide
// tile's 512 both leave 2^-46 of sum |a| |y| (2^-42 and 2^-38 at worst); the sweeps' double-float products
// keep 2^-44 at worst.  Ordinary columns stay above the lines but for one output in 1000 of the diagonal
// blocks (seven digits there: one in 40, hence the eight); n = 4096, 16 right-hand sides: 562 -> 601 us
// with the estimate (1926 by the sweeps).
// What bounds it: latency, 5 us a step with few rows and 8 to 11 us with many (at n = 4096 and one
// right-hand side 170 us of inverses, most of it the last doubling, then 30 steps); from n = 8192 on the
// wide kernel's tiles, 3 to 5 us each of load latency and integer work at two warps per scheduler (with
// the warps' sums converted and added in FP64, ~2000 instead of ~1600 instructions a tile: n = 4096 560
// -> 542 us, 8192 1246 -> 1186, 16384 3232 -> 2995 with 16 right-hand sides).  Solves against the
// sweeps', us with 1, 4 and 16 right-hand sides:
//   n = 64 21 21 29 (56 61 85), 128 43 43 50 (105 113 144), 2048 238 243 303 (249 367 997),
//   4 and 16: 4096 436 590 (636 1908), 8192 933 1314 (1204 3788), 16384 2225 3306 (3191 8756).
// Backward errors entry by entry are at or below 1e-14 of |A| |x| where the sweeps' (whose double-float
// products keep 44 bits and drop what is 2^-74 below its group) reach 1e-13 for ordinary matrices and 1 for
// ones in mixed units.  Tiles that meet a NaN or an infinity use FP64 FMAs.
#include <cooperative_groups.h>

#include <climits>

#include "digits.cuh"
#include "hrp_internal.cuh"

namespace cg = cooperative_groups;

namespace hrp {
namespace {

constexpr int kThreads = 256;
constexpr int kRows = 16;
constexpr int kSd = kByteDig, kWd = kDig;        // digits per operand (few rows, many), weights s + t below kept
// smallest sum |a| |y| against the scales that the digits cover, of a warp's 16 terms and of a wide tile's, in
// units of the first digits' product
constexpr float kCoveredStep = 0x1p-13f * 4096.f, kCoveredWide = 0x1p-4f * 4096.f;
constexpr int kManyLow = 4;                      // lanes with outputs to recompute above which a warp recomputes all
constexpr int kNone = -4096;                     // below every exponent of a right-hand side against its term's
constexpr int kNoRow = -(1 << 20);               // the scale of a row of zeros

// The inverse of a 64 x 64 diagonal block of L (block blockIdx.y), 8 of its columns per CTA: columns
// blockIdx.x + 8 u, two to a warp, so that every CTA has as much to do.  16 lanes hold a column, rows
// q, q + 16, ..; substitution in FP64, a step costs one reciprocal product, a broadcast and up to four
// FMAs, and what bounds it is that chain (64 steps of ~150 clocks), from n = 4096 on the FP64 pipe.
// Row i goes to W + i blk at the block's columns, zeros after it.
__global__ void __launch_bounds__(128)
inverse64_kernel(const double* __restrict__ L, int ldl, int n, double* __restrict__ W, int blk) {
  __shared__ double Ls[64][65];                  // [k][i]
  __shared__ double rinv[64];
  pdl_wait();
  pdl_trigger();
  const int c0 = 64 * blockIdx.y, m = min(64, n - c0), off = c0 % blk;
  const int tid = threadIdx.x, lane = tid & 31, q = lane & 15;
#pragma unroll
  for (int u = 0; u < 32; ++u) {
    const int i = tid & 63, k = (tid >> 6) + 2 * u;
    Ls[k][i] = (i < m && k <= i) ? L[(size_t)(c0 + k) * ldl + c0 + i] : 0.0;
  }
  for (int e = tid; e < 8 * (blk - off - 64); e += 128) {
    const int i = (int)blockIdx.x + 8 * (e / (blk - off - 64));
    if (i < m) W[(size_t)(c0 + i) * blk + off + 64 + e % (blk - off - 64)] = 0.0;
  }
  __syncthreads();
  if (tid < 64) rinv[tid] = tid < m ? 1.0 / Ls[tid][tid] : 1.0;
  __syncthreads();
  const int first = (int)blockIdx.x + 16 * (tid >> 5), c = first + 8 * (lane >> 4);
  double y[4];
#pragma unroll
  for (int p = 0; p < 4; ++p) y[p] = q + 16 * p == c ? 1.0 : 0.0;
#pragma unroll
  for (int p = 0; p < 4; ++p) {
    if (16 * p + 15 < first) continue;           // whole warps
    for (int kk = 0; kk < 16; ++kk) {
      const int k = 16 * p + kk;
      const double v = __shfl_sync(0xffffffffu, y[p], (lane & 16) | kk) * rinv[k];
      if (q == kk) y[p] = v;
      else if (q > kk) y[p] = fma(-Ls[k][q + 16 * p], v, y[p]);
#pragma unroll
      for (int r = p + 1; r < 4; ++r) y[r] = fma(-Ls[k][q + 16 * r], v, y[r]);
    }
  }
#pragma unroll
  for (int p = 0; p < 4; ++p) {
    const int i = q + 16 * p;
    if (i < m && c < 64) W[(size_t)(c0 + i) * blk + off + c] = i >= c ? y[p] : 0.0;
  }
}

// What the two product kernels share: the fragments of a warp's 16 KS terms from k0.
// A: element (half-row h, k step s, j) is row r0 + g + 8 h, k = k0 + 16 s + t2 + (j & 1) + 8 (j >> 1), with
// g = lane / 4, t2 = 2 (lane % 4); P(i, k) at P[k ldp + i], or TRANS: P[i ldp + k]
template <bool TRANS, int KS>
__device__ __forceinline__ void load_rows(double (&a)[2][KS][4], const double* __restrict__ P, int ldp, int r0, int rows, int k0,
                                          int K) {
  const int g = (threadIdx.x & 31) >> 2, t2 = 2 * (threadIdx.x & 3);
#pragma unroll
  for (int s = 0; s < KS; ++s)
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int k = k0 + 16 * s + t2 + (j & 1) + 8 * (j >> 1);
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int i = r0 + g + 8 * h;
        a[h][s][j] = (i < rows && k < K) ? (TRANS ? P[(size_t)i * ldp + k] : P[(size_t)k * ldp + i]) : 0.0;
      }
    }
}
// Y: element (half h, s, j) is right-hand side g + 8 h, the same k
template <int NH, int KS>
__device__ __forceinline__ void load_rhs(double (&y)[NH][KS][4], const double* __restrict__ Y, int ldy, int nrhs, int k0, int K) {
  const int g = (threadIdx.x & 31) >> 2, t2 = 2 * (threadIdx.x & 3);
#pragma unroll
  for (int s = 0; s < KS; ++s)
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int k = k0 + 16 * s + t2 + (j & 1) + 8 * (j >> 1);
#pragma unroll
      for (int h = 0; h < NH; ++h) {
        const int c = g + 8 * h;
        y[h][s][j] = (c < nrhs && k < K) ? Y[(size_t)c * ldy + k] : 0.0;
      }
    }
}
// The scales: of term k the largest exponent field among its right-hand sides, over the eight lanes (and
// halves) that hold them, two terms a word of ek; of a right-hand side (ey) the largest of its fields
// against the terms' scales; of a row (ea) the largest field times its term's scale.  special: a NaN or
// an infinity (in some lane).
template <int KS>
__device__ __forceinline__ int term(const unsigned (&ek)[KS][2], int s, int j) {
  return (int)((ek[s][j >> 1] >> (16 * (j & 1))) & 0xffffu);
}
template <int NH, int KS>
__device__ __forceinline__ void rhs_scales(const double (&y)[NH][KS][4], unsigned (&ek)[KS][2], int (&ey)[NH], bool& special) {
#pragma unroll
  for (int s = 0; s < KS; ++s)
#pragma unroll
    for (int p = 0; p < 2; ++p) {
      unsigned w = 0x00010001u;
#pragma unroll
      for (int h = 0; h < NH; ++h)
        w = __vmaxu2(w, (unsigned)dig_field(y[h][s][2 * p]) | ((unsigned)dig_field(y[h][s][2 * p + 1]) << 16));
#pragma unroll
      for (int o = 4; o < 32; o <<= 1) w = __vmaxu2(w, __shfl_xor_sync(0xffffffffu, w, o));
      special |= (w & 0xffffu) == 0x7ffu || (w >> 16) == 0x7ffu;
      ek[s][p] = w;
    }
#pragma unroll
  for (int h = 0; h < NH; ++h) {
    ey[h] = kNone;
#pragma unroll
    for (int s = 0; s < KS; ++s)
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const double v = y[h][s][j];             // (words: a 64-bit test becomes a comparison on the FP64 pipe)
        if (((unsigned)__double2hiint(v) << 1) | (unsigned)__double2loint(v)) ey[h] = max(ey[h], max(dig_field(v), 1) - term<KS>(ek, s, j));
      }
#pragma unroll
    for (int o = 1; o < 4; o <<= 1) ey[h] = max(ey[h], __shfl_xor_sync(0xffffffffu, ey[h], o));
  }
}
template <int KS>
__device__ __forceinline__ void row_scales(const double (&a)[2][KS][4], const unsigned (&ek)[KS][2], int (&ea)[2], bool& special) {
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    ea[h] = INT_MIN;
    unsigned any = 0;
#pragma unroll
    for (int s = 0; s < KS; ++s)
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const int f = dig_field(a[h][s][j]);
        special |= f == 0x7ff;
        any |= (unsigned)__double2hiint(a[h][s][j]) | (unsigned)__double2loint(a[h][s][j]);
        ea[h] = max(ea[h], max(f, 1) + term<KS>(ek, s, j));
      }
    if (any == 0) ea[h] = kNoRow;
#pragma unroll
    for (int o = 1; o < 4; o <<= 1) ea[h] = max(ea[h], __shfl_xor_sync(0xffffffffu, ea[h], o));
  }
}
// the digits of a k step of the right-hand sides
template <int ND, int NH, int KS>
__device__ __forceinline__ void rhs_digits(const double (&y)[NH][KS][4], const unsigned (&ek)[KS][2], const int (&ey)[NH], int s,
                                           uint32_t (&bf)[ND][NH][2]) {
#pragma unroll
  for (int h = 0; h < NH; ++h) {
    unsigned long long m[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) m[j] = (unsigned long long)dig_fix(y[h][s][j], ey[h] + term<KS>(ek, s, j)) + kByteBias;
#pragma unroll
    for (int d = 0; d < ND; ++d) {
      bf[d][h][0] = byte_pair(m[0], m[1], d);
      bf[d][h][1] = byte_pair(m[2], m[3], d);
    }
  }
}
// |first digit| + 2^-8 |second| of a pair: the magnitudes behind the estimate of sum |a| |y|
__device__ __forceinline__ uint32_t pair_abs(uint32_t d0, uint32_t d1) {
  d0 &= 0x7fff7fffu;
  d1 &= 0x7fff7fffu;
  const __half2 v = __hfma2(*reinterpret_cast<const __half2*>(&d1), __half2half2(__ushort_as_half(0x1c00)),      // 2^-8
                            *reinterpret_cast<const __half2*>(&d0));
  return *reinterpret_cast<const uint32_t*>(&v);
}
__device__ __forceinline__ void row_fragment(const unsigned long long (&m0)[4], const unsigned long long (&m1)[4], int d,
                                             uint32_t (&af)[4]) {
  af[0] = byte_pair(m0[0], m0[1], d);
  af[1] = byte_pair(m1[0], m1[1], d);
  af[2] = byte_pair(m0[2], m0[3], d);
  af[3] = byte_pair(m1[2], m1[3], d);
}
// the products of a k step: rows(d) gives digit d of the rows, bf[d] the right-hand sides'; est: the estimate, from
// the first digits or (FINE) the first two
template <int ND, bool FINE, int NH, class Rows>
__device__ __forceinline__ void step_products(float (&acc)[ND][NH][4], float (&est)[NH][4], const Rows& rows,
                                              const uint32_t (&bf)[ND][NH][2]) {
  uint32_t first[4];
#pragma unroll
  for (int d = 0; d < ND; ++d) {
    uint32_t af[4];
    rows(d, af);
#pragma unroll
    for (int e = 0; e < ND - d; ++e)
#pragma unroll
      for (int h = 0; h < NH; ++h) dig_mma(acc[d + e][h], af, bf[e][h][0], bf[e][h][1]);
    if (d == 0) {
#pragma unroll
      for (int q = 0; q < 4; ++q) first[q] = FINE ? af[q] : af[q] & 0x7fff7fffu;
    }
    if (FINE && d == 1) {
#pragma unroll
      for (int q = 0; q < 4; ++q) first[q] = pair_abs(first[q], af[q]);
    }
    if (d == (FINE ? 1 : 0)) {
#pragma unroll
      for (int h = 0; h < NH; ++h)
        dig_mma(est[h], first, FINE ? pair_abs(bf[0][h][0], bf[1][h][0]) : bf[0][h][0] & 0x7fff7fffu,
                FINE ? pair_abs(bf[0][h][1], bf[1][h][1]) : bf[0][h][1] & 0x7fff7fffu);
    }
  }
}
// the warp's sums to part[row][right-hand side]: weights 2^(-12 - 8 w) joined in units of 2^-28 (w < 3) and
// 2^-68, and these in units of 2^-58 (16 terms below 1).  Returns the outputs that the digits do not
// cover: bit 4 h + register.
template <int NH>
__device__ __forceinline__ unsigned store_sums(const float (&acc)[kSd][NH][4], const float (&est)[NH][4], const int (&ea)[2],
                                               const int (&ey)[NH], bool estimate, double (*part)[8 * NH]) {
  const int lane = threadIdx.x & 31, g = lane >> 2, t2 = 2 * (lane & 3);
  unsigned low = 0;
#pragma unroll
  for (int h = 0; h < NH; ++h)
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      long long hi = 0, lo = 0;
#pragma unroll
      for (int w = 0; w < 3; ++w) hi = (hi << 8) + __float2int_rn(acc[w][h][q]);
#pragma unroll
      for (int w = 3; w < kSd; ++w) lo = (lo << 8) + __float2int_rn(acc[w][h][q]);
      const int c = t2 + (q & 1), ec = __shfl_sync(0xffffffffu, ey[h], 4 * c);
      part[g + 8 * (q >> 1)][8 * h + c] = dig_to_double((hi << 30) + ((lo + 512) >> 10), ea[q >> 1] + ec - 2 * 1022 - 58);
      if (estimate && est[h][q] < kCoveredStep && ea[q >> 1] != kNoRow && ec != kNone) low |= 1u << (4 * h + q);
    }
  return low;
}
// the same sums by FP64 FMAs over the terms kb .. ke - 1 (row i: from lo(i), below hi(i))
template <int NH, bool TRANS, class Lo, class Hi>
__device__ __forceinline__ void plain_sums(const double* __restrict__ P, int ldp, int r0, int rows, const double* __restrict__ Y, int ldy,
                                           int nrhs, Lo lo, Hi hi, double (*part)[8 * NH]) {
  for (int e = threadIdx.x & 31; e < kRows * 8 * NH; e += 32) {
    const int i = r0 + e / (8 * NH), c = e % (8 * NH);
    double v = 0.0;
    if (i < rows && c < nrhs)
      for (int k = lo(i); k < hi(i); ++k)
        v = fma(TRANS ? P[(size_t)i * ldp + k] : P[(size_t)k * ldp + i], Y[(size_t)c * ldy + k], v);
    part[e / (8 * NH)][c] = v;
  }
}
template <int NH>
__device__ __forceinline__ double sum_parts(const double (*part)[kRows][8 * NH], int i, int c) {
  return ((part[0][i][c] + part[1][i][c]) + (part[2][i][c] + part[3][i][c])) +
         ((part[4][i][c] + part[5][i][c]) + (part[6][i][c] + part[7][i][c]));
}

// O(i, c) = sum_k P(i, k) Y(k, c) (ADD: O -= ...) for few rows i < rows, k < K <= 512, c < nrhs <= 8 NH.
// TRI 1: P(i, k) = 0 for k > i; TRI 2: for k < i.  A CTA covers 128 terms, a warp 16, and a cluster of
// ceil(K / 128) CTAs in y the row tile; the others leave their sums in CTA 0's shared memory.
template <int NH, bool TRANS, bool ADD, int TRI>
__global__ void __launch_bounds__(kThreads, 2)
solve_step_kernel(const double* __restrict__ P, int ldp, int rows, int K, const double* __restrict__ Y, int ldy,
                  double* __restrict__ O, int ldo, int nrhs) {
  // CTA 0 of a cluster must have started before the others write to its shared memory
  asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory");
  pdl_wait();
  pdl_trigger();
  __shared__ double part[8][kRows][8 * NH];
  __shared__ double from[3][kRows * 8 * NH];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int r0 = blockIdx.x * kRows, k0 = 128 * (int)blockIdx.y + 16 * warp;
  if (k0 < K && !(TRI == 1 && k0 > r0 + kRows - 1) && !(TRI == 2 && k0 + 15 < r0)) {
    double a[2][1][4], y[NH][1][4];
    load_rows<TRANS, 1>(a, P, ldp, r0, rows, k0, K);
    load_rhs<NH, 1>(y, Y, ldy, nrhs, k0, K);
    unsigned ek[1][2];
    int ea[2], ey[NH];
    bool special = false;
    rhs_scales<NH, 1>(y, ek, ey, special);
    row_scales<1>(a, ek, ea, special);
    if (__any_sync(0xffffffffu, special)) {
      plain_sums<NH, TRANS>(P, ldp, r0, rows, Y, ldy, nrhs, [&](int i) { return TRI == 2 ? max(k0, i) : k0; },
                            [&](int i) { return min(min(K, k0 + 16), TRI == 1 ? i + 1 : K); }, part[warp]);
    } else {
      float acc[kSd][NH][4] = {}, est[NH][4] = {};
      uint32_t bf[kSd][NH][2];
      rhs_digits<kSd, NH, 1>(y, ek, ey, 0, bf);
      unsigned long long m[2][4];
#pragma unroll
      for (int j = 0; j < 4; ++j)
#pragma unroll
        for (int h = 0; h < 2; ++h) m[h][j] = (unsigned long long)dig_fix(a[h][0][j], ea[h] - term<1>(ek, 0, j)) + kByteBias;
      const bool estimate = nrhs > 1;                            // alone, a column sets its own terms' scales
      step_products<kSd, true, NH>(acc, est, [&](int d, uint32_t (&af)[4]) { row_fragment(m[0], m[1], d, af); }, bf);
      const unsigned low = store_sums<NH>(acc, est, ea, ey, estimate, part[warp]);
      const unsigned lanes = __ballot_sync(0xffffffffu, low != 0);
      if (lanes) {
        auto lo = [&](int i) { return TRI == 2 ? max(k0, i) : k0; };
        auto hi = [&](int i) { return min(min(K, k0 + 16), TRI == 1 ? i + 1 : K); };
        __syncwarp();
        if (__popc(lanes) > kManyLow) {
          plain_sums<NH, TRANS>(P, ldp, r0, rows, Y, ldy, nrhs, lo, hi, part[warp]);
        } else {
          // a term per lane
#pragma unroll 1
          for (int q = 0; q < 4 * NH; ++q)
            for (unsigned who = __ballot_sync(0xffffffffu, (low >> q) & 1); who; who &= who - 1) {
              const int src = __ffs(who) - 1, i = (src >> 2) + 8 * ((q >> 1) & 1), c = 8 * (q >> 2) + 2 * (src & 3) + (q & 1);
              const int k = lo(r0 + i) + (lane & 15);
              double v = 0.0;
              if (k < hi(r0 + i)) v = (TRANS ? P[(size_t)(r0 + i) * ldp + k] : P[(size_t)k * ldp + r0 + i]) * Y[(size_t)c * ldy + k];
#pragma unroll
              for (int o = 8; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
              if (lane == 0) part[warp][i][c] = v;
            }
        }
      }
    }
  } else {
    for (int e = lane; e < kRows * 8 * NH; e += 32) part[warp][e / (8 * NH)][e % (8 * NH)] = 0.0;
  }
  __syncthreads();
  const int i = tid % kRows, c = tid / kRows;
  const bool out = c < 8 * NH && r0 + i < rows && c < nrhs;
  double v = out ? sum_parts<NH>(part, i, c) : 0.0;
  cg::cluster_group cluster = cg::this_cluster();
  const int rank = (int)cluster.block_rank();
  asm volatile("barrier.cluster.wait.aligned;" ::: "memory");
  if (rank > 0 && out) cluster.map_shared_rank(&from[rank - 1][0], 0)[tid] = v;
  cluster.sync();
  if (rank > 0 || !out) return;
  for (int q = 1; q < (int)gridDim.y; ++q) v += from[q - 1][tid];
  double* o = O + (size_t)c * ldo + r0 + i;
  *o = ADD ? *o - v : v;
}
static_assert(kRows * 16 == kThreads, "one output per thread at 16 right-hand sides");

// O -= P Y for many rows: a warp keeps 64 terms, whose right-hand sides' digits it cuts once and holds in
// shared memory as mma fragments, and the CTA runs over row tiles, the next tile's entries in flight
// during the products.  The warps share the tile's scales (a row's largest entry over all terms, found
// a tile ahead), so that their sums are added as 64-bit integers and converted once.
constexpr int kWide = 4;                         // k steps per warp
template <int NH>
constexpr int wide_smem() {
  return 8 * kWide * kWd * NH * 32 * 8 + 2 * 8 * kRows * 8 * NH * (8 + 4);
}
template <int NH, bool TRANS>
__global__ void __launch_bounds__(kThreads, 1)
solve_wide_kernel(const double* __restrict__ P, int ldp, int rows, int K, const double* __restrict__ Y, int ldy,
                  double* __restrict__ O, int ldo, int nrhs) {
  pdl_wait();
  pdl_trigger();
  extern __shared__ __align__(16) unsigned char smem[];
  // by tile modulo 3: a tile's rows are scaled while the one before is multiplied and the words of the one
  // after it are cleared
  __shared__ int s_ea[3][kRows], s_special[3];
  __shared__ int s_ey[8 * NH], s_yspecial;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, g = lane >> 2;
  uint2 (*bfs)[kWd][NH][32] = reinterpret_cast<uint2 (*)[kWd][NH][32]>(smem) + warp * kWide;       // [s][digit][half][lane]
  // [parity]: the warps' sums, and their estimates of sum |a| |y|
  long long (*parts)[8][kRows][8 * NH] =
      reinterpret_cast<long long (*)[8][kRows][8 * NH]>(smem + 8 * kWide * kWd * NH * 32 * 8);
  float (*ests)[8][kRows][8 * NH] = reinterpret_cast<float (*)[8][kRows][8 * NH]>(parts + 2);
  const bool estimate = nrhs > 1;
  const int k0 = 16 * kWide * warp;
  const bool act = k0 < K;
  const int step = (int)gridDim.x * kRows;
  int r0 = (int)blockIdx.x * kRows;
  if (tid < 3 * kRows) (&s_ea[0][0])[tid] = kNoRow;
  if (tid < 3) s_special[tid] = 0;
  if (tid < 8 * NH) s_ey[tid] = kNone;
  if (tid == 0) s_yspecial = 0;
  double a[2][kWide][4];
  if (act) load_rows<TRANS, kWide>(a, P, ldp, r0, rows, k0, K);
  unsigned ek[kWide][2];
  int ey[NH];
  double y[NH][kWide][4];
  __syncthreads();
  if (act) {
    bool special = false;
    load_rhs<NH, kWide>(y, Y, ldy, nrhs, k0, K);
    rhs_scales<NH, kWide>(y, ek, ey, special);
    if ((lane & 3) == 0) {
#pragma unroll
      for (int h = 0; h < NH; ++h) atomicMax(&s_ey[8 * h + g], ey[h]);
    }
    if (special) s_yspecial = 1;
  }
  auto scale_rows = [&](int buf) {
    int ea[2];
    bool special = false;
    row_scales<kWide>(a, ek, ea, special);
    if ((lane & 3) == 0) {
      atomicMax(&s_ea[buf][g], ea[0]);
      atomicMax(&s_ea[buf][g + 8], ea[1]);
    }
    if (special) s_special[buf] = 1;
  };
  if (act) scale_rows(0);
  __syncthreads();
  if (act && !s_yspecial) {
#pragma unroll
    for (int h = 0; h < NH; ++h) ey[h] = s_ey[8 * h + g];
#pragma unroll
    for (int s = 0; s < kWide; ++s) {
      uint32_t bf[kWd][NH][2];
      rhs_digits<kWd, NH, kWide>(y, ek, ey, s, bf);
#pragma unroll
      for (int d = 0; d < kWd; ++d)
#pragma unroll
        for (int h = 0; h < NH; ++h) bfs[s][d][h][lane] = make_uint2(bf[d][h][0], bf[d][h][1]);
    }
    __syncwarp();
  }
  const int i = tid % kRows, c = tid / kRows;
  for (int t = 0, par = 0, buf = 0; r0 < rows; r0 += step, ++t, par ^= 1) {
    const bool out = c < 8 * NH && r0 + i < rows && c < nrhs;
    double* o = O + (size_t)c * ldo + r0 + i;
    const double o0 = out ? *o : 0.0;
    const int next = buf == 2 ? 0 : buf + 1, after = 3 - buf - next;
    const bool plain = s_yspecial || s_special[buf];             // the same in every warp
    const bool more = r0 + step < rows;
    if (tid < kRows) s_ea[after][tid] = kNoRow;
    if (tid == 0) s_special[after] = 0;
    if (plain) {
      double (*part)[8 * NH] = reinterpret_cast<double (*)[8 * NH]>(parts[par][warp]);
      plain_sums<NH, TRANS>(P, ldp, r0, rows, Y, ldy, nrhs, [&](int) { return k0; },
                            [&](int) { return min(K, k0 + 16 * kWide); }, part);
      if (act && more) {
        load_rows<TRANS, kWide>(a, P, ldp, r0 + step, rows, k0, K);
        scale_rows(next);
      }
    } else if (act) {
      const int ea[2] = {s_ea[buf][g], s_ea[buf][g + 8]};
      unsigned long long m[kWide][2][4];
#pragma unroll
      for (int s = 0; s < kWide; ++s)
#pragma unroll
        for (int j = 0; j < 4; ++j)
#pragma unroll
          for (int h = 0; h < 2; ++h)
            m[s][h][j] = (unsigned long long)dig_fix(a[h][s][j], ea[h] - term<kWide>(ek, s, j)) + kByteBias;
      if (more) load_rows<TRANS, kWide>(a, P, ldp, r0 + step, rows, k0, K);
      float acc[kWd][NH][4] = {}, est[NH][4] = {};
#pragma unroll
      for (int s = 0; s < kWide; ++s) {
        uint32_t bf[kWd][NH][2];
#pragma unroll
        for (int d = 0; d < kWd; ++d)
#pragma unroll
          for (int h = 0; h < NH; ++h) {
            const uint2 v = bfs[s][d][h][lane];
            bf[d][h][0] = v.x;
            bf[d][h][1] = v.y;
          }
        step_products<kWd, false, NH>(acc, est, [&](int d, uint32_t (&af)[4]) { row_fragment(m[s][0], m[s][1], d, af); }, bf);
      }
      // weights 2^(-12 - 8 w) joined in units of 2^-54 (512 terms below 1)
#pragma unroll
      for (int h = 0; h < NH; ++h)
#pragma unroll
        for (int q = 0; q < 4; q += 2) {
          long long v[2];
#pragma unroll
          for (int u = 0; u < 2; ++u) {
            long long hi = 0, lo = 0;
#pragma unroll
            for (int w = 0; w < 3; ++w) hi = (hi << 8) + __float2int_rn(acc[w][h][q + u]);
#pragma unroll
            for (int w = 3; w < kWd; ++w) lo = (lo << 8) + __float2int_rn(acc[w][h][q + u]);
            v[u] = (hi << 26) + (lo >> 6);
          }
          const int i = g + 4 * q, c = 8 * h + 2 * (lane & 3);
          *reinterpret_cast<longlong2*>(&parts[par][warp][i][c]) = make_longlong2(v[0], v[1]);
          *reinterpret_cast<float2*>(&ests[par][warp][i][c]) = make_float2(est[h][q], est[h][q + 1]);
        }
      if (more) scale_rows(next);
    } else {
      for (int e = lane; e < kRows * 8 * NH; e += 32) {
        parts[par][warp][e / (8 * NH)][e % (8 * NH)] = 0;
        ests[par][warp][e / (8 * NH)][e % (8 * NH)] = 0.f;
      }
    }
    // one barrier per tile: the sums of the next go to the other half
    const int er = s_ea[buf][i];
    bool low = false;
    __syncthreads();
    if (out) {
      if (plain) {
        *o = o0 - sum_parts<NH>(reinterpret_cast<const double (*)[kRows][8 * NH]>(parts[par]), i, c);
      } else {
        long long v = 0;
#pragma unroll
        for (int w = 0; w < 8; ++w) v += parts[par][w][i][c];
        float est = 0.f;
#pragma unroll
        for (int w = 0; w < 8; ++w) est += ests[par][w][i][c];
        low = estimate && est < kCoveredWide && er != kNoRow && s_ey[c] != kNone;
        if (!low) *o = o0 - dig_to_double(v, er + s_ey[c] - 2 * 1022 - 54);
      }
    }
    // outputs the digits do not cover: FP64 FMAs, the terms over the warp's lanes
    for (unsigned who = __ballot_sync(0xffffffffu, low); who; who &= who - 1) {
      const int src = __ffs(who) - 1, si = r0 + src % kRows, sc = (tid - lane + src) / kRows;
      double f = 0.0;
      for (int k = lane; k < K; k += 32) f = fma(TRANS ? P[(size_t)si * ldp + k] : P[(size_t)k * ldp + si], Y[(size_t)sc * ldy + k], f);
#pragma unroll
      for (int d = 16; d > 0; d >>= 1) f += __shfl_xor_sync(0xffffffffu, f, d);
      if (lane == src) *o = o0 - f;
    }
    buf = next;
  }
}

template <int NH, bool TRANS, bool ADD, int TRI>
cudaError_t launch_step(const double* P, int ldp, int rows, int K, const double* Y, int ldy, double* O, int ldo, int nrhs,
                        cudaStream_t s) {
  if (rows <= 0) return cudaSuccess;
  const int tiles = (rows + kRows - 1) / kRows, ky = (K + 127) / 128;
  cudaLaunchConfig_t cfg = {};
  cfg.blockDim = dim3(kThreads);
  cfg.stream = s;
  cudaLaunchAttribute at[2];
  const int np = launch_ctx().pdl ? 1 : 0;
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = np;
  if constexpr (ADD) {
    // the wide kernel where the clusters would be more than two CTAs per SM (n = 3000 .. 8192 with 16
    // right-hand sides: 2 to 4 % above lines at one half, one and four CTAs)
    if (tiles * ky > 2 * device_sm_count()) {
      static unsigned long long attr_mask = 0;
      const unsigned long long attr_bit = dev_bit();
      if (!(attr_mask & attr_bit)) {
        cudaError_t e = cudaFuncSetAttribute(solve_wide_kernel<NH, TRANS>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             wide_smem<NH>());
        if (e != cudaSuccess) return e;
        attr_mask |= attr_bit;
      }
      const int per = (tiles + device_sm_count() - 1) / device_sm_count();
      cfg.gridDim = dim3((tiles + per - 1) / per);
      cfg.dynamicSmemBytes = wide_smem<NH>();
      return cudaLaunchKernelEx(&cfg, solve_wide_kernel<NH, TRANS>, P, ldp, rows, K, Y, ldy, O, ldo, nrhs);
    }
  }
  cfg.gridDim = dim3(tiles, ky);
  at[np].id = cudaLaunchAttributeClusterDimension;
  at[np].val.clusterDim.x = 1;
  at[np].val.clusterDim.y = ky;
  at[np].val.clusterDim.z = 1;
  cfg.numAttrs = np + 1;
  return cudaLaunchKernelEx(&cfg, solve_step_kernel<NH, TRANS, ADD, TRI>, P, ldp, rows, K, Y, ldy, O, ldo, nrhs);
}

template <int NH>
cudaError_t solve_group(const double* L, int ldl, double* B, int ldb, int n, int nrhs, int blk, const double* W, double* Z,
                        cudaStream_t s) {
  const int nb = (n + blk - 1) / blk;
  cudaError_t e;
  for (int r = 0; r < nb; ++r) {                 // Z = L^{-1} B, B's rows updated as they come
    const int R0 = r * blk, m = n - R0 < blk ? n - R0 : blk;
    if ((e = launch_step<NH, true, false, 1>(W + (size_t)R0 * blk, blk, m, m, B + R0, ldb, Z + R0, n, nrhs, s)) != cudaSuccess)
      return e;
    if ((e = launch_step<NH, false, true, 0>(L + (size_t)R0 * ldl + R0 + m, ldl, n - R0 - m, m, Z + R0, n, B + R0 + m, ldb,
                                             nrhs, s)) != cudaSuccess)
      return e;
  }
  for (int r = nb - 1; r >= 0; --r) {            // B = L^{-T} Z
    const int R0 = r * blk, m = n - R0 < blk ? n - R0 : blk;
    if ((e = launch_step<NH, false, false, 2>(W + (size_t)R0 * blk, blk, m, m, Z + R0, n, B + R0, ldb, nrhs, s)) != cudaSuccess)
      return e;
    if ((e = launch_step<NH, true, true, 0>(L + R0, ldl, R0, m, B + R0, ldb, Z, n, nrhs, s)) != cudaSuccess) return e;
  }
  return cudaSuccess;
}

}  // namespace

// FP64 inverses of the diagonal blocks of solve_block(n) rows
cudaError_t launch_solve_inverses(const double* L, int ldl, int n, void* work, cudaStream_t s) {
  const int blk = solve_block(n), ldt = solve_scratch(n);
  double* W = static_cast<double*>(work);
  double* T = W + (size_t)n * blk;
  // the first kernel may follow a join with another stream (see LaunchCtx): launched plainly
  LaunchCtx& lc = launch_ctx();
  const bool pdl = lc.pdl;
  lc.pdl = false;
  (void)launch_pdl(inverse64_kernel, dim3(8, (n + 63) / 64), dim3(128), 0, s, L, ldl, n, W, blk);
  lc.pdl = pdl;
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  for (int h = 64; h < blk; h *= 2) {
    // T(c, i) = sum_k W11(k, c) L21(i, k), then W21(i, c) = -sum_k T(c, k) W22(i, k)
    GemmProducts p1, p2;
    for (int g0 = 0; g0 + h < n; g0 += 2 * h) {
      const int n2 = n - g0 - h < h ? n - g0 - h : h, off = g0 % blk;
      const long long w11 = (long long)g0 * blk + off, w22 = (long long)(g0 + h) * blk + off + h;
      const long long w21 = (long long)(g0 + h) * blk + off, tt = (long long)g0 * ldt;
      p1.b[p1.count++] = GemmProduct{w11, (long long)g0 * ldl + g0 + h, tt, h, n2, h, 0};
      p2.b[p2.count++] = GemmProduct{tt, w22, w21, h, n2, n2, 0};
      if (p1.count == kMaxGemmProducts || g0 + 3 * h >= n) {
        if ((e = launch_gemm_f64_products(T, ldt, W, blk, L, ldl, false, p1, s)) != cudaSuccess) return e;
        if ((e = launch_gemm_f64_products(W, blk, T, ldt, W, blk, true, p2, s)) != cudaSuccess) return e;
        p1.count = p2.count = 0;
      }
    }
  }
  return cudaSuccess;
}

cudaError_t launch_solve(const double* L, int ldl, double* B, int ldb, int n, int nrhs, void* work, cudaStream_t s) {
  const int blk = solve_block(n);
  const double* W = static_cast<const double*>(work);
  double* Z = static_cast<double*>(work) + (size_t)n * (blk + solve_scratch(n));
  for (int c0 = 0; c0 < nrhs; c0 += kPotrsMaxRhs) {
    const int nc = nrhs - c0 < kPotrsMaxRhs ? nrhs - c0 : kPotrsMaxRhs;
    double* Bc = B + (size_t)c0 * ldb;
    const cudaError_t e = nc <= 8 ? solve_group<1>(L, ldl, Bc, ldb, n, nc, blk, W, Z, s)
                                  : solve_group<2>(L, ldl, Bc, ldb, n, nc, blk, W, Z, s);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

// Single solves gain at every size (figures above) but with one right-hand side on large factors, whose
// sweeps read L once and whose links are short: n = 2048 238 us against 249, 4096 about equal (417),
// 8192 870 against 795.  In a batch, whose systems overlap on streams, the launches count: 24 FP64
// systems of 64 .. 1024, factored and solved with 4 right-hand sides, take 3.01 ms with the block solve up
// to 256 rows, 2.91 up to 512, 3.31 up to 1024.  Up to 8 right-hand sides and 1024 rows single solves do as
// batched ones, so that both agree to the bit there (at 1024 rows that costs a single solve 45 us of
// 175, at 512 the blocks take 88 us against 133).
bool solve_blocked(int n, int nrhs) { return n <= kSolveSmall || nrhs > 8 || (n > 1024 && (nrhs > 1 || n <= 3072)); }

int solve_launches(int n, int nrhs, bool inverses) {
  const int blk = solve_block(n), nb = (n + blk - 1) / blk;
  int l = (nrhs + kPotrsMaxRhs - 1) / kPotrsMaxRhs * (4 * nb - 2);
  if (inverses) {
    l += 1;
    for (int h = 64; h < blk && h < n; h *= 2) l += 2 * ((n + 2 * h * kMaxGemmProducts - 1) / (2 * h * kMaxGemmProducts));
  }
  return l;
}

}  // namespace hrp
