// The leaf POTRF by refinement: an FP32 Cholesky corrected to FP64 accuracy with exact residuals
// (used by potrf_leaf_cluster_kernel before its direct schedules, see there).
//
// The direct schedules of k_leaf_cluster.cu carry the accuracy of the result through all 128
// pivots, in FP64 (~820 cycles a column) or in pairs of binary32 (~420).  Here the chain runs in
// plain binary32 (about 60 cycles a column, one warp, two columns at a time) and the digits come
// afterwards, from products:
//   L0 = chol_32(A), W0 = L0^{-1}                       binary32, every CTA of the cluster the same
//   repeat  R  = A - L L^T                              exact (digit products, digits.cuh)
//           E  = W0 R W0^T,  F = its lower triangle with half the diagonal
//           L += L0 F                                   binary16 pairs (22 bits) on the tensor pipe
// (L (I + F) (I + F)^T L^T = A to first order in F.)  Each step multiplies the error by the relative
// error of L0 and W0, about 2^-21 for the leaves of dominant matrices, so two steps pass FP64's
// unit roundoff; the loop stops when the next error is below 2^-57.  L is held in 62-bit fixed
// point against the scales 2^e_i, e_i = ceil(ex_i / 2) for a_ii < 2^ex_i, so that |l_ij| < 2^e_i
// exactly, whatever the range of A (the fixed point keeps one more bit for binary32's rounding).
//
// Work split: the 36 residual tiles (I, J) belong to CTA (I + J) mod 8; the corrections of column
// block J to CTA J.  Every CTA needs all residuals and all corrections; they are exchanged through
// a scratch array in global memory (36 KB each, L2 resident; distributed shared memory was
// measured at ~9 bytes per clock and SM for this all-to-all pattern), two cluster barriers a step;
// nothing else waits.
//
// The error is relative to the scales, and an entry of L far below its own (weakly coupled unknowns) keeps
// fewer digits than in an FP64 factorization.  So sum |l_ik| |l_jk| + |a_ij| is estimated for every entry from L0
// (one mma a 16 x 8 tile and 16 terms); where it is zero, so is l_ij; entries below 2^-kFineBits or
// 2^-kCoarseBits are computed again in FP64 at the end, l_ij = (a_ij - sum_{k<j} l_ik l_jk) / l_jj, up to kMaxRepair
// of them (~1 us each; a leaf with more is factored directly).  The others are accurate to 2^-57 of the scale, so
// to 2^-31 of themselves at the line.  Factors of dominant matrices of order n have entries of 2^-16 at n = 8192,
// and one in 10^4 of those below 2^-30; all-FP64 trees are for the smaller orders.
//
// A leaf whose diagonal is not positive, with |a_ij| > sqrt(a_ii a_jj), a binary32 pivot that is not
// positive, or that would not converge soon (a kernel matrix with nugget below ~10^-3) is left untouched and
// factored by the direct schedules in the same launch.
#pragma once
#include <cooperative_groups.h>

#include "digits.cuh"
#include "hrp_internal.cuh"

namespace hrp {
namespace leafref {

namespace cg = cooperative_groups;

constexpr int kThreads = 256;
constexpr int kCtas = 8;
constexpr int kTiles = 36;
constexpr int kTtLd = 136;             // halves per row of the staged column block
constexpr int kMaxStep = 6;
constexpr float kTol = 0x1p-57f;
// A leaf gives up where the loop would take longer than the direct schedules: with a scaled pivot of binary32
// below kMinPivot, or a first correction above kMaxFirst (each step gains that factor: five steps of
// ~12 us).  Kernel matrices of order 128, nugget 1e-2, 1e-3 and 1e-4, us: refined 74, given up 133 and 112
// (186 and 186 when every leaf ran to its sixth step); FP64 schedule alone 106, double-float 70, where
// giving up costs 97 and 78.
constexpr float kMinPivot = 0x1p-12f, kMaxFirst = 0x1p-12f;

// Entries of L below their scale by kFineBits (all-FP64 trees) or kCoarseBits (others, whose off-diagonal blocks carry
// binary32's 2^-24) are computed again in FP64; a leaf with more than kMaxRepair is factored directly
constexpr int kMaxRepair = 16, kFineBits = 26, kCoarseBits = 30;

struct Smem {
  unsigned long long Lx[kTiles][256];  // L in units of 2^(e_i - 62) plus kByteBias, rows swizzled
  union {
    float f[kTiles][256];              // binary32 tiles not yet eliminated, row-major with ft()
    __half h[kTiles][2][256];          // L0 as binary16 pairs hi + lo 2^-11, row-major with ht()
  } L0;
  __half W0[kTiles][2][256];           // L0^{-1}, pairs
  __half R[kTiles][2][256];            // R (lower tiles, the diagonal ones whole), scaled, pairs
  __half Tt[2][16][kTtLd];             // T = R W0_J^T, then F, transposed: [column][row]; rows of H
  float Wrow[16][132];                 // rows 16 rank .. of the inverse, binary32
  __half Sbuf[12][2][256];             // phase 1: sums for the off-diagonal blocks of W0, pairs
  float4 xy[16][16];                   // phase 1: the diagonal block's column pairs, rows 2 j, 2 j + 1
  float4 rr[16];                       // phase 1: 1 / l_kk, 1 / l_{k+1,k+1}, l_{k+1,k} of a pair
  int e[128];                          // scales
  unsigned zero[8][2][4];              // this column block's entries of L that are zero (half tiles, as the words of xC)
  double rep_a[kMaxRepair];            // CTA 0: the entries to compute again, by column, and their values in A
  int rep[kMaxRepair], nrep;
  int nlow;                            // such entries found here, half tiles with zeros times 2^16, with lost ones times 2^24
  unsigned rmax[2], emax[2];           // largest |R| and scaled |E| here (bits), by step parity
};

__device__ __forceinline__ int tix(int I, int J) { return I * (I + 1) / 2 + J; }
// element (i, j) of a binary32 tile: 16-byte groups swizzled so that 8 rows read without conflicts
__device__ __forceinline__ int ft(int i, int j) { return i * 16 + ((((j >> 2) ^ (i >> 1)) & 3) << 2) + (j & 3); }
// element (i, j) of a binary16 tile: the two 16-byte halves of a row swapped on rows 4-7 and 12-15
__device__ __forceinline__ int ht(int i, int j) { return i * 16 + ((((j >> 3) ^ (i >> 2)) & 1) << 3) + (j & 7); }
// element (i, k) of a fixed-point tile: halves of a row swapped on odd rows
__device__ __forceinline__ int lx(int i, int k) { return i * 16 + (k ^ ((i & 1) << 3)); }

__device__ __forceinline__ float rsqrt_fast(float x) {
  float r;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}

// x as hi + lo 2^-11, both binary16 (22 bits of x; lo keeps binary16's normal range)
__device__ __forceinline__ void half_pair(float x, __half& hi, __half& lo) {
  hi = __float2half_rn(x);
  lo = __float2half_rn((x - __half2float(hi)) * 2048.f);
}
__device__ __forceinline__ void half_pair2(float2 x, __half2& hi, __half2& lo) {
  hi = __float22half2_rn(x);
  const float2 b = __half22float2(hi);
  lo = __float22half2_rn(make_float2((x.x - b.x) * 2048.f, (x.y - b.y) * 2048.f));
}
// x (|x| < 1 up to rounding) in units of 2^-62, truncated
__device__ __forceinline__ unsigned long long fix62(float x) {
  const unsigned b = __float_as_uint(x);
  const int F = (int)(b >> 23) & 0xff, sh = F - 88;          // x = m 2^(F - 150)
  const long long m = F ? (long long)((b & 0x7fffffu) | 0x800000u) : 0;
  const long long M = sh >= 0 ? m << min(sh, 39) : (sh > -24 ? m >> -sh : 0);
  return (unsigned long long)((int)b < 0 ? -M : M);
}

// fragments of a 16 x 16 binary16 tile: as the A operand (rows x terms), its transpose as A, as the B
// operand (columns x terms), its transpose as B
enum class Op { A, At, B, Bt };
template <Op O>
__device__ __forceinline__ void frag(uint32_t (&r)[4], const __half* t, int lane) {
  if constexpr (O == Op::A) {
    const int i = lane & 15;
    dig_ldmatrix(r, t + ht(i, (lane >> 4) * 8));
  } else if constexpr (O == Op::At) {
    const int i = ((lane >> 4) & 1) * 8 + (lane & 7);
    dig_ldmatrix_t(r, t + ht(i, ((lane >> 3) & 1) * 8));
  } else if constexpr (O == Op::B) {
    const int i = (lane & 7) + ((lane >> 4) << 3);
    dig_ldmatrix(r, t + ht(i, ((lane >> 3) & 1) * 8));
  } else {
    const int i = ((lane >> 3) & 1) * 8 + (lane & 7);
    dig_ldmatrix_t(r, t + ht(i, (lane >> 4) * 8));
  }
}
// acc0 += hi hi, acc1 += hi lo + lo hi (weight 2^-11) for a 16 x 16 output and 16 terms
__device__ __forceinline__ void pair_mm(float (&acc0)[2][4], float (&acc1)[2][4], const uint32_t (&ah)[4],
                                        const uint32_t (&al)[4], const uint32_t (&bh)[4], const uint32_t (&bl)[4]) {
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    dig_mma(acc0[h], ah, bh[2 * h], bh[2 * h + 1]);
    dig_mma(acc1[h], ah, bl[2 * h], bl[2 * h + 1]);
    dig_mma(acc1[h], al, bh[2 * h], bh[2 * h + 1]);
  }
}
// the value of a pair product
__device__ __forceinline__ float pair_value(float c0, float c1) { return fmaf(c1, 0x1p-11f, c0); }
// a warp's 16 x 16 result (scaled by f) as pairs to a tile
__device__ __forceinline__ void put_pairs(__half (*t)[256], const float (&c0)[2][4], const float (&c1)[2][4], float f,
                                          int lane) {
#pragma unroll
  for (int h = 0; h < 2; ++h)
#pragma unroll
    for (int q = 0; q < 4; q += 2) {
      const int i = (lane >> 2) + 4 * q, j = 8 * h + 2 * (lane & 3);
      __half2 hi, lo;
      half_pair2(make_float2(f * pair_value(c0[h][q], c1[h][q]), f * pair_value(c0[h][q + 1], c1[h][q + 1])), hi, lo);
      *reinterpret_cast<__half2*>(t[0] + ht(i, j)) = hi;
      *reinterpret_cast<__half2*>(t[1] + ht(i, j)) = lo;
    }
}
// A-operand fragments of a binary32 tile, split into pairs in registers
__device__ __forceinline__ void frag_f32(uint32_t (&ah)[4], uint32_t (&al)[4], const float* t, int lane) {
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const int i = (lane >> 2) + 8 * (q & 1), j = 2 * (lane & 3) + 8 * (q >> 1);
    __half2 hi, lo;
    half_pair2(*reinterpret_cast<const float2*>(t + ft(i, j)), hi, lo);
    ah[q] = *reinterpret_cast<const uint32_t*>(&hi);
    al[q] = *reinterpret_cast<const uint32_t*>(&lo);
  }
}
template <Op OA, Op OB>
__device__ __forceinline__ void tile_pair_mm(float (&c0)[2][4], float (&c1)[2][4], const __half (*A)[256],
                                             const __half (*B)[256], int lane) {
  uint32_t ah[4], al[4], bh[4], bl[4];
  frag<OA>(ah, A[0], lane);
  frag<OA>(al, A[1], lane);
  frag<OB>(bh, B[0], lane);
  frag<OB>(bl, B[1], lane);
  pair_mm(c0, c1, ah, al, bh, bl);
}

// Cholesky of the 32 x 32 diagonal block p (tiles 2p, 2p + 1) by warp 0, and its inverse W by warp 1.
// Warp 0's lane i holds row i; columns two at a time: every lane forms the pair's pivots (both
// reciprocal square roots at once, 1 / l_11 = l_00 (a_00 a_11 - a_10^2)^{-1/2}), the lanes' entries of
// the two columns go through shared memory (16-byte broadcast reads; a shuffle costs four issue slots of the
// sub-partition) and update the rest, columns 16 .. 31 once for the first sixteen.  The entries that
// the next pair's pivots need are shuffled instead, and its reciprocal square roots started before
// the exchange and the update: the chain of a pair is one reciprocal square root and one shuffle.  Warp 1's lane c holds column
// c of W and applies the same column pairs to it one step behind, told by named barriers 1 .. 15
// (one per pair: the producer only arrives).  False (warp 0) when a pivot is not positive and finite;
// both warps pass every barrier in any case.
__device__ __forceinline__ void pair_arrive(int id) { asm volatile("bar.arrive %0, 64;" ::"r"(id) : "memory"); }
__device__ __forceinline__ void pair_wait(int id) { asm volatile("bar.sync %0, 64;" ::"r"(id) : "memory"); }
__device__ __forceinline__ bool potrf32(Smem& sm, int p, int lane) {
  const unsigned full = 0xffffffffu;
  const int ti = lane >> 4, ri = lane & 15;
  float a[32];
#pragma unroll
  for (int j4 = 0; j4 < 8; ++j4) {
    const int tj = j4 >> 2;
    float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
    if (tj <= ti) v = *reinterpret_cast<const float4*>(&sm.L0.f[tix(2 * p + ti, 2 * p + tj)][ft(ri, 4 * (j4 & 3))]);
    a[4 * j4] = v.x;
    a[4 * j4 + 1] = v.y;
    a[4 * j4 + 2] = v.z;
    a[4 * j4 + 3] = v.w;
  }
  bool ok = true;
  float d0 = __shfl_sync(full, a[0], 0), q = __shfl_sync(full, a[0], 1), s = __shfl_sync(full, a[1], 1);
  float det = fmaf(s, d0, -q * q);
  float r0 = rsqrt_fast(d0), rd = rsqrt_fast(det);
#pragma unroll
  for (int k = 0; k < 32; k += 2) {
    const int end = k < 16 ? 16 : 32;            // columns 16 .. 31 get columns 0 .. 15 all at once
    float nd0 = 0.f, nq = 0.f, ns = 0.f;         // the next pair's block before this pair's update
    if (k + 2 < end) {
      nd0 = __shfl_sync(full, a[k + 2], k + 2);
      nq = __shfl_sync(full, a[k + 2], k + 3);
      ns = __shfl_sync(full, a[k + 3], k + 3);
    }
    ok = ok && d0 > kMinPivot && det > kMinPivot * d0;   // scaled pivots: false for NaN too
    const float m = q * r0, r1 = d0 * r0 * rd;
    const float4 rr = make_float4(r0, r1, m, 0.f);
    const float x = a[k] * r0;                   // column k of L (rows >= k)
    const float y = fmaf(-x, m, a[k + 1]) * r1;  // column k + 1 (rows > k)
    a[k] = x;
    a[k + 1] = y;
    if (k + 2 < end) {
      // the next pair, as far as its reciprocal square roots: the chain
      const float vx = __shfl_sync(full, x, k + 2), vy = __shfl_sync(full, y, k + 2);
      const float vz = __shfl_sync(full, x, k + 3), vw = __shfl_sync(full, y, k + 3);
      d0 = fmaf(-vy, vy, fmaf(-vx, vx, nd0));
      q = fmaf(-vw, vy, fmaf(-vz, vx, nq));
      s = fmaf(-vw, vw, fmaf(-vz, vz, ns));
      det = fmaf(s, d0, -q * q);
      r0 = rsqrt_fast(d0);
      rd = rsqrt_fast(det);
      a[k + 2] = fmaf(-y, vy, fmaf(-x, vx, a[k + 2]));
      a[k + 3] = fmaf(-y, vw, fmaf(-x, vz, a[k + 3]));
    }
    reinterpret_cast<float2*>(sm.xy[k >> 1])[lane] = make_float2(x, y);
    if (lane == 0) sm.rr[k >> 1] = rr;
    __syncwarp();
    if (k < 28) pair_arrive((k >> 1) + 1);       // 15 is the caller's, after the last two pairs
    if ((k >> 4) <= ti) {                        // the columns as pairs (zero above the diagonal), over the binary32 tile
      __half2 hi, lo;
      half_pair2(make_float2(k <= lane ? x : 0.f, k + 1 <= lane ? y : 0.f), hi, lo);
      __half (*t)[256] = sm.L0.h[tix(2 * p + ti, 2 * p + (k >> 4))];
      *reinterpret_cast<__half2*>(t[0] + ht(ri, k & 15)) = hi;
      *reinterpret_cast<__half2*>(t[1] + ht(ri, k & 15)) = lo;
    }
#pragma unroll
    for (int j = k + 4; j < end; j += 2) {
      const float4 v = sm.xy[k >> 1][j >> 1];    // rows j and j + 1 of the two columns
      a[j] = fmaf(-y, v.y, fmaf(-x, v.x, a[j]));
      a[j + 1] = fmaf(-y, v.w, fmaf(-x, v.z, a[j + 1]));
    }
    if (k == 14) {
#pragma unroll
      for (int j = 16; j < 32; j += 2)
#pragma unroll
        for (int c = 0; c < 16; c += 2) {
          const float4 v = sm.xy[c >> 1][j >> 1];
          a[j] = fmaf(-a[c + 1], v.y, fmaf(-a[c], v.x, a[j]));
          a[j + 1] = fmaf(-a[c + 1], v.w, fmaf(-a[c], v.z, a[j + 1]));
        }
      d0 = __shfl_sync(full, a[16], 16);
      q = __shfl_sync(full, a[16], 17);
      s = __shfl_sync(full, a[17], 17);
      det = fmaf(s, d0, -q * q);
      r0 = rsqrt_fast(d0);
      rd = rsqrt_fast(det);
    }
  }
  return ok;
}
// warp 1: W = L^{-1} of the block as pairs
__device__ __forceinline__ void inverse32(Smem& sm, int p, int lane) {
  const int ti = lane >> 4, ri = lane & 15;
  float w[32];
#pragma unroll
  for (int r = 0; r < 32; ++r) w[r] = r == lane ? 1.f : 0.f;
#pragma unroll
  for (int k = 0; k < 32; k += 2) {
    if (k < 30) pair_wait((k >> 1) + 1);         // barrier 15 covers the last two pairs
    const float4 rr = sm.rr[k >> 1];
    w[k] *= rr.x;
    w[k + 1] = fmaf(-rr.z, w[k], w[k + 1]) * rr.y;
    if (ti <= (k >> 4)) {                        // rows k and k + 1 are final
      __half (*t)[256] = sm.W0[tix(2 * p + (k >> 4), 2 * p + ti)];
      __half2 hi, lo;
      half_pair2(make_float2(w[k], w[k + 1]), hi, lo);
      t[0][ht(k & 15, ri)] = __low2half(hi);
      t[0][ht((k & 15) + 1, ri)] = __high2half(hi);
      t[1][ht(k & 15, ri)] = __low2half(lo);
      t[1][ht((k & 15) + 1, ri)] = __high2half(lo);
    }
#pragma unroll
    for (int j = k + 2; j < 32; j += 2) {
      const float4 v = sm.xy[k >> 1][j >> 1];
      w[j] = fmaf(-v.y, w[k + 1], fmaf(-v.x, w[k], w[j]));
      w[j + 1] = fmaf(-v.w, w[k + 1], fmaf(-v.z, w[k], w[j + 1]));
    }
  }
}

// C (binary32 tile) -= the pair products
__device__ __forceinline__ void sub_tile(float* C, const float (&c0)[2][4], const float (&c1)[2][4], int lane) {
#pragma unroll
  for (int h = 0; h < 2; ++h)
#pragma unroll
    for (int q = 0; q < 4; q += 2) {
      float2* o = reinterpret_cast<float2*>(C + ft((lane >> 2) + 4 * q, 8 * h + 2 * (lane & 3)));
      float2 v = *o;
      v.x -= pair_value(c0[h][q], c1[h][q]);
      v.y -= pair_value(c0[h][q + 1], c1[h][q + 1]);
      *o = v;
    }
}

// L0 and W0 of the scaled leaf in L0.f (NB blocks of 32), both as pairs; false when a pivot failed.  Right-looking by blocks of 32 columns; the products run on
// the tensor pipe from the pairs (22 bits: a little below binary32, which the refinement makes up
// for; in binary32 FMAs they were bound by shared-memory reads, 36000 of 51000 cycles).
__device__ __forceinline__ bool factor32(Smem& sm, int NB, int tid) {
  const int warp = tid >> 5, lane = tid & 31;
  for (int p = 0; p < NB; ++p) {
    // the diagonal block's update with panel p - 1
    if (p > 0) {
      if (warp < 3) {
        const int I = 2 * p + (warp > 0), J = 2 * p + (warp == 2);
        float c0[2][4] = {}, c1[2][4] = {};
        tile_pair_mm<Op::A, Op::B>(c0, c1, sm.L0.h[tix(I, 2 * p - 2)], sm.L0.h[tix(J, 2 * p - 2)], lane);
        tile_pair_mm<Op::A, Op::B>(c0, c1, sm.L0.h[tix(I, 2 * p - 1)], sm.L0.h[tix(J, 2 * p - 1)], lane);
        sub_tile(sm.L0.f[tix(I, J)], c0, c1, lane);
      }
      __syncthreads();
    }
    int fail = 0;
    if (warp == 0) {
      fail = !potrf32(sm, p, lane);
      pair_arrive(15);
    } else if (warp == 1) {
      inverse32(sm, p, lane);
    } else if (p > 0) {
      // the other tiles' update with panel p - 1, and the sums S(I, J) = sum_K L(I, K) W(K, J) of
      // tile rows 2p, 2p + 1
      int u = 0;
      for (int J = 2 * p; J < 2 * NB; ++J)
        for (int I = max(J, 2 * p + 2); I < 2 * NB; ++I)
          if (u++ % 6 == warp - 2) {
            float c0[2][4] = {}, c1[2][4] = {};
            tile_pair_mm<Op::A, Op::B>(c0, c1, sm.L0.h[tix(I, 2 * p - 2)], sm.L0.h[tix(J, 2 * p - 2)], lane);
            tile_pair_mm<Op::A, Op::B>(c0, c1, sm.L0.h[tix(I, 2 * p - 1)], sm.L0.h[tix(J, 2 * p - 1)], lane);
            sub_tile(sm.L0.f[tix(I, J)], c0, c1, lane);
          }
      for (int h = 0; h < 2; ++h)
        for (int J = 0; J < 2 * p; ++J)
          if (u++ % 6 == warp - 2) {
            float c0[2][4] = {}, c1[2][4] = {};
            for (int K = J; K < 2 * p; ++K)
              tile_pair_mm<Op::A, Op::Bt>(c0, c1, sm.L0.h[tix(2 * p + h, K)], sm.W0[tix(K, J)], lane);
            put_pairs(sm.Sbuf[2 * J + h], c0, c1, 1.f, lane);
          }
    }
    if (__syncthreads_or(fail)) return false;
    // panel: L(I, 2p), L(I, 2p + 1) = A(I, ..) Wpp^T, a warp per tile row; and the blocks of W left of
    // the diagonal block, W(I, J) = -sum_K Wpp(I, K) S(K, J)
    int u = 0;
    for (int I = 2 * p + 2; I < 2 * NB; ++I)
      if (u++ % 8 == warp) {
        float x0[2][4] = {}, x1[2][4] = {}, y0[2][4] = {}, y1[2][4] = {};
        uint32_t ah[4], al[4], bh[4], bl[4];
        frag_f32(ah, al, sm.L0.f[tix(I, 2 * p)], lane);
        frag<Op::B>(bh, sm.W0[tix(2 * p, 2 * p)][0], lane);
        frag<Op::B>(bl, sm.W0[tix(2 * p, 2 * p)][1], lane);
        pair_mm(x0, x1, ah, al, bh, bl);
        frag<Op::B>(bh, sm.W0[tix(2 * p + 1, 2 * p)][0], lane);
        frag<Op::B>(bl, sm.W0[tix(2 * p + 1, 2 * p)][1], lane);
        pair_mm(y0, y1, ah, al, bh, bl);
        frag_f32(ah, al, sm.L0.f[tix(I, 2 * p + 1)], lane);
        frag<Op::B>(bh, sm.W0[tix(2 * p + 1, 2 * p + 1)][0], lane);
        frag<Op::B>(bl, sm.W0[tix(2 * p + 1, 2 * p + 1)][1], lane);
        pair_mm(y0, y1, ah, al, bh, bl);
        __syncwarp();                                       // every lane has read both tiles
        put_pairs(sm.L0.h[tix(I, 2 * p)], x0, x1, 1.f, lane);
        put_pairs(sm.L0.h[tix(I, 2 * p + 1)], y0, y1, 1.f, lane);
      }
    for (int J = 0; J < 2 * p; ++J)
      for (int h = 0; h < 2; ++h)
        if (u++ % 8 == warp) {
          float c0[2][4] = {}, c1[2][4] = {};
          for (int K = 0; K <= h; ++K)
            tile_pair_mm<Op::A, Op::Bt>(c0, c1, sm.W0[tix(2 * p + h, 2 * p + K)], sm.Sbuf[2 * J + K], lane);
          put_pairs(sm.W0[tix(2 * p + h, J)], c0, c1, -1.f, lane);
        }
    __syncthreads();
  }
  return true;
}

// B fragments of the staged column block (columns x rows 16 k ..), hi or lo plane
__device__ __forceinline__ void frag_tt(uint32_t (&r)[4], const __half (*t)[kTtLd], int kt, int lane) {
  dig_ldmatrix(r, &t[(lane & 7) + ((lane >> 4) << 3)][16 * kt + ((lane >> 3) & 1) * 8]);
}
// a warp's 16 x 16 result (rows 16 I ..) into the staged column block
__device__ __forceinline__ void put_tt(Smem& sm, int I, const float (&v)[2][4], int lane) {
#pragma unroll
  for (int h = 0; h < 2; ++h)
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int c = 8 * h + 2 * (lane & 3) + (q & 1), r = 16 * I + (lane >> 2) + 8 * (q >> 1);
      __half hi, lo;
      half_pair(v[h][q], hi, lo);
      sm.Tt[0][c][r] = hi;
      sm.Tt[1][c][r] = lo;
    }
}

// sum over the 16 (J + 1) inner terms of L(I, :) L(J, :)^T for one half tile (rows 0 .. 15, columns
// j0 .. + 7), in units of 2^-60 of the fixed points' scales, modulo 2^64.  ND digits, weights s + t <
// ND kept: 8 is exact to the fixed point; 6 (an error of 2^-49) is enough for the first residual,
// whose L carries binary32's error (with 5 the loop takes a third step).
template <int ND>
__device__ __forceinline__ void half_tile_product(const Smem& sm, int I, int J, int j0, int lane, long long (&sum)[4]) {
  float acc[ND][4];
#pragma unroll
  for (int w = 0; w < ND; ++w)
#pragma unroll
    for (int q = 0; q < 4; ++q) acc[w][q] = 0.f;
  const int ra = lane >> 2, kk = 2 * (lane & 3);
  const unsigned long long* la = sm.Lx[tix(I, 0)];
  const unsigned long long* lb = sm.Lx[tix(J, 0)];
#pragma unroll 1
  for (int kt = 0; kt <= J; ++kt, la += 256, lb += 256) {
    const ulonglong2 a0 = *reinterpret_cast<const ulonglong2*>(la + lx(ra, kk));
    const ulonglong2 a1 = *reinterpret_cast<const ulonglong2*>(la + lx(ra + 8, kk));
    const ulonglong2 a2 = *reinterpret_cast<const ulonglong2*>(la + lx(ra, kk + 8));
    const ulonglong2 a3 = *reinterpret_cast<const ulonglong2*>(la + lx(ra + 8, kk + 8));
    const ulonglong2 b0 = *reinterpret_cast<const ulonglong2*>(lb + lx(j0 + ra, kk));
    const ulonglong2 b1 = *reinterpret_cast<const ulonglong2*>(lb + lx(j0 + ra, kk + 8));
    uint32_t bf[ND][2];
#pragma unroll
    for (int s = 0; s < ND; ++s) {
      bf[s][0] = byte_pair(b0.x, b0.y, s);
      bf[s][1] = byte_pair(b1.x, b1.y, s);
    }
#pragma unroll
    for (int s = 0; s < ND; ++s) {
      const uint32_t af[4] = {byte_pair(a0.x, a0.y, s), byte_pair(a1.x, a1.y, s), byte_pair(a2.x, a2.y, s),
                              byte_pair(a3.x, a3.y, s)};
#pragma unroll
      for (int t = 0; t < ND - s; ++t) dig_mma(acc[s + t], af, bf[t][0], bf[t][1]);
    }
  }
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    // weights 2^(-14 - 8 w): w = 0 .. 2 joined in units of 2^-30, the others of 2^(-14 - 8 (ND - 1))
    long long hi = 0, lo = 0;
#pragma unroll
    for (int w = 0; w < 3; ++w) hi = (hi << 8) + __float2int_rn(acc[w][q]);
#pragma unroll
    for (int w = 3; w < ND; ++w) lo = (lo << 8) + __float2int_rn(acc[w][q]);
    constexpr int kLo = 60 - 14 - 8 * (ND - 1);
    sum[q] = (hi << 30) + (kLo >= 0 ? lo << (kLo >= 0 ? kLo : 0) : lo >> (kLo < 0 ? -kLo : 0));
  }
}

// x 2^e truncated to binary32 (0 below its normal range)
__device__ __forceinline__ float scaled_float(double x, int e) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(x);
  const int F = ((int)(b >> 52) & 0x7ff) - 1023 + 127 + e;
  if (F <= 0) return 0.f;
  return __uint_as_float(((unsigned)(b >> 32) & 0x80000000u) | ((unsigned)min(F, 254) << 23) | ((unsigned)(b >> 29) & 0x7fffffu));
}

// the largest of the CTAs' words (bits of non-negative floats)
__device__ __forceinline__ float cluster_max(cg::cluster_group& cluster, unsigned* w) {
  unsigned q[kCtas], m = 0;
#pragma unroll
  for (int u = 0; u < kCtas; ++u) q[u] = *(volatile unsigned*)cluster.map_shared_rank(w, u);
#pragma unroll
  for (int u = 0; u < kCtas; ++u) m = max(m, q[u]);
  return __uint_as_float(m);
}

// floats of global scratch the refinement exchanges through: residual tiles, corrections, and 8 words per half tile
constexpr int kScratch = 2 * kTiles * 256 + 2 * kTiles * 8;

// Entry classes of a half tile (rows 16 I .., columns 16 J + 8 h ..), from est = |a_ij| + sum_k |l_ik| |l_jk| with the
// binary32 factor's upper halves (a: A's entries in units of 2^-58 of their scales, bit q of nz: a_ij is not zero): bits (lane, q) of low[q] where est is below thr, of zero[q] where it is zero
// (then so is l_ij); any entry that its upper half cannot hold sets `lost`.
__device__ __forceinline__ void entry_classes(const Smem& sm, int I, int J, int h, const long long (&a)[4], int nz, int n, float thr, int lane,
                                              unsigned (&low)[4], unsigned (&zero)[4], bool& lost) {
  float c[4] = {};
#pragma unroll 2
  for (int k = 0; k <= J; ++k) {
    uint32_t ah[4], bh[4];
    frag<Op::A>(ah, sm.L0.h[tix(I, k)][0], lane);
    frag<Op::B>(bh, sm.L0.h[tix(J, k)][0], lane);
#pragma unroll
    for (int q = 0; q < 4; ++q) ah[q] &= 0x7fff7fffu;
    dig_mma(c, ah, (h ? bh[2] : bh[0]) & 0x7fff7fffu, (h ? bh[3] : bh[1]) & 0x7fff7fffu);
  }
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const int gi = 16 * I + (lane >> 2) + 8 * (q >> 1), gj = 16 * J + 8 * h + 2 * (lane & 3) + (q & 1);
    const bool in = gi < n && gi > gj;
    float est = c[q];
    if (in && ((nz >> q) & 1)) {
      const unsigned long long v = (unsigned long long)(a[q] < 0 ? -a[q] : a[q]);
      est += fmaxf(fmaf((float)(unsigned)(v >> 32), 0x1p-26f, (float)(unsigned)v * 0x1p-58f), 0x1p-120f);
    }
    low[q] = __ballot_sync(0xffffffffu, in && est > 0.f && est < thr);
    zero[q] = __ballot_sync(0xffffffffu, in && est == 0.f);
    lost |= in && est > 0.f && est < 0x1p-24f;
  }
}

// The leaf.  Returns true when A holds L (and W32 its FP32 inverse); false, the same in every CTA,
// with nothing written, when the direct schedules must factor it.  Every thread of the cluster
// takes the same path through the cluster barriers.
__device__ bool leaf_refine(double* __restrict__ A, int ld, int n, float* __restrict__ W32, int ldw,
                            float* scratch, float thr, unsigned char* smem_raw) {
  Smem& sm = *reinterpret_cast<Smem*>(smem_raw);
  cg::cluster_group cluster = cg::this_cluster();
  const int rank = (int)cluster.block_rank();
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int NB = (n + 31) / 32, T = 2 * NB, NTL = T * (T + 1) / 2;
  float* xR = scratch;                        // residual tiles
  float* xD = scratch + kTiles * 256;         // corrections of L
  unsigned* xC = reinterpret_cast<unsigned*>(scratch + 2 * kTiles * 256);   // entry classes
  int total = 0;                              // entries to compute again

  // this warp's residual units: half tiles (16 rows, 8 columns) of the CTA's tiles, longest products
  // first; the tile's entries in fixed point (unit 2^(e_i + e_j - 58)) stay in registers
  int uI[2] = {-1, -1}, uJ[2] = {0, 0}, uH[2] = {0, 0};
  {
    int slot = 0;
    for (int J = T - 1; J >= 0; --J) {
      const int I = (rank - J) & 7;
      if (I < J || I >= T) continue;
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int u = 2 * slot + h;
        if (u == warp) {
          uI[0] = I;
          uJ[0] = J;
          uH[0] = h;
        } else if (15 - u == warp) {
          uI[1] = I;
          uJ[1] = J;
          uH[1] = h;
        }
      }
      ++slot;
    }
  }
  // ---- load: every lower tile (one entry per thread and tile, all loads in flight), the
  // diagonal's scales, then scaled binary32 ----
  int bad = 0;
  const int li = tid & 15, lk = tid >> 4;
  double araw[2][4];
  {
    double v[kTiles];
    int t = 0;
#pragma unroll
    for (int I = 0; I < 8; ++I)
#pragma unroll
      for (int J = 0; J <= I; ++J, ++t) {
        const int gi = 16 * I + li, gk = 16 * J + lk;
        v[t] = (gi < n && gk <= gi) ? A[(size_t)gk * ld + gi] : 0.0;
      }
#pragma unroll
    for (int x = 0; x < 2; ++x)
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const int gi = 16 * uI[x] + (lane >> 2) + 8 * (q >> 1), gj = 16 * uJ[x] + 8 * uH[x] + 2 * (lane & 3) + (q & 1);
        // a diagonal tile's residual is formed whole, from A's lower triangle
        const int gr = max(gi, gj), gc = min(gi, gj);
        araw[x][q] = (uI[x] >= 0 && gr < n) ? A[(size_t)gc * ld + gr] : 0.0;
      }
    if (tid < 2) sm.rmax[tid] = sm.emax[tid] = 0;
    if (tid == 0) sm.nlow = sm.nrep = 0;
    if (tid < 128) {
      int e = 0;
      if (tid < n) {
        const long long b = __double_as_longlong(A[(size_t)tid * ld + tid]);
        const int F = (int)(b >> 52);                          // negative for a negative entry
        bad = F <= 0 || F >= 0x7ff;
        e = bad ? 0 : (F - 1022 + 1) >> 1;
      }
      sm.e[tid] = e;
    }
    if (__syncthreads_or(bad)) return false;
    t = 0;
#pragma unroll
    for (int I = 0; I < 8; ++I) {
      if (I >= T) break;
      const int gi = 16 * I + li, ei = sm.e[gi];
#pragma unroll
      for (int J = 0; J <= I; ++J) {
        const int gk = 16 * J + lk, ee = ei + sm.e[gk];
        const double x = v[I * (I + 1) / 2 + J];
        // a positive definite leaf has |a_ij| < 2^(e_i + e_j)
        bad |= dig_field(x) > ee + 1022;
        float f = scaled_float(x, -ee);
        if (gi >= n) f = gi == gk ? 0.5f : 0.f;                // rows past n: a unit block of its own
        sm.L0.f[I * (I + 1) / 2 + J][ft(li, lk)] = f;
      }
    }
  }
  if (__syncthreads_or(bad)) return false;
  long long afix[2][4];
  int nz = 0;
#pragma unroll
  for (int x = 0; x < 2; ++x) {
    if (uI[x] < 0) continue;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int gi = 16 * uI[x] + (lane >> 2) + 8 * (q >> 1), gj = 16 * uJ[x] + 8 * uH[x] + 2 * (lane & 3) + (q & 1);
      afix[x][q] = 0;
      if (gi < n && gj < n) afix[x][q] = dig_fix(araw[x][q], sm.e[gi] + sm.e[gj] + 2 + 1022) >> 2;
      if (((unsigned)__double2hiint(araw[x][q]) << 1) | (unsigned)__double2loint(araw[x][q])) nz |= 1 << (4 * x + q);
      if (gi >= n && gi == gj) afix[x][q] = 1ll << 57;         // 0.5
    }
  }
  if (!factor32(sm, NB, tid)) return false;                    // the same in every CTA
  // ---- L to fixed point: a lane takes two adjacent columns of a row ----
  for (int t = warp; t < NTL; t += 8) {
    const int j = 2 * (lane & 7), ib = lane >> 3;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int i = 4 * q + ib, at = ht(i, j);
      const float2 hi = __half22float2(*reinterpret_cast<const __half2*>(&sm.L0.h[t][0][at]));
      const float2 lo = __half22float2(*reinterpret_cast<const __half2*>(&sm.L0.h[t][1][at]));
      *reinterpret_cast<ulonglong2*>(&sm.Lx[t][lx(i, j)]) =
          make_ulonglong2(fix62(pair_value(hi.x, lo.x)) + kByteBias, fix62(pair_value(hi.y, lo.y)) + kByteBias);
    }
  }
  __syncthreads();

  float first = 1.f, last = 1.f;
  const bool mine = rank < T;                                  // this CTA's column block exists
  bool good = false;
  for (int step = 0; step < kMaxStep; ++step) {
    // ---- R = A - L L^T: this CTA's tiles, to the scratch ----
    const int par = step & 1;
    float mx = 0.f;
    if (step == 0) {
#pragma unroll
      for (int x = 0; x < 2; ++x) {
        if (uI[x] < 0) continue;
        unsigned low[4], zero[4], w = 0;
        bool lost = false;
        entry_classes(sm, uI[x], uJ[x], uH[x], afix[x], nz >> (4 * x), n, thr, lane, low, zero, lost);
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          if (lane == q) w = low[q];
          if (lane == 4 + q) w = zero[q];
        }
        if (lane < 8) __stcg(xC + (tix(uI[x], uJ[x]) * 2 + uH[x]) * 8 + lane, w);
        const int c = __popc(low[0]) + __popc(low[1]) + __popc(low[2]) + __popc(low[3]) +
                      (zero[0] | zero[1] | zero[2] | zero[3] ? 1 << 16 : 0) + (__any_sync(0xffffffffu, lost) ? 1 << 24 : 0);
        if (lane == 0 && c) atomicAdd(&sm.nlow, c);
      }
    }
#pragma unroll
    for (int x = 0; x < 2; ++x) {
      if (uI[x] < 0) continue;
      const int I = uI[x], J = uJ[x], j0 = 8 * uH[x];
      long long sum[4];
      if (step == 0) half_tile_product<6>(sm, I, J, j0, lane, sum);
      else half_tile_product<8>(sm, I, J, j0, lane, sum);
      float res[4];
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const long long d = afix[x][q] - sum[q];
        const unsigned long long a = (unsigned long long)(d < 0 ? -d : d);
        res[q] = fmaf((float)(unsigned)(a >> 32), 0x1p32f, (float)(unsigned)a) * (d < 0 ? -0x1p-58f : 0x1p-58f);
        mx = fmaxf(mx, fabsf(res[q]));
      }
      float* o = xR + tix(I, J) * 256 + (lane >> 2) * 16 + j0 + 2 * (lane & 3);
      __stcg(reinterpret_cast<float2*>(o), make_float2(res[0], res[1]));
      __stcg(reinterpret_cast<float2*>(o + 128), make_float2(res[2], res[3]));
    }
    {
      // non-negative floats order as their bits
      const unsigned m = __reduce_max_sync(0xffffffffu, __float_as_uint(mx));
      if (lane == 0) atomicMax(&sm.rmax[par], m);
    }
    cluster.sync();                                            // B1: the residual tiles are written
    // ---- all of R, scaled by a power of two, as pairs ----
    float4 g[9];
#pragma unroll
    for (int u = 0; u < 9; ++u) {
      const int idx = tid + kThreads * u;
      g[u] = (idx >> 6) < NTL ? __ldcg(reinterpret_cast<const float4*>(xR) + idx) : make_float4(0.f, 0.f, 0.f, 0.f);
    }
    mx = cluster_max(cluster, &sm.rmax[par]);
    if (step == 0) {
      int w[kCtas];
      bool zeros = false, lost = false;
#pragma unroll
      for (int u = 0; u < kCtas; ++u) w[u] = *(volatile int*)cluster.map_shared_rank(&sm.nlow, u);
#pragma unroll
      for (int u = 0; u < kCtas; ++u) {
        total += w[u] & 0xffff;
        zeros |= ((w[u] >> 16) & 0xff) != 0;
        lost |= (w[u] >> 24) != 0;
      }
      // the same in every CTA.  (Fill from an entry that its upper half cannot hold would pass for a zero.)
      if (total > kMaxRepair || (zeros && (lost || total > 0))) break;
      if (mine && tid < 64) {
        const int I = tid >> 3;
        (&sm.zero[0][0][0])[tid] = I >= rank && I < T ? __ldcg(xC + (tix(I, rank) * 2 + ((tid >> 2) & 1)) * 8 + 4 + (tid & 3)) : 0u;
      }
      if (rank == 0 && total > 0) {
        // half tile u / 4, word u % 4
        for (int u = tid; u < 2 * NTL * 4; u += kThreads) {
          const int t = u >> 3, h = (u >> 2) & 1, q = u & 3;
          int I = 0;
          while ((I + 1) * (I + 2) / 2 <= t) ++I;
          const int J = t - I * (I + 1) / 2;
          for (unsigned m = __ldcg(xC + (t * 2 + h) * 8 + q); m; m &= m - 1) {
            const int l = __ffs(m) - 1, i = 16 * I + (l >> 2) + 8 * (q >> 1), j = 16 * J + 8 * h + 2 * (l & 3) + (q & 1);
            const int at = atomicAdd(&sm.nrep, 1);
            sm.rep[at] = (j << 8) | i;
          }
        }
        __syncthreads();
        if (warp == 0) {                                       // by column, then row
          const int v = lane < total ? sm.rep[lane] : INT_MAX;
          int at = 0;
          for (int u = 0; u < total; ++u) at += __shfl_sync(0xffffffffu, v, u) < v;
          __syncwarp();
          if (lane < total) {
            sm.rep[at] = v;
            sm.rep_a[at] = A[(size_t)(v >> 8) * ld + (v & 255)];
          }
        }
      }
    }
    // scale 2^s with max |R| 2^s in [0.5, 1)
    const int xe = max((int)(__float_as_uint(mx) >> 23) & 0xff, 1) - 126;
    const int s = min(-xe, 100);
    const float fs = __uint_as_float((unsigned)(s + 127) << 23), fsi = __uint_as_float((unsigned)(127 - s) << 23);
    if (mx > 0.f) {
#pragma unroll
      for (int u = 0; u < 9; ++u) {
        const int idx = tid + kThreads * u, t = idx >> 6, i = (idx & 63) >> 2, j = 4 * (idx & 3);
        if (t >= NTL) continue;
        __half2 h0, l0, h1, l1;
        half_pair2(make_float2(g[u].x * fs, g[u].y * fs), h0, l0);
        half_pair2(make_float2(g[u].z * fs, g[u].w * fs), h1, l1);
        __half2* p = reinterpret_cast<__half2*>(&sm.R[t][0][ht(i, j)]);
        p[0] = h0;
        p[1] = h1;
        p = reinterpret_cast<__half2*>(&sm.R[t][1][ht(i, j)]);
        p[0] = l0;
        p[1] = l1;
      }
    }
    __syncthreads();
    const int J = rank;
    const int I = warp;
    float em = 0.f;
    float dl[2][4] = {};                                       // this warp's corrections L0 F
    const bool below = mine && mx > 0.f && I >= J && I < T;
    if (mine && mx > 0.f) {
      uint32_t ah[4], al[4], bh[4], bl[4];
      // T = R W0_J^T, row tile I
      if (I < T) {
        float c0[2][4] = {}, c1[2][4] = {};
        for (int k = 0; k <= J; ++k) {
          if (k <= I) {
            frag<Op::A>(ah, sm.R[tix(I, k)][0], lane);
            frag<Op::A>(al, sm.R[tix(I, k)][1], lane);
          } else {
            frag<Op::At>(ah, sm.R[tix(k, I)][0], lane);
            frag<Op::At>(al, sm.R[tix(k, I)][1], lane);
          }
          frag<Op::B>(bh, sm.W0[tix(J, k)][0], lane);
          frag<Op::B>(bl, sm.W0[tix(J, k)][1], lane);
          pair_mm(c0, c1, ah, al, bh, bl);
        }
#pragma unroll
        for (int h = 0; h < 2; ++h)
#pragma unroll
          for (int q = 0; q < 4; ++q) c0[h][q] = fmaf(c1[h][q], 0x1p-11f, c0[h][q]);
        put_tt(sm, I, c0, lane);
      }
      __syncthreads();
      // E = W0 T (row tiles I >= J), F: lower triangle with half the diagonal
      float f0[2][4] = {}, f1[2][4] = {};
      if (below) {
        for (int k = 0; k <= I; ++k) {
          frag<Op::A>(ah, sm.W0[tix(I, k)][0], lane);
          frag<Op::A>(al, sm.W0[tix(I, k)][1], lane);
          frag_tt(bh, sm.Tt[0], k, lane);
          frag_tt(bl, sm.Tt[1], k, lane);
          pair_mm(f0, f1, ah, al, bh, bl);
        }
#pragma unroll
        for (int h = 0; h < 2; ++h)
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            float E = fmaf(f1[h][q], 0x1p-11f, f0[h][q]);
            if (!(fabsf(E) < 1e30f)) em = __uint_as_float(0x7f800000u);   // not finite: gives up
            em = fmaxf(em, fabsf(E));
            const int c = 8 * h + 2 * (lane & 3) + (q & 1), r = (lane >> 2) + 8 * (q >> 1);
            if (I == J) E = r > c ? E : (r == c ? 0.5f * E : 0.f);
            f0[h][q] = E;
          }
      }
      __syncthreads();
      if (below) put_tt(sm, I, f0, lane);
      __syncthreads();
      // the correction of column block J, L0 F
      if (below) {
        float c1[2][4] = {};
        for (int k = J; k <= I; ++k) {
          frag<Op::A>(ah, sm.L0.h[tix(I, k)][0], lane);
          frag<Op::A>(al, sm.L0.h[tix(I, k)][1], lane);
          frag_tt(bh, sm.Tt[0], k, lane);
          frag_tt(bl, sm.Tt[1], k, lane);
          pair_mm(dl, c1, ah, al, bh, bl);
        }
        float* o = xD + tix(I, J) * 256 + (lane >> 2) * 16 + 2 * (lane & 3);
#pragma unroll
        for (int h = 0; h < 2; ++h) {
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            const int c = 8 * h + 2 * (lane & 3) + (q & 1), r = (lane >> 2) + 8 * (q >> 1);
            dl[h][q] = (I > J || r >= c) ? fmaf(c1[h][q], 0x1p-11f, dl[h][q]) * fsi : 0.f;
          }
          __stcg(reinterpret_cast<float2*>(o + 8 * h), make_float2(dl[h][0], dl[h][1]));
          __stcg(reinterpret_cast<float2*>(o + 8 * h + 128), make_float2(dl[h][2], dl[h][3]));
        }
      }
    }
    {
      const unsigned m = __reduce_max_sync(0xffffffffu, __float_as_uint(em));
      if (lane == 0) atomicMax(&sm.emax[par], m);
      // the other parity's words were read before the last barrier and are used again after this one
      if (tid == 0) sm.rmax[par ^ 1] = sm.emax[par ^ 1] = 0;
    }
    cluster.sync();                                            // B2: the corrections are written
    em = cluster_max(cluster, &sm.emax[par]) * fsi;          // the scale is the same in every CTA
    if (!(em < (step == 0 ? kMaxFirst : 0.25f))) break;
    if (step == 0) first = fmaxf(em, 0x1p-24f);
    else if (em > 0.25f * last && em > 0x1p-50f) break;
    last = em;
    good = em * first <= kTol;
    if (good) {
      // no further residual: the last correction goes into this CTA's own columns only
      if (below) {
#pragma unroll
        for (int h = 0; h < 2; ++h)
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            const int c = 8 * h + 2 * (lane & 3) + (q & 1), r = (lane >> 2) + 8 * (q >> 1);
            sm.Lx[tix(I, J)][lx(r, c)] += fix62(dl[h][q]);
          }
      }
    } else if (mx > 0.f) {
#pragma unroll
      for (int u = 0; u < 9; ++u) {
        const int idx = tid + kThreads * u;
        g[u] = (idx >> 6) < NTL ? __ldcg(reinterpret_cast<const float4*>(xD) + idx) : make_float4(0.f, 0.f, 0.f, 0.f);
      }
#pragma unroll
      for (int u = 0; u < 9; ++u) {
        const int idx = tid + kThreads * u, t = idx >> 6, i = (idx & 63) >> 2, j = 4 * (idx & 3);
        if (t >= NTL) continue;
        ulonglong2* p = reinterpret_cast<ulonglong2*>(&sm.Lx[t][lx(i, j)]);   // 4 terms stay together
        ulonglong2 y0 = p[0], y1 = p[1];
        y0.x += fix62(g[u].x);
        y0.y += fix62(g[u].y);
        y1.x += fix62(g[u].z);
        y1.y += fix62(g[u].w);
        p[0] = y0;
        p[1] = y1;
        if (step == 0 && W32 != nullptr) {                      // for the inverse below, times 2^22
          __half2* o = reinterpret_cast<__half2*>(&sm.R[t][0][ht(i, j)]);
          o[0] = __float22half2_rn(make_float2(g[u].x * 0x1p22f, g[u].y * 0x1p22f));
          o[1] = __float22half2_rn(make_float2(g[u].z * 0x1p22f, g[u].w * 0x1p22f));
        }
      }
    }
    __syncthreads();
    if (step == 0 && W32 != nullptr && mine) {
      // W = W0 + H W0, H = I - W0 L (a Newton step on the inverse), rows 16 rank ..: L = L0 plus the
      // first correction; every product down to 2^-32, the sums of magnitude 1 start from -I
      const int C = warp;
      const bool delta = mx > 0.f && !good;                    // else the correction is below 2^-33 and R still the residual
      if (C <= rank) {
        float c0[2][4] = {}, c1[2][4] = {}, c2[2][4] = {};
        uint32_t ah[4], al[4], bh[4], bl[4], bd[4];
        if (C == rank) {
#pragma unroll
          for (int h = 0; h < 2; ++h)
#pragma unroll
            for (int q = 0; q < 4; ++q)
              if ((lane >> 2) + 8 * (q >> 1) == 8 * h + 2 * (lane & 3) + (q & 1)) c0[h][q] = -1.f;
        }
        for (int K = C; K <= rank; ++K) {
          frag<Op::A>(ah, sm.W0[tix(rank, K)][0], lane);
          frag<Op::A>(al, sm.W0[tix(rank, K)][1], lane);
          frag<Op::Bt>(bh, sm.L0.h[tix(K, C)][0], lane);
          frag<Op::Bt>(bl, sm.L0.h[tix(K, C)][1], lane);
          pair_mm(c0, c1, ah, al, bh, bl);
          if (delta) frag<Op::Bt>(bd, sm.R[tix(K, C)][0], lane);
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            dig_mma(c2[h], al, bl[2 * h], bl[2 * h + 1]);
            if (delta) dig_mma(c2[h], ah, bd[2 * h], bd[2 * h + 1]);
          }
        }
        // -H times 2^16 as one binary16 plane, rows of H
#pragma unroll
        for (int h = 0; h < 2; ++h)
#pragma unroll
          for (int q = 0; q < 4; q += 2) {
            const float x0 = fmaf(c2[h][q], 0x1p-22f, pair_value(c0[h][q], c1[h][q])) * -0x1p16f;
            const float x1 = fmaf(c2[h][q + 1], 0x1p-22f, pair_value(c0[h][q + 1], c1[h][q + 1])) * -0x1p16f;
            *reinterpret_cast<__half2*>(&sm.Tt[0][(lane >> 2) + 4 * q][16 * C + 8 * h + 2 * (lane & 3)]) =
                __float22half2_rn(make_float2(x0, x1));
          }
      }
      __syncthreads();
      if (C <= rank) {
        float c0[2][4] = {};
        uint32_t ah[4], bh[4];
        for (int K = C; K <= rank; ++K) {
          dig_ldmatrix(ah, &sm.Tt[0][lane & 15][16 * K + (lane >> 4) * 8]);
          frag<Op::Bt>(bh, sm.W0[tix(K, C)][0], lane);
#pragma unroll
          for (int h = 0; h < 2; ++h) dig_mma(c0[h], ah, bh[2 * h], bh[2 * h + 1]);
        }
#pragma unroll
        for (int h = 0; h < 2; ++h)
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            const int c = 8 * h + 2 * (lane & 3) + (q & 1), r = (lane >> 2) + 8 * (q >> 1), at = ht(r, c);
            const float w = pair_value(__half2float(sm.W0[tix(rank, C)][0][at]), __half2float(sm.W0[tix(rank, C)][1][at]));
            sm.Wrow[r][16 * C + c] = fmaf(c0[h][q], 0x1p-16f, w);
          }
      }
    }
    __syncthreads();
    if (good) break;
  }
  if (good && mine) {
    // this CTA's column block of L, and its rows of W
    const int J = rank, gj = 16 * J + lk;
#pragma unroll
    for (int I = 0; I < 8; ++I) {
      const int gi = 16 * I + li;
      if (I >= J && I < T && gi < n && gj <= gi) {
        // bit of entry (li, lk) in its half tile's words: lane 4 (li mod 8) + (lk mod 8) / 2, register 2 (li / 8) + lk mod 2
        const bool z = (sm.zero[I][lk >> 3][2 * (li >> 3) + (lk & 1)] >> (4 * (li & 7) + ((lk & 7) >> 1))) & 1;
        A[(size_t)gj * ld + gi] = z ? 0.0 : dig_to_double((long long)(sm.Lx[tix(I, J)][lx(li, lk)] - kByteBias), sm.e[gi] - 62);
      }
    }
    if (W32 != nullptr) {
      const int gi = 16 * rank + li;
      if (gi < n)
        for (int c = lk; c < n; c += 16)
          W32[(size_t)c * ldw + gi] = c <= gi ? ldexpf(sm.Wrow[li][c], -sm.e[c]) : 0.f;
    }
  }
  cluster.sync();                       // no CTA leaves (or reuses its memory) while others may read it
  if (good && total > 0 && rank == 0 && warp == 0) {
    // l_ij = (a_ij - sum_{k<j} l_ik l_jk) / l_jj from the finished entries, column by column
    for (int u = 0; u < total; ++u) {
      const int i = sm.rep[u] & 255, j = sm.rep[u] >> 8;
      double t = 0.0;
      for (int k = lane; k < j; k += 32) t = fma(__ldcg(A + (size_t)k * ld + i), __ldcg(A + (size_t)k * ld + j), t);
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
      if (lane == 0) A[(size_t)j * ld + i] = (sm.rep_a[u] - t) / __ldcg(A + (size_t)j * ld + j);
      __threadfence_block();
      __syncwarp();
    }
  }
  return good;
}

}  // namespace leafref
}  // namespace hrp
