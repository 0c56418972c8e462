// FP64 leaf TRSM of Alg. 2, B <- B L^{-T} with L a diagonal leaf of order nc <= 128, by refinement
// on the tensor pipe instead of a substitution on the FP64 pipe.
//
// The rows of B are independent.  A CTA takes 16 or 32 of them and, with W the FP32 inverse of L
// (from the leaf POTRF, or launch_trtri_leaves for a standalone solve):
//   X = fl32(B) W^T                                     FP32
//   repeat  R = B - X L^T                               exact (digit products, 64-bit integers)
//           X += R W^T                                  correction in FP32, X in 62-bit fixed point
// Each correction multiplies the error by the relative error rho of an FP32 solve (about
// 2^-24 times the condition number of L), so two of them pass FP64's unit roundoff for the leaves
// of ordinary matrices, and the loop goes on until the next error is below 2^-54 of the row.
// Unlike the substitution this has no chain along the columns: every step is a product.  What
// bounds it is latency of the staged phases at few rows, and the mma and splitting work (28
// products per entry and pass) at many.  Against the right-looking FP64 substitution
// (trsm_rl64_kernel, FP64 pipe and a 63-step chain), 128 columns: 1000 rows 66 -> ~28 us, 3000
// rows 188 -> ~50 us; a standalone TRSM of 3000 x 2048 (three levels, 16 leaves of 128) 3.51 ->
// 1.22 ms, the n = 1024 FP64 factor and solve with leaf 64 1.96 -> 1.84 ms.  Its error against
// extended precision is 2 to 10 times smaller than the substitution's.
//
// Scales are powers of two, applied exactly: 2^beta_r from the largest entry of row r of B, c_j
// from the largest entry of column j of the first X over the CTA's rows, rho_r of row r of that X
// after the columns' scales, and El_j of row j of L with the columns' scales.  X is held to
// 2^-62 of its row's and column's scale.  Rows whose first X is not finite, whose B does not fit the
// scales, or that do not converge (an ill-conditioned or singular leaf) are solved by FP64
// substitution in the same CTA.
//
// A column's scale comes from all rows of the CTA, and an entry whose own terms are far below its row's and
// column's scales (rows or columns in different units) would be left with their error.  So sum |x| |l|
// is estimated for every entry beside the first residual (one mma per 16 terms on bfloat16 magnitudes),
// and the entries below 2^-12 of the scales are computed again, x_j = (b_j - sum_{k<j} x_k l_jk) / l_jj in FP64,
// once the others are done; a row with more than kMaxLow of them sends its CTA to the substitution.  The line:
// a residual is good to 2^-59.8 of its scales (128 terms, ordinary digits; nc 2^-59.7 at worst), so 2^-47.8 of
// sum |x| |l| at it, under the substitution's bound of nc 2^-53; of 2000 entries of an ordinary panel one is
// below it or fewer (up to 13 at 2^-10).  It costs 4 % of the n = 1024 FP64 factorization (1470 -> 1530 us) and 8 %
// of the TRSM of 3000 x 2048 (1127 -> 1224).
#include <climits>

#include "digits.cuh"
#include "hrp_internal.cuh"

namespace hrp {
namespace {

// fractional bits of the residual's fixed point.  B and X L^T are formed modulo 2^64 and may wrap
// (up to 2^7 units); their difference is below 2^-2 or the rows go to the substitution.
constexpr int kRFrac = 60;
constexpr int kMaxPass = 8;
// Entries below 2^-12 of their scales (kCovered) are computed again by FP64 FMAs, up to kMaxLow in a row
constexpr float kCovered = 0x1p-12f;
constexpr int kMaxLow = 6;
// the scale of a column whose first X is zero in every row: it must weigh nothing in the rows of L
constexpr int kNoScale = -4096;

struct T64Layout {                            // byte offsets into dynamic shared memory
  int lx, w, xd, b, r, total, xd_ld, xd_plane;
};
__host__ __device__ inline T64Layout t64_layout(int nc, int rows) {
  const int T = (nc + 15) / 16, ncp = 16 * T;
  T64Layout l;
  l.lx = 0;                                   // L: lower 16 x 16 tiles of 64-bit values
  l.w = l.lx + T * (T + 1) / 2 * 256 * 8;     // W: groups of 8 rows j, [k][8] for k < 8 (g + 1)
  l.xd = l.w + 32 * (2 * T) * (2 * T + 1) * 4;
  l.xd_ld = ncp + 8;                          // X's digits [7][rows][ncp + 8], and its magnitudes
  l.xd_plane = rows * l.xd_ld;
  l.b = l.xd + (kDig + 1) * l.xd_plane * 2;         // B: [k][rows] doubles
  l.r = l.b + ncp * rows * 8;                 // R (and fl32(B)): [k][rows] floats
  l.total = l.r + ncp * rows * 4;
  return l;
}
// entry (j, k) of a 16 x 16 tile of L: rows of 128 bytes, halves swapped on odd rows so that a
// fragment's 16-byte reads do not conflict
__device__ __forceinline__ int lx_at(int j, int k) { return j * 16 + (k ^ ((j & 1) << 3)); }
// exponent e of x with |x| < 2^e (INT_MIN for zero), and for binary32
__device__ __forceinline__ int ex_of(float x) {
  const int F = (int)(__float_as_uint(x) >> 23) & 0xff;
  return (__float_as_uint(x) << 1) == 0 ? INT_MIN : max(F, 1) - 126;
}
// (zero is tested on the bits: an FP64 comparison runs on the FP64 pipe, 19 clocks a warp and SM)
__device__ __forceinline__ bool is_zero(double x) { return ((unsigned long long)__double_as_longlong(x) << 1) == 0; }
__device__ __forceinline__ int ex_of(double x) { return is_zero(x) ? INT_MIN : max(dig_field(x), 1) - 1022; }

// x 2^e truncated to binary32 (0 below its normal range), and x in units of 2^(E - 62), |x| < 2^E,
// both by integer operations (conversions run on the FP64 pipe)
__device__ __forceinline__ float seed_float(double x, int e) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(x);
  const int F = ((int)(b >> 52) & 0x7ff) - 1023 + 127 + e;
  if (F <= 0) return 0.f;
  if (F >= 255) return __uint_as_float(0x7fc00000u);
  return __uint_as_float(((unsigned)(b >> 32) & 0x80000000u) | ((unsigned)F << 23) | ((unsigned)(b >> 29) & 0x7fffffu));
}
__device__ __forceinline__ long long fix_float(float x, int E) {
  const unsigned b = __float_as_uint(x);
  const int F = (int)(b >> 23) & 0xff;
  if (F == 0) return 0;
  const long long m = (long long)((b & 0x7fffffu) | 0x800000u);
  const int sh = F - 150 + 62 - E;                            // x = m 2^(F - 150)
  const long long v = sh >= 0 ? m << min(sh, 39) : (sh > -25 ? m >> -sh : 0);
  return (int)b < 0 ? -v : v;
}

// |v| of a fixed-point entry (unit 2^-62, plus kDigBias) as a bfloat16, truncated, at least 2^-60 unless zero
__device__ __forceinline__ uint32_t fix_abs(unsigned long long v) {
  const long long d = (long long)(v - kDigBias);
  const unsigned long long a = (unsigned long long)(d < 0 ? -d : d);
  const unsigned hi = (unsigned)(a >> 32);                    // units 2^-30
  const int b = (int)(__float_as_uint((float)hi * 0x1p-30f) >> 16);
  return a == 0 ? 0u : (uint32_t)max(b, kAbsMin);
}

// unit u of the packed W -> its group and column: 4 g (g + 1) units come before group g
__device__ __forceinline__ void w_unit(int u, int& g, int& k) {
  g = (int)((sqrtf((float)(u + 1)) - 1.0f) * 0.5f);
  while (4 * (g + 1) * (g + 2) <= u) ++g;
  while (4 * g * (g + 1) > u) --g;
  k = u - 4 * g * (g + 1);
}
__device__ __forceinline__ void cp_async16(void* dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src)
               : "memory");
}
__device__ __forceinline__ void cp_async_wait_all() {
  asm volatile("cp.async.commit_group;\ncp.async.wait_group 0;" ::: "memory");
}

// float scale 2^e (saturating: values past binary32's range make the refinement give up)
__device__ __forceinline__ float pow2f(int e) { return __uint_as_float((unsigned)(max(-126, min(127, e)) + 127) << 23); }

// The CTA's rows by FP64 substitution, 16 lanes per row: lane q holds columns q, q + 16, ..  L and its reciprocal
// pivots are staged first (over L, W and X's digits, and over R); what bounds it is then the FP64 pipe, 4.5 FMAs
// a column and pair of rows.  200 rows of 128 columns in units far apart take 120 us, refined ones 76 and
// trsm_rl64_kernel 80; 3000 rows 178, 97 and 202.  (With L read from global memory, a division per
// column in every lane and idle rows computed too: 437 and 363.)
template <int TM, int ROWS, int NT>
__device__ __noinline__ bool substitute(double* X, int ld, int r0, int m, int c0, int nc, const double* __restrict__ L, int ldl,
                                        unsigned char* smem, __half* s16, int lds, float* s32, int ld32) {
  const T64Layout lay = t64_layout(nc, ROWS);
  double* Ls = reinterpret_cast<double*>(smem);
  double* rinv = reinterpret_cast<double*>(smem + lay.r);
  const double* Bs = reinterpret_cast<const double*>(smem + lay.b);
  const int row0 = blockIdx.x * ROWS, live = min(ROWS, m - row0);
  X += (size_t)c0 * ld + r0 + row0;
  L += (size_t)c0 * ldl + c0;
  if (s16 != nullptr) s16 += (size_t)(r0 + row0) * lds + c0;
  if (s32 != nullptr) s32 += (size_t)c0 * ld32 + r0 + row0;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, q = tid & 15, ncp = (nc + 15) / 16 * 16;
  bool over16 = false;
  __syncthreads();
#pragma unroll 4
  for (int k = warp; k < nc; k += NT / 32)
#pragma unroll
    for (int u = 0; u < TM / 2; ++u) {
      const int j = lane + 32 * u;
      if (j < ncp) Ls[k * ncp + j] = (j >= k && j < nc) ? L[(size_t)k * ldl + j] : 0.0;
    }
  __syncthreads();
  if (tid < nc) rinv[tid] = 1.0 / Ls[tid * ncp + tid];
  __syncthreads();
  for (int rb = 0; rb < ROWS; rb += NT / 16) {
    if (rb + 2 * warp >= live) continue;                      // whole warps
    const int r = rb + (tid >> 4);
    double y[TM];
#pragma unroll
    for (int c = 0; c < TM; ++c) y[c] = q + 16 * c < nc ? Bs[(q + 16 * c) * ROWS + r] : 0.0;
#pragma unroll
    for (int p = 0; p < TM; ++p)
      for (int kk = 0; kk < 16; ++kk) {
        const int k = 16 * p + kk;
        if (k >= nc) break;
        const double* lk = Ls + k * ncp + q;
        const double v = __shfl_sync(0xffffffffu, y[p], (lane & 16) | kk) * rinv[k];
        if (q == kk) y[p] = v;
        else if (q > kk) y[p] = fma(-v, lk[16 * p], y[p]);
#pragma unroll
        for (int c = p + 1; c < TM; ++c)
          if (16 * c < nc) y[c] = fma(-v, lk[16 * c], y[c]);
      }
    if (r >= live) continue;
#pragma unroll
    for (int c = 0; c < TM; ++c) {
      const int j = q + 16 * c;
      if (j >= nc) continue;
      X[(size_t)j * ld + r] = y[c];
      if (s32 != nullptr) s32[(size_t)j * ld32 + r] = (float)y[c];
      if (s16 != nullptr) {
        over16 |= fabs(y[c]) > (double)kF16Max;
        s16[(size_t)r * lds + j] = __double2half(y[c]);
      }
    }
  }
  return over16;
}

// MR: 16-row tiles per CTA.  NT: threads, one warp per group of 8 columns (nc <= NT / 4).
template <int MR, int NT>
__global__ void __launch_bounds__(NT, 1)
trsm_refine64_kernel(double* __restrict__ A, int ld, int r0, int m, int c0, int nc, const double* __restrict__ Lm,
                     int ldl, const float* __restrict__ W, int ldw, __half* __restrict__ S, int lds,
                     float* __restrict__ S32, int ld32, const int* __restrict__ info, unsigned* __restrict__ err) {
  constexpr int ROWS = 16 * MR;
  constexpr int TM = NT / 64;                 // tiles of 16 columns at most
  constexpr int TS = NT / 256;                // tiles staged per step
  pdl_wait();
  pdl_trigger();
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ int s_beta[ROWS], s_rho[ROWS], s_c[16 * TM], s_el[16 * TM];
  __shared__ unsigned s_max, s_low[ROWS][TM / 2];            // entries to compute again, a bit per column
  __shared__ int s_nlow[ROWS];
  if (*(volatile const int*)info != INT_MAX) return;
  const T64Layout lay = t64_layout(nc, ROWS);
  const int T = (nc + 15) / 16, ncp = 16 * T, G = 2 * T, nt = T * (T + 1) / 2;
  double* Ld = reinterpret_cast<double*>(smem + lay.lx);
  long long* Lx = reinterpret_cast<long long*>(smem + lay.lx);
  float* Ws = reinterpret_cast<float*>(smem + lay.w);
  __half* Xd = reinterpret_cast<__half*>(smem + lay.xd);
  double* Bs = reinterpret_cast<double*>(smem + lay.b);
  float* Rs = reinterpret_cast<float*>(smem + lay.r);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int row0 = blockIdx.x * ROWS;
  const double* Bg = A + (size_t)c0 * ld + r0 + row0;
  const int live = min(ROWS, m - row0);

  // B: a thread holds one row's entries (lanes along rows); L's lower tiles (raw): one entry of a
  // tile per thread, lanes along j (a column of L is contiguous); all of a batch in flight together
  constexpr int kU = 4 * MR, kS = NT / ROWS;
  const int br = tid % ROWS, bk = tid / ROWS;
  double bv[kU];
#pragma unroll
  for (int u = 0; u < kU; ++u) {
    const int k = bk + kS * u;
    bv[u] = (k < nc && br < live) ? Bg[(size_t)k * ld + br] : 0.0;
  }
  // W in its packed groups: unit u = (group g, k), 8 consecutive rows of column k of W, by
  // asynchronous 16-byte copies (both sides 16-byte aligned: ldw a multiple of 4)
  const bool wvec = (ldw & 3) == 0 && (reinterpret_cast<uintptr_t>(W) & 15) == 0;
  const int nunit = 4 * G * (G + 1);
  for (int u = tid; u < nunit; u += NT) {
    int g, k;
    w_unit(u, g, k);
    float* dst = Ws + 8 * u;
    if (wvec && 8 * g + 8 <= nc && k < nc) {
      cp_async16(dst, W + (size_t)k * ldw + 8 * g);
      cp_async16(dst + 4, W + (size_t)k * ldw + 8 * g + 4);
    } else {
#pragma unroll
      for (int q = 0; q < 8; ++q) dst[q] = (8 * g + q < nc && k < nc) ? W[(size_t)k * ldw + 8 * g + q] : 0.f;
    }
  }
  {
    const int j = tid & 15, k = (tid >> 4) & 15;
    int I = 0, J = 0;
    auto step = [&]() {
      if (++J > I) {
        ++I;
        J = 0;
      }
    };
    if (TS == 2 && tid >= 256) step();
    constexpr int kB = TS == 2 ? 18 : 10;      // all of a thread's entries in flight at once
    for (int t0 = tid >> 8; t0 < nt; t0 += kB * TS) {
      double v[kB];
#pragma unroll
      for (int u = 0; u < kB; ++u) {
        const int gj = 16 * I + j, gk = 16 * J + k;
        v[u] = (gj < nc && gk <= gj) ? Lm[(size_t)(c0 + gk) * ldl + c0 + gj] : (gj == gk ? 1.0 : 0.0);
#pragma unroll
        for (int w = 0; w < TS; ++w) step();
      }
#pragma unroll
      for (int u = 0; u < kB; ++u)
        if (t0 + TS * u < nt) Ld[(t0 + TS * u) * 256 + lx_at(j, k)] = v[u];
    }
  }
  if (tid < ROWS) s_beta[tid] = s_rho[tid] = INT_MIN;
  if (tid < ROWS) s_nlow[tid] = 0;
  if (tid < ROWS * (TM / 2)) s_low[tid / (TM / 2)][tid % (TM / 2)] = 0;
  if (tid < 16 * TM) s_c[tid] = INT_MIN;
  if (tid == 0) s_max = 0;
  __syncthreads();
  {
    int ex = INT_MIN;
#pragma unroll
    for (int u = 0; u < kU; ++u) ex = max(ex, ex_of(bv[u]));
    atomicMax(&s_beta[br], ex);
    __syncthreads();
    const int be = s_beta[br] == INT_MIN ? 0 : s_beta[br];
#pragma unroll
    for (int u = 0; u < kU; ++u) {
      const int k = bk + kS * u;
      // |B 2^-beta| < 1; entries below binary32's range are zero here and come back with R
      if (k < ncp) {
        Bs[k * ROWS + br] = bv[u];
        Rs[k * ROWS + br] = seed_float(bv[u], -be);
      }
    }
  }
  cp_async_wait_all();
  __syncthreads();
  // the warp's group of 8 columns: short and long ones share the sub-partitions evenly.  A
  // lane's outputs: row lane % 16 (and + 16), columns 4 (lane / 16) .. + 3 of the group
  const int g = NT == 512 && warp >= 8 ? 23 - warp : (NT == 256 && warp >= 4 ? 11 - warp : warp);
  const bool act = g < G;                     // whole warps
  const int rr = lane & 15, cq = 4 * (lane >> 4);
  // o = R W^T
  auto product = [&](float (&o)[MR][4]) {
#pragma unroll
    for (int h = 0; h < MR; ++h)
#pragma unroll
      for (int q = 0; q < 4; ++q) o[h][q] = 0.f;
    const float* wp = Ws + 32 * g * (g + 1) + cq;
    const float* rp = Rs + rr;
    for (int k0 = 0; k0 <= g; ++k0, wp += 64, rp += 8 * ROWS) {
      float4 w[8];
      float b[8][MR];
#pragma unroll
      for (int k = 0; k < 8; ++k) {
        w[k] = *reinterpret_cast<const float4*>(wp + 8 * k);
#pragma unroll
        for (int h = 0; h < MR; ++h) b[k][h] = rp[k * ROWS + 16 * h];
      }
#pragma unroll
      for (int k = 0; k < 8; ++k)
#pragma unroll
        for (int h = 0; h < MR; ++h) {
          o[h][0] = fmaf(b[k][h], w[k].x, o[h][0]);
          o[h][1] = fmaf(b[k][h], w[k].y, o[h][1]);
          o[h][2] = fmaf(b[k][h], w[k].z, o[h][2]);
          o[h][3] = fmaf(b[k][h], w[k].w, o[h][3]);
        }
    }
  };
  float x0[MR][4];
  int bad = 0;
  if (tid < nc) {                             // an inverse near the ends of binary32's range is no seed
    const float d = fabsf(W[(size_t)tid * ldw + tid]);
    bad = !(d > 0x1p-100f && d < 0x1p100f);
  }
  if (act) {
    product(x0);
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      int ex = INT_MIN;
#pragma unroll
      for (int h = 0; h < MR; ++h) {
        bad |= !isfinite(x0[h][q]);
        ex = max(ex, ex_of(x0[h][q]));
      }
      // the 16 lanes of this column
#pragma unroll
      for (int o = 8; o > 0; o >>= 1) ex = max(ex, __shfl_xor_sync(0xffffffffu, ex, o));
      if (rr == 0) s_c[8 * g + cq + q] = ex == INT_MIN ? kNoScale : ex;
    }
  }
  bad = __syncthreads_or(bad);
  if (!bad) {
    if (act) {
#pragma unroll
      for (int h = 0; h < MR; ++h) {
        int ex = INT_MIN;
#pragma unroll
        for (int q = 0; q < 4; ++q)
          if (x0[h][q] != 0.f) ex = max(ex, ex_of(x0[h][q]) - s_c[8 * g + cq + q]);
        atomicMax(&s_rho[rr + 16 * h], ex);
      }
    }
    // rows of L against the columns' scales, then in fixed point: thread (j, k) of every tile of a
    // tile row (two tile rows at a time with 512 threads)
    const int k = tid & 15, j = (tid >> 4) & 15;
    int ck[TM];
#pragma unroll
    for (int J = 0; J < TM; ++J) ck[J] = J < T ? s_c[16 * J + k] : 0;
#pragma unroll
    for (int i = 0; i < TM / TS; ++i) {
      // tile rows 0, 1, .. (256 threads), or i and 7 - i on the two halves: as many tiles each
      const int I = TS == 2 ? (tid >= 256 ? TM - 1 - i : i) : i;
      if (I >= T) continue;                                     // whole warps
      double v[TM];
      int ex = INT_MIN;
#pragma unroll
      for (int J = 0; J < TM; ++J) {
        v[J] = J <= I ? Ld[(I * (I + 1) / 2 + J) * 256 + lx_at(j, k)] : 0.0;
        bad |= dig_field(v[J]) == 0x7ff;
        if (!is_zero(v[J])) ex = max(ex, ex_of(v[J]) + ck[J]);
      }
#pragma unroll
      for (int o = 8; o > 0; o >>= 1) ex = max(ex, __shfl_xor_sync(0xffffffffu, ex, o));
      if (ex == INT_MIN) ex = 0;                                // a zero row: W is not finite there
      if (k == 0) s_el[16 * I + j] = ex;
#pragma unroll
      for (int J = 0; J < TM; ++J)
        if (J <= I)
          Lx[(I * (I + 1) / 2 + J) * 256 + lx_at(j, k)] =
              (long long)((unsigned long long)dig_fix(v[J], ex + 1022 - ck[J]) + kDigBias);
    }
    bad = __syncthreads_or(bad);
  }
  // X in fixed point, unit 2^(E - 62) with E = beta_r + rho_r + c_j + 1, and its digits
  long long X[MR][4];
  auto put_digits = [&]() {
#pragma unroll
    for (int h = 0; h < MR; ++h) {
      __half* d = Xd + (size_t)(rr + 16 * h) * lay.xd_ld + 8 * g + cq;
      unsigned long long Mb[4];
#pragma unroll
      for (int q = 0; q < 4; ++q) Mb[q] = (unsigned long long)X[h][q] + kDigBias;
#pragma unroll
      for (int s = 0; s < kDig; ++s)
        *reinterpret_cast<uint2*>(d + (size_t)s * lay.xd_plane) =
            make_uint2(dig_pair(Mb[0], Mb[1], s), dig_pair(Mb[2], Mb[3], s));
    }
  };
  if (!bad) {
    if (tid < ROWS && s_rho[tid] == INT_MIN) s_rho[tid] = 0;
    if (tid < ROWS && s_beta[tid] == INT_MIN) s_beta[tid] = 0;
    for (int u = tid; u < nunit; u += NT) {
      int gu, ku;
      w_unit(u, gu, ku);
      const int el = s_el[ku];
      float4 w0 = *reinterpret_cast<float4*>(Ws + 8 * u), w1 = *reinterpret_cast<float4*>(Ws + 8 * u + 4);
      const int* cc = s_c + 8 * gu;
      // columns without a scale take no correction (a residual there goes to the substitution)
      auto f = [&](int q) { return cc[q] == kNoScale ? 0.f : pow2f(el - cc[q]); };
      w0 = make_float4(w0.x * f(0), w0.y * f(1), w0.z * f(2), w0.w * f(3));
      w1 = make_float4(w1.x * f(4), w1.y * f(5), w1.z * f(6), w1.w * f(7));
      *reinterpret_cast<float4*>(Ws + 8 * u) = w0;
      *reinterpret_cast<float4*>(Ws + 8 * u + 4) = w1;
    }
    __syncthreads();
    if (act) {
#pragma unroll
      for (int h = 0; h < MR; ++h)
#pragma unroll
        for (int q = 0; q < 4; ++q) X[h][q] = fix_float(x0[h][q], s_rho[rr + 16 * h] + s_c[8 * g + cq + q] + 1);
      put_digits();
      // the magnitudes of the first X against the same scales, as bfloat16 (dig_abs)
#pragma unroll
      for (int h = 0; h < MR; ++h) {
        uint32_t b[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const int e = s_rho[rr + 16 * h] + s_c[8 * g + cq + q] + 1, v = (int)(__float_as_uint(fabsf(x0[h][q])) >> 16);
          b[q] = x0[h][q] == 0.f ? 0u : (uint32_t)max(v - e * 128, kAbsMin);
        }
        *reinterpret_cast<uint2*>(Xd + kDig * lay.xd_plane + (size_t)(rr + 16 * h) * lay.xd_ld + 8 * g + cq) =
            make_uint2(b[0] | (b[1] << 16), b[2] | (b[3] << 16));
      }
    }
  }
  __syncthreads();

  // sum |x| |l| of every entry of X L^T against the scales (a fifth of a pass): where an entry's own terms are
  // far below them, the residual's digits do not cover it
  int many = 0;                               // too many of them in a row: joins `bad` with the first pass
  if (!bad && act) {
    const int I = g >> 1, jrow = 8 * (g & 1) + (lane >> 2);
    float est[MR][4] = {};
    const __half* xa = Xd + kDig * lay.xd_plane + (size_t)(lane & 15) * lay.xd_ld + (lane >> 4) * 8;
#pragma unroll 2
    for (int kt = 0; kt <= I; ++kt) {
      const long long* lt = Lx + (I * (I + 1) / 2 + kt) * 256;
      const ulonglong2 p0 = *reinterpret_cast<const ulonglong2*>(lt + lx_at(jrow, 2 * (lane & 3)));
      const ulonglong2 p1 = *reinterpret_cast<const ulonglong2*>(lt + lx_at(jrow, 2 * (lane & 3) + 8));
      const uint32_t b0 = fix_abs(p0.x) | (fix_abs(p0.y) << 16), b1 = fix_abs(p1.x) | (fix_abs(p1.y) << 16);
#pragma unroll
      for (int h = 0; h < MR; ++h) {
        uint32_t a[4];
        dig_ldmatrix(a, xa + (size_t)(16 * h) * lay.xd_ld + 16 * kt);
        dig_mma_bf16(est[h], a, b0, b1);
      }
    }
#pragma unroll
    for (int h = 0; h < MR; ++h)
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const int r = 16 * h + (lane >> 2) + 8 * (q >> 1), j = 8 * g + 2 * (lane & 3) + (q & 1);
        // (all terms and the right-hand side zero: so is the entry)
        if (j < nc && r < live && est[h][q] < kCovered && (est[h][q] > 0.f || !is_zero(Bs[j * ROWS + r]))) {
          atomicOr(&s_low[r][j >> 5], 1u << (j & 31));
          if (atomicAdd(&s_nlow[r], 1) >= kMaxLow) many = 1;
        }
      }
  }

  float first = 1.f, last = 1.f;
  bool done = false;
  for (int pass = 0; pass < kMaxPass && !bad && !done; ++pass) {
    // ---- R = B - X L^T, the warp's 8 columns ----
    if (act) {
      const int I = g >> 1, jrow = 8 * (g & 1) + (lane >> 2);
      long long sum[MR][4];
#pragma unroll
      for (int h = 0; h < MR; ++h)
#pragma unroll
        for (int q = 0; q < 4; ++q) sum[h][q] = 0;
      const __half* xa = Xd + (size_t)(lane & 15) * lay.xd_ld + (lane >> 4) * 8;
#pragma unroll 1
      for (int ks = 0; ks <= I; ks += 2) {
        float acc[kDig][MR][4];
#pragma unroll
        for (int w = 0; w < kDig; ++w)
#pragma unroll
          for (int h = 0; h < MR; ++h)
#pragma unroll
            for (int q = 0; q < 4; ++q) acc[w][h][q] = 0.f;
#pragma unroll
        for (int k2 = 0; k2 < 2; ++k2) {
          const int kt = ks + k2;
          if (kt > I) break;
          // L(j, 2t), (j, 2t + 1), (j, 2t + 8), (j, 2t + 9) of tile (I, kt)
          const long long* lt = Lx + (I * (I + 1) / 2 + kt) * 256;
          const ulonglong2 p0 = *reinterpret_cast<const ulonglong2*>(lt + lx_at(jrow, 2 * (lane & 3)));
          const ulonglong2 p1 = *reinterpret_cast<const ulonglong2*>(lt + lx_at(jrow, 2 * (lane & 3) + 8));
          uint32_t bf[kDig][2];
#pragma unroll
          for (int s = 0; s < kDig; ++s) {
            bf[s][0] = dig_pair(p0.x, p0.y, s);
            bf[s][1] = dig_pair(p1.x, p1.y, s);
          }
#pragma unroll
          for (int s = 0; s < kDig; ++s)
#pragma unroll
            for (int h = 0; h < MR; ++h) {
              uint32_t a[4];
              dig_ldmatrix(a, xa + (size_t)s * lay.xd_plane + (size_t)(16 * h) * lay.xd_ld + 16 * kt);
#pragma unroll
              for (int t = 0; t < kDig - s; ++t) dig_mma(acc[s + t][h], a, bf[t][0], bf[t][1]);
            }
        }
#pragma unroll
        for (int h = 0; h < MR; ++h)
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            // weights 2^(-16 - 9 w): w = 0 .. 2 and 3 .. 6 joined first
            long long hi = 0, lo = 0;
#pragma unroll
            for (int w = 0; w < 3; ++w) hi = (hi << 9) + __float2int_rn(acc[w][h][q]);
#pragma unroll
            for (int w = 3; w < kDig; ++w) lo = (lo << 9) + __float2int_rn(acc[w][h][q]);
            sum[h][q] += (hi << (kRFrac - 34)) + (lo >> (70 - kRFrac));
          }
      }
#pragma unroll
      for (int h = 0; h < MR; ++h)
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const int r = 16 * h + (lane >> 2) + 8 * (q >> 1), j = 8 * g + 2 * (lane & 3) + (q & 1);
          float res = 0.f;
          if (j < nc && r < live) {
            // unit of the residual: 2^(beta + rho + 1 + El_j - kRFrac)
            const int z = s_beta[r] + s_rho[r] + 1 + s_el[j];
            const double x = Bs[j * ROWS + r];
            const int F = dig_field(x);
            const int sh = max(F, 1) - 1075 + kRFrac - z;
            long long mb = (long long)(((unsigned long long)__double_as_longlong(x) & 0xfffffffffffffull) |
                                       (F ? 0x10000000000000ull : 0ull));
            if (mb != 0 && (sh > 18 || F == 0x7ff)) bad = 1;            // B outside the scales
            else if (sh >= 0) mb <<= min(sh, 63);
            else mb = (mb + (1ll << (min(-sh, 62) - 1))) >> min(-sh, 62);
            if (__double_as_longlong(x) < 0) mb = -mb;
            // |d| to binary32 by halves (of d itself the halves would cancel)
            const long long d = mb - sum[h][q];
            const unsigned long long a = (unsigned long long)(d < 0 ? -d : d);
            res = fmaf((float)(unsigned)(a >> 32), 0x1p32f, (float)(unsigned)a) * (d < 0 ? -0x1p-60f : 0x1p-60f);
            if (!(fabsf(res) < 0.25f) || (s_c[j] == kNoScale && res != 0.f)) bad = 1;
          }
          Rs[j * ROWS + r] = res;
        }
    }
    __syncthreads();
    // ---- X += R W^T ----
    float mx = 0.f;
    if (act) {
      float o[MR][4];
      product(o);
#pragma unroll
      for (int h = 0; h < MR; ++h)
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          if (!(fabsf(o[h][q]) < 0.25f)) {
            bad = 1;
          } else {
            mx = fmaxf(mx, fabsf(o[h][q]));
            X[h][q] += __float2ll_rn(o[h][q] * 0x1p62f);
          }
        }
      // non-negative floats order as their bits
      const unsigned mb = __reduce_max_sync(0xffffffffu, __float_as_uint(mx));
      if (lane == 0) atomicMax(&s_max, mb);
    }
    bad = __syncthreads_or(bad | many);
    const float delta = __uint_as_float(s_max);
    if (pass == 0) first = fmaxf(delta, 0x1p-24f);
    else if (delta > 0.25f * last && delta > 0x1p-50f) bad = 1;        // does not converge
    last = delta;
    done = delta * first <= 0x1p-57f;
    if (!done && !bad) {
      if (act) put_digits();
      __syncthreads();
      if (tid == 0) s_max = 0;                 // read by all before this barrier, written after the next
    }
  }
  bool over16 = false;
  if (!bad && done) {
    if (act) {
#pragma unroll
      for (int h = 0; h < MR; ++h)
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const int r = rr + 16 * h, j = 8 * g + cq + q;
          if (r >= live || j >= nc) continue;
          const double x = dig_to_double(X[h][q], s_beta[r] + s_rho[r] + s_c[j] + 1 - 62);
          A[(size_t)(c0 + j) * ld + r0 + row0 + r] = x;
          if (S32 != nullptr) S32[(size_t)(c0 + j) * ld32 + r0 + row0 + r] = (float)x;
          if (S != nullptr) {
            over16 |= fabs(x) > (double)kF16Max;
            S[(size_t)(r0 + row0 + r) * lds + c0 + j] = __double2half(x);
          }
        }
    }
    // the entries that the digits do not cover, from the others of their row: x_j = (b_j - sum_{k<j} x_k l_jk) / l_jj,
    // a row per warp, the terms over its lanes
    __syncthreads();
    for (int r = warp; r < live; r += NT / 32) {
      if (s_nlow[r] == 0) continue;
      double* xr = A + (size_t)c0 * ld + r0 + row0 + r;
      for (int w = 0; w < TM / 2; ++w)
        for (unsigned m = s_low[r][w]; m; m &= m - 1) {
          const int j = 32 * w + __ffs(m) - 1;
          const double* lj = Lm + (size_t)c0 * ldl + c0 + j;
          const double b = Bs[j * ROWS + r], d = lj[(size_t)j * ldl];
          double xk[TM / 2], lk[TM / 2], t = 0.0;             // a row's terms, 32 apart, all in flight at once
#pragma unroll
          for (int u = 0; u < TM / 2; ++u) {
            const int k = lane + 32 * u;
            xk[u] = k < j ? __ldcg(xr + (size_t)k * ld) : 0.0;
            lk[u] = k < j ? lj[(size_t)k * ldl] : 0.0;
          }
          const double rd = 1.0 / d;                          // off the chain
#pragma unroll
          for (int u = 0; u < TM / 2; ++u) t = fma(xk[u], lk[u], t);
#pragma unroll
          for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
          if (lane == 0) {
            const double x = (b - t) * rd;
            xr[(size_t)j * ld] = x;
            if (S32 != nullptr) S32[(size_t)(c0 + j) * ld32 + r0 + row0 + r] = (float)x;
            if (S != nullptr) {
              over16 |= fabs(x) > (double)kF16Max;
              S[(size_t)(r0 + row0 + r) * lds + c0 + j] = __double2half(x);
            }
          }
          __syncwarp();
        }
    }
  } else {
    over16 = substitute<TM, ROWS, NT>(A, ld, r0, m, c0, nc, Lm, ldl, smem, S, lds, S32, ld32);
  }
  if (S != nullptr && __any_sync(0xffffffffu, over16) && lane == 0) atomicOr(err, DEV_ERR_RANGE16);
}

template <int MR, int NT>
cudaError_t launch_refine(double* A, int ld, int r0, int m, int c0, int nc, const double* Lm, int ldl, const float* W,
                          int ldw, __half* S, int lds, float* S32, int ld32, const int* info, unsigned* err,
                          cudaStream_t s) {
  static unsigned long long attr_mask = 0;
  const unsigned long long attr_bit = dev_bit();
  if (!(attr_mask & attr_bit)) {
    cudaError_t e = cudaFuncSetAttribute(trsm_refine64_kernel<MR, NT>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         t64_layout(NT / 4, 16 * MR).total);
    if (e != cudaSuccess) return e;
    attr_mask |= attr_bit;
  }
  (void)launch_pdl(trsm_refine64_kernel<MR, NT>, dim3((m + 16 * MR - 1) / (16 * MR)), dim3(NT),
                   t64_layout(nc, 16 * MR).total, s, A, ld, r0, m, c0, nc, Lm, ldl, W, ldw, S, lds, S32, ld32, info, err);
  return cudaGetLastError();
}

}  // namespace

cudaError_t launch_trsm_refine64(double* A, int ld, int r0, int m, int c0, int nc, const float* W, int ldw,
                                 __half* shadow16, int lds, float* shadow32, int ld32, const int* info, unsigned* err,
                                 cudaStream_t s, const double* Lm, int ldl) {
  if (!Lm) {
    Lm = A;
    ldl = ld;
  }
  if (m <= 0 || nc <= 0) return cudaSuccess;
  if (nc > 128) return cudaErrorInvalidValue;
  // 16 rows per CTA while that fits one wave of SMs, else 32 (every CTA stages and splits all of L);
  // a warp per 8 columns
  const bool wide = (m + 15) / 16 > device_sm_count();
#define HRP_REFINE(MR_, NT_) launch_refine<MR_, NT_>(A, ld, r0, m, c0, nc, Lm, ldl, W, ldw, shadow16, lds, shadow32, ld32, info, err, s)
  if (nc <= 64) return wide ? HRP_REFINE(2, 256) : HRP_REFINE(1, 256);
  return wide ? HRP_REFINE(2, 512) : HRP_REFINE(1, 512);
#undef HRP_REFINE
}

}  // namespace hrp
