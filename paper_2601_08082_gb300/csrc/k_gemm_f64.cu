// FP64 GEMM C -= X Y^T of the FP64 levels (the updates of Alg. 2 and 3) by error-free digit
// products on the FP16 tensor pipe (digits.cuh), one launch for one block or for a list of
// independent blocks.
//
// One CTA of 4 warps computes one 32 x 32 tile (a warp 16 x 16).  Per chunk of 32 inner terms the
// CTA loads its 64 operand rows from the master (coalesced along rows), takes the rows' largest
// exponents, writes the digits and magnitudes to shared memory (41 KB) and multiplies them; the next chunk's
// loads are in flight during the products.  What bounds it: 56 mma per warp and 16 terms (8 clocks
// each per sub-partition) against ~45 integer instructions per entry of splitting; two or three
// CTAs per SM overlap the two.  The small tile is for the small products this library runs in
// FP64 (orders 64 to 1024): a 64 x 64 tile would leave most SMs idle.
//
// Measured against the FP64 SIMT kernel it replaces (32 x 32 tiles, FP64 FMAs): the 32 diagonal
// blocks of 125 x 125 x 1024 of a SYRK 10.3 ms one after another -> one launch, the whole SYRK
// (n = 4000, k = 1024, three levels) 10.40 -> 0.457 ms; the n = 1024 FP64 factorization and solve
// 2.58 -> 1.96 ms.  Relative error against extended precision 5e-17 .. 7e-17, where the FMA
// chains had 1.2e-16 (k = 16) .. 8.5e-16 (k = 1000).
//
// A row's scale carries a bit of headroom over its largest entry so far.  When a later chunk
// holds a larger entry still, the CTA moves its integer sums to FP64 first (at the old scales)
// and goes on with the new ones.  A tile whose operand rows hold a NaN or an infinity is computed
// by plain FP64 FMAs instead, so that those propagate as they would there.
//
// Outputs that the digits do not cover.  A term is held to 2^-59.7 of the product of the two rows'
// scales; where sum |x| |y| (estimated beside the digit products, two mma per warp and 16 terms)
// is below 2^-8 of that product, the output is computed by FP64 FMAs, by the warp's lanes together for up to
// four lanes' outputs, else for the warp's whole part.  The rest is then within k 2^-51.7 sum |x| |y| at
// worst, and a few 2^-53 sum |x| |y| for ordinary digits.  The line: factors of dominant matrices stay
// 2^4 above it and those of kernel matrices 2^0 to 2^3; one bit of headroom instead of two (and 2^-10)
// costs no time.  OPs 1 and 2 take 2^-14: their triangle's rows are mostly their diagonal entry, and one
// output in 100 of an ordinary factor is below 2^-10, one in 10^4 below 2^-14, where ordinary digits
// still leave 2^-46 (the sweeps' double-float products 2^-44).  The estimate costs 2 to 2.5 % (the SYRK 424 -> 435 us, n = 1024 1434 -> 1463).
#include "digits.cuh"
#include "hrp_internal.cuh"

namespace hrp {
namespace {

constexpr int kT = 32;                         // tile edge
constexpr int kThreads = 128;
constexpr int kPlane = kT * kDigLd;            // halves per digit plane of one operand
constexpr int kSpecial = 1 << 20;              // OPs 1 and 2: the exponent of a NaN or an infinity
constexpr float kCovered = 0x1p-8f;            // smallest sum |x| |y| against the scales that the digits cover
constexpr float kCoveredInv = 0x1p-14f;        // the same in OPs 1 and 2
constexpr int kManyLow = 4;                    // lanes with uncovered outputs above which the warp computes all by FMAs
constexpr int kFlush = 64;                     // chunks the 32-bit sums hold (2^24 each) before a move to FP64

// OP 0: C -= X Y^T.  OP 1: C = X Y^T with term kk of X's row r zero for kk < r.  OP 2: C = -X Y^T with Y
// given by rows (term kk of row r at Y[r ldy + kk]), zero for kk > r.  OPs 1 and 2 (the doubling of
// triangular inverses, launch_solve_inverses) skip the chunks of 32 terms that are all zero.  They
// also scale term kk, X's entries by 2^t and Y's by 2^-t, by the largest entry of the term in the tile's
// rows of the operand that is no triangle (Y in OP 1, X in OP 2): rows then keep their digits whatever
// powers of two scale the rows or the columns of the triangle that is inverted.
template <int OP, class List>
__global__ void __launch_bounds__(kThreads, 2)
gemm_f64_digits_kernel(double* __restrict__ C, int ldc, const double* __restrict__ X, int ldx,
                       const double* __restrict__ Y, int ldy, int k, const __grid_constant__ List bl) {
  pdl_wait();
  pdl_trigger();
  constexpr int kOperand = (kDig + 1) * kPlane;                  // halves of one operand
  extern __shared__ __align__(16) __half dig[];                  // [2 operands][7 digits, magnitude][32][kDigLd]
  __shared__ int rowmax[2][2 * kT];                              // largest exponent field of the chunk, by parity
  __shared__ int scale[2 * kT];                                  // the rows' scales (biased exponent)
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;

  // this CTA's block and tile
  int b = 0;
  while (b + 1 < bl.count && (int)blockIdx.x >= bl.b[b + 1].tile0) ++b;
  const auto blk = bl.b[b];
  const int ti = (int)blockIdx.x - blk.tile0;
  int ty, tx;
  const double* Xb;
  const double* Yb;
  double* Cb;
  int lower = 0;
  if constexpr (OP == 0) {
    gemm_block_tile(blk, kT, ti, tx, ty);
    lower = blk.lower;
    Xb = X + blk.xr;
    Yb = Y + blk.yr;
    Cb = C + (size_t)blk.yr * ldc + blk.xr;
  } else {
    const int gm = (blk.m + kT - 1) / kT;
    ty = ti / gm;
    tx = ti - ty * gm;
    k = blk.k;
    Xb = X + blk.xo;
    Yb = Y + blk.yo;
    Cb = C + blk.co;
  }
  const int m0 = tx * kT, n0 = ty * kT, m = blk.m, n = blk.n;

  if (tid < 2 * kT) {
    rowmax[0][tid] = rowmax[1][tid] = 0;
    scale[tid] = 0;
  }
  // warp w holds inner terms 8 w .. 8 w + 7 of the chunk, lane = operand row
  const bool okx = m0 + lane < m, oky = n0 + lane < n;
  double px[8], py[8];
  auto fetch = [&](int k0) {
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      const int kk = k0 + 8 * warp + q;
      px[q] = (okx && kk < k) ? Xb[(size_t)kk * ldx + m0 + lane] : 0.0;
      if (OP == 2) py[q] = (oky && kk < k) ? Yb[(size_t)(n0 + lane) * ldy + kk] : 0.0;
      else py[q] = (oky && kk < k) ? Yb[(size_t)kk * ldy + n0 + lane] : 0.0;
    }
  };
  int iacc[kDig][8];
  float est[2][4] = {};                                          // sum |x| |y| against the scales
  double vacc[8];
#pragma unroll
  for (int j = 0; j < 8; ++j) {
    vacc[j] = 0.0;
#pragma unroll
    for (int g = 0; g < kDig; ++g) iacc[g][j] = 0;
  }
  // the warp's 16 x 16 part: rows 16 (warp / 2), columns 16 (warp % 2); register j of a lane is
  // row g + 8 ((j >> 1) & 1), column 8 (j >> 2) + 2 t + (j & 1), g = lane / 4, t = lane % 4
  const int a0 = 16 * (warp >> 1), b0 = 16 * (warp & 1);
  const int gr = a0 + (lane >> 2), gc = b0 + 2 * (lane & 3);
  auto flush = [&]() {
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      double f0, f1;
      dig_scale(scale[gr + 8 * ((j >> 1) & 1)], scale[kT + gc + 8 * (j >> 2) + (j & 1)], f0, f1);
      vacc[j] += dig_value(iacc, j) * f0 * f1;
#pragma unroll
      for (int g = 0; g < kDig; ++g) iacc[g][j] = 0;
    }
  };
  bool flushed = false, special = false;
  int held = 0;
  const int c0 = OP == 1 ? m0 / kDigK : 0;
  const int nchunk = OP == 2 ? (min(k, n0 + kT) + kDigK - 1) / kDigK : (k + kDigK - 1) / kDigK;
  fetch(c0 * kDigK);
  __syncthreads();
  for (int c = c0; c < nchunk; ++c) {
    int fx = 0, fy = 0, tk[8];
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      const int gx = dig_field(px[q]), gy = dig_field(py[q]);
      if constexpr (OP == 0) {
        fx = max(fx, gx);
        fy = max(fy, gy);
      } else {
        const int g = (int)__reduce_max_sync(0xffffffffu, (unsigned)(OP == 1 ? gy : gx));
        tk[q] = g == 0 ? -4096 : g - 1023;                       // a term that is zero throughout: negligible
        if (OP == 2) tk[q] = -tk[q];
        fx = max(fx, gx == 0x7ff ? kSpecial : (gx == 0 ? 0 : gx + tk[q]));
        fy = max(fy, gy == 0x7ff ? kSpecial : (gy == 0 ? 0 : gy - tk[q]));
      }
    }
    atomicMax(&rowmax[c & 1][lane], fx);
    atomicMax(&rowmax[c & 1][kT + lane], fy);
    __syncthreads();                                             // also: the last chunk's products are done
    int need = 0, mx = 0;
    if (tid < 2 * kT) {
      mx = rowmax[c & 1][tid];
      rowmax[(c + 1) & 1][tid] = 0;
      need = mx == (OP == 0 ? 0x7ff : kSpecial) ? 2 : (max(mx, 1) > scale[tid] ? 1 : 0);
    }
    const bool grow = __syncthreads_or(need) != 0;
    if (grow && __syncthreads_or(need == 2)) {
      special = true;
      break;
    }
    if (grow || held == kFlush) {
      if (held > 0) {
        flush();
        flushed = true;
        held = 0;
      }
      int old[2][2][2];                                          // [row half][column half][column]
#pragma unroll
      for (int j = 0; j < 8; ++j) old[(j >> 1) & 1][j >> 2][j & 1] = scale[gr + 8 * ((j >> 1) & 1)] + scale[kT + gc + 8 * (j >> 2) + (j & 1)];
      __syncthreads();
      if (need) scale[tid] = max(mx, 1) + kDigHead;
      __syncthreads();
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        const int d = old[(j >> 1) & 1][j >> 2][j & 1] - scale[gr + 8 * ((j >> 1) & 1)] - scale[kT + gc + 8 * (j >> 2) + (j & 1)];
        float& t = est[j >> 2][j & 3];
        if (t > 0.f) t = fmaxf(t * __int_as_float((max(d, -126) + 127) << 23), 0x1p-126f);        // zero means none
      }
    }
    {
      int ex[8], ey[8];
#pragma unroll
      for (int q = 0; q < 8; ++q) {
        ex[q] = scale[lane] - (OP == 0 ? 0 : tk[q]);
        ey[q] = scale[kT + lane] + (OP == 0 ? 0 : tk[q]);
      }
      __half* dx = dig + lane * kDigLd + 8 * warp;
      dig_split8(px, ex, dx, kPlane);
      dig_split8(py, ey, dx + kOperand, kPlane);
      dig_abs8(px, ex, dx + kDig * kPlane);
      dig_abs8(py, ey, dx + kOperand + kDig * kPlane);
    }
    if (c + 1 < nchunk) fetch((c + 1) * kDigK);
    __syncthreads();
    dig_chunk(dig, kPlane, a0, dig + kOperand, kPlane, b0, iacc, est);
    ++held;
  }
  // outputs whose terms are all too far below the scales of their row and column
  unsigned low = 0;
  if (!special) {
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      const int r = m0 + gr + 8 * ((j >> 1) & 1), cl = n0 + gc + 8 * (j >> 2) + (j & 1);
      const float t = est[j >> 2][j & 3];
      if (r < m && cl < n && !(lower && r < cl) && t > 0.f && t < (OP == 0 ? kCovered : kCoveredInv)) low |= 1u << j;
    }
    special = __popc(__ballot_sync(0xffffffffu, low != 0)) > kManyLow;       // this warp's part
  }
  auto yv = [&](int cl, int kk) { return OP == 2 ? Yb[(size_t)cl * ldy + kk] : Yb[(size_t)kk * ldy + cl]; };
  auto store = [&](int r, int cl, double s) {
    double* p = Cb + (size_t)cl * ldc + r;
    if (OP == 0) *p -= s;
    else *p = OP == 1 ? s : -s;
  };
  if (special) {
    double s[8] = {};
    for (int kk = 0; kk < k; ++kk) {
      double x[2], y[4];
#pragma unroll
      for (int h = 0; h < 2; ++h) x[h] = Xb[(size_t)kk * ldx + min(m0 + gr + 8 * h, m - 1)];
#pragma unroll
      for (int h = 0; h < 4; ++h) y[h] = yv(min(n0 + gc + 8 * (h >> 1) + (h & 1), n - 1), kk);
#pragma unroll
      for (int j = 0; j < 8; ++j) s[j] = fma(x[(j >> 1) & 1], y[2 * (j >> 2) + (j & 1)], s[j]);
    }
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      const int r = m0 + gr + 8 * ((j >> 1) & 1), cl = n0 + gc + 8 * (j >> 2) + (j & 1);
      if (r < m && cl < n && !(lower && r < cl)) store(r, cl, s[j]);
    }
    return;
  }
  if (__any_sync(0xffffffffu, low != 0)) {
    // a few: FP64 FMAs by the whole warp, the terms over its lanes
#pragma unroll 1
    for (int j = 0; j < 8; ++j)
      for (unsigned who = __ballot_sync(0xffffffffu, (low >> j) & 1); who; who &= who - 1) {
        const int src = __ffs(who) - 1;
        const int r = m0 + a0 + (src >> 2) + 8 * ((j >> 1) & 1), cl = n0 + b0 + 2 * (src & 3) + 8 * (j >> 2) + (j & 1);
        double s = 0.0;
        for (int kk = lane; kk < k; kk += 32) s = fma(Xb[(size_t)kk * ldx + r], yv(cl, kk), s);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        if (lane == 0) store(r, cl, s);
      }
  }
  double cv[8];
#pragma unroll
  for (int j = 0; j < 8; ++j) {
    const int r = m0 + gr + 8 * ((j >> 1) & 1), cl = n0 + gc + 8 * (j >> 2) + (j & 1);
    cv[j] = (OP == 0 && r < m && cl < n && !(lower && r < cl) && !((low >> j) & 1)) ? Cb[(size_t)cl * ldc + r] : 0.0;
  }
#pragma unroll
  for (int j = 0; j < 8; ++j) {
    const int rr = gr + 8 * ((j >> 1) & 1), cc = gc + 8 * (j >> 2) + (j & 1);
    const int r = m0 + rr, cl = n0 + cc;
    if (r >= m || cl >= n || (lower && r < cl) || ((low >> j) & 1)) continue;
    double f0, f1;
    dig_scale(scale[rr], scale[kT + cc], f0, f1);
    double v = dig_value(iacc, j);
    if (f1 != 1.0) v *= f1;
    double* p = Cb + (size_t)cl * ldc + r;
    if (OP == 0) {
      if (flushed) *p = cv[j] - fma(v, f0, vacc[j]);
      else *p = fma(-v, f0, cv[j]);
    } else {
      const double x = flushed ? fma(v, f0, vacc[j]) : v * f0;
      *p = OP == 1 ? x : -x;
    }
  }
}

}  // namespace

constexpr int kSmem = 2 * (kDig + 1) * kPlane * (int)sizeof(__half);

cudaError_t launch_gemm_f64_blocks(double* C, int ldc, const double* X, int ldx, const double* Y, int ldy, int k,
                                   GemmBlocks& bl, cudaStream_t s) {
  if (k <= 0 || bl.count <= 0) return cudaSuccess;
  const int tiles = gemm_block_offsets(bl, kT);
  if (tiles <= 0) return cudaSuccess;
  (void)launch_pdl(gemm_f64_digits_kernel<0, GemmBlocks>, dim3(tiles), dim3(kThreads), kSmem, s, C, ldc, X, ldx, Y, ldy,
                   k, bl);
  return cudaGetLastError();
}

cudaError_t launch_gemm_f64_products(double* C, int ldc, const double* X, int ldx, const double* Y, int ldy, bool neg_rows,
                                     GemmProducts& bl, cudaStream_t s) {
  int tiles = 0;
  for (int i = 0; i < bl.count; ++i) {
    bl.b[i].tile0 = tiles;
    tiles += ((bl.b[i].m + kT - 1) / kT) * ((bl.b[i].n + kT - 1) / kT);
  }
  if (tiles <= 0) return cudaSuccess;
  if (neg_rows)
    (void)launch_pdl(gemm_f64_digits_kernel<2, GemmProducts>, dim3(tiles), dim3(kThreads), kSmem, s, C, ldc, X, ldx, Y, ldy,
                     0, bl);
  else
    (void)launch_pdl(gemm_f64_digits_kernel<1, GemmProducts>, dim3(tiles), dim3(kThreads), kSmem, s, C, ldc, X, ldx, Y, ldy,
                     0, bl);
  return cudaGetLastError();
}

}  // namespace hrp
