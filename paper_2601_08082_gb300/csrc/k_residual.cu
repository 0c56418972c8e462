// The residual R = B - A X of the refinement (Sec. 1-2: FP64 residual with the original A), A
// symmetric and read once from its lower triangle, by error-free digit products on the FP16
// tensor pipe (digits.cuh).
//
// What bounded the FP64 FMA kernel this replaces was the FP64 pipe: n^2 nrhs FMAs at 1.7 per clock
// and SM, 29.0 ms at n = 32768 with 16 right-hand sides, where reading A takes 0.63 ms.  The
// digit products run ~20 times faster, and the sums inside a tile are exact: 5.4 ms (hrp_posv at
// n = 32768, 134.9 -> 87.7 ms; n = 4096, 16 right-hand sides, 5.60 -> 4.84 ms).
//
// Scales: e_i = ceil(ex_i / 2) for a_ii < 2^ex_i.  A positive definite A has |a_ij| <=
// sqrt(a_ii a_jj) < 2^(e_i + e_j), so every entry is written in digits against 2^(e_i + e_j + 1),
// whatever the rows' ranges, and one set of digits serves the product with A_IJ (rows of block I)
// and with its transpose (rows of block J).  X enters as 2^(e_j) x_j against the largest of its
// 64-row block and column.  A tile with an entry beyond that bound, a diagonal entry that is not
// positive and normal, or a NaN or infinity in A or X is computed by FP64 FMAs instead (an
// indefinite matrix, a solve that gave up).  So a row's error is about 2^-59 sqrt(a_ii) times its largest
// sqrt(a_jj) |x_j| per block of 64: invariant under scaling A to D A D, and far below what the norms that
// end a refinement see; terms that are small only by a weak a_ij are not followed beyond it.
//
// Launches: a prologue (one CTA per 64-row block: R = B, the e_i, X's digits in the order the mma
// fragments read them, 14 KB per block), then one CTA of 4 warps per 64 x 64 lower tile: 63 KB of
// digits in shared memory, three CTAs per SM so that one CTA's loads and splitting run under
// another's products.  Both products' results are added to R with FP64 atomics.
#include "digits.cuh"
#include "hrp_internal.cuh"

namespace hrp {
namespace {

constexpr int kB = kResBlock;
constexpr int kLd = kB + 8;                       // halves per staged row: 144 bytes, conflict-free ldmatrix
constexpr int kTilePlane = kB * kLd;
constexpr int kThreads = 128;

// largest e with a tile's bound: scale of entry (i, j) is 2^(e_i + e_j + 1)
__device__ __forceinline__ int half_exponent(double d, bool& bad) {
  const long long b = __double_as_longlong(d);
  const int F = (int)(b >> 52);                   // negative for d < 0
  bad = F <= 0 || F >= 0x7ff;
  return bad ? 0 : (F - 1022 + 1) >> 1;
}

// blk: e[64 blk ..], xs[16 blk ..] (biased scales of X's columns), flag[blk], frag[blk]
__global__ void __launch_bounds__(kThreads)
residual_prologue_kernel(const double* __restrict__ A, int lda, const double* __restrict__ X, int ldx,
                         const double* __restrict__ B, int ldb, double* __restrict__ R, int ldr, int n, int nrhs,
                         int* __restrict__ e, int* __restrict__ xs, int* __restrict__ flag, uint2* __restrict__ frag) {
  pdl_wait();
  pdl_trigger();
  __shared__ __align__(16) __half dx[kDig * kResRhs * kLd];
  __shared__ int se[kB], top[kResRhs];
  const int blk = blockIdx.x, R0 = blk * kB, tid = threadIdx.x;
  int bad = 0;
  if (tid < kB) {
    bool b = false;
    const int gi = R0 + tid;
    se[tid] = gi < n ? half_exponent(A[(size_t)gi * lda + gi], b) : 0;
    bad = b;
    e[R0 + tid] = se[tid];
  }
  if (tid < kResRhs) top[tid] = 1;
  __syncthreads();
  // unit (column c, 8 rows): c = tid / 8, rows 8 (tid % 8) ..
  const int c = tid >> 3, r0 = 8 * (tid & 7);
  double v[8];
  int eb[8], mx = 1;
#pragma unroll
  for (int q = 0; q < 8; ++q) {
    const int gi = R0 + r0 + q;
    const bool in = c < nrhs && gi < n;
    v[q] = in ? X[(size_t)c * ldx + gi] : 0.0;
    if (in) R[(size_t)c * ldr + gi] = B[(size_t)c * ldb + gi];
    const int F = dig_field(v[q]);
    bad |= F == 0x7ff;
    if (__double_as_longlong(v[q]) << 1) mx = max(mx, max(F, 1) + se[r0 + q]);
  }
  atomicMax(&top[c], mx);
  bad = __syncthreads_or(bad);
#pragma unroll
  for (int q = 0; q < 8; ++q) eb[q] = (__double_as_longlong(v[q]) << 1) ? top[c] - se[r0 + q] : 1;
  if (!bad) dig_split8(v, eb, dx + (size_t)c * kLd + r0, kResRhs * kLd);
  if (tid < kResRhs) xs[blk * kResRhs + tid] = top[tid];
  if (tid == 0) flag[blk] = bad;
  __syncthreads();
  if (bad) return;
  // fragment order [k step][digit][8 columns][lane]: lane (g, t) holds terms 2t, 2t+1, 2t+8, 2t+9
  // of column g
  uint2* out = frag + (size_t)blk * (kResFragBytes / sizeof(uint2));
  for (int idx = tid; idx < (kB / 16) * kDig * 2 * 32; idx += kThreads) {
    const int lane = idx & 31, h = (idx >> 5) & 1, st = idx >> 6;
    const int t = st % kDig, ks = st / kDig;
    const __half* p = dx + (size_t)t * kResRhs * kLd + (size_t)(8 * h + (lane >> 2)) * kLd + 16 * ks + 2 * (lane & 3);
    out[idx] = make_uint2(*reinterpret_cast<const uint32_t*>(p), *reinterpret_cast<const uint32_t*>(p + 8));
  }
}

__device__ __forceinline__ void tile_of(long long t, int& I, int& J) {
  long long i = (long long)((sqrt(8.0 * (double)t + 1.0) - 1.0) * 0.5);
  while (i * (i + 1) / 2 > t) --i;
  while ((i + 1) * (i + 2) / 2 <= t) ++i;
  I = (int)i;
  J = (int)(t - i * (i + 1) / 2);
}

// NH: groups of 8 right-hand sides (1 or 2)
template <int NH>
__global__ void __launch_bounds__(kThreads, 3)
residual_tile_kernel(const double* __restrict__ A, int lda, const double* __restrict__ X, int ldx,
                     double* __restrict__ R, int ldr, int n, int nrhs, const int* __restrict__ e,
                     const int* __restrict__ xs, const int* __restrict__ flag, const uint2* __restrict__ frag) {
  pdl_wait();
  pdl_trigger();
  extern __shared__ __align__(16) unsigned char smem[];
  __half* dig = reinterpret_cast<__half*>(smem);       // [7][64][kLd], row i, column j
  int I, J;
  tile_of(blockIdx.x, I, J);
  const int I0 = I * kB, J0 = J * kB;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  // entry (i, j) of the tile, mirrored above the diagonal of a diagonal tile
  auto entry = [&](int i, int j) {
    const int gi = I0 + i, gj = J0 + j;
    if (gi >= n || gj >= n) return 0.0;
    return (gi >= gj) ? A[(size_t)gj * lda + gi] : A[(size_t)gi * lda + gj];
  };
  int bad = flag[I] | flag[J];
  {
    // warp w: rows 32 (w % 2) + lane, columns 32 (w / 2) .. + 31 in four units of 8
    const int i = 32 * (warp & 1) + lane;
    const int ei = e[I0 + i];
#pragma unroll
    for (int u = 0; u < 4; u += 2) {
      double v[2][8];
#pragma unroll
      for (int h = 0; h < 2; ++h)
#pragma unroll
        for (int q = 0; q < 8; ++q) v[h][q] = entry(i, 32 * (warp >> 1) + 8 * (u + h) + q);
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int j0 = 32 * (warp >> 1) + 8 * (u + h);
        int eb[8];
#pragma unroll
        for (int q = 0; q < 8; ++q) {
          eb[q] = ei + __ldg(e + J0 + j0 + q) + 1 + 1022;
          bad |= dig_field(v[h][q]) > eb[q];
          eb[q] = max(eb[q], dig_field(v[h][q]));
        }
        dig_split8(v[h], eb, dig + (size_t)i * kLd + j0, kTilePlane);
      }
    }
  }
  if (__syncthreads_or(bad)) {
    // FP64 FMAs, a row of the tile (and of its transpose) per thread and right-hand side
    double (*As)[kB + 1] = reinterpret_cast<double (*)[kB + 1]>(smem);
    for (int idx = tid; idx < kB * kB; idx += kThreads) As[idx % kB][idx / kB] = entry(idx % kB, idx / kB);
    __syncthreads();
    const int i = tid % kB;
    for (int c = tid / kB; c < nrhs; c += kThreads / kB) {
      double y = 0.0, z = 0.0;
      for (int j = 0; j < kB; ++j) {
        if (J0 + j < n) y = fma(As[i][j], X[(size_t)c * ldx + J0 + j], y);
        if (I0 + j < n) z = fma(As[j][i], X[(size_t)c * ldx + I0 + j], z);
      }
      if (I0 + i < n) atomicAdd(R + (size_t)c * ldr + I0 + i, -y);
      if (I != J && J0 + i < n) atomicAdd(R + (size_t)c * ldr + J0 + i, -z);
    }
    return;
  }
#pragma unroll 1
  for (int side = 0; side < 2; ++side) {
    if (side == 1 && I == J) break;
    // side 0: R_I -= A_IJ X_J (rows of the staged digits); side 1: R_J -= A_IJ^T X_I (columns)
    const int kb = side ? I : J, rb = side ? J : I, m0 = 16 * warp;
    const uint2* xf = frag + (size_t)kb * (kResFragBytes / sizeof(uint2)) + lane;
    const __half* ap = side ? dig + (size_t)(((lane >> 4) & 1) * 8 + (lane & 7)) * kLd + m0 + ((lane >> 3) & 1) * 8
                            : dig + (size_t)(m0 + (lane & 15)) * kLd + (lane >> 4) * 8;
    const int astep = side ? 16 * kLd : 16;            // 16 inner terms on
    int iacc[kDig][4 * NH];
#pragma unroll
    for (int g = 0; g < kDig; ++g)
#pragma unroll
      for (int j = 0; j < 4 * NH; ++j) iacc[g][j] = 0;
#pragma unroll 1
    for (int ch = 0; ch < kB / kDigK; ++ch) {
      float acc[kDig][NH][4];
#pragma unroll
      for (int g = 0; g < kDig; ++g)
#pragma unroll
        for (int h = 0; h < NH; ++h)
#pragma unroll
          for (int q = 0; q < 4; ++q) acc[g][h][q] = 0.f;
#pragma unroll
      for (int k2 = 0; k2 < kDigK / 16; ++k2) {
        const int ks = 2 * ch + k2;
        uint2 b[kDig][NH];
#pragma unroll
        for (int t = 0; t < kDig; ++t)
#pragma unroll
          for (int h = 0; h < NH; ++h) b[t][h] = __ldg(xf + ((ks * kDig + t) * 2 + h) * 32);
#pragma unroll
        for (int s = 0; s < kDig; ++s) {
          uint32_t a[4];
          const __half* p = ap + (size_t)s * kTilePlane + ks * astep;
          if (side) dig_ldmatrix_t(a, p);
          else dig_ldmatrix(a, p);
#pragma unroll
          for (int t = 0; t < kDig - s; ++t)
#pragma unroll
            for (int h = 0; h < NH; ++h) dig_mma(acc[s + t][h], a, b[t][h].x, b[t][h].y);
        }
      }
#pragma unroll
      for (int g = 0; g < kDig; ++g)
#pragma unroll
        for (int j = 0; j < 4 * NH; ++j) iacc[g][j] += __float2int_rn(acc[g][j >> 2][j & 3]);
    }
    const int rr = rb * kB + m0 + (lane >> 2);
    const int e0 = e[rr], e1 = e[rr + 8];
#pragma unroll
    for (int j = 0; j < 4 * NH; ++j) {
      const int c = 8 * (j >> 2) + 2 * (lane & 3) + (j & 1), row = rr + 8 * ((j >> 1) & 1);
      if (c >= nrhs || row >= n) continue;
      const int sh = (((j >> 1) & 1) ? e1 : e0) + 1 + xs[kb * kResRhs + c] - 1022 - 34;
      const double v = dig_shift(dig_value(iacc, j), sh);
      if (__double_as_longlong(v) << 1) atomicAdd(R + (size_t)c * ldr + row, -v);
    }
  }
}

}  // namespace

cudaError_t launch_residual(const double* A, int lda, const double* X, int ldx, const double* B, int ldb,
                            double* R, int ldr, int n, int nrhs, void* work, cudaStream_t s) {
  if (n <= 0 || nrhs <= 0) return cudaSuccess;
  const long long nb = (n + kB - 1) / kB;
  uint2* frag = static_cast<uint2*>(work);
  int* e = reinterpret_cast<int*>(static_cast<unsigned char*>(work) + (size_t)nb * kResFragBytes);
  int* xs = e + nb * kB;
  int* flag = xs + nb * kResRhs;
  const int smem = kDig * kTilePlane * (int)sizeof(__half);
  static unsigned long long attr_mask = 0;
  const unsigned long long attr_bit = dev_bit();
  cudaError_t err;
  if (!(attr_mask & attr_bit)) {
    if ((err = cudaFuncSetAttribute(residual_tile_kernel<1>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem)) != cudaSuccess ||
        (err = cudaFuncSetAttribute(residual_tile_kernel<2>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem)) != cudaSuccess)
      return err;
    attr_mask |= attr_bit;
  }
  const dim3 tiles((unsigned)(nb * (nb + 1) / 2));
  for (int c0 = 0; c0 < nrhs; c0 += kResRhs) {
    const int nc = nrhs - c0 < kResRhs ? nrhs - c0 : kResRhs;
    const double* Xc = X + (size_t)c0 * ldx;
    double* Rc = R + (size_t)c0 * ldr;
    (void)launch_pdl(residual_prologue_kernel, dim3((unsigned)nb), dim3(kThreads), 0, s, A, lda, Xc, ldx,
                     B + (size_t)c0 * ldb, ldb, Rc, ldr, n, nc, e, xs, flag, frag);
    if ((err = cudaGetLastError()) != cudaSuccess) return err;
    if (nc <= 8)
      (void)launch_pdl(residual_tile_kernel<1>, tiles, dim3(kThreads), smem, s, A, lda, Xc, ldx, Rc, ldr, n, nc, e, xs,
                       flag, frag);
    else
      (void)launch_pdl(residual_tile_kernel<2>, tiles, dim3(kThreads), smem, s, A, lda, Xc, ldx, Rc, ldr, n, nc, e, xs,
                       flag, frag);
    if ((err = cudaGetLastError()) != cudaSuccess) return err;
  }
  return cudaSuccess;
}

}  // namespace hrp
