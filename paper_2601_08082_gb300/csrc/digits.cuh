// FP64 products on the FP16 tensor pipe, by error-free splitting (Ozaki, Ogita, Oishi and Rump,
// "Error-free transformations of matrix multiplication by using fast routines of matrix
// multiplication", 2012).
//
// This GPU's FP64 pipe retires about 1.7 lane-FMAs per clock and SM (1.2 TFLOP/s in all), its
// FP16 mma.sync pipe 1019 (measured), so 28 FP16 products per FP64 product are still ~21 times
// faster.  Every operand entry of a row is written against the row's scale 2^E (|x| < 2^E) as
//   x = 2^E sum_{s=0..6} d_s 2^(-8 - 9 s),   d_s an integer in [-256, 256],
// which keeps 62 fractional bits below the row's scale (all 53 of x when x is within 2^-9 of
// it).  The digit products d_s d_t are integers of at most 2^16; those of one weight s + t = g
// <= 6 are summed by the tensor cores in FP32, exactly: at most 7 pairs x 32 terms x 2^16 < 2^24
// per chunk of 32 inner terms (checked against 64-bit integers on the device for the largest
// magnitudes).  Chunk sums are then carried in 32-bit integers.  Per term, the dropped pairs (six of
// weight 7: 2^-60.4) and the digits' tails (2^-62 each) are below 2^-59.7 of the two scales' product.
//
// A scale is shared by the terms of a row, and the error is relative to it: FP64 sums give every term its
// own exponent, a digit product does not.  An output whose terms are all far below its row's scale times
// its column's (rows or columns in different units) would lose the digits that matter, so the kernels
// also sum bfloat16 magnitudes (dig_abs), an estimate of sum |x| |y| against the same scales, and
// compute by FP64 FMAs the outputs where it is too small.
#pragma once
#include <stdint.h>

#include <cuda_fp16.h>

namespace hrp {

constexpr int kDig = 7;        // digits per operand, and weights s + t = 0 .. 6 kept
constexpr int kDigK = 32;      // inner terms per chunk (exactness bound above)
constexpr int kDigLd = 40;     // halves per staged row of 32: 80 bytes, conflict-free for ldmatrix
constexpr int kDigHead = 1;    // bits of headroom of a row's scale over its largest entry so far

__device__ __forceinline__ int dig_field(double x) {         // biased exponent field
  return (int)((unsigned long long)__double_as_longlong(x) >> 52) & 0x7ff;
}

// x in units of 2^(E - 62), E = eb - 1022 (the fixed point the digits are cut from), |x| < 2^E; bits
// below the unit are dropped.  x finite.  The significand is placed at the top once and only ever
// shifted right (its exponent field is at most eb; zero may have any eb), the sign applied by xor and
// carry.
__device__ __forceinline__ long long dig_fix(double x, int eb) {
  const uint32_t h = (uint32_t)__double2hiint(x), l = (uint32_t)__double2loint(x);
  const int F = (int)(h >> 20) & 0x7ff;
  const uint32_t mh = (h & 0xfffffu) | ((uint32_t)min(F, 1) << 20);
  const unsigned long long m = ((unsigned long long)__funnelshift_l(l, mh, 9) << 32) | (l << 9);
  const unsigned long long v = m >> min((unsigned)(eb - max(F, 1)), 63u);
  const long long s = (long long)(int)h >> 63;                 // 0 or -1
  return (long long)(v ^ (unsigned long long)s) - s;
}
// the s-th digits of two fixed-point values as a pair of halves.  M must already hold kDigBias
// (256 at every digit position), which makes the digits come out unsigned, u = d + 256.
constexpr unsigned long long kDigBias = 0x4020100804020100ull;
__device__ __forceinline__ uint32_t dig_pair(unsigned long long M0, unsigned long long M1, int s) {
  const int o = 54 - 9 * s;
  uint32_t u0 = (uint32_t)(M0 >> o), u1 = (uint32_t)(M1 >> o);
  if (s > 0) {
    u0 &= 511u;
    u1 &= 511u;
  }
  // 0x6400 | u is the half 1024 + u (u <= 512); subtracting 1280 leaves d exactly
  const uint32_t h = 0x64006400u | u0 | (u1 << 16);
  const __half2 d = __hsub2(*reinterpret_cast<const __half2*>(&h), __half2half2(__ushort_as_half(0x6500)));
  return *reinterpret_cast<const uint32_t*>(&d);
}

// The 7 digits of 8 consecutive inner terms v[0..7] of one row, eb[i] = the scale of v[i] as a
// biased exponent (field(v[i]) <= eb[i]; E = eb - 1022), to dst[s * plane .. + 8) halves (16-byte
// stores).  Entries are finite.
__device__ __forceinline__ void dig_split8(const double (&v)[8], const int (&eb)[8], __half* dst, int plane) {
  uint32_t w[kDig][4];
#pragma unroll
  for (int p = 0; p < 4; ++p) {
    const unsigned long long M0 = (unsigned long long)dig_fix(v[2 * p], eb[2 * p]) + kDigBias;
    const unsigned long long M1 = (unsigned long long)dig_fix(v[2 * p + 1], eb[2 * p + 1]) + kDigBias;
#pragma unroll
    for (int s = 0; s < kDig; ++s) w[s][p] = dig_pair(M0, M1, s);
  }
#pragma unroll
  for (int s = 0; s < kDig; ++s)
    *reinterpret_cast<uint4*>(dst + (size_t)s * plane) = make_uint4(w[s][0], w[s][1], w[s][2], w[s][3]);
}

// the same with one scale for all 8
__device__ __forceinline__ void dig_split8(const double (&v)[8], int eb, __half* dst, int plane) {
  const int e[8] = {eb, eb, eb, eb, eb, eb, eb, eb};
  dig_split8(v, e, dst, plane);
}

// |x| against the same scale as a bfloat16, truncated, not below 2^-60 unless x is zero: the operands
// of the estimate of sum |x| |y| that tells which outputs the digits cover.  A sum of such products
// is zero only where every product is.
constexpr int kAbsMin = (127 - 60) << 7;
__device__ __forceinline__ uint32_t dig_abs(double x, int eb) {
  const uint32_t h = (uint32_t)__double2hiint(x) & 0x7fffffffu;
  const int b = max((int)(h >> 13) + ((126 - eb) << 7), kAbsMin);
  return (h | (uint32_t)__double2loint(x)) ? (uint32_t)b : 0u;
}
__device__ __forceinline__ void dig_abs8(const double (&v)[8], const int (&eb)[8], __half* dst) {
  uint32_t w[4];
#pragma unroll
  for (int p = 0; p < 4; ++p) w[p] = dig_abs(v[2 * p], eb[2 * p]) | (dig_abs(v[2 * p + 1], eb[2 * p + 1]) << 16);
  *reinterpret_cast<uint4*>(dst) = make_uint4(w[0], w[1], w[2], w[3]);
}

__device__ __forceinline__ void dig_ldmatrix(uint32_t (&r)[4], const __half* p) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"((uint32_t)__cvta_generic_to_shared(p))
               : "memory");
}
__device__ __forceinline__ void dig_ldmatrix_t(uint32_t (&r)[4], const __half* p) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"((uint32_t)__cvta_generic_to_shared(p))
               : "memory");
}
__device__ __forceinline__ void dig_mma(float (&d)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

__device__ __forceinline__ void dig_mma_bf16(float (&d)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// One chunk of a warp's 16 x 16 output: rows a0 .. a0 + 15 of the staged digits A ([s][row][k],
// `aplane` halves per digit), columns = rows b0 .. b0 + 15 of B.  The weights' sums over the
// chunk are added to iacc[g][j], j = 4 (column half) + the mma accumulator's register, and those of
// the bfloat16 magnitudes (plane kDig of both operands) to est.
__device__ __forceinline__ void dig_chunk(const __half* A, int aplane, int a0, const __half* B, int bplane, int b0,
                                          int (&iacc)[kDig][8], float (&est)[2][4]) {
  const int lane = threadIdx.x & 31;
  float acc[kDig][2][4];
#pragma unroll
  for (int g = 0; g < kDig; ++g)
#pragma unroll
    for (int h = 0; h < 2; ++h)
#pragma unroll
      for (int q = 0; q < 4; ++q) acc[g][h][q] = 0.f;
  // ldmatrix addresses: A tiles (rows 0-7, k 0-7), (8-15, 0-7), (0-7, 8-15), (8-15, 8-15);
  // B tiles (columns 0-7, k 0-7), (0-7, 8-15), (8-15, 0-7), (8-15, 8-15)
  const __half* ap = A + (size_t)(a0 + (lane & 15)) * kDigLd + (lane >> 4) * 8;
  const __half* bp = B + (size_t)(b0 + (lane & 7) + ((lane >> 4) << 3)) * kDigLd + ((lane >> 3) & 1) * 8;
#pragma unroll
  for (int ks = 0; ks < kDigK; ks += 16) {
    {
      uint32_t a[4], e[4];
      dig_ldmatrix(a, ap + (size_t)kDig * aplane + ks);
      dig_ldmatrix(e, bp + (size_t)kDig * bplane + ks);
      dig_mma_bf16(est[0], a, e[0], e[1]);
      dig_mma_bf16(est[1], a, e[2], e[3]);
    }
    uint32_t b[kDig][4];
#pragma unroll
    for (int t = 0; t < kDig; ++t) dig_ldmatrix(b[t], bp + (size_t)t * bplane + ks);
#pragma unroll
    for (int s = 0; s < kDig; ++s) {
      uint32_t a[4];
      dig_ldmatrix(a, ap + (size_t)s * aplane + ks);
#pragma unroll
      for (int t = 0; t < kDig - s; ++t) {
        dig_mma(acc[s + t][0], a, b[t][0], b[t][1]);
        dig_mma(acc[s + t][1], a, b[t][2], b[t][3]);
      }
    }
  }
#pragma unroll
  for (int g = 0; g < kDig; ++g)
#pragma unroll
    for (int j = 0; j < 8; ++j) iacc[g][j] += __float2int_rn(acc[g][j >> 2][j & 3]);
}

// The product sum of one output in units of 2^(Ex + Ey - 34): weights g = 0 .. 2 and 3 .. 6 are
// joined in 64-bit integers and converted by the 1.5 2^52 offset (two FP64 additions; the
// conversion instructions run on the FP64 pipe too).  Up to 2^15 inner terms.
template <int NJ>
__device__ __forceinline__ double dig_value(const int (&iacc)[kDig][NJ], int j) {
  const long long hi = ((long long)iacc[0][j] << 18) + ((long long)iacc[1][j] << 9) + (long long)iacc[2][j];
  const long long lo = ((long long)iacc[3][j] << 27) + ((long long)iacc[4][j] << 18) +
                       ((long long)iacc[5][j] << 9) + (long long)iacc[6][j];      // units 2^-36 of hi's
  constexpr long long kMagic = 0x4338000000000000ll;                               // 1.5 2^52
  const double hm = __longlong_as_double(kMagic + hi);
  const double lm = __longlong_as_double(kMagic + ((lo + 128) >> 8));              // units 2^-28
  // hm - 1.5 2^52 - 1.5 2^24 is exact; the FMA adds lm 2^-28 = 1.5 2^24 + lo 2^-36
  return fma(lm, 0x1p-28, hm - (0x1.8p52 + 0x1.8p24));
}
// 2^(Ex + Ey - 34) for biased row scales ebx, eby, as two factors (their product may leave the
// normal range on its own)
__device__ __forceinline__ void dig_scale(int ebx, int eby, double& f0, double& f1) {
  const int e = ebx + eby - 2 * 1022 - 34;
  const int e0 = max(-1022, min(1023, e));
  const int e1 = max(-1022, min(1023, e - e0));
  f0 = __longlong_as_double((long long)(e0 + 1023) << 52);
  f1 = __longlong_as_double((long long)(e1 + 1023) << 52);
}

// a fixed-point value M 2^u (|M| < 2^63) as the nearest double, by integer operations; results
// outside the normal range go through ldexp
__device__ __forceinline__ double dig_to_double(long long M, int u) {
  if (M == 0) return 0.0;
  const unsigned long long sgn = (unsigned long long)M & 0x8000000000000000ull;
  unsigned long long a = (unsigned long long)(M < 0 ? -M : M);
  const int z = __clzll((long long)a);                        // a 2^z in [2^63, 2^64)
  a <<= z;
  // leading 53 bits, rounded to nearest even at the 11 below
  unsigned long long q = a >> 11;
  const unsigned rest = (unsigned)a & 0x7ffu;
  q += (rest > 0x400u) | ((rest == 0x400u) & (unsigned)(q & 1));
  const int e = 63 - z + u;                                   // value in [2^e, 2^(e+1)) (2^(e+1) after a carry)
  if (e >= -1021 && e <= 1021)
    return __longlong_as_double((long long)(sgn | (((unsigned long long)(e + 1022) << 52) + q)));
  return ldexp(sgn ? -(double)q : (double)q, e - 52);
}

// Digits of 8 bits: byte s of a fixed-point value with kByteBias (128 at every byte) added is d + 128,
// weight 2^(8 (7 - s)); a pair of digits takes a byte permutation, a mask and a subtraction, less
// than half of the 9-bit ones, for kernels where every value is split once per use.  Eight digits,
// weights s + t <= 7 kept (36 products); a product of 128 terms sums to at most 8 x 128 x 2^14 = 2^24
// per weight, exact in binary32 without intermediate moves.
constexpr int kByteDig = 8;
constexpr unsigned long long kByteBias = 0x8080808080808080ull;
// digits s of M0 and M1 as a pair of halves
__device__ __forceinline__ uint32_t byte_pair(unsigned long long M0, unsigned long long M1, int s) {
  const int byte = 7 - s;                // from the low end
  const uint32_t w0 = byte >= 4 ? (uint32_t)(M0 >> 32) : (uint32_t)M0, w1 = byte >= 4 ? (uint32_t)(M1 >> 32) : (uint32_t)M1;
  const uint32_t b = byte & 3;
  const uint32_t x = (__byte_perm(w0, w1, b | (b << 4) | ((4 + b) << 8) | ((4 + b) << 12)) & 0x00ff00ffu) | 0x64006400u;
  const __half2 d = __hsub2(*reinterpret_cast<const __half2*>(&x), __half2half2(__ushort_as_half(0x6480)));   // 1152
  return *reinterpret_cast<const uint32_t*>(&d);
}

// v 2^e by integer addition to the exponent (the FP64 pipe is the slow one); exact unless the
// result leaves the normal range, where ldexp rounds it
__device__ __forceinline__ double dig_shift(double v, int e) {
  const long long b = __double_as_longlong(v);
  const int F = (int)(b >> 52) & 0x7ff;
  if (F == 0) return v;                          // a sum of digits: zero, never subnormal
  if (F + e >= 1 && F + e <= 2046) return __longlong_as_double(b + ((long long)e << 52));
  return ldexp(v, e);
}

}  // namespace hrp
