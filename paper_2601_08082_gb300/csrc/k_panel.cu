// A whole FP32-level TRSM node of Alg. 2 (two to eight diagonal leaves) in one launch.
//
// The recursion alternates leaf TRSMs (X = fl32(B) W^T, W the FP32 inverse of the leaf) with updates
// of the columns to the right, 2 nleaf - 1 launches in a chain of 7 to 9 us each, whatever the size.
// The rows of B are independent, so a row tile can run through the chain on its own: a cluster of 4
// CTAs takes 16 rows, CTA r the columns 32 r .. 32 r + 31 of every leaf, and they exchange the tile's
// rounded right-hand side and its solution, 2 KB a CTA, through distributed shared memory before and
// after each leaf.  Every entry is the same chain of FMAs, in the same order, as in the launches
// it replaces (launch_trsm_leaf32, launch_gemm_simt): a thread holds 4 rows of one column and reads
// per term one word of the operand and one float4 of the tile (a broadcast).  The operands (W or a
// block of L, 128 terms x 32 columns) of the next product are in flight during this one.
// What bounds it: issue and shared-memory reads, two wavefronts for four FMAs per warp, one warp per
// scheduler and CTA; ~0.6 us per 128 terms, and two cluster barriers a leaf.
#include <algorithm>
#include <climits>
#include <type_traits>

#include <cooperative_groups.h>

#include "hrp_internal.cuh"

namespace cg = cooperative_groups;

namespace hrp {
namespace {

constexpr int kTh = 128, kRows = 16, kCol = 32, kRanks = 4;

struct PanelLayout {
  int xs, fb, ys, bd, total;
};
__host__ __device__ inline PanelLayout panel_layout(int nc, int nleaf) {
  PanelLayout l;
  l.xs = 0;                                       // X, [column][16 rows] floats
  l.fb = l.xs + nc * kRows * 4;                   // the leaf's rounded right-hand side, the same
  l.ys = l.fb + 128 * kRows * 4;                  // operands, two buffers [term][32 columns]
  l.bd = l.ys + 2 * 128 * kCol * 4;               // B, [leaf][4 rows][thread] doubles
  l.total = l.bd + nleaf * 4 * kTh * 8;
  return l;
}

// binary64 to binary32, round to nearest even, and back, by integer operations (the conversions run on
// the FP64 pipe, 19 clocks a warp and SM)
__device__ __forceinline__ float to_float(double x) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(x);
  const int F = (int)(b >> 52) & 0x7ff;
  if (F < 897 || F > 1149) return (float)x;       // zero, subnormal or near the ends of binary32
  const unsigned long long v = b & 0x7fffffffffffffffull;
  const unsigned q = (unsigned)(v >> 29) - (896u << 23), rest = (unsigned)v & 0x1fffffffu;
  return __uint_as_float(((unsigned)(b >> 32) & 0x80000000u) | (q + ((rest > 0x10000000u) | ((rest == 0x10000000u) & q & 1u))));
}
__device__ __forceinline__ double to_double(float x) {
  const unsigned b = __float_as_uint(x);
  const unsigned F = (b >> 23) & 0xffu;
  if (F == 0 || F == 0xff) return (double)x;
  return __hiloint2double((int)((b & 0x80000000u) | (((b & 0x7fffffffu) >> 3) + (896u << 20))), (int)(b << 29));
}

// F64: the blocks of L come from the master and are rounded here; else from its FP32 copy L32
template <bool F64>
__global__ void __cluster_dims__(1, kRanks, 1) __launch_bounds__(kTh, F64 ? 2 : 3)
trsm_panel32_kernel(double* __restrict__ A, int ld, int r0, int m, int c0, int nc, const float* __restrict__ W32,
                    const float* __restrict__ L32, int ldl32, __half* __restrict__ S, int lds, float* __restrict__ S32, int ld32,
                    const int* __restrict__ info, unsigned* __restrict__ err, const __grid_constant__ PanelPlan plan) {
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ int s_stop;
  const PanelLayout lay = panel_layout(nc, plan.nleaf);
  float* Xs = reinterpret_cast<float*>(smem + lay.xs);
  float* Fb = reinterpret_cast<float*>(smem + lay.fb);
  float* Ys = reinterpret_cast<float*>(smem + lay.ys);
  double* Bd = reinterpret_cast<double*>(smem + lay.bd);
  cg::cluster_group cluster = cg::this_cluster();
  const int rank = (int)cluster.block_rank();
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  // every CTA of the cluster has started before any writes to another's shared memory
  asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory");
  pdl_wait();
  pdl_trigger();
  const int row0 = blockIdx.x * kRows + 4 * warp;                // this thread's rows row0 .. row0 + 3
  const int live = min(4, m - row0);
  double* Ab = A + (size_t)c0 * ld + r0 + row0;                  // column c of the node at + c ld
  for (int t = 0; t < plan.nleaf; ++t) {
    const int c = kCol * rank + lane;
#pragma unroll
    for (int q = 0; q < 4; ++q)
      Bd[(4 * t + q) * kTh + tid] = (c < plan.sz[t] && q < live) ? __ldcg(Ab + (size_t)(plan.off[t] + c) * ld + q) : 0.0;
  }
  // operand of unit u: terms warp + 4 e of its block, column `lane` of this CTA's slice
  using Reg = typename std::conditional<F64, double, float>::type;
  Reg pre[32];
  auto fetch = [&](int u) {
    const int t = plan.t[u], kl = plan.k[u], c = kCol * rank + lane;
    const bool ok = c < plan.sz[t];
    if (kl == t) {                                               // the leaf's inverse
      const float* w = W32 + (size_t)(c0 + plan.off[t]) * 128 + c;
#pragma unroll
      for (int e = 0; e < 32; ++e) {
        const int k = warp + 4 * e;
        const float v = (ok && k < plan.sz[t]) ? w[(size_t)k * 128] : 0.f;
        if constexpr (F64) pre[e] = __hiloint2double(0, __float_as_int(v));
        else pre[e] = v;
      }
    } else {
      const size_t i = (size_t)c0 + plan.off[t] + c, k0 = (size_t)c0 + plan.off[kl];
#pragma unroll
      for (int e = 0; e < 32; ++e) {
        const int k = warp + 4 * e;
        const bool in = ok && k < plan.sz[kl];
        if constexpr (F64) pre[e] = in ? A[(k0 + k) * ld + i] : 0.0;
        else pre[e] = in ? L32[(k0 + k) * ldl32 + i] : 0.f;
      }
    }
  };
  auto put = [&](int u) {
    float* y = Ys + (u & 1) * 128 * kCol;
    const bool inv = plan.k[u] == plan.t[u];
#pragma unroll
    for (int e = 0; e < 32; ++e) {
      float v;
      if constexpr (F64) v = inv ? __int_as_float(__double2loint(pre[e])) : to_float(pre[e]);
      else v = pre[e];
      y[(warp + 4 * e) * kCol + lane] = v;
    }
  };
  // o += rows of src (columns of 16 rows) times the staged operand
  float o[4];
  auto product = [&](const float* src, int u, int kn) {
    const float* y = Ys + (u & 1) * 128 * kCol + lane;
    const float* x = src + 4 * warp;
#pragma unroll 16
    for (int k = 0; k < kn; ++k) {
      const float b = y[k * kCol];
      const float4 a = *reinterpret_cast<const float4*>(x + k * kRows);
      o[0] = fmaf(a.x, b, o[0]);
      o[1] = fmaf(a.y, b, o[1]);
      o[2] = fmaf(a.z, b, o[2]);
      o[3] = fmaf(a.w, b, o[3]);
    }
  };
  // this thread's four values of column c to [c][16 rows] of every CTA
  auto send = [&](float* dst, int c, float4 v) {
    float4* p = reinterpret_cast<float4*>(dst + c * kRows + 4 * warp);
#pragma unroll
    for (int r = 0; r < kRanks; ++r) *cluster.map_shared_rank(p, r) = v;
  };
  fetch(0);
  asm volatile("barrier.cluster.wait.aligned;" ::: "memory");
  // the cluster stops as one where an earlier leaf has failed
  if (rank == 0 && tid < kRanks) *cluster.map_shared_rank(&s_stop, tid) = *(volatile const int*)info != INT_MAX;
  bool over16 = false;
  for (int u = 0; u < plan.nunit; ++u) {
    const int t = plan.t[u], kl = plan.k[u], c = kCol * rank + lane, n = plan.sz[t];
    put(u);
    if (kl == t) {
      if (c < n) {
        float4 f;
        f.x = to_float(Bd[(4 * t + 0) * kTh + tid]);
        f.y = to_float(Bd[(4 * t + 1) * kTh + tid]);
        f.z = to_float(Bd[(4 * t + 2) * kTh + tid]);
        f.w = to_float(Bd[(4 * t + 3) * kTh + tid]);
        send(Fb, c, f);
      }
      cluster.sync();
      if (u == 0 && s_stop) return;                              // all CTAs: nothing is sent any more
      if (u + 1 < plan.nunit) fetch(u + 1);
      o[0] = o[1] = o[2] = o[3] = 0.f;
      product(Fb, u, n);
      if (c < n) {
        if (u + 1 < plan.nunit) send(Xs, plan.off[t] + c, make_float4(o[0], o[1], o[2], o[3]));
        double* a = Ab + (size_t)(plan.off[t] + c) * ld;
#pragma unroll
        for (int q = 0; q < 4; ++q)
          if (q < live) {
            a[q] = to_double(o[q]);
            if (S32 != nullptr) S32[(size_t)(c0 + plan.off[t] + c) * ld32 + r0 + row0 + q] = o[q];
            if (S != nullptr) {
              over16 |= fabsf(o[q]) > kF16Max;
              S[(size_t)(r0 + row0 + q) * lds + c0 + plan.off[t] + c] = __float2half_rn(o[q]);
            }
          }
      }
      if (u + 1 < plan.nunit) cluster.sync();
    } else {
      __syncthreads();
      if (u + 1 < plan.nunit) fetch(u + 1);
      if (plan.flag[u] & 1) o[0] = o[1] = o[2] = o[3] = 0.f;
      product(Xs + plan.off[kl] * kRows, u, plan.sz[kl]);
      if (plan.flag[u] & 2) {
#pragma unroll
        for (int q = 0; q < 4; ++q) Bd[(4 * t + q) * kTh + tid] -= to_double(o[q]);
      }
    }
  }
  if (S != nullptr && __any_sync(0xffffffffu, over16) && lane == 0) atomicOr(err, DEV_ERR_RANGE16);
}

template <bool F64>
cudaError_t launch_panel(double* A, int ld, int r0, int m, int c0, int nc, const float* W32, __half* S, int lds, float* S32,
                         int ld32, const int* info, unsigned* err, const PanelPlan& plan, cudaStream_t s) {
  static unsigned long long attr_mask = 0;
  const unsigned long long attr_bit = dev_bit();
  if (!(attr_mask & attr_bit)) {
    cudaError_t e = cudaFuncSetAttribute(trsm_panel32_kernel<F64>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         panel_layout(128 * kPanelLeaves, kPanelLeaves).total);
    if (e != cudaSuccess) return e;
    attr_mask |= attr_bit;
  }
  (void)launch_pdl(trsm_panel32_kernel<F64>, dim3((m + kRows - 1) / kRows, kRanks), dim3(kTh),
                   panel_layout(nc, plan.nleaf).total, s, A, ld, r0, m, c0, nc, W32, S32, ld32, S, lds, S32, ld32, info, err,
                   plan);
  return cudaGetLastError();
}

}  // namespace

int panel_max_rows(int nc, int nleaf, bool shadow32) {
  const int per = std::min(shadow32 ? 3 : 2, (227 * 1024) / (panel_layout(nc, nleaf).total + 2048));
  return device_sm_count() * per / kRanks * kRows;
}

cudaError_t launch_trsm_panel32(double* A, int ld, int r0, int m, int c0, int nc, const float* W32, __half* S, int lds,
                                float* S32, int ld32, const int* info, unsigned* err, const PanelPlan& plan, cudaStream_t s) {
  if (m <= 0 || nc <= 0) return cudaSuccess;
  return S32 != nullptr ? launch_panel<false>(A, ld, r0, m, c0, nc, W32, S, lds, S32, ld32, info, err, plan, s)
                        : launch_panel<true>(A, ld, r0, m, c0, nc, W32, S, lds, S32, ld32, info, err, plan, s);
}

}  // namespace hrp
