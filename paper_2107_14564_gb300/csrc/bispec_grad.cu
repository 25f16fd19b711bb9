// Kernels of the adjoint (gradient) of the estimator with respect to delta(x).
//
// For an upstream gradient g_t = dL/dB_t and c_t = V_c^3 / (V T_t) (Eq. (2.7) with Eq. (2.10)),
// B_t = c_t sum_x d_a d_b d_c is trilinear in the shell fields, so
//   dL/d delta(y) = sum_k [ sum_n S_n(k) K(k) G^_n(k) ] e^{+i k.y},
//   G_n(x) = sum_t g_t c_t sum_{positions of n in t} (product of the other two fields),
// with G^_n the forward DFT of G_n over the grid and K the optional Kaiser factor (Eq. (3.4)).
// G_n is formed on the evaluation grid as a small dense product G[n](x) = sum_p W[p][n] P_p(x)
// over pairs p = (a, b), a >= b, with P_p = d_a d_b and W[p][n] collecting the g_t c_t of every
// bin position whose other two shells are p.
#include <algorithm>

#include "common.cuh"

namespace bsp {
namespace {

constexpr int kAdjThreads = 128;

// VPT neighbouring voxels in one load.
template <int VPT> struct AdjVec;
template <> struct AdjVec<4> {
  using type = float4;
  static __device__ __forceinline__ float at(const float4& v, int j) { return j == 0 ? v.x : j == 1 ? v.y : j == 2 ? v.z : v.w; }
  static __device__ __forceinline__ float4 make(const float* v) { return make_float4(v[0], v[1], v[2], v[3]); }
};
template <> struct AdjVec<2> {
  using type = float2;
  static __device__ __forceinline__ float at(const float2& v, int j) { return j == 0 ? v.x : v.y; }
  static __device__ __forceinline__ float2 make(const float* v) { return make_float2(v[0], v[1]); }
};

// W[e] = sum over the bins listed for entry e of g_t c_t, in list order (deterministic).
__global__ void build_w_kernel(const double* g, const double* cnorm, const int* ptr, const int* idx, int n_entries,
                               float* W) {
  const int e = blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= n_entries) return;
  double s = 0.0;
  for (int i = ptr[e]; i < ptr[e + 1]; ++i) s += g[idx[i]] * cnorm[idx[i]];
  W[e] = (float)s;
}

// G[n][v] = sum_p W[p][n] d_a(v) d_b(v): a thread holds G of VPT neighbouring voxels for all n < 4 NQ in
// registers and walks the pairs; the block's voxels of every field lie in shared memory, a pair's row
// of W comes from L1 (one address a warp) one pair ahead. A pair only reaches the n of its bins, so the
// pairs are listed by the range of quads of n they need (adj_range) and each list's loop leaves out
// the rest, a fifth of the work at 24 shells.
// What bounds it: the FMA pipe (multiply-adds with three register reads reach 67% of its rate) and the
// loads' latency at 12 warps an SM. With 2 voxels a thread, every row of W padded to 32 and read when it
// was needed the adjoint products took 5.06 ms at Ng = 256 and 24 shells, now 2.15. Skipping quads by
// a test per pair instead of by lists cost as much as it saved (2.84 against 2.58 ms), packed
// multiply-adds on rows stored twice more (3.7 ms: twice the loads).
template <int NQ, int VPT>
struct AdjBlock {
  using Vec = typename AdjVec<VPT>::type;
  static constexpr int VB = kAdjThreads * VPT;  // voxels per block pass
  float acc[4 * NQ][VPT];
  // The pairs p0 .. p1 - 1 (an even number), whose n lie in the quads of adj_range(RANGE, NQ).
  template <int RANGE>
  __device__ __forceinline__ void walk(const int2* __restrict__ pairs, const float4* __restrict__ W, int p0, int p1,
                                       const float* fs) {
    constexpr AdjRange r = adj_range(RANGE, NQ);
    constexpr int N = r.q1 - r.q0;
    auto load = [&](int p, int2& ab, float4 (&w)[N]) {
      ab = pairs[p];
#pragma unroll
      for (int q = 0; q < N; ++q) w[q] = __ldg(W + (size_t)p * NQ + r.q0 + q);
    };
    auto add = [&](const int2& ab, const float4 (&w)[N]) {
      const Vec x = *reinterpret_cast<const Vec*>(fs + ab.x * VB);
      const Vec y = *reinterpret_cast<const Vec*>(fs + ab.y * VB);
#pragma unroll
      for (int j = 0; j < VPT; ++j) {
        const float prod = AdjVec<VPT>::at(x, j) * AdjVec<VPT>::at(y, j);
#pragma unroll
        for (int q = 0; q < N; ++q) {
          float(*g)[VPT] = acc + 4 * (r.q0 + q);
          g[0][j] = fmaf(w[q].x, prod, g[0][j]);
          g[1][j] = fmaf(w[q].y, prod, g[1][j]);
          g[2][j] = fmaf(w[q].z, prod, g[2][j]);
          g[3][j] = fmaf(w[q].w, prod, g[3][j]);
        }
      }
    };
    if (p0 >= p1) return;
    int2 ab0, ab1;
    float4 w0[N], w1[N];
    load(p0, ab0, w0);
    for (int p = p0; p < p1; p += 2) {
      load(p + 1, ab1, w1);
      add(ab0, w0);
      load(p + 2 < p1 ? p + 2 : p, ab0, w0);
      add(ab1, w1);
    }
  }
};

template <int NQ, int VPT>
__global__ void __launch_bounds__(kAdjThreads, NQ <= 6 ? 3 : 2) adjoint_products_kernel(
    const float* __restrict__ fields, long long nvox, int ns, const int2* __restrict__ pairs, AdjLists lists,
    const float4* __restrict__ W, float* __restrict__ G) {
  using B = AdjBlock<NQ, VPT>;
  using Vec = typename B::Vec;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  float* fs = reinterpret_cast<float*>(smem_raw) + threadIdx.x * VPT;  // [ns][VB], this thread's voxels
  for (long long base = (long long)blockIdx.x * B::VB; base < nvox; base += (long long)gridDim.x * B::VB) {
    const long long v = base + (long long)threadIdx.x * VPT;
    const bool in = v < nvox;  // nvox is a multiple of VPT
    for (int n = 0; n < ns; ++n)  // each thread reads back what it stored: no barrier
      *reinterpret_cast<Vec*>(fs + n * B::VB) = in ? *reinterpret_cast<const Vec*>(fields + (long long)n * nvox + v) : Vec{};
    B b;
#pragma unroll
    for (int n = 0; n < 4 * NQ; ++n)
#pragma unroll
      for (int j = 0; j < VPT; ++j) b.acc[n][j] = 0.f;
    b.template walk<0>(pairs, W, lists.p[0], lists.p[1], fs);
    b.template walk<1>(pairs, W, lists.p[1], lists.p[2], fs);
    b.template walk<2>(pairs, W, lists.p[2], lists.p[3], fs);
    b.template walk<3>(pairs, W, lists.p[3], lists.p[4], fs);
    b.template walk<4>(pairs, W, lists.p[4], lists.p[5], fs);
    if (in) {
#pragma unroll
      for (int n = 0; n < 4 * NQ; ++n)
        if (n < ns) *reinterpret_cast<Vec*>(G + (long long)n * nvox + v) = AdjVec<VPT>::make(b.acc[n]);
    }
  }
}

template <int NQ, int VPT>
bsp_status launch_adjoint(const float* fields, long long nvox, int ns, const int2* pairs, const AdjLists& lists,
                          const float* W, float* G, int n_sm, cudaStream_t s) {
  constexpr int VB = kAdjThreads * VPT;
  const size_t smem = (size_t)ns * VB * sizeof(float);
  auto kern = adjoint_products_kernel<NQ, VPT>;
  const bsp_status st = allow_shared(kern, (size_t)4 * NQ * VB * sizeof(float));
  if (st != BSP_OK) return st;
  int per_sm = 0;
  BSP_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, kAdjThreads, smem));
  const long long blocks = std::min<long long>((nvox + VB - 1) / VB, (long long)std::max(per_sm, 1) * std::max(n_sm, 1) * 4);
  kern<<<(unsigned)blocks, kAdjThreads, smem, s>>>(fields, nvox, ns, pairs, lists, reinterpret_cast<const float4*>(W), G);
  BSP_CUDA(cudaGetLastError());
  return BSP_OK;
}

}  // namespace

bsp_status launch_build_w(const double* g, const double* cnorm, const int* ptr, const int* idx, int n_entries,
                          float* W, cudaStream_t s) {
  if (n_entries == 0) return BSP_OK;
  build_w_kernel<<<(n_entries + 255) / 256, 256, 0, s>>>(g, cnorm, ptr, idx, n_entries, W);
  BSP_CUDA(cudaGetLastError());
  return BSP_OK;
}

int adjoint_padded_shells(int ns) { return ns <= 32 ? (ns + 7) / 8 * 8 : (ns + 15) / 16 * 16; }

bsp_status launch_adjoint_products(const float* fields, long long nvox, int ns, int np, const int2* pairs,
                                   const AdjLists& lists, const float* W, float* G, int n_sm, cudaStream_t s) {
  if (lists.p[kAdjRanges] == 0) {
    BSP_CUDA(cudaMemsetAsync(G, 0, (size_t)ns * (size_t)nvox * sizeof(float), s));
    return BSP_OK;
  }
  switch (np) {
    case 8: return launch_adjoint<2, 4>(fields, nvox, ns, pairs, lists, W, G, n_sm, s);
    case 16: return launch_adjoint<4, 4>(fields, nvox, ns, pairs, lists, W, G, n_sm, s);
    case 24: return launch_adjoint<6, 4>(fields, nvox, ns, pairs, lists, W, G, n_sm, s);
    case 32: return launch_adjoint<8, 4>(fields, nvox, ns, pairs, lists, W, G, n_sm, s);
    case 48: return launch_adjoint<12, 2>(fields, nvox, ns, pairs, lists, W, G, n_sm, s);
    case 64: return launch_adjoint<16, 2>(fields, nvox, ns, pairs, lists, W, G, n_sm, s);
  }
  return fail_c(BSP_ERR_NOT_SUPPORTED, "gradient: at most 64 shells");
}

}  // namespace bsp
