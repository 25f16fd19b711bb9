// Triple-product reduction on CUDA cores and the final normalisation.
//
// msum[t] = sum_x d_a(x) d_b(x) d_c(x) for every kept bin t = (a, b, c) (numerator of Eq. (2.7);
// with counting fields, the T_abc of Eq. (2.10)). One launch sums the bins of every contraction
// level, sampling the coarser levels' voxels from the evaluation grid's fields with their stride;
// a second adds the partial sums in FP64 in a fixed order (deterministic results).
//
// FP32: an output's products are added in voxel order over runs of kSumRun voxels, the runs in
// FP64. A lane owns one run and a warp one tile of 2 x 4 x 8 outputs (a, b, c), so 32 runs go
// through the same 8 pair products and 64 multiply-adds per voxel and no lane idles for want of bins;
// tiles at the edge of the triangle region take 4 c. One block of 12 warps an SM (8 warps: 1.34 ms
// per estimate at Ng = 256 and 24 shells, 12: 1.30, 16, which leaves 128 registers: 1.62; blocks of
// tiles of 2 b as well were shorter and fewer fitted one block: 1.33 with 12).
//   * What bounds it: the FMA units (at most 67% of their rate with three register reads each,
//     measured on an outer product), then the warps' waits at the stages' barriers. Shared memory
//     delivers 32 words per cycle whatever lanes share (measured: LDS.128 takes 4 cycles a warp even
//     when its lanes read 8 distinct quads), so a tile has to use a word often: 2 x 4 x 8 reads 14
//     words a voxel for 72 operations, 2 x 4 x 4 reads 10 for 40, 1 x 4 x 4 reads 9 for 20.
//   * Also measured at Ng = 256 and 24 shells: two runs packed in a lane's registers (1.38 ms), tiles
//     in threads with lanes on different tiles of one voxel (1.36); the earlier layout was of that
//     kind with 1 x 4 x 4 tiles, 118 of 256 threads in use.
// FP64 (1/64 of the FP32 rate: 2 multiply-adds per SM and cycle): any order of additions will do,
// so lanes own voxels and a warp exactly the pair products and multiply-adds its bins need, none
// for tile padding; loads go straight to L1. Ng = 128 and 16 shells 2.43 -> 1.04 ms, Ng = 32 and 8
// shells 46.6 -> 13.1 us (there the earlier blocks summed 64 voxels in 11 threads).
#include <algorithm>

#include "common.cuh"
#include "tc_ptx.cuh"

namespace bsp {

namespace {

constexpr int kSumThreads = 32 * kSumWarps;
constexpr int kSumVox = 32;     // voxels of a run per stage: whole cache lines
constexpr int kSumQuads = kSumVox / 4;
constexpr int kSumRow = 4 * kSumVox;          // bytes of a run in a staged field
constexpr int kSumFieldBytes = 32 * kSumRow;  // one field of a stage: 32 runs
// Run r's quad q lies in place q ^ sum_swz(r): eight lanes' 16-byte reads of one field meet all banks.
static_assert(kSumRow == 128, "a run's stage is one row of all banks");
__host__ __device__ constexpr int sum_swz(int r) { return r & (kSumQuads - 1); }
constexpr int kF64Warps = 4;
constexpr int kF64Run = 64;  // 32-voxel steps summed lane by lane

// The level of work item w.
__device__ __forceinline__ const SumLevel& level_of(const SumArgs& a, int w) {
  int l = 0;
  while (l + 1 < a.n_lv && w >= a.lv[l + 1].w0) ++l;
  return a.lv[l];
}

// Lane l ends with the sum over the warp of its v[l]: halves are exchanged, so 31 additions in
// all instead of 5 per output.
__device__ __forceinline__ double warp_transpose_sum(const float* v, int lane) {
  double d[16];
  {
    const bool up = (lane & 16) != 0;
#pragma unroll
    for (int i = 0; i < 16; ++i) {
      const float send = up ? v[i] : v[i + 16];
      const float keep = up ? v[i + 16] : v[i];
      d[i] = (double)keep + (double)__shfl_xor_sync(0xffffffffu, send, 16);
    }
  }
#pragma unroll
  for (int o = 8; o > 0; o >>= 1) {
    const bool up = (lane & o) != 0;
#pragma unroll
    for (int i = 0; i < o; ++i) {
      const double send = up ? d[i] : d[i + o];
      const double keep = up ? d[i + o] : d[i];
      d[i] = keep + __shfl_xor_sync(0xffffffffu, send, o);
    }
  }
  return d[0];
}
__device__ __forceinline__ double warp_transpose_sum(const double* v, int lane) {
  double d[16];
  {
    const bool up = (lane & 16) != 0;
#pragma unroll
    for (int i = 0; i < 16; ++i) {
      const double send = up ? v[i] : v[i + 16];
      const double keep = up ? v[i + 16] : v[i];
      d[i] = keep + __shfl_xor_sync(0xffffffffu, send, 16);
    }
  }
#pragma unroll
  for (int o = 8; o > 0; o >>= 1) {
    const bool up = (lane & o) != 0;
#pragma unroll
    for (int i = 0; i < o; ++i) {
      const double send = up ? d[i] : d[i + o];
      const double keep = up ? d[i + o] : d[i];
      d[i] = keep + __shfl_xor_sync(0xffffffffu, send, o);
    }
  }
  return d[0];
}

// ---------------------------------------------------------------- FP32
// Four voxels of this lane's row of a staged field: one 16-byte load.
__device__ __forceinline__ void lds_quad(uint32_t addr, float (&v)[4]) {
  asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v[0]), "=f"(v[1]), "=f"(v[2]), "=f"(v[3]) : "r"(addr));
}

// One quad of a tile whose fields are in registers: two neighbouring voxels' pair products are one
// packed multiplication; their triple products are added in voxel order.
template <int NC>
__device__ __forceinline__ void sum_quad(const float (&a)[2][4], const float (&b)[4][4], const float (&c)[NC][4],
                                         float (&acc)[64]) {
#pragma unroll
  for (int h = 0; h < 4; h += 2) {
    uint64_t p[2][4];
#pragma unroll
    for (int i = 0; i < 2; ++i)
#pragma unroll
      for (int j = 0; j < 4; ++j)
        p[i][j] = ptx::f2_mul(ptx::f2_pack(a[i][h], a[i][h + 1]), ptx::f2_pack(b[j][h], b[j][h + 1]));
#pragma unroll
    for (int e = 0; e < 2; ++e)
#pragma unroll
      for (int i = 0; i < 2; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          const float x = __uint_as_float((uint32_t)(e ? p[i][j] >> 32 : p[i][j]));
#pragma unroll
          for (int k = 0; k < NC; ++k) acc[32 * i + 8 * j + k] = fmaf(x, c[k][h + e], acc[32 * i + 8 * j + k]);
        }
  }
}

// A stage, two quads at a time: the second's loads are under way while the first is summed. A, B, C
// are the shared-memory addresses of this lane's row of the tile's fields, swz the exchange of its
// quads (see contract_f32_kernel).
template <int NC>
__device__ __forceinline__ void sum_stage(const uint32_t (&A)[2], const uint32_t (&B)[4], const uint32_t (&C)[8],
                                          uint32_t off, uint32_t swz, float (&acc)[64]) {
#pragma unroll 1
  for (uint32_t q = 0; q < kSumVox * 4; q += 32) {
    float a[2][2][4], b[2][4][4], c[2][NC][4];
#pragma unroll
    for (int t = 0; t < 2; ++t) {
      const uint32_t o = off + ((q + 16 * t) ^ swz);
#pragma unroll
      for (int i = 0; i < 2; ++i) lds_quad(A[i] + o, a[t][i]);
#pragma unroll
      for (int i = 0; i < 4; ++i) lds_quad(B[i] + o, b[t][i]);
#pragma unroll
      for (int i = 0; i < NC; ++i) lds_quad(C[i] + o, c[t][i]);
    }
    sum_quad<NC>(a[0], b[0], c[0], acc);
    sum_quad<NC>(a[1], b[1], c[1], acc);
  }
}

// Block = (level, sub, gps groups of 32 runs). A stage holds kSumVox voxels of every run of the group
// for the sub's fields, [field][run][voxel], the quads of a run exchanged so that eight lanes' 16-byte
// reads of one field meet all banks. 128 bytes a run and stage: a copy that brings less than a
// cache line still occupies shared memory for a cycle (8 voxels a stage: 1.45 ms, 16: 1.25, 32:
// 1.13, at Ng = 256 and 24 shells). One block an SM, two stages of up to 27 fields (12 warps: 0.95 ms).
// Copies go two runs a thread per look at a field's offset: 1.37 -> 1.30 ms per estimate, with 12 warps.
__global__ void __launch_bounds__(kSumThreads, 1) contract_f32_kernel(SumArgs a) {
  extern __shared__ __align__(128) unsigned char smem[];
  __shared__ long long foff[kSumMaxFields];
  const int tid = threadIdx.x;
  const int lane = tid & 31;
  const SumLevel L = level_of(a, blockIdx.x);
  const int unit = (int)(blockIdx.x - L.w0);
  const int split = unit / L.units;  // the subs of a group run side by side: its fields stay in L2
  const SumSub sub = L.subs[unit - split * L.units];
  const float* fields = static_cast<const float*>(a.fields);
  if (tid < sub.nf) foff[tid] = (long long)L.sub_fields[sub.field0 + tid] * L.fstride;
  // copies: this thread takes quad cq of runs cr and cr + 16 of every (kSumThreads / 128)-th field
  const int stage_bytes = sub.nf * kSumFieldBytes;
  const int cq = tid % kSumQuads, cr = (tid / kSumQuads) & 15;
  constexpr int kStep = kSumThreads / (16 * kSumQuads);
  static_assert(kStep >= 1 && kStep * 16 * kSumQuads == kSumThreads, "a thread copies one quad of two runs");
  const int f0 = tid / (16 * kSumQuads);
  unsigned char* const cdst = smem + cr * kSumRow + ((cq ^ sum_swz(cr)) << 4);
  static_assert(sum_swz(0) == sum_swz(16), "runs 16 apart exchange quads alike");
  const int warp = tid >> 5;
  uint32_t A[2], B[4], C[8];
  const bool active = warp < sub.ntiles;
  const uint32_t swz = (uint32_t)sum_swz(lane) << 4;
  {
    const SumTile t = L.tiles[sub.tile0 + (active ? warp : 0)];
    const uint32_t row = ptx::smem_u32(smem) + lane * kSumRow;
#pragma unroll
    for (int i = 0; i < 2; ++i) A[i] = row + t.a[i] * kSumFieldBytes;
#pragma unroll
    for (int i = 0; i < 4; ++i) B[i] = row + t.b[i] * kSumFieldBytes;
#pragma unroll
    for (int i = 0; i < 8; ++i) C[i] = row + t.c[i] * kSumFieldBytes;
  }
  const int g0 = split * L.gps, g1 = min(g0 + L.gps, L.ngrp);
#pragma unroll 1
  for (int grp = g0; grp < g1; ++grp) {
    // the runs of the group: whole runs first, then the summation blocks' remainders; lane r sums run r
    const bool whole = grp < L.ngf;
    const int len = whole ? kSumRun : L.vpb - L.nfull * kSumRun;
    __shared__ int2 runs[32];
    if (grp > g0) __syncthreads();  // the last group's runs and stages have been read
    if (tid < 32) {
      const int i = (whole ? grp : grp - L.ngf) * 32 + tid;
      const int b = whole ? i / L.nfull : i;
      int2 v = make_int2(0, 0);
      if (b < L.nblk) {
        const long long first = (long long)b * L.vpb;
        const long long start = first + (long long)(whole ? i - b * L.nfull : L.nfull) * kSumRun;
        const long long end = min(min(first + (long long)L.vpb, L.nvox), start + (long long)len);
        if (end > start) v = make_int2((int)start, (int)end);
      }
      runs[tid] = v;
    }
    __syncthreads();
    const int2 run0 = runs[cr], run1 = runs[cr + 16];
    auto issue = [&](int k, int buf) {
      unsigned char* dst = cdst + buf * stage_bytes;
      const int v0 = run0.x + k * kSumVox + 4 * cq, v1 = run1.x + k * kSumVox + 4 * cq;
      const bool in0 = v0 < run0.y, in1 = v1 < run1.y;
      if (L.t == 1) {
        const float *src0 = fields + (in0 ? v0 : 0), *src1 = fields + (in1 ? v1 : 0);
        const uint32_t n0 = in0 ? 16u : 0u, n1 = in1 ? 16u : 0u;
#pragma unroll 2
        for (int f = f0; f < sub.nf; f += kStep) {
          const long long o = foff[f];
          ptx::cp_async16_zfill(dst + f * kSumFieldBytes, src0 + o, n0);
          ptx::cp_async16_zfill(dst + f * kSumFieldBytes + 16 * kSumRow, src1 + o, n1);
        }
      } else {
        auto at = [&](int v) {  // g is a multiple of 8: the quad lies in one row of the level's grid
          const unsigned g = (unsigned)L.g, u = (unsigned)v;
          const unsigned xy = u / g, z = u - xy * g, x = xy / g, y = xy - x * g;
          return ((long long)x * L.t * L.s + (long long)y * L.t) * L.s + (long long)z * L.t;
        };
        const float *src0 = fields + (in0 ? at(v0) : 0), *src1 = fields + (in1 ? at(v1) : 0);
        for (int f = f0; f < sub.nf; f += kStep) {
          const long long o = foff[f];
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            ptx::cp_async_zfill<4>(dst + f * kSumFieldBytes + 4 * e, in0 ? src0 + o + e * L.t : fields, in0 ? 4u : 0u);
            ptx::cp_async_zfill<4>(dst + f * kSumFieldBytes + 16 * kSumRow + 4 * e, in1 ? src1 + o + e * L.t : fields,
                                   in1 ? 4u : 0u);
          }
        }
      }
      ptx::cp_async_commit();
    };
    float acc[64];
#pragma unroll
    for (int i = 0; i < 64; ++i) acc[i] = 0.f;
    const int nst = len / kSumVox;
    issue(0, 0);
    for (int k = 0; k < nst; ++k) {
      ptx::cp_async_wait<0>();  // stage k has landed
      __syncthreads();          // for every thread, and stage k - 1 has been read
      if (k + 1 < nst) issue(k + 1, (k + 1) & 1);
      if (active) {
        const uint32_t off = (uint32_t)((k & 1) * stage_bytes);
        if (sub.nc == 8) sum_stage<8>(A, B, C, off, swz, acc);
        else sum_stage<4>(A, B, C, off, swz, acc);
      }
    }
    if (active) {
      float half[32];
#pragma unroll
      for (int m = 0; m < 2; ++m) {
#pragma unroll
        for (int i = 0; i < 32; ++i) half[i] = acc[32 * m + i];
        const double s = warp_transpose_sum(half, lane);
        double* out = L.partial + (long long)split * L.n_ent + (sub.tile0 + warp) * 64 + 32 * m + lane;
        *out = grp > g0 ? *out + s : s;  // this lane's alone
      }
    }
  }
}

// ---------------------------------------------------------------- FP64
// Warp = (level, set of kSumJobs jobs, run of spw steps of 32 voxels), lane = voxel.
__global__ void __launch_bounds__(32 * kF64Warps, 4) contract_f64_kernel(SumArgs a) {
  __shared__ long long foff[kF64Warps][kSumJobs][6];
  __shared__ int fcnt[kF64Warps][kSumJobs];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int w = blockIdx.x * kF64Warps + warp;
  if (w >= a.items) return;  // warp-uniform; no block barrier below
  const SumLevel L = level_of(a, w);
  const int unit = w - L.w0;
  const int split = unit / L.units, set = unit - split * L.units;
  const double* fields = static_cast<const double*>(a.fields);
  if (lane < kSumJobs) {
    const int j = set * kSumJobs + lane;
    SumJob job{};
    if (j < L.njobs) job = L.jobs[j];
    fcnt[warp][lane] = job.n;
#pragma unroll
    for (int i = 0; i < 6; ++i) foff[warp][lane][i] = (long long)job.f[i] * L.fstride;
  }
  __syncwarp();
  // Sums of kF64Run steps are added over the warp before they join the total: a lane that meets the
  // counting fields' peak at the origin would otherwise round every later addition at its size. The
  // total keeps its additions' rounding errors: at Ng = 768 and 24 shells a warp adds 1600 such sums,
  // and what those after the peak lost to rounding, all the same way, moved a count off its integer.
  double total = 0.0, lost = 0.0;
  const long long v0 = (long long)split * L.spw * 32;
  for (int k0 = 0; k0 < L.spw; k0 += kF64Run) {
    double acc[4 * kSumJobs];
#pragma unroll
    for (int i = 0; i < 4 * kSumJobs; ++i) acc[i] = 0.0;
    const int k1 = min(k0 + kF64Run, L.spw);
    for (int k = k0; k < k1; ++k) {
      const long long v = v0 + 32LL * k + lane;
      const bool in = v < L.nvox;
      long long o = in ? v : 0;
      if (L.t > 1 && in) {
        const unsigned g = (unsigned)L.g, u = (unsigned)v;
        const unsigned xy = u / g, z = u - xy * g, x = xy / g, y = xy - x * g;
        o = ((long long)x * L.t * L.s + (long long)y * L.t) * L.s + (long long)z * L.t;
      }
      if (!in) continue;  // the ragged end: the lane adds nothing
      const double* f = fields + o;
#pragma unroll
      for (int j = 0; j < kSumJobs; ++j) {
        const int n = fcnt[warp][j];  // warp-uniform
        if (n == 0) break;
        const long long* fo = foff[warp][j];
        const double p = f[fo[0]] * f[fo[1]];
        const double d0 = f[fo[2]], d1 = f[fo[3]], d2 = f[fo[4]], d3 = f[fo[5]];
        acc[4 * j] = fma(p, d0, acc[4 * j]);
        if (n > 1) acc[4 * j + 1] = fma(p, d1, acc[4 * j + 1]);
        if (n > 2) acc[4 * j + 2] = fma(p, d2, acc[4 * j + 2]);
        if (n > 3) acc[4 * j + 3] = fma(p, d3, acc[4 * j + 3]);
      }
    }
    const double x = warp_transpose_sum(acc, lane), t = total + x, y = t - total;
    lost += (total - (t - y)) + (x - y);
    total = t;
  }
  const int e = set * 4 * kSumJobs + lane;
  // once a total is infinite, the differences above are NaN: it has no rounding errors to add
  if (e < L.n_ent) L.partial[(long long)split * L.n_ent + e] = isfinite(lost) ? total + lost : total;
}

// msum[map[e]] = scale * sum over the splits of partial[.][e] (added to msum when accumulating
// x-slabs). A block takes 8 neighbouring outputs, 32 threads each: thread (e, k) adds splits k,
// k + 32, ..., then the 32 sums are added in order. (A warp of outputs a block, 8 threads each, left
// small plans with 5 blocks of long dependent chains: 18.5 us of an Ng = 32 FP64 estimate.)
constexpr int kReduceOuts = 8;
__global__ void __launch_bounds__(256) reduce_sums_kernel(SumArgs a) {
  __shared__ double part[32][kReduceOuts + 1];
  const int o = threadIdx.x % kReduceOuts, k = threadIdx.x / kReduceOuts;
  const int idx = blockIdx.x * kReduceOuts + o;
  int l = 0;
  while (l + 1 < a.n_lv && idx >= a.lv[l + 1].ent0) ++l;
  const SumLevel L = a.lv[l];
  const int e = idx - L.ent0;
  const int dst = idx < a.n_ent ? L.map[e] : -1;
  double s = 0.0;
  if (dst >= 0) {
#pragma unroll 4
    for (int b = k; b < L.splits; b += 32) s += L.partial[(long long)b * L.n_ent + e];
  }
  part[k][o] = s;
  __syncthreads();
  if (k == 0 && dst >= 0) {
#pragma unroll
    for (int w = 1; w < 32; ++w) s += part[w][o];
    a.msum[dst] = a.accumulate ? a.msum[dst] + L.scale * s : L.scale * s;
  }
}

}  // namespace

template <>
bsp_status launch_contract_simt<float>(const SumArgs& a, cudaStream_t s) {
  if (a.items == 0) return BSP_OK;
  const bsp_status st = allow_shared(contract_f32_kernel, (size_t)sum_stage_bytes(kSumMaxFields));
  if (st != BSP_OK) return st;
  contract_f32_kernel<<<a.items, kSumThreads, a.smem, s>>>(a);
  BSP_CUDA(cudaGetLastError());
  return BSP_OK;
}

template <>
bsp_status launch_contract_simt<double>(const SumArgs& a, cudaStream_t s) {
  if (a.items == 0) return BSP_OK;
  contract_f64_kernel<<<(a.items + kF64Warps - 1) / kF64Warps, 32 * kF64Warps, 0, s>>>(a);
  BSP_CUDA(cudaGetLastError());
  return BSP_OK;
}

bsp_status launch_reduce_sums(const SumArgs& a, cudaStream_t s) {
  if (a.n_ent == 0) return BSP_OK;
  reduce_sums_kernel<<<(a.n_ent + kReduceOuts - 1) / kReduceOuts, 32 * kReduceOuts, 0, s>>>(a);
  BSP_CUDA(cudaGetLastError());
  return BSP_OK;
}

int sum_stage_bytes(int nf) { return 2 * nf * kSumFieldBytes; }

// ---------------------------------------------------------------- product fields (order 4)
template <typename T>
__global__ void pair_fields_kernel(const T* __restrict__ f, long long nvox, const int2* __restrict__ pairs, int np,
                                   T* __restrict__ out) {
  const long long total = nvox * np;
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < total;
       i += (long long)gridDim.x * blockDim.x) {
    const int j = (int)(i / nvox);
    const long long v = i - (long long)j * nvox;
    const int2 ab = pairs[j];
    out[i] = f[(long long)ab.x * nvox + v] * f[(long long)ab.y * nvox + v];
  }
}

template <typename T>
bsp_status launch_pair_fields(const void* f, long long nvox, const int2* pairs, int np, void* out, int n_sm,
                              cudaStream_t s) {
  if (np == 0 || nvox == 0) return BSP_OK;
  const long long need = (nvox * np + 255) / 256;
  const long long blocks = std::min<long long>(need, 8LL * std::max(n_sm, 1));
  pair_fields_kernel<T><<<(unsigned)blocks, 256, 0, s>>>(static_cast<const T*>(f), nvox, pairs, np,
                                                         static_cast<T*>(out));
  BSP_CUDA(cudaGetLastError());
  return BSP_OK;
}

template bsp_status launch_pair_fields<float>(const void*, long long, const int2*, int, void*, int, cudaStream_t);
template bsp_status launch_pair_fields<double>(const void*, long long, const int2*, int, void*, int, cudaStream_t);

// ---------------------------------------------------------------- level fields
// dst[j][x][y][z] = src[shells[j]][t x][t y][t z]: the split fields of a coarser level sampled from
// the evaluation grid (side S) with stride t.
__global__ void decimate_kernel(const uint16_t* __restrict__ src, int S, const int* __restrict__ shells, int nsh,
                                uint16_t* __restrict__ dst, int g, int t) {
  const long long per = (long long)g * g * g;
  const long long total = per * nsh;
  const long long plane = (long long)S * S;
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < total;
       i += (long long)gridDim.x * blockDim.x) {
    const int j = (int)(i / per);
    const long long v = i - (long long)j * per;
    const int x = (int)(v / ((long long)g * g));
    const int y = (int)((v / g) % g);
    const int z = (int)(v % g);
    dst[i] = src[(long long)shells[j] * plane * S + ((long long)x * t * S + (long long)y * t) * S + (long long)z * t];
  }
}

bsp_status launch_decimate(const uint16_t* src, int S, const int* shells, int nsh, uint16_t* dst, int g, int t,
                           int n_sm, cudaStream_t s) {
  const long long total = (long long)g * g * g * nsh;
  if (total == 0) return BSP_OK;
  long long blocks = std::min<long long>((total + 255) / 256, 16LL * n_sm);
  decimate_kernel<<<(unsigned)blocks, 256, 0, s>>>(src, S, shells, nsh, dst, g, t);
  BSP_CUDA(cudaGetLastError());
  return BSP_OK;
}

// ---------------------------------------------------------------- finalize
// b_trip[t] = norm msum[t] / tsum[t]                     (Eq. (2.7) with Eq. (2.10))
// b_grid[cell] = norm sum msum / sum tsum over the cell's bins, NaN if it has none.
__global__ void finalize_kernel(FinalizeArgs a) {
  const int idx = blockIdx.x * blockDim.x + threadIdx.x;
  if (idx < a.n_trip) a.b_trip[idx] = a.norm * a.msum[idx] / a.tsum[idx];
  if (a.b_grid != nullptr && idx < a.n_cells) {
    const int lo = a.cell_ptr[idx], hi = a.cell_ptr[idx + 1];
    if (lo == hi) {
      a.b_grid[idx] = __longlong_as_double(0x7ff8000000000000ULL);
    } else {
      double num = 0.0, den = 0.0;
      for (int i = lo; i < hi; ++i) {
        const int t = a.cell_idx[i];
        num += a.msum[t];
        den += a.tsum[t];
      }
      a.b_grid[idx] = a.norm * num / den;
    }
  }
}

bsp_status launch_finalize(const FinalizeArgs& a, cudaStream_t s) {
  const int n = a.n_trip > a.n_cells ? a.n_trip : a.n_cells;
  if (n == 0) return BSP_OK;
  finalize_kernel<<<(n + 255) / 256, 256, 0, s>>>(a);
  BSP_CUDA(cudaGetLastError());
  return BSP_OK;
}

}  // namespace bsp
