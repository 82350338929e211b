// SIMT GEMM C = A . B^T (fp32 FMA) for the fp32 path: the projections of the
// memory, the query, the scores and the two fusion layers when the workload
// stores fp32 (tensor cores would round fp32 operands).
//
// One CTA of 256 threads computes a tile of 64 features x 64 rows, 4 x 4 sums
// per thread.  k-tiles of 32 arrive by 16-byte asynchronous copies in a ring
// of kSimtStages, rows of both operands k-major as they lie in memory; a
// thread reads four consecutive k of its four features and four rows at once
// (16-byte shared loads, a pitch of 36 floats: the 16 feature rows of a warp's
// read fall on distinct banks), so 64 FMAs follow eight loads and the FMA
// pipe bounds a full GPU (128 per cycle and SM).
//
// Split K: a draft step's 64-row batch has 16 tiles, so without a split 16 SMs
// work and each walks the whole contraction.  S <= 8 CTAs of one cluster share
// a tile, each contracting a slice of k; their partial tiles meet in
// distributed shared memory, CTA r summing rows [64 r / S, 64 (r + 1) / S) in
// rank order (deterministic).  The four GEMMs of a 64-row step at d = 1024
// (0.5 GF) took 774 us without the split or the ring, now 68 us (each with
// ~5 us of event-bracketed launch).
#include <algorithm>

#include "gemm_epilogue.cuh"
#include "tc_ptx.cuh"

namespace fovea {

constexpr int kSimtTile = 64, kSimtK = 32, kSimtThreads = 256, kSimtStages = 4;
constexpr int kSimtPitch = kSimtK + 4;                       // floats
constexpr int kSimtStageFloats = 2 * kSimtTile * kSimtPitch;
constexpr int kSimtSmem = kSimtStages * kSimtStageFloats * (int)sizeof(float);
constexpr int kSimtSumPitch = kSimtTile + 4;
static_assert(kSimtTile * kSimtSumPitch <= kSimtStages * kSimtStageFloats, "partial tile in the ring");

// 16 bytes global -> shared, zeros when !real.
__device__ __forceinline__ void simt_copy16(float* dst, const float* src, bool real) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(tc::smem_u32(dst)), "l"(src),
               "r"(real ? 16 : 0)
               : "memory");
}

template <int EPI>
__global__ void __launch_bounds__(kSimtThreads) simt_gemm_kernel(const __grid_constant__ GemmArgs a) {
  extern __shared__ __align__(16) float simt_sm[];
  const int S = a.splits;
  const int rank = (int)blockIdx.x % S;
  const GemmGroup& g = a.groups[blockIdx.z];
  const int m0 = ((int)blockIdx.x / S) * kSimtTile, n0 = blockIdx.y * kSimtTile;
  if (m0 >= g.m || n0 >= g.n) return;                        // the whole cluster
  pdl_wait();
  pdl_trigger();
  const int kt_total = a.k_total / kSimtK;
  const int kt0 = rank * kt_total / S, kt1 = (rank + 1) * kt_total / S;
  const int tid = threadIdx.x;
  // copies: thread tid brings 16-byte piece tid % 8 of rows tid / 8 and + 32
  // of both operands
  const int cr = tid >> 3, ck = (tid & 7) * 4;
  auto load = [&](int kt) {
    float* st = simt_sm + (kt - kt0) % kSimtStages * kSimtStageFloats;
    const int k = kt * kSimtK;                               // b_split is a multiple of kSimtK
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int r = cr + 32 * h, m = m0 + r, n = n0 + r;
      const bool am = m < g.m, bn = n < g.n;
      const float* pa = m < a.a_split || !am
                            ? static_cast<const float*>(a.A0) + (long long)(g.a_row0 + (am ? m : 0)) * a.lda0
                            : static_cast<const float*>(a.A1) + (long long)(m - a.a_split) * a.lda1;
      const long long row = (long long)g.b_row0 + (bn ? n : 0);
      const float* pb = k < a.b_split ? static_cast<const float*>(a.B0) + row * a.ldb0 + k
                                      : static_cast<const float*>(a.B1) + row * a.ldb1 + (k - a.b_split);
      simt_copy16(st + r * kSimtPitch + ck, pa + k + ck, am);
      simt_copy16(st + (kSimtTile + r) * kSimtPitch + ck, pb + ck, bn);
    }
  };
  const int tx = tid & 15, ty = tid >> 4;                    // features tx + 16 i, rows ty + 16 j
  float acc[4][4] = {};
#pragma unroll
  for (int p = 0; p < kSimtStages - 1; ++p) {
    if (kt0 + p < kt1) load(kt0 + p);
    asm volatile("cp.async.commit_group;" ::: "memory");
  }
  for (int kt = kt0; kt < kt1; ++kt) {
    asm volatile("cp.async.wait_group %0;" ::"n"(kSimtStages - 2) : "memory");
    __syncthreads();                     // the tile has landed; the slot read last is free
    if (kt + kSimtStages - 1 < kt1) load(kt + kSimtStages - 1);
    asm volatile("cp.async.commit_group;" ::: "memory");
    const float* as = simt_sm + (kt - kt0) % kSimtStages * kSimtStageFloats;
    const float* bs = as + kSimtTile * kSimtPitch;
#pragma unroll
    for (int k = 0; k < kSimtK; k += 4) {
      float4 av[4], bv[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        av[i] = *reinterpret_cast<const float4*>(as + (tx + 16 * i) * kSimtPitch + k);
        bv[i] = *reinterpret_cast<const float4*>(bs + (ty + 16 * i) * kSimtPitch + k);
      }
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          acc[i][j] = fmaf(av[i].x, bv[j].x, acc[i][j]);
          acc[i][j] = fmaf(av[i].y, bv[j].y, acc[i][j]);
          acc[i][j] = fmaf(av[i].z, bv[j].z, acc[i][j]);
          acc[i][j] = fmaf(av[i].w, bv[j].w, acc[i][j]);
        }
    }
  }
  if (S == 1) {
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const int m = m0 + tx + 16 * i, n = n0 + ty + 16 * j;
        if (m < g.m && n < g.n) gemm_epilogue<float, EPI>(a, g, m, n, acc[i][j]);
      }
    return;
  }
  // the partial tile [row][feature] over the ring
  asm volatile("cp.async.wait_all;" ::: "memory");
  __syncthreads();
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) simt_sm[(ty + 16 * j) * kSimtSumPitch + tx + 16 * i] = acc[i][j];
  tc::cluster_sync();
  const int r0 = rank * kSimtTile / S, rows = (rank + 1) * kSimtTile / S - r0;
  for (int it = tid; it < rows * (kSimtTile / 4); it += kSimtThreads) {
    const int r = r0 + it / (kSimtTile / 4), c = it % (kSimtTile / 4) * 4;
    if (n0 + r >= g.n) break;            // rows ascend with it
    const uint32_t local = tc::smem_u32(simt_sm + r * kSimtSumPitch + c);
    float4 t[8];
#pragma unroll
    for (int q = 0; q < 8; ++q)
      if (q < S) t[q] = tc::ld_dsmem_f4(tc::map_dsmem(local, (uint32_t)q));
    float4 s = t[0];
#pragma unroll
    for (int q = 1; q < 8; ++q)
      if (q < S) {
        s.x += t[q].x;
        s.y += t[q].y;
        s.z += t[q].z;
        s.w += t[q].w;
      }
    const float v[4] = {s.x, s.y, s.z, s.w};
#pragma unroll
    for (int e = 0; e < 4; ++e)
      if (m0 + c + e < g.m) gemm_epilogue<float, EPI>(a, g, m0 + c + e, n0 + r, v[e]);
  }
  tc::cluster_sync();                    // no CTA leaves while its partial tile is read
}

template <int EPI>
static cudaError_t launch_simt(const GemmArgs& args, int max_m, int max_n, cudaStream_t s) {
  static thread_local GemmArgs a;
  a = args;
  const int tiles_m = (max_m + kSimtTile - 1) / kSimtTile, tiles_n = (max_n + kSimtTile - 1) / kSimtTile;
  int dev = 0, sms = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(simt_gemm_kernel<EPI>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSimtSmem);
  if (e != cudaSuccess) return e;
  // tiles with work; split while they leave half of the GPU's two CTAs per SM
  // idle and every slice keeps at least two k-tiles
  long long tiles = 0;
  for (int i = 0; i < a.ngroups; ++i)
    tiles += (long long)((a.groups[i].m + kSimtTile - 1) / kSimtTile) *
             ((a.groups[i].n + kSimtTile - 1) / kSimtTile);
  int S = 1;
  while (S < 8 && tiles * S * 2 <= 2 * sms && a.k_total / kSimtK >= 4 * S) S *= 2;
  a.splits = S;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(tiles_m * S, tiles_n, a.ngroups);
  cfg.blockDim = dim3(kSimtThreads);
  cfg.dynamicSmemBytes = kSimtSmem;
  cfg.stream = s;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.x = S;
  attr[1].val.clusterDim.y = 1;
  attr[1].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 2;
  return cudaLaunchKernelEx(&cfg, simt_gemm_kernel<EPI>, a);
}

cudaError_t launch_gemm_simt(int epi, const GemmArgs& a, int max_m, int max_n, cudaStream_t s) {
  if (max_m <= 0 || max_n <= 0 || a.ngroups <= 0) return cudaSuccess;
  switch (epi) {
    case kEpiStore: return launch_simt<kEpiStore>(a, max_m, max_n, s);
    case kEpiScores: return launch_simt<kEpiScores>(a, max_m, max_n, s);
    case kEpiBiasSilu: return launch_simt<kEpiBiasSilu>(a, max_m, max_n, s);
    case kEpiBiasF32: return launch_simt<kEpiBiasF32>(a, max_m, max_n, s);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace fovea
