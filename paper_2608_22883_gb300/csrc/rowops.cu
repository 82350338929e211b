// Row-wise kernels of the FOVEA path: LayerNorm (+ depth embedding), mask
// compaction, the gather-and-weighted-sum readout, and the gate + gated
// residual + RMSNorm finalisation.
#include "rowmath.cuh"

namespace fovea {

// ---------------------------------------------------------------------------
// LN over rows of d elements (memory equation: LN(v_i)), an optional gather of
// source rows.  sum(x) and sum(x^2) are taken in double-float (var = E[x^2] -
// mean^2, free of cancellation at that precision) and the affine map is
// evaluated in double-float, so the single rounding to the stored type is
// taken on an almost exact value (the value a float64 evaluation rounds).
//
// fp32 (ln_rows_kernel): one CTA per row, every element in double-float.
// bf16 (ln_tokens_kernel): the same stored values at the cost of fp32
// arithmetic.  In bf16, fp32 rounds an element as the exact value would
// unless it lies within the fp32 error bound of a rounding midpoint (about
// one element in 2000); only those take the double-float map.
// ---------------------------------------------------------------------------
constexpr int kLnThreads = 512;

template <class T> struct LnVec;     // elements per 16-byte vector, vectors per thread
template <> struct LnVec<__nv_bfloat16> {
  static constexpr int N = 8, MAX = FOVEA_MAX_D / 8 / kLnThreads;
};
template <> struct LnVec<float> {
  static constexpr int N = 4, MAX = FOVEA_MAX_D / 4 / kLnThreads;
};

template <class T>
__global__ void __launch_bounds__(kLnThreads) ln_rows_kernel(
    const T* __restrict__ x, const int32_t* __restrict__ src_row, int d,
    const T* __restrict__ gamma, const T* __restrict__ beta, float eps, T* __restrict__ out) {
  constexpr int V = LnVec<T>::N;
  constexpr int kLnMaxVec = LnVec<T>::MAX;
  __shared__ dfloat red[2][kLnThreads / 32];
  const int row = blockIdx.x;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int nvec = d / V;
  float xv[kLnMaxVec][V], gv[kLnMaxVec][V], bv[kLnMaxVec][V];
#pragma unroll
  for (int j = 0; j < kLnMaxVec; ++j) {      // weights: independent of the predecessor
    const int vi = tid + j * kLnThreads;
    if (vi < nvec) {
      ln_load<T>(gamma + vi * V, gv[j]);
      ln_load<T>(beta + vi * V, bv[j]);
    }
  }
  pdl_wait();
  pdl_trigger();
  const long long src = src_row ? (long long)src_row[row] : (long long)row;
  const T* xr = x + src * d;
#pragma unroll
  for (int j = 0; j < kLnMaxVec; ++j) {
    const int vi = tid + j * kLnThreads;
    if (vi < nvec) {
      ln_load<T>(xr + vi * V, xv[j]);
    }
  }
  dfloat s1 = {0.0f, 0.0f}, s2 = {0.0f, 0.0f};
#pragma unroll
  for (int j = 0; j < kLnMaxVec; ++j) {
    if (tid + j * kLnThreads < nvec) {
#pragma unroll
      for (int i = 0; i < V; ++i) {
        s1 = df_add_f(s1, xv[j][i]);
        s2 = df_add(s2, df_two_prod(xv[j][i], xv[j][i]));
      }
    }
  }
  s1 = warp_sum_df(s1);
  s2 = warp_sum_df(s2);
  if (lane == 0) {
    red[0][warp] = s1;
    red[1][warp] = s2;
  }
  __syncthreads();
  if (warp == 0) {
    constexpr int NW = kLnThreads / 32;
    dfloat a = lane < NW ? red[0][lane] : dfloat{0.0f, 0.0f};
    dfloat b = lane < NW ? red[1][lane] : dfloat{0.0f, 0.0f};
    a = warp_sum_df(a);
    b = warp_sum_df(b);
    if (lane == 0) {
      const dfloat mean = df_div_f(a, (float)d);
      const dfloat ex2 = df_div_f(b, (float)d);
      const dfloat var = df_add(ex2, df_mul(dfloat{-mean.hi, -mean.lo}, mean));
      red[0][0] = mean;
      red[1][0] = df_rsqrt(df_add_f(var, eps));
    }
  }
  __syncthreads();
  const dfloat neg_mean = {-red[0][0].hi, -red[0][0].lo};
  const dfloat rstd = red[1][0];
  T* o = out + (long long)row * d;
#pragma unroll
  for (int j = 0; j < kLnMaxVec; ++j) {
    const int vi = tid + j * kLnThreads;
    if (vi < nvec) {
      T res[V];
#pragma unroll
      for (int i = 0; i < V; ++i) {
        dfloat y = df_mul(df_add_f(neg_mean, xv[j][i]), rstd);
        y = df_add_f(df_mul_f(y, gv[j][i]), bv[j][i]);
        res[i] = df_store<T>(y);
      }
      *reinterpret_cast<uint4*>(o + vi * V) = *reinterpret_cast<const uint4*>(res);
    }
  }
}

// Packed pairs of fp32 values (one instruction per pair on sm_100 and later).
struct f32x2 {
  unsigned long long v;
};
__device__ __forceinline__ f32x2 x2_pack(float lo, float hi) {
  f32x2 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r.v) : "f"(lo), "f"(hi));
  return r;
}
__device__ __forceinline__ float2 x2_unpack(f32x2 a) {
  float2 r;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(a.v));
  return r;
}
__device__ __forceinline__ f32x2 x2_add(f32x2 a, f32x2 b) {
  f32x2 r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
  return r;
}
__device__ __forceinline__ f32x2 x2_sub(f32x2 a, f32x2 b) {
  f32x2 r;
  asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
  return r;
}
__device__ __forceinline__ f32x2 x2_mul(f32x2 a, f32x2 b) {
  f32x2 r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
  return r;
}
// The running sum s and the sum c of its rounding errors (Ogita, Rump and
// Oishi, Sum2), two independent sums at once.
__device__ __forceinline__ void x2_sum2(f32x2& s, f32x2& c, f32x2 x) {
  const f32x2 t = x2_add(s, x);
  const f32x2 bb = x2_sub(t, s);
  c = x2_add(c, x2_add(x2_sub(s, x2_sub(t, bb)), x2_sub(x, bb)));
  s = t;
}
__device__ __forceinline__ void sum2_join(float& s, float& c, float s2, float c2) {
  const dfloat t = df_two_sum(s, s2);
  s = t.hi;
  c = __fadd_rn(__fadd_rn(c, c2), t.lo);
}

// One warp per row (kRowWarps = 1; for few rows the CTA's four), the row, gamma
// and beta in shared memory; CTAs of four warps loop over the rows.  Bound by
// its instructions and by HBM alike: per element 8 packed operations of the two
// compensated sums (the squares are exact: a bf16 value has 8 significant bits)
// and about 15 of the map and its midpoint test.  A row per warp needs no CTA
// barrier and one reduction, where a CTA per row took two barriers and
// double-float arithmetic on every element: 32768 rows of 4096 took 932 us, now
// 225 us (2.4 TB/s; 6 of them for the RMS of the results).
constexpr int kLnTokWarps = 4;
constexpr int kLnTokLoads = 8;          // 16-byte loads in flight per lane
// Rows per SM up to which the four warps of a CTA share a row: with a row per
// warp 576 rows leave an SM four warps, each with 128 elements per lane in
// series.  A build of 576 tokens at d = 4096 takes 242 us with shared rows, 252
// with a row per warp; 2304 tokens 558 and 581, 4608 tokens 862 and 882.
constexpr int kLnTokSplitRows = 16;

template <int kRowWarps>
__global__ void __launch_bounds__(32 * kLnTokWarps) ln_tokens_kernel(
    const __nv_bfloat16* __restrict__ x, const int32_t* __restrict__ src_row, int rows, int d,
    const __nv_bfloat16* __restrict__ gamma, const __nv_bfloat16* __restrict__ beta, float eps,
    __nv_bfloat16* __restrict__ out, float* __restrict__ rms) {
  extern __shared__ __align__(16) uint4 ln_sm[];     // gamma [d], beta [d], the rows in work
  __shared__ float4 parts[kLnTokWarps];
  constexpr int kRows = kLnTokWarps / kRowWarps;     // rows a CTA works on at a time
  constexpr int kLanes = 32 * kRowWarps;             // threads of a row
  constexpr int kLoads = kLnTokLoads / (kRowWarps > 1 ? 2 : 1);
  const int nvec = d / 8, lane = threadIdx.x % kLanes, mine = threadIdx.x / kLanes;
  uint4* g_s = ln_sm;
  uint4* b_s = ln_sm + nvec;
  uint4* x_s = ln_sm + (2 + mine) * nvec;
  for (int i = threadIdx.x; i < nvec; i += 32 * kLnTokWarps) {
    g_s[i] = reinterpret_cast<const uint4*>(gamma)[i];
    b_s[i] = reinterpret_cast<const uint4*>(beta)[i];
  }
  pdl_wait();
  pdl_trigger();
  __syncthreads();
  for (int row = blockIdx.x * kRows + mine; row < rows; row += gridDim.x * kRows) {
    const uint4* xr = reinterpret_cast<const uint4*>(x + (long long)src_row[row] * d);
    f32x2 s1 = x2_pack(0.0f, 0.0f), c1 = s1, s2 = s1, c2 = s1;
#pragma unroll 1
    for (int j0 = lane; j0 < nvec; j0 += kLanes * kLoads) {
      uint4 raw[kLoads];
#pragma unroll
      for (int j = 0; j < kLoads; ++j) {
        const int vi = j0 + kLanes * j;
        raw[j] = vi < nvec ? __ldg(xr + vi) : make_uint4(0u, 0u, 0u, 0u);   // zeros add nothing
      }
#pragma unroll
      for (int j = 0; j < kLoads; ++j) {
        const int vi = j0 + kLanes * j;
        if (vi < nvec) x_s[vi] = raw[j];
        const uint32_t w[4] = {raw[j].x, raw[j].y, raw[j].z, raw[j].w};
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const f32x2 v = x2_pack(__uint_as_float(w[q] << 16), __uint_as_float(w[q] & 0xFFFF0000u));
          x2_sum2(s1, c1, v);
          x2_sum2(s2, c2, x2_mul(v, v));
        }
      }
    }
    float a = x2_unpack(s1).x, ac = x2_unpack(c1).x, b = x2_unpack(s2).x, bc = x2_unpack(c2).x;
    sum2_join(a, ac, x2_unpack(s1).y, x2_unpack(c1).y);
    sum2_join(b, bc, x2_unpack(s2).y, x2_unpack(c2).y);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      sum2_join(a, ac, __shfl_xor_sync(0xffffffffu, a, o), __shfl_xor_sync(0xffffffffu, ac, o));
      sum2_join(b, bc, __shfl_xor_sync(0xffffffffu, b, o), __shfl_xor_sync(0xffffffffu, bc, o));
    }
    if constexpr (kRowWarps > 1) {                   // the CTA's one row: its warps' sums in order
      if ((threadIdx.x & 31) == 0) parts[threadIdx.x >> 5] = make_float4(a, ac, b, bc);
      __syncthreads();
      a = parts[0].x; ac = parts[0].y; b = parts[0].z; bc = parts[0].w;
#pragma unroll
      for (int w = 1; w < kRowWarps; ++w) {
        sum2_join(a, ac, parts[w].x, parts[w].y);
        sum2_join(b, bc, parts[w].z, parts[w].w);
      }
      __syncthreads();                               // before the next row's parts
    }
    const dfloat mean = df_div_f(df_two_sum(a, ac), (float)d);
    const dfloat ex2 = df_div_f(df_two_sum(b, bc), (float)d);
    const dfloat neg_mean = {-mean.hi, -mean.lo};
    const dfloat rstd = df_rsqrt(df_add_f(df_add(ex2, df_mul(neg_mean, mean)), eps));
    // fp32 error of y = (x - mean) rstd gamma + beta: at most three times 2^-24
    // of the product (x - mean_hi, rstd_hi for rstd, their product), 2^-24 of
    // the result, and mean_lo <= 2^-24 |mean|: inside the window
    // 2^-22 (|product| + |y|) + 2^-23 |mean| rstd |gamma|
    const float mr = fabsf(mean.hi) * rstd.hi * 1.1920929e-7f;
    __nv_bfloat16* o = out + (long long)row * d;
    f32x2 sq = x2_pack(0.0f, 0.0f);                        // of the results, for their RMS
#pragma unroll 1                                       // a lane reads the vectors it stored above
    for (int vi = lane; vi < nvec; vi += kLanes) {
      const uint4 xv = x_s[vi], gr = g_s[vi], br = b_s[vi];
      const uint32_t xw[4] = {xv.x, xv.y, xv.z, xv.w};
      const uint32_t gw[4] = {gr.x, gr.y, gr.z, gr.w}, bw[4] = {br.x, br.y, br.z, br.w};
      uint32_t ow[4], slow = 0u;
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        float y[2];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const float xf = __uint_as_float(h ? xw[q] & 0xFFFF0000u : xw[q] << 16);
          const float gf = __uint_as_float(h ? gw[q] & 0xFFFF0000u : gw[q] << 16);
          const float bf = __uint_as_float(h ? bw[q] & 0xFFFF0000u : bw[q] << 16);
          const float u = (xf - mean.hi) * rstd.hi;
          y[h] = fmaf(u, gf, bf);
          const float window =
              fmaf(fmaf(fabsf(u), fabsf(gf), fabsf(y[h])), 2.3841858e-7f, mr * fabsf(gf));
          // midpoint of the two bf16 values around y; a window that reaches
          // their spacing, or a value that is not finite, is recomputed too
          const float mid = __uint_as_float((__float_as_uint(y[h]) & 0xFFFF0000u) | 0x8000u);
          if (!(fabsf(y[h] - mid) > window && fabsf(y[h]) * 0.001953125f > window))
            slow |= 1u << (2 * q + h);
        }
        const __nv_bfloat162 p = __floats2bfloat162_rn(y[0], y[1]);
        ow[q] = *reinterpret_cast<const uint32_t*>(&p);
        const f32x2 yy = x2_pack(y[0], y[1]);
        sq = x2_add(sq, x2_mul(yy, yy));
      }
      reinterpret_cast<uint4*>(o)[vi] = make_uint4(ow[0], ow[1], ow[2], ow[3]);
      while (slow != 0u) {                             // the exact value, after the vector store
        const int e = 8 * vi + __ffs(slow) - 1;
        slow &= slow - 1u;
        const float xf = __bfloat162float(reinterpret_cast<const __nv_bfloat16*>(x_s)[e]);
        const float gf = __bfloat162float(reinterpret_cast<const __nv_bfloat16*>(g_s)[e]);
        const float bf = __bfloat162float(reinterpret_cast<const __nv_bfloat16*>(b_s)[e]);
        const dfloat t = df_mul(df_add_f(neg_mean, xf), rstd);
        o[e] = df_to_bf16(df_add_f(df_mul_f(t, gf), bf));
      }
    }
    float ssq = warp_sum(x2_unpack(sq).x + x2_unpack(sq).y);
    if constexpr (kRowWarps > 1) {
      if ((threadIdx.x & 31) == 0) parts[threadIdx.x >> 5].x = ssq;
      __syncthreads();
      ssq = 0.0f;
#pragma unroll
      for (int w = 0; w < kRowWarps; ++w) ssq += parts[w].x;
      __syncthreads();                               // before the next row's parts
    }
    if (lane == 0) rms[row] = sqrtf(ssq / (float)d);
  }
}

// LN of the draft hidden states plus the depth embedding (query equation:
// LN(h_n) + E_dep[l_n]), fp32: the mean and the variance in two passes over
// the register-resident row (sum of x, then sum of (x - mean)^2; fixed-order
// warp and block reductions), the affine map in fp32, rounded once to the
// stored type.  Against the float64 evaluation the stored value differs by
// one unit in the last place only where the exact value lies within fp32
// rounding of a midpoint of the stored type (for bf16 about one element in
// 10^4; the query it feeds moves by ~1e-6 of its scale).  One CTA per row;
// 16-byte loads, all requested before any arithmetic.  When the depth
// embedding table fits (<= 64 KB) and the rows are few, each thread copies its
// columns of every row of it into shared memory before griddepcontrol.wait
// (weights: not written by the previous kernel), so the depth lookup adds no
// dependent global load.  An invalid depth sets kErrDepth and uses depth 0.
template <class T>
__global__ void __launch_bounds__(kLnThreads, 2) ln_query_kernel(
    const T* __restrict__ x, int d, const T* __restrict__ gamma, const T* __restrict__ beta,
    float eps, const T* __restrict__ E, const int32_t* __restrict__ depth, int max_depth,
    int e_smem, int* err, T* __restrict__ out) {
  constexpr int V = LnVec<T>::N;
  constexpr int kLnMaxVec = LnVec<T>::MAX;
  constexpr int NW = kLnThreads / 32;
  __shared__ float red[2][NW];
  extern __shared__ __align__(16) uint8_t ln_dyn[];
  T* e_s = reinterpret_cast<T*>(ln_dyn);            // [max_depth + 1, d] when e_smem
  const int row = blockIdx.x;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int nvec = d / V;
  // the row in fp32; gamma, beta and the depth row kept as loaded (16-byte
  // vectors) and widened in the last pass: two CTAs fit on an SM
  float xv[kLnMaxVec][V];
  uint4 gv[kLnMaxVec], bv[kLnMaxVec], ev[kLnMaxVec];
#pragma unroll
  for (int j = 0; j < kLnMaxVec; ++j) {      // weights: independent of the predecessor
    const int vi = tid + j * kLnThreads;
    if (vi < nvec) {
      gv[j] = *reinterpret_cast<const uint4*>(gamma + vi * V);
      bv[j] = *reinterpret_cast<const uint4*>(beta + vi * V);
      if (e_smem)
        for (int r = 0; r <= max_depth; ++r)
          cp_async16(e_s + (long long)r * d + vi * V, E + (long long)r * d + vi * V);
    }
  }
  pdl_wait();
  pdl_trigger();
  // the row and the depth are requested together; the depth embedding row
  // (from the staged table) is read once the depth is known
  const T* xr = x + (long long)row * d;
#pragma unroll
  for (int j = 0; j < kLnMaxVec; ++j) {
    const int vi = tid + j * kLnThreads;
    if (vi < nvec) ln_load<T>(xr + vi * V, xv[j]);
  }
  int dep = depth[row];
  if (dep < 0 || dep > max_depth) {
    if (tid == 0) atomicOr(err, kErrDepth);
    dep = 0;
  }
  const T* er = (e_smem ? e_s : E) + (long long)dep * d;
  if (e_smem) cp_async_wait_all();          // this thread's own copies
#pragma unroll
  for (int j = 0; j < kLnMaxVec; ++j) {
    const int vi = tid + j * kLnThreads;
    if (vi < nvec) ev[j] = *reinterpret_cast<const uint4*>(er + vi * V);
  }
  // pass 1: mean
  float s = 0.0f;
#pragma unroll
  for (int j = 0; j < kLnMaxVec; ++j)
    if (tid + j * kLnThreads < nvec)
#pragma unroll
      for (int i = 0; i < V; ++i) s += xv[j][i];
  s = warp_sum(s);
  if (lane == 0) red[0][warp] = s;
  __syncthreads();
  float tot = 0.0f;
#pragma unroll
  for (int w = 0; w < NW; ++w) tot += red[0][w];
  const float mean = tot / (float)d;
  // pass 2: variance about the mean
  float q = 0.0f;
#pragma unroll
  for (int j = 0; j < kLnMaxVec; ++j)
    if (tid + j * kLnThreads < nvec)
#pragma unroll
      for (int i = 0; i < V; ++i) {
        const float c = xv[j][i] - mean;
        q = fmaf(c, c, q);
      }
  q = warp_sum(q);
  if (lane == 0) red[1][warp] = q;
  __syncthreads();
  float qt = 0.0f;
#pragma unroll
  for (int w = 0; w < NW; ++w) qt += red[1][w];
  const float rstd = 1.0f / sqrtf(qt / (float)d + eps);
  T* o = out + (long long)row * d;
#pragma unroll
  for (int j = 0; j < kLnMaxVec; ++j) {
    const int vi = tid + j * kLnThreads;
    if (vi < nvec) {
      T res[V];
      float gf[V], bf[V], ef[V];
      ln_unpack<T>(gv[j], gf);
      ln_unpack<T>(bv[j], bf);
      ln_unpack<T>(ev[j], ef);
#pragma unroll
      for (int i = 0; i < V; ++i) {
        const float y = fmaf((xv[j][i] - mean) * rstd, gf[i], bf[i]) + ef[i];
        res[i] = from_f32<T>(y);
      }
      *reinterpret_cast<uint4*>(o + vi * V) = *reinterpret_cast<const uint4*>(res);
    }
  }
}

cudaError_t launch_ln_query(int dtype, const void* h, int rows, int d, const void* gamma,
                            const void* beta, float eps, const void* E, const int32_t* depth,
                            int max_depth, int* err, void* out, cudaStream_t s) {
  if (rows == 0) return cudaSuccess;
  constexpr int kESmemMax = 64 * 1024;
  const size_t es = dtype == FOVEA_BF16 ? 2 : 4;
  const size_t e_bytes = (size_t)(max_depth + 1) * d * es;
  // the depth table staged in shared memory by every CTA when the rows are
  // few (it hides the dependent load of the row's depth embedding); for many
  // rows the CTAs read the one row they need instead
  static int sms = 0;
  if (sms == 0) {
    int dev = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  }
  const int e_smem = e_bytes <= (size_t)kESmemMax && rows <= 2 * sms ? 1 : 0;
  const size_t smem = e_smem ? e_bytes : 0;
  if (dtype == FOVEA_BF16) {
    using T = __nv_bfloat16;
    static bool configured = false;
    if (!configured) {
      cudaError_t e = cudaFuncSetAttribute(ln_query_kernel<T>,
                                           cudaFuncAttributeMaxDynamicSharedMemorySize, kESmemMax);
      if (e != cudaSuccess) return e;
      configured = true;
    }
    return launch_pdl(ln_query_kernel<T>, dim3(rows), dim3(kLnThreads), smem, s, (const T*)h, d,
                      (const T*)gamma, (const T*)beta, eps, (const T*)E, depth, max_depth, e_smem,
                      err, (T*)out);
  }
  static bool configured_f = false;
  if (!configured_f) {
    cudaError_t e = cudaFuncSetAttribute(ln_query_kernel<float>,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize, kESmemMax);
    if (e != cudaSuccess) return e;
    configured_f = true;
  }
  return launch_pdl(ln_query_kernel<float>, dim3(rows), dim3(kLnThreads), smem, s, (const float*)h,
                    d, (const float*)gamma, (const float*)beta, eps, (const float*)E, depth,
                    max_depth, e_smem, err, (float*)out);
}

cudaError_t launch_ln_rows(int dtype, const void* x, const int32_t* src_row, int rows, int d,
                           const void* gamma, const void* beta, float eps, void* out, float* rms,
                           cudaStream_t s) {
  if (rows == 0) return cudaSuccess;
  if (dtype != FOVEA_BF16)
    return launch_pdl(ln_rows_kernel<float>, dim3(rows), dim3(kLnThreads), 0, s, (const float*)x,
                      src_row, d, (const float*)gamma, (const float*)beta, eps, (float*)out);
  int dev = 0, sms = 0, per_sm = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (e != cudaSuccess) return e;
  const bool split = rows <= kLnTokSplitRows * sms;
  const int at_once = split ? 1 : kLnTokWarps;
  const auto kern = split ? ln_tokens_kernel<kLnTokWarps> : ln_tokens_kernel<1>;
  const size_t smem = (size_t)d * 2 * (2 + at_once);           // at most 96 KB
  e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                           FOVEA_MAX_D * 2 * (2 + at_once));
  if (e == cudaSuccess)
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, 32 * kLnTokWarps, smem);
  if (e != cudaSuccess) return e;
  const int ctas = (rows + at_once - 1) / at_once;
  const int most = sms * (per_sm > 0 ? per_sm : 1);
  return launch_pdl(kern, dim3(ctas < most ? ctas : most), dim3(32 * kLnTokWarps),
                    smem, s, (const __nv_bfloat16*)x, src_row, rows, d, (const __nv_bfloat16*)gamma,
                    (const __nv_bfloat16*)beta, eps, (__nv_bfloat16*)out, rms);
}

// ---------------------------------------------------------------------------
// Mask compaction (memory validity m_i and the valid set V): per-image valid
// counts, then an ordered compaction of valid positions.
// ---------------------------------------------------------------------------
constexpr int kScanThreads = 256;

// Norms of the rows of W, a warp each: CTA `cta` of the extra ones of a launch.
__device__ __forceinline__ void row_norms(const RowNorms& nw, int cta) {
  const int r = cta * (kScanThreads / 32) + (int)(threadIdx.x >> 5), lane = threadIdx.x & 31;
  if (r >= nw.d) return;
  const uint4* w = static_cast<const uint4*>(nw.W) + (long long)r * (nw.d / 8);
  float ss = 0.0f;
  for (int v = lane; v < nw.d / 8; v += 32) {
    float x[8];
    ln_unpack<__nv_bfloat16>(__ldg(w + v), x);
#pragma unroll
    for (int i = 0; i < 8; ++i) ss = fmaf(x[i], x[i], ss);
  }
  ss = warp_sum(ss);
  if (lane == 0) nw.norms[r] = sqrtf(ss);
}

__global__ void __launch_bounds__(kScanThreads) count_valid_kernel(const uint8_t* __restrict__ mask,
                                                                  int M_max,
                                                                  int32_t* __restrict__ counts) {
  __shared__ float scratch[32];
  const int b = blockIdx.x;
  int c = 0;
  for (int i = threadIdx.x; i < M_max; i += kScanThreads)
    c += mask[(long long)b * M_max + i] != 0;
  const float tot = block_sum((float)c, scratch);   // exact: counts < 2^24
  if (threadIdx.x == 0) counts[b] = (int32_t)tot;
}

__global__ void __launch_bounds__(kScanThreads) compact_kernel(const uint8_t* __restrict__ mask,
                                                              int M_max,
                                                              const __grid_constant__ ImageTable tab,
                                                              int32_t* __restrict__ orig_index,
                                                              int32_t* __restrict__ src_row,
                                                              const RowNorms nw) {
  __shared__ int warp_tot[kScanThreads / 32];
  const int b = blockIdx.x;
  if (b >= tab.B) return row_norms(nw, b - tab.B);
  const int chunk = (M_max + kScanThreads - 1) / kScanThreads;
  const int beg = min(M_max, threadIdx.x * chunk), end = min(M_max, beg + chunk);
  const uint8_t* mb = mask ? mask + (long long)b * M_max : nullptr;
  int c = 0;
  for (int i = beg; i < end; ++i) c += mb ? (mb[i] != 0) : 1;
  // exclusive scan of c over the block (thread order = position order)
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  int incl = c;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int t = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += t;
  }
  if (lane == 31) warp_tot[warp] = incl;
  __syncthreads();
  int base = 0;
  for (int w = 0; w < warp; ++w) base += warp_tot[w];
  int rank = base + incl - c;
  const int off = tab.off[b];
  for (int i = beg; i < end; ++i) {
    if (mb == nullptr || mb[i] != 0) {
      orig_index[off + rank] = i;
      src_row[off + rank] = b * M_max + i;
      ++rank;
    }
  }
}

cudaError_t launch_count_valid(const uint8_t* mask, int B, int M_max, int32_t* counts,
                               cudaStream_t s) {
  count_valid_kernel<<<B, kScanThreads, 0, s>>>(mask, M_max, counts);
  return cudaGetLastError();
}

cudaError_t launch_compact(const uint8_t* mask, int B, int M_max, const ImageTable& tab,
                           int32_t* orig_index, int32_t* src_row, const RowNorms& nw, cudaStream_t s) {
  const int norm_ctas = nw.norms != nullptr ? (nw.d + kScanThreads / 32 - 1) / (kScanThreads / 32) : 0;
  compact_kernel<<<B + norm_ctas, kScanThreads, 0, s>>>(mask, M_max, tab, orig_index, src_row, nw);
  return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// The gathers of a selection made by select_kernel (sel_cnt, sel_pos, sel_w):
// the readout r_n = sum_{t < K} alpha_t u_{pi(t)} (the alpha / r_n equation)
// and, in bf16 with the projected values, the first fusion layer
// SiLU(G_h + sum alpha_t p_{pi(t)} + [b_f1 ; b_g1]).
// Grid (N rows, chunks of 32 x vector width columns: those of P first, then
// those of U); 8 warps per CTA split the selected entries (warp w takes t = w,
// w + 8, ...), each lane owns one 16-byte vector of columns and keeps eight
// gathers in flight; the warps' partial sums are combined in warp order (fixed
// order, fp32).  Bound by the latency of its gathers out of L2: a row's work
// spreads over up to 20 CTAs, where the selection + gather kernel has two.
// ---------------------------------------------------------------------------
constexpr int kReadoutWarps = 8;
constexpr int kReadoutThreads = 32 * kReadoutWarps;
constexpr int kReadoutUnroll = 8;

template <class T>
struct Vec16;
template <> struct Vec16<__nv_bfloat16> { static constexpr int N = 8; };
template <> struct Vec16<float> { static constexpr int N = 4; };

template <class T>
__global__ void __launch_bounds__(kReadoutThreads, 4) readout_kernel(const __grid_constant__ RowGather a) {
  constexpr int V = Vec16<T>::N;
  __shared__ float part[kReadoutWarps][32 * V];
  const int n = blockIdx.x;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int p_chunks = a.P != nullptr ? (2 * a.H + 32 * V - 1) / (32 * V) : 0;
  const bool proj = (int)blockIdx.y < p_chunks;
  const int chunk = proj ? blockIdx.y : (int)blockIdx.y - p_chunks;
  const int width = proj ? 2 * a.H : a.d;              // columns, and the row stride
  const T* X = static_cast<const T*>(proj ? a.P : a.U);
  const int col = (chunk * 32 + lane) * V;
  pdl_wait();
  pdl_trigger();
  const int K = a.sel_cnt[n];
  const int32_t* pos = a.sel_pos + (long long)n * a.k_max;
  const float* w = a.sel_w + (long long)n * a.k_max;
  float acc[V];
#pragma unroll
  for (int i = 0; i < V; ++i) acc[i] = 0.0f;
  if (col < width) {
    for (int t = warp; t < K; t += kReadoutUnroll * kReadoutWarps) {
      uint4 raw[kReadoutUnroll];               // as loaded: few registers, more CTAs per SM
      float wt[kReadoutUnroll];
#pragma unroll
      for (int j = 0; j < kReadoutUnroll; ++j) {
        const int tj = t + j * kReadoutWarps;
        wt[j] = 0.0f;
        raw[j] = make_uint4(0u, 0u, 0u, 0u);
        if (tj < K) {
          wt[j] = w[tj];
          raw[j] = __ldg(reinterpret_cast<const uint4*>(X + (long long)pos[tj] * width + col));
        }
      }
#pragma unroll
      for (int j = 0; j < kReadoutUnroll; ++j) {
        float u[V];
        ln_unpack<T>(raw[j], u);
#pragma unroll
        for (int i = 0; i < V; ++i) acc[i] = fmaf(wt[j], u[i], acc[i]);
      }
    }
  }
#pragma unroll
  for (int i = 0; i < V; ++i) part[warp][lane * V + i] = acc[i];
  __syncthreads();
  // combine the warps' partial sums in warp order; thread i of the CTA owns
  // element i of the chunk
  for (int e = threadIdx.x; e < 32 * V; e += kReadoutThreads) {
    const int c = chunk * 32 * V + e;
    if (c >= width) continue;
    float sum = 0.0f;
#pragma unroll
    for (int wi = 0; wi < kReadoutWarps; ++wi) sum += part[wi][e];
    const long long o = (long long)n * width + c;
    if (proj) {
      const float bias = to_f32(c < a.H ? static_cast<const T*>(a.b_f1)[c]
                                        : static_cast<const T*>(a.b_g1)[c - a.H]);
      const float z = sum + a.Gh[o] + bias;
      static_cast<T*>(a.act)[o] = from_f32<T>(siluf_(z));
    } else {
      if (a.r_out != nullptr) a.r_out[o] = sum;
      if (a.r_lo != nullptr) static_cast<T*>(a.r_lo)[o] = from_f32<T>(sum);
    }
  }
}

cudaError_t launch_readout(int dtype, const RowGather& a, int N, cudaStream_t s) {
  if (N == 0) return cudaSuccess;
  const int cols = 32 * (dtype == FOVEA_BF16 ? 8 : 4);
  const int chunks = (a.P != nullptr ? (2 * a.H + cols - 1) / cols : 0) +
                     (a.U != nullptr ? (a.d + cols - 1) / cols : 0);
  const dim3 grid(N, chunks);
  if (dtype == FOVEA_BF16)
    return launch_pdl(readout_kernel<__nv_bfloat16>, grid, dim3(kReadoutThreads), 0, s, a);
  return launch_pdl(readout_kernel<float>, grid, dim3(kReadoutThreads), 0, s, a);
}

// ---------------------------------------------------------------------------
// Exact rounding of the marked key elements (memory equation k_i = W_K
// LN(v_i)): a CTA per token, one warp per marked element, the token's row in
// shared memory and the element's weight row by 16-byte loads.  Products of two bf16
// values are exact in fp32; each lane sums its products with the cascaded
// (compensated) summation of Ogita, Rump and Oishi ("Accurate sum and dot
// product", 2005, Algorithm Sum2: TwoSum of the running sum and the product,
// the rounding errors added separately), whose error is below
// eps |S| + (n eps)^2 sum |p| -- about 2^-27 of the key for d <= 8192, far
// inside the distance of any marked element from a bf16 midpoint that matters
// -- and the lanes' (sum, error) pairs are combined in double-float before
// the single rounding to bf16.
//
// Bound by the L2 reads of the weight rows (19 marked elements per token of d
// = 4096, 8 KB each) and by the summation's instructions, two products side by
// side in packed fp32 arithmetic.  A warp per element of a list in no order
// read both rows from L2 and summed one product at a time: 1025 us at 32768
// tokens of d = 4096, now 864 (846 before the window of the marks was widened),
// and 291 us at 10368 tokens of d = 3584, now 231.
// ---------------------------------------------------------------------------
constexpr int kRefineThreads = 256;
// Tokens per SM up to which two CTAs share a token: five CTAs fit an SM, so
// few tokens leave each warp three elements in a row.  A build of 576 tokens
// at d = 4096 takes 287 us with two CTAs per token, 291 with one (10368
// tokens: 1066 and 1070).
constexpr int kRefineSplitRows = 8;
static_assert(FOVEA_MAX_D <= 32 * kRefineThreads, "one word of marks per thread");

// Eight products of two bf16 vectors into the running sums s and error sums c,
// two independent sums side by side (packed fp32 arithmetic).
__device__ __forceinline__ void sum2_bf16x8(const uint4& xa, const uint4& wa, f32x2& s, f32x2& c) {
  const uint32_t xs[4] = {xa.x, xa.y, xa.z, xa.w}, ws[4] = {wa.x, wa.y, wa.z, wa.w};
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const f32x2 x = x2_pack(__uint_as_float(xs[q] << 16), __uint_as_float(xs[q] & 0xFFFF0000u));
    const f32x2 w = x2_pack(__uint_as_float(ws[q] << 16), __uint_as_float(ws[q] & 0xFFFF0000u));
    x2_sum2(s, c, x2_mul(x, w));                                // the products are exact
  }
}

__global__ void __launch_bounds__(kRefineThreads) refine_keys_kernel(
    const __nv_bfloat16* __restrict__ xv, const __nv_bfloat16* __restrict__ W, int d,
    const uint32_t* __restrict__ bits, __nv_bfloat16* __restrict__ K) {
  extern __shared__ uint4 refine_sm[];                           // [d / 8] the token's row, [d] columns
  __shared__ int n_cols;
  const int nv = d / 8;                                          // d % 64 == 0
  uint16_t* cols = reinterpret_cast<uint16_t*>(refine_sm + nv);
  const int tid = threadIdx.x, lane = tid & 31;
  const long long row = blockIdx.x;
  const uint4* x = reinterpret_cast<const uint4*>(xv + row * d);
  // d <= 32 kRefineThreads; of several CTAs of a token each takes every
  // gridDim.y-th word of marks
  uint32_t m = tid < d / 32 && tid % (int)gridDim.y == (int)blockIdx.y ? bits[row * (d / 32) + tid] : 0u;
  if (tid == 0) n_cols = 0;
  for (int l = tid; l < nv; l += kRefineThreads) refine_sm[l] = x[l];
  __syncthreads();
  if (m != 0u) {
    int at = atomicAdd(&n_cols, __popc(m));
    for (; m != 0u; m &= m - 1u) cols[at++] = (uint16_t)(32 * tid + __ffs(m) - 1);
  }
  __syncthreads();
  const int n = n_cols;
  for (int it = tid >> 5; it < n; it += kRefineThreads / 32) {
    const int col = cols[it];
    const uint4* w = reinterpret_cast<const uint4*>(W + (long long)col * d);
    f32x2 s0 = x2_pack(0.0f, 0.0f), c0 = s0, s1 = s0, c1 = s0;
    int l = lane;
    for (; l + 96 < nv; l += 128) {
      uint4 wv[4];
#pragma unroll
      for (int j = 0; j < 4; ++j) wv[j] = __ldg(w + l + 32 * j);
#pragma unroll
      for (int j = 0; j < 4; ++j)
        sum2_bf16x8(refine_sm[l + 32 * j], wv[j], j & 1 ? s1 : s0, j & 1 ? c1 : c0);
    }
#pragma unroll 1
    for (; l < nv; l += 32) sum2_bf16x8(refine_sm[l], __ldg(w + l), s0, c0);
    const float2 sa = x2_unpack(s0), ca = x2_unpack(c0), sb = x2_unpack(s1), cb = x2_unpack(c1);
    dfloat acc = df_add(df_add(df_two_sum(sa.x, ca.x), df_two_sum(sa.y, ca.y)),
                        df_add(df_two_sum(sb.x, cb.x), df_two_sum(sb.y, cb.y)));
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      const dfloat t = {__shfl_xor_sync(0xffffffffu, acc.hi, o), __shfl_xor_sync(0xffffffffu, acc.lo, o)};
      acc = df_add(acc, t);
    }
    if (lane == 0) K[row * d + col] = df_to_bf16(acc);
  }
}

// Per image b: out[(b C + c) * ld + j] = in[(off_b + j) * C + c] for entries
// j < m_b and columns c < C, zero for m_b <= j < ld: the transposed projected
// values the weighted-sum GEMM reads, K-major over the image's entries.  Bound
// by HBM: each CTA moves a 64 x 64 tile with 16-byte accesses on both sides (a row of the
// tile is a full 128-byte line), and its pitch of 33 words keeps the 4-byte
// stores free of bank conflicts and the 2-byte reads at two ways.  A 4096 x 4096
// matrix (67 MB moved): 21 us against 42 us with 2-byte global accesses.
__global__ void __launch_bounds__(256) transpose_images_kernel(const __nv_bfloat16* __restrict__ in,
                                                               int C, int ld,
                                                               const __grid_constant__ ImageTable tab,
                                                               __nv_bfloat16* __restrict__ out) {
  constexpr int kPitch = 33;                         // words
  __shared__ uint32_t t[64 * kPitch];
  const int b = blockIdx.z;
  const int j0 = blockIdx.x * 64, c0 = blockIdx.y * 64;
  const int row = threadIdx.x >> 3, v = threadIdx.x & 7;
  const int m = tab.m[b];
#pragma unroll
  for (int k = 0; k < 64; k += 32) {
    const int j = j0 + row + k;
    uint4 u = make_uint4(0u, 0u, 0u, 0u);
    if (j < m) u = __ldg(reinterpret_cast<const uint4*>(in + ((long long)tab.off[b] + j) * C + c0) + v);
    uint32_t* d = t + (row + k) * kPitch + 4 * v;
    d[0] = u.x; d[1] = u.y; d[2] = u.z; d[3] = u.w;
  }
  __syncthreads();
  const unsigned short* t16 = reinterpret_cast<const unsigned short*>(t);
#pragma unroll
  for (int k = 0; k < 64; k += 32) {
    const int c = row + k;                           // output row; v: its vector of 8 entries
    uint32_t w[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const uint32_t lo = t16[(8 * v + 2 * q) * 2 * kPitch + c];
      const uint32_t hi = t16[(8 * v + 2 * q + 1) * 2 * kPitch + c];
      w[q] = lo | (hi << 16);
    }
    reinterpret_cast<uint4*>(out + ((long long)b * C + c0 + c) * ld + j0)[v] =
        make_uint4(w[0], w[1], w[2], w[3]);
  }
}

cudaError_t launch_transpose_images(const void* in, int C, int ld, const ImageTable& tab,
                                    void* out, cudaStream_t s) {
  if (tab.B <= 0 || C <= 0 || ld <= 0) return cudaSuccess;
  if (C % 64 != 0 || ld % 64 != 0) return cudaErrorInvalidValue;
  transpose_images_kernel<<<dim3(ld / 64, C / 64, tab.B), 256, 0, s>>>(
      (const __nv_bfloat16*)in, C, ld, tab, (__nv_bfloat16*)out);
  return cudaGetLastError();
}

cudaError_t launch_refine_keys(const void* xv, const void* W, int d, const uint32_t* bits, int rows,
                               void* K, cudaStream_t s) {
  if (rows == 0 || d == 0) return cudaSuccess;
  int dev = 0, sms = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  const int parts = rows <= kRefineSplitRows * sms ? 2 : 1;
  refine_keys_kernel<<<dim3(rows, parts), kRefineThreads, 4 * d, s>>>((const __nv_bfloat16*)xv,
                                                         (const __nv_bfloat16*)W, d, bits,
                                                         (__nv_bfloat16*)K);
  return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// Gate, gated residual and RMSNorm (Eq. hidden_correction):
// g = sigma(a_g . w_g2 + b_g2), y = h + g c, h_hat = y / sqrt(mean(y^2) + eps) * gamma.
// One CTA per row; `act` is [N, 2H] with a_f in columns 0..H-1 and a_g in
// H..2H-1.  Every operand of the row is requested before the first reduction.
// A row past the depth gate is copied (h_hat = h, gate 0).
// ---------------------------------------------------------------------------
constexpr int kFinThreads = 512;

template <class T>
__global__ void __launch_bounds__(kFinThreads, 2) finalize_kernel(
    const T* __restrict__ h, const float* __restrict__ c, const T* __restrict__ act, int H, int d,
    const T* __restrict__ w_g2, const T* __restrict__ b_g2, const T* __restrict__ rms_gamma,
    float eps, const __grid_constant__ DepthGate gate_rows, T* __restrict__ h_out,
    float* __restrict__ gate_out) {
  constexpr int V = LnVec<T>::N;
  constexpr int MV = LnVec<T>::MAX;
  __shared__ float scratch[32];
  const int n = blockIdx.x, tid = threadIdx.x;
  const int nvec = d / V;
  const T* hr = h + (long long)n * d;
  const float* cr = c + (long long)n * d;
  float hv[MV][V], cv[MV][V], gv[MV][V];
#pragma unroll
  for (int j = 0; j < MV; ++j) {
    const int vi = tid + j * kFinThreads;
    if (vi < nvec) {
      ln_load<T>(hr + vi * V, hv[j]);
      ln_load<T>(rms_gamma + vi * V, gv[j]);
    }
  }
  pdl_wait();
  pdl_trigger();
  if (row_gated(gate_rows, n)) {          // not corrected: h_hat = h, gate 0
    T* o = h_out + (long long)n * d;
#pragma unroll
    for (int j = 0; j < MV; ++j) {
      const int vi = tid + j * kFinThreads;
      if (vi < nvec) *reinterpret_cast<uint4*>(o + vi * V) = *reinterpret_cast<const uint4*>(hr + vi * V);
    }
    if (gate_out != nullptr && tid == 0) gate_out[n] = 0.0f;
    return;
  }
#pragma unroll
  for (int j = 0; j < MV; ++j) {
    const int vi = tid + j * kFinThreads;
    if (vi < nvec) {
#pragma unroll
      for (int i = 0; i < V; i += 4) {
        const float4 c4 = *reinterpret_cast<const float4*>(cr + vi * V + i);
        cv[j][i] = c4.x; cv[j][i + 1] = c4.y; cv[j][i + 2] = c4.z; cv[j][i + 3] = c4.w;
      }
    }
  }
  const T* a_g = act + (long long)n * 2 * H + H;
  float part = 0.0f;
  for (int k = tid; k < H; k += kFinThreads) part = fmaf(to_f32(a_g[k]), to_f32(w_g2[k]), part);
  const float z = block_sum(part, scratch) + to_f32(b_g2[0]);
  const float g = sigmoidf_(z);
  float ss = 0.0f;
#pragma unroll
  for (int j = 0; j < MV; ++j) {
    if (tid + j * kFinThreads < nvec) {
#pragma unroll
      for (int i = 0; i < V; ++i) {
        hv[j][i] = fmaf(g, cv[j][i], hv[j][i]);          // y = h + g c
        ss = fmaf(hv[j][i], hv[j][i], ss);
      }
    }
  }
  const float tot = block_sum(ss, scratch);
  const float inv = 1.0f / sqrtf(tot / (float)d + eps);
  T* o = h_out + (long long)n * d;
#pragma unroll
  for (int j = 0; j < MV; ++j) {
    const int vi = tid + j * kFinThreads;
    if (vi < nvec) {
      T res[V];
#pragma unroll
      for (int i = 0; i < V; ++i) res[i] = from_f32<T>(hv[j][i] * inv * gv[j][i]);
      *reinterpret_cast<uint4*>(o + vi * V) = *reinterpret_cast<const uint4*>(res);
    }
  }
  if (gate_out != nullptr && tid == 0) gate_out[n] = g;
}

cudaError_t launch_finalize(int dtype, const void* h, const float* c, const void* act, int H, int d,
                            const void* w_g2, const void* b_g2, const void* rms_gamma, float eps,
                            int N, const DepthGate& gate, void* h_out, float* gate_out,
                            cudaStream_t s) {
  if (N == 0) return cudaSuccess;
  if (dtype == FOVEA_BF16) {
    using T = __nv_bfloat16;
    return launch_pdl(finalize_kernel<T>, dim3(N), dim3(kFinThreads), 0, s, (const T*)h, c,
                      (const T*)act, H, d, (const T*)w_g2, (const T*)b_g2, (const T*)rms_gamma,
                      eps, gate, (T*)h_out, gate_out);
  }
  return launch_pdl(finalize_kernel<float>, dim3(N), dim3(kFinThreads), 0, s, (const float*)h, c,
                    (const float*)act, H, d, (const float*)w_g2, (const float*)b_g2,
                    (const float*)rms_gamma, eps, gate, (float*)h_out, gate_out);
}

}  // namespace fovea
