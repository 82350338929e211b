// The memory build's GEMMs C = X . W^T (bf16, fp32 sums) on CTA pairs: the
// keys and values (W_K ; W_U against LN(v)), then, in one launch, the folded
// keys (W_Q^T against the keys) and the projected values ([W_f1 ; W_g1]_r
// against the values): a one-image build's 48 and 12 tiles fill one wave of
// pairs together (build 266 us, 291 with two launches; 32768 tokens: the same).
// Thousands of token rows meet thousands of features, so, unlike the draft
// step's GEMMs (gemm_tc.cu), these are bound by the tensor pipe and by what
// feeds it.
//
// Tile and split.  A pair of CTAs (one cluster, tcgen05 cta_group::2) owns a
// tile of 256 tokens x 256 features: each CTA stages its 128 token rows and
// its half of the features, and the pair's MMA (M = 256, N = 256) reads both
// halves.  A one-CTA tile of 128 x 256 moves 48 KB through shared memory per
// k-block twice (TMA write, tensor-core read), 750 cycles at 128 B/cycle
// against the MMA's 516; the pair moves 32 KB per CTA, which the MMA covers.
// The grid is persistent, one pair per two SMs, and the accumulator is
// double-buffered in tensor memory (2 x 256 columns), so the epilogue of one
// buffer runs under the MMAs of the other.
//
// Chunked sums.  The tensor core adds a product sum to its fp32 accumulator
// with truncation, once per 16 elements of the contraction, so a long
// contraction falls short by about 2^-26 of the result per addition.  For the
// keys every chunk of kChunkSu * KPS * 64 = 256 elements starts a fresh
// accumulator, and the epilogue threads add the chunks in registers with rounded
// fp32 additions.  The projected values, and the folded keys of up to
// kChunkFoldRows tokens, take about eight chunks (of at least 256 elements): the
// accumulators that a split contraction of one-CTA tiles gave them.  The first
// is twice as long, so that its MMAs cover the epilogue's stores of the tile
// before: a build of 10368 tokens of d = 3584 takes 1039 us (1034 with one
// accumulator, 1066 with equal chunks), one image 242 (241), 32768 tokens 3400
// (3402).  The values and the folded keys of more tokens keep one
// accumulator: draining one every 256 elements costs a tile a sixth of its rate
// (folded keys of 32768 tokens 820 us instead of 628).
// A key must be the correctly rounded bf16 of its exact sum; the keys whose
// sum lies so near a rounding midpoint that the GEMM cannot tell are marked
// and recomputed exactly (refine_keys_kernel).  The window of the marks
// follows the error of the sum (kKeyWindow below).
//
// Roles (320 threads): warp 0 lanes 0 and 1 issue the TMA loads of this CTA's
// features and tokens, warp 1 allocates the tensor memory and, in the leader
// CTA (cluster rank 0), an elected lane issues the MMAs of the pair; warps 2 .. 9
// run the epilogue: warp w reads accumulator lanes (tokens) 32 (w % 4) .. +31
// and one half of the columns, 128 fp32 sums per thread.  Stage barriers
// (`full`) live in the leader and count both CTAs' bytes; commits signal
// both CTAs (`empty`, `tfull`); the epilogue warps of both release a buffer
// to the leader (`tempty`).
//
// Every wait is bounded.  A role whose wait gives up sets its CTA's abort
// flag and leaves its loop; the pair meets at a cluster barrier, which both
// CTAs reach because all waits are bounded, and when either has aborted the
// leader commits the MMAs it issued, both wait for them and for the copies
// in flight (bounded), and only then is the tensor memory freed.
#include <algorithm>

#include "tc_ptx.cuh"

namespace fovea {
namespace pair {

using namespace tc;

constexpr int BM = 128;                  // token rows per CTA (256 per pair)
constexpr int BN = 256;                  // features per pair
constexpr int BNH = BN / 2;              // features each CTA stages
constexpr int KPS = 2;                   // k-blocks of 64 per stage
constexpr int kSmemRows = BM * 128;      // bytes of one k-block of tokens
constexpr int kSmemFeat = BNH * 128;     // bytes of one k-block of this CTA's features
constexpr int kStageBytes = KPS * (kSmemRows + kSmemFeat);
constexpr int kStages = 3;
constexpr int kChunkSu = 2;              // stages per accumulator chunk of the keys
constexpr int kChunks = 8;               // accumulator chunks of the projected values ...
constexpr int kChunkFoldRows = 8192;     // ... and of the folded keys of up to this many tokens
constexpr int kEpiWarps = 8;
constexpr int kThreads = 64 + 32 * kEpiWarps;
constexpr int kWarpStage = 32 * 128;     // an epilogue warp's staging: 32 rows x 64 bf16
constexpr int kSmemBytes = 1024 + kStages * kStageBytes + kEpiWarps * kWarpStage + 256;
constexpr int kBandRows = 8;             // row tiles a wave of pairs shares
constexpr uint32_t kTmemCols = 512;
// kind::f16: D fp32, A and B bf16, both K-major, N = 256, M = 256
constexpr uint32_t kIdesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(BN >> 3) << 17) |
                            ((uint32_t)(2 * BM >> 4) << 24);
// The folded part's features are W_Q read as it lies, the contraction along its
// rows: B MN-major (bit 16).  A stage holds two blocks of 64 features, each
// KPS * 64 contraction rows of 128 bytes (128-byte swizzle): 16 KB from one
// block of features to the next, 1 KB from 8 contraction rows to the next.
constexpr uint32_t kIdescMn = kIdesc | (1u << 16);
constexpr uint64_t kMnBlock = (uint64_t)(KPS * 64 * 128 >> 4);
static_assert(BNH == KPS * 64, "one box for both orders of the features");

// Key window: an element is marked when its sum lies within
// kKeyWindow * max(|sum|, scale) of a bf16 rounding midpoint.  The error of a sum
// follows its partial sums, so scale is the largest of three sizes of theirs: the
// RMS of the token's sums over its half of the tile, the same of the chunks that
// they are made of (a component that every token shares and the row cancels), and
// |x| |w| / sqrt(d) of the element's own token and feature (rows of unequal size).
// With chunked sums the farthest mis-rounded key from its midpoint, over 3.7e8
// keys of independent normal data at d = 256 .. 8192 (none refined, compared with
// float64), lay 2^-20.4 of the first size away, with no trend in d (0.017 % of the
// keys were mis-rounded); 2^-19 keeps a margin of 2.6x.  Of 2.1e6 keys at d = 4096
// with a shared component 10 and 33 times the rest, the first size alone left 176
// and 3820 wrong, and with rows 64 times their neighbours that the tokens cancel
// 261; with all three none is.  (Products whose signs are arranged along the
// contraction within a chunk, so that every chunk cancels by itself, can err by
// more: no bound short of |x| |w| holds for them, and that marks a third of the
// keys.)  The two further sizes cost a build of 32768 tokens about 45 us here, 22 in
// the recomputation and 6 for the norms, of 3410.  One accumulator over the whole
// contraction needs 2^-15 and marks 5 % instead of 0.5: at 32768 tokens, d = 4096
// their recomputation took 11.0 ms of a 17.5 ms build, now 0.87 ms.
constexpr float kKeyWindow = 1.0f / 524288.0f;   // 2^-19

__device__ __forceinline__ uint32_t cta_rank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ void tma_load_pair(uint32_t dst, const CUtensorMap* map, uint32_t bar,
                                              int x, int y, int z) {
  asm volatile(
      "cp.async.bulk.tensor.3d.cta_group::2.shared::cluster.global.tile.mbarrier::complete_tx::bytes"
      " [%0], [%1, {%3, %4, %5}], [%2];" ::"r"(dst),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(bar), "r"(x), "r"(y), "r"(z)
      : "memory");
}
__device__ __forceinline__ void umma_pair(uint32_t tmem_d, uint64_t adesc, uint64_t bdesc,
                                          uint32_t idesc, uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(tmem_d),
      "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate)
      : "memory");
}
// Completion of the MMAs issued so far, signalled to the barrier at this
// offset in both CTAs of the pair.
__device__ __forceinline__ void commit_pair(uint64_t* bar) {
  asm volatile(
      "tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64"
      " [%0], %1;" ::"r"(smem_u32(bar)), "h"((unsigned short)3)
      : "memory");
}
__device__ __forceinline__ void arrive_cluster(uint32_t caddr) {
  asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(caddr) : "memory");
}
__device__ __forceinline__ uint32_t try_wait_cluster(uint64_t* bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n}\n"
      : "=r"(ok)
      : "r"(smem_u32(bar)), "r"(parity)
      : "memory");
  return ok;
}
// The same without suspending the thread while the phase is incomplete.
__device__ __forceinline__ uint32_t test_wait_cluster(uint64_t* bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.test_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n}\n"
      : "=r"(ok)
      : "r"(smem_u32(bar)), "r"(parity)
      : "memory");
  return ok;
}
// mbar_wait with cluster-scope acquire: the barrier is signalled by the peer.
static __device__ __noinline__ bool wait_cluster(uint64_t* bar, uint32_t parity,
                                                 volatile int* abort_flag, uint64_t limit_ns) {
  if (test_wait_cluster(bar, parity)) return true;
  const uint64_t t0 = globaltimer_ns();
  while (true) {
    if (limit_ns < kSuspendNs ? test_wait_cluster(bar, parity) : try_wait_cluster(bar, parity)) return true;
    if (abort_flag != nullptr && *abort_flag) return false;
    if (globaltimer_ns() - t0 > limit_ns) return false;
  }
}
// 16 consecutive fp32 accumulator columns of this thread's lane.
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, float (&v)[16]) {
  uint32_t r[16];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
      "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
        "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]),
        "=r"(r[14]), "=r"(r[15])
      : "r"(taddr));
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
  for (int i = 0; i < 16; ++i) v[i] = __uint_as_float(r[i]);
}
__device__ __forceinline__ uint32_t ld_dsmem_u32(uint32_t caddr) {
  uint32_t v;
  asm volatile("ld.shared::cluster.u32 %0, [%1];" : "=r"(v) : "r"(caddr) : "memory");
  return v;
}
__device__ __forceinline__ uint32_t pack_bf16(float a, float b) {
  const __nv_bfloat162 p = __floats2bfloat162_rn(a, b);
  return *reinterpret_cast<const uint32_t*>(&p);
}

// The midpoint of the two bf16 values around a finite fp32 value is its upper
// 16 bits followed by 0x8000.  An element whose window reaches the spacing of
// the bf16 values around it (a sum far below the scale) is always marked, as
// is one that is not finite.
__device__ __forceinline__ bool near_midpoint(float acc, float scale) {
  const float mid = __uint_as_float((__float_as_uint(acc) & 0xFFFF0000u) | 0x8000u);
  const float window = kKeyWindow * fmaxf(fabsf(acc), scale);
  return !(fabsf(acc - mid) > window && fabsf(acc) * 0.001953125f >= window);
}

// One tile of the output: where it lies.
struct Tile {
  int part, m0, n_cols, row0;
};
__device__ __forceinline__ Tile tile_at(const PairGemm& a, int t) {
  // bands of kBandRows row tiles; within a band consecutive tiles walk the
  // rows, so that the pairs of a wave share both operands through L2
  const int per_band = kBandRows * a.feat_tiles;
  const int band = t / per_band;
  const int rows_here = min(kBandRows, a.row_tiles - band * kBandRows);
  const int local = t - band * per_band;
  const int ft = local / rows_here;
  Tile r;
  r.row0 = (band * kBandRows + local % rows_here) * 2 * BM;
  r.part = ft < a.tile_end[0] ? 0 : ft < a.tile_end[1] ? 1 : 2;
  r.m0 = (r.part ? ft - a.tile_end[r.part - 1] : ft) * BN;
  r.n_cols = min(BN, a.cols[r.part] - r.m0);
  return r;
}

// KEYS: part 0 is the keys (rounded, near-midpoint elements marked); HILO: part
// 0's sums are stored as hi = bf16(sum) to out[0] and bf16(sum - hi) to out_lo,
// and its feature matrix lies as [K, cols].  The
// other parts are rounded sums.  Part 0 reads the tokens of tmR0, the others
// those of tmR1.
template <bool KEYS, bool HILO>
__global__ void __launch_bounds__(kThreads, 1) __cluster_dims__(2, 1, 1)
    pair_gemm_kernel(const __grid_constant__ CUtensorMap tmF0,
                     const __grid_constant__ CUtensorMap tmF1,
                     const __grid_constant__ CUtensorMap tmF2,
                     const __grid_constant__ CUtensorMap tmR0,
                     const __grid_constant__ CUtensorMap tmR1, const __grid_constant__ PairGemm a) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);
  uint8_t* staging = smem + kStages * kStageBytes;
  uint64_t* full = reinterpret_cast<uint64_t*>(staging + kEpiWarps * kWarpStage);
  uint64_t* empty = full + kStages;
  uint64_t* tfull = empty + kStages;
  uint64_t* tempty = tfull + 2;
  uint64_t* drain = tempty + 2;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(drain + 1);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t rank = cta_rank();
  const int pairs = (int)gridDim.x >> 1, pid = (int)blockIdx.x >> 1;
  if (threadIdx.x == 0) {
    for (int i = 0; i < kStages; ++i) {
      mbar_init(&full[i], 1);
      mbar_init(&empty[i], 1);
    }
    for (int i = 0; i < 2; ++i) {
      mbar_init(&tfull[i], 1);
      mbar_init(&tempty[i], 2 * kEpiWarps);
    }
    mbar_init(drain, 1);
    *abort_flag = 0;
    fence_mbar_init();
    prefetch_tmap(&tmF0);
    prefetch_tmap(&tmR0);
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     smem_u32(tmem_slot)), "r"(kTmemCols) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  cluster_sync();                        // the peer's barriers are initialised
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;
  pdl_wait();
  pdl_trigger();
  const int tiles = a.feat_tiles * a.row_tiles;
  const int su_total = (a.k_blocks + KPS - 1) / KPS;   // past the last k-block the maps fill zeros

  if (warp == 0 && lane < 2) {
    // ---- TMA producers: lane 0 features, lane 1 tokens.  The leader's lane 0
    // posts the bytes of both CTAs on its full barrier.
    int i = 0;
    bool go = true;
    for (int t = pid; go && t < tiles; t += pairs) {
      const Tile ti = tile_at(a, t);
      const CUtensorMap* map = lane == 1 ? (ti.part ? &tmR1 : &tmR0)
                                         : ti.part == 0 ? &tmF0 : ti.part == 1 ? &tmF1 : &tmF2;
      const int y = lane == 1 ? ti.row0 + (int)rank * BM : ti.m0 + (int)rank * BNH;
      for (int su = 0; su < su_total; ++su, ++i) {
        const int st = i % kStages;
        if (i >= kStages &&
            !wait_cluster(&empty[st], ((uint32_t)(i / kStages) & 1u) ^ 1u, abort_flag, a.wait_ns)) {
          *abort_flag = 1;
          go = false;
          break;
        }
        if (lane == 0 && rank == 0) mbar_expect_tx(&full[st], 2u * kStageBytes);
        const uint32_t dst = smem_u32(smem + st * kStageBytes) + (lane == 1 ? 0u : (uint32_t)(KPS * kSmemRows));
        if (HILO && lane == 0 && ti.part == 0)
          tma_load_pair(dst, map, map_dsmem(smem_u32(&full[st]), 0), 0, su * KPS * 64, y / 64);
        else
          tma_load_pair(dst, map, map_dsmem(smem_u32(&full[st]), 0), 0, y, su * KPS);
      }
    }
    // the last stages' releases have arrived here before the CTA may leave
    if (go && lane == 0)
      for (int j = i > kStages ? i - kStages : 0; j < i; ++j)
        if (!wait_cluster(&empty[j % kStages], (uint32_t)(j / kStages) & 1u, abort_flag, a.wait_ns)) {
          *abort_flag = 1;
          break;
        }
  } else if (warp == 1 && rank == 0) {
    // ---- MMA issuer of the pair: the warp runs the loop converged (stage
    // addresses and descriptors in uniform registers), one elected lane issues
    const uint64_t desc0 = sw128_desc(smem_u32(smem));
    uint32_t st = 0, ph = 0;
    int c = 0;
    bool go = true;
    for (int t = pid; go && t < tiles; t += pairs) {
      const int part = tile_at(a, t).part;
      const int chunk = a.chunk[part];
      const bool mn = HILO && part == 0;
      int su0 = 0;
      for (int len = a.chunk0[part]; go && su0 < su_total; su0 += len, len = chunk, ++c) {
        const int buf = c & 1;
        const uint32_t d = tmem_base + (uint32_t)(buf * BN);
        if (c >= 2 &&
            !__all_sync(0xffffffffu, wait_cluster(&tempty[buf], ((uint32_t)(c >> 1) & 1u) ^ 1u,
                                                  abort_flag, a.wait_ns))) {
          *abort_flag = 1;
          go = false;
          break;
        }
        tc_fence_after();
        const int su1 = min(su0 + len, su_total);
        for (int su = su0; su < su1; ++su) {
          if (!__all_sync(0xffffffffu, wait_cluster(&full[st], ph, abort_flag, a.wait_ns))) {
            *abort_flag = 1;
            go = false;
            break;
          }
          if (elect_one()) {
            // descriptor start addresses are in units of 16 bytes
            const uint64_t ad = desc0 + (uint64_t)(st * (uint32_t)(kStageBytes >> 4));
            const uint64_t bd = ad + (uint64_t)((KPS * kSmemRows) >> 4) +
                                (mn ? (kMnBlock - 1) << 16 : 0);   // its leading-dimension offset
            const uint32_t idesc = mn ? kIdescMn : kIdesc;
            // per 16 elements of the contraction: 32 bytes of a K-major row,
            // 16 rows of an MN-major block
#pragma unroll
            for (int j = 0; j < KPS; ++j)
#pragma unroll
              for (int k = 0; k < 4; ++k)
                umma_pair(d, ad + (uint64_t)((j * kSmemRows >> 4) + 2 * k),
                          bd + (uint64_t)(mn ? (4 * j + k) * (16 * 128 >> 4)
                                             : (j * kSmemFeat >> 4) + 2 * k),
                          idesc, (su > su0 || j > 0 || k > 0) ? 1u : 0u);
            commit_pair(&empty[st]);
          }
          __syncwarp();
          if (++st == (uint32_t)kStages) {
            st = 0;
            ph ^= 1u;
          }
        }
        if (go && elect_one()) commit_pair(&tfull[buf]);
        __syncwarp();
      }
    }
  } else if (warp >= 2) {
    // ---- epilogue ----
    const int quarter = warp & 3, half = (warp - 2) >> 2;
    uint8_t* stg = staging + (warp - 2) * kWarpStage;
    const uint32_t lanes = tmem_base + ((uint32_t)(quarter * 32) << 16) + (uint32_t)(half * BNH);
    int c = 0;
    bool go = true;
    for (int t = pid; go && t < tiles; t += pairs) {
      const Tile ti = tile_at(a, t);
      float acc[BNH];
#pragma unroll
      for (int j = 0; j < BNH; ++j) acc[j] = 0.0f;
      float cs[2] = {};                          // keys: squares of every fourth column's chunk sums
      const int chunk = a.chunk[ti.part];
      int su0 = 0;
      for (int len = a.chunk0[ti.part]; su0 < su_total; su0 += len, len = chunk, ++c) {
        const int buf = c & 1;
        const bool ok = wait_cluster(&tfull[buf], (uint32_t)(c >> 1) & 1u, abort_flag, a.wait_ns);
        if (!__all_sync(0xffffffffu, ok)) {      // tcgen05.ld below is a .sync.aligned instruction
          *abort_flag = 1;
          go = false;
          break;
        }
        tc_fence_after();
        const uint32_t src = lanes + (uint32_t)(buf * BN);
#pragma unroll
        for (int q = 0; q < BNH / 16; ++q) {
          float v[16];
          tmem_ld16(src + (uint32_t)(16 * q), v);
#pragma unroll
          for (int j = 0; j < 16; ++j) acc[16 * q + j] += v[j];
          if (KEYS) {
#pragma unroll
            for (int j = 0; j < 16; j += 4) cs[(j >> 2) & 1] = fmaf(v[j], v[j], cs[(j >> 2) & 1]);
          }
        }
        tc_fence_before();
        __syncwarp();
        if (lane == 0) arrive_cluster(map_dsmem(smem_u32(&tempty[buf]), 0));
      }
      if (!go) break;
      const int row = ti.row0 + (int)rank * BM + quarter * 32;   // first token of this warp
      const int cols = min(BNH, ti.n_cols - half * BNH);         // valid columns of this half
      if (cols <= 0) continue;                                   // uniform in the warp
      const int col0 = ti.m0 + half * BNH;
      uint32_t need[BNH / 32];
      if (KEYS && ti.part == 0) {
        float ss = 0.0f;                       // columns past the matrix are zeros
#pragma unroll
        for (int j = 0; j < BNH; ++j) ss = fmaf(acc[j], acc[j], ss);
        const float scale = sqrtf(fmaxf(ss, 4.0f * (cs[0] + cs[1])) / (float)cols);
        const float rms = row + lane < a.rows ? a.row_rms[row + lane] : 0.0f;
#pragma unroll
        for (int q = 0; q < BNH / 32; ++q) {
          uint32_t bits = 0u;
          if (row + lane < a.rows && 32 * q < cols) {
#pragma unroll
            for (int j = 0; j < 32; j += 4) {
              const float4 w = __ldg(reinterpret_cast<const float4*>(a.feat_norm + col0 + 32 * q + j));
              if (near_midpoint(acc[32 * q + j], fmaxf(scale, rms * w.x))) bits |= 1u << j;
              if (near_midpoint(acc[32 * q + j + 1], fmaxf(scale, rms * w.y))) bits |= 2u << j;
              if (near_midpoint(acc[32 * q + j + 2], fmaxf(scale, rms * w.z))) bits |= 4u << j;
              if (near_midpoint(acc[32 * q + j + 3], fmaxf(scale, rms * w.w))) bits |= 8u << j;
            }
          }
          need[q] = bits;
        }
        // every word of the token's row is written, 8 bytes at a time (columns
        // come in multiples of 64)
        if (row + lane < a.rows) {
          uint32_t* m = a.fix_bits + (long long)(row + lane) * (a.ldc[0] >> 5) + (col0 >> 5);
#pragma unroll
          for (int q = 0; q < BNH / 32; q += 2)
            if (32 * q < cols) *reinterpret_cast<uint2*>(m + q) = make_uint2(need[q], need[q + 1]);
        }
      }
      // 32 rows x 64 columns at a time through the warp's staging (16-byte
      // chunks swizzled by row: conflict-free both ways), written out 128
      // bytes of a row per eight lanes
      const bool hilo = HILO && ti.part == 0;
      const long long ldc = a.ldc[ti.part];
#pragma unroll
      for (int g = 0; g < BNH / 64; ++g) {
        if (64 * g >= cols) break;
#pragma unroll
        for (int w = 0; w < (HILO ? 2 : 1); ++w) {
          if (w == 1 && !hilo) break;
          __nv_bfloat16* dst = static_cast<__nv_bfloat16*>(w == 0 ? a.out[ti.part] : a.out_lo) +
                               col0 + 64 * g;
#pragma unroll
          for (int ch = 0; ch < 8; ++ch) {
            uint32_t p[4];
#pragma unroll
            for (int e = 0; e < 4; ++e) {
              float& x = acc[64 * g + 8 * ch + 2 * e];
              float& y = acc[64 * g + 8 * ch + 2 * e + 1];
              p[e] = pack_bf16(x, y);
              if (HILO && w == 0 && hilo) {      // what hi leaves, for the second pass
                x -= __uint_as_float(p[e] << 16);
                y -= __uint_as_float(p[e] & 0xFFFF0000u);
              }
            }
            *reinterpret_cast<uint4*>(stg + lane * 128 + ((ch ^ (lane & 7)) << 4)) =
                make_uint4(p[0], p[1], p[2], p[3]);
          }
          __syncwarp();
#pragma unroll
          for (int it = 0; it < 8; ++it) {
            const int r = it * 4 + (lane >> 3), ch = lane & 7;
            const uint4 u = *reinterpret_cast<const uint4*>(stg + r * 128 + ((ch ^ (r & 7)) << 4));
            if (row + r < a.rows)
              *reinterpret_cast<uint4*>(dst + (long long)(row + r) * ldc + 8 * ch) = u;
          }
          __syncwarp();
        }
      }
    }
  }
  __syncwarp();
  // ---- both CTAs' roles have ended ----
  tc_fence_before();
  cluster_sync();
  tc_fence_after();
  const uint32_t mine = smem_u32(const_cast<int*>(abort_flag));
  const bool aborted = *abort_flag != 0 || ld_dsmem_u32(map_dsmem(mine, rank ^ 1u)) != 0u;
  if (aborted) {
    if (threadIdx.x == 0) atomicOr(a.err, kErrTimeout);
    if (rank == 0 && warp == 1 && elect_one()) commit_pair(drain);   // the issuing lane's MMAs
    if (lane == 0) {
      wait_cluster(drain, 0, nullptr, kDefaultWaitLimitNs);
      const uint64_t t0 = globaltimer_ns();          // copies in flight land
      while (globaltimer_ns() - t0 < 2000000ull) {}
    }
    __syncwarp();
  }
  tc_fence_before();
  cluster_sync();                        // no CTA leaves while the peer may still signal it
  tc_fence_after();
  if (warp == 1)
    asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem_base),
                 "r"(kTmemCols) : "memory");
}

// Pairs of this kernel resident on the GPU at once (per device).
template <bool KEYS, bool HILO>
static cudaError_t launch(PairGemm& a, const CUtensorMap* maps, cudaStream_t s) {
  auto kern = pair_gemm_kernel<KEYS, HILO>;
  static int resident[64] = {};
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg = {};
  cfg.blockDim = dim3(kThreads);
  cfg.dynamicSmemBytes = kSmemBytes;
  cfg.stream = s;
  int n = dev < 64 ? resident[dev] : 0;
  if (n == 0) {
    e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemBytes);
    if (e != cudaSuccess) return e;
    cudaLaunchAttribute cl[1];
    cl[0].id = cudaLaunchAttributeClusterDimension;
    cl[0].val.clusterDim.x = 2;
    cl[0].val.clusterDim.y = 1;
    cl[0].val.clusterDim.z = 1;
    cfg.gridDim = dim3(2);
    cfg.attrs = cl;
    cfg.numAttrs = 1;
    e = cudaOccupancyMaxActiveClusters(&n, kern, &cfg);
    if (e != cudaSuccess) return e;
    if (n <= 0) return cudaErrorInvalidConfiguration;
    if (dev < 64) resident[dev] = n;
  }
  const int tiles = a.feat_tiles * a.row_tiles;
  // equal rounds: as many pairs as the tiles of a round need
  const int rounds = (tiles + n - 1) / n;
  cfg.gridDim = dim3(2 * ((tiles + rounds - 1) / rounds));
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kern, maps[0], maps[1], maps[2], maps[3], maps[4], a);
}

}  // namespace pair

cudaError_t launch_pair_gemm(bool keys, PairGemm a, const TmaOperand (&F)[3], const TmaOperand& R0,
                             const TmaOperand& R1, cudaStream_t s) {
  a.feat_tiles = 0;
  CUtensorMap maps[5];                 // F0, F1, F2, R0, R1; absent parts repeat a present one
  const TmaOperand* some = &F[0];
  for (const TmaOperand& f : F)
    if (f.base != nullptr) some = &f;
  for (int i = 0; i < 3; ++i) {
    a.cols[i] = F[i].base != nullptr ? (int)F[i].rows : 0;
    a.feat_tiles += (a.cols[i] + pair::BN - 1) / pair::BN;
    a.tile_end[i] = a.feat_tiles;
    if (!encode_kblock_map(&maps[i], F[i].base != nullptr ? F[i] : *some, pair::BNH, pair::KPS))
      return cudaErrorInvalidValue;
  }
  if (a.rows <= 0 || a.feat_tiles == 0) return cudaSuccess;
  a.k_blocks = (int)(some->cols / 64);
  const int su_total = (a.k_blocks + pair::KPS - 1) / pair::KPS;
  for (int i = 0; i < 3; ++i) {
    const bool chunked = i > 0 || a.rows <= pair::kChunkFoldRows;
    a.chunk[i] = keys ? (i == 0 ? pair::kChunkSu : su_total)
                      : chunked ? std::max(pair::kChunkSu, su_total / pair::kChunks) : su_total;
    a.chunk0[i] = keys ? a.chunk[i] : 2 * a.chunk[i];
  }
  a.row_tiles = (a.rows + 2 * pair::BM - 1) / (2 * pair::BM);
  a.wait_ns = wait_limit_ns();
  const TmaOperand& r0 = R0.base != nullptr ? R0 : R1;
  const TmaOperand& r1 = R1.base != nullptr ? R1 : R0;
  if (!encode_kblock_map(&maps[3], r0, pair::BM, pair::KPS) ||
      !encode_kblock_map(&maps[4], r1, pair::BM, pair::KPS))
    return cudaErrorInvalidValue;
  return keys ? pair::launch<true, false>(a, maps, s) : pair::launch<false, true>(a, maps, s);
}

}  // namespace fovea
