// C ABI of libfovea (include/fovea.h): argument checks, the memory handle,
// the workspace layout, and the launch sequence of one draft step.
#include <cstdarg>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <algorithm>
#include <mutex>
#include <string>
#include <vector>

#include <atomic>

#include "common.cuh"

using namespace fovea;

// ---------------------------------------------------------------------------
// Errors
// ---------------------------------------------------------------------------
static thread_local std::string g_last_error;

static fovea_status fail(fovea_status st, const char* fmt, ...) {
  char buf[512];
  va_list ap;
  va_start(ap, fmt);
  vsnprintf(buf, sizeof(buf), fmt, ap);
  va_end(ap);
  g_last_error = buf;
  return st;
}
namespace fovea {
// Records the message fovea_last_error() returns (for other translation units).
fovea_status report_error(fovea_status st, const char* msg) {
  g_last_error = msg;
  return st;
}
}  // namespace fovea

static fovea_status cuda_fail(cudaError_t e, const char* where) {
  return fail(FOVEA_ERR_CUDA, "%s: %s", where, cudaGetErrorString(e));
}
#define FOVEA_CUDA(call, where)                   \
  do {                                            \
    cudaError_t e_ = (call);                      \
    if (e_ != cudaSuccess) return cuda_fail(e_, where); \
  } while (0)

// ---------------------------------------------------------------------------
// Per-launch timing (CUDA events on the launching stream)
// ---------------------------------------------------------------------------
namespace {
struct TimingRec {
  const char* name;
  cudaEvent_t start, stop;
};
std::mutex g_tmu;
bool g_timing = false;
std::vector<TimingRec> g_recs;
std::vector<cudaEvent_t> g_free_events;

cudaEvent_t take_event() {
  if (!g_free_events.empty()) {
    cudaEvent_t e = g_free_events.back();
    g_free_events.pop_back();
    return e;
  }
  cudaEvent_t e = nullptr;
  cudaEventCreate(&e);
  return e;
}

bool capturing(cudaStream_t s) {
  cudaStreamCaptureStatus st = cudaStreamCaptureStatusNone;
  cudaStreamIsCapturing(s, &st);
  return st != cudaStreamCaptureStatusNone;
}

// Records start/stop events around one launch when timing is enabled.  While
// the stream is being captured into a CUDA graph the records become external
// event nodes of the graph, re-recorded by every replay.
struct KernelTimer {
  const char* name;
  cudaStream_t s;
  bool on, graph;
  KernelTimer(const char* n, cudaStream_t st) : name(n), s(st), on(false), graph(false) {
    std::lock_guard<std::mutex> lk(g_tmu);
    if (!g_timing) return;
    graph = capturing(s);
    TimingRec r{name, take_event(), take_event()};
    if (graph) cudaEventRecordWithFlags(r.start, s, cudaEventRecordExternal);
    else cudaEventRecord(r.start, s);
    g_recs.push_back(r);
    on = true;
  }
  ~KernelTimer() {
    if (!on) return;
    std::lock_guard<std::mutex> lk(g_tmu);
    for (auto it = g_recs.rbegin(); it != g_recs.rend(); ++it)
      if (it->name == name) {
        if (graph) cudaEventRecordWithFlags(it->stop, s, cudaEventRecordExternal);
        else cudaEventRecord(it->stop, s);
        break;
      }
  }
};
}  // namespace

// ---------------------------------------------------------------------------
// Memory handle
// ---------------------------------------------------------------------------
struct MemoryBlock {                 // a cudaMalloc allocation
  void* ptr = nullptr;
  size_t bytes = 0;
};
constexpr size_t kBlockGrain = 64 << 10;

struct fovea_memory {
  int device = 0;
  MemoryBlock block;                 // what the buffers below lie in
  int B = 0, M_max = 0, d = 0, dtype = 0;
  int total = 0;
  std::vector<int32_t> counts;       // valid entries per image (host)
  std::vector<int64_t> offsets;      // first entry of each image, B + 1 (host)
  void* keys = nullptr;              // [total, d]
  void* values = nullptr;            // [total, d]
  int32_t* orig_index = nullptr;     // [total]
  // bf16: the values projected through the r-half of the first fusion layer,
  // p_i = [W_f1 ; W_g1][:, d:2d] u_i  ([total, 2H]), and the weights they
  // were built with (a call with other W_f1 / W_g1 pointers or H does not
  // use them)
  void* proj = nullptr;
  // the projected values transposed per image, [B, 2H, proj_ld] with
  // proj_ld = max valid count rounded up to 64 (zero-padded): the feature
  // operand of the weighted-sum GEMM over dense selection weights
  void* projT = nullptr;
  int proj_ld = 0;
  const void* proj_wf1 = nullptr;
  const void* proj_wg1 = nullptr;
  int proj_h = 0;
  // bf16: the keys folded through the query projection, kappa_i = W_Q^T k_i,
  // as a hi / lo pair of bf16 values ([total, 2d]: row i holds kappa_hi then
  // kappa_lo = bf16(kappa - kappa_hi), about 16 significant bits), and the
  // W_Q they were built with: q . k_i = x . kappa_i, so a call with that W_Q
  // scores x = LN(h) + E_dep against them directly
  void* folded = nullptr;
  const void* fold_wq = nullptr;
};

// Caps up to this select and gather in one kernel (two CTAs a row at most);
// above it the gathers have a kernel of their own over the whole GPU.  Step of
// 64 rows, d = 4096, one kernel against two: K = 128 27.6 / 25.9 us, K = 256
// 31.3 / 28.5, with the readout 42.5 / 38.3; the paper's setting behind its
// depth gate 43.9 / 30.9.  At K = 64 two kernels are 0.7 us faster on the GPU
// (25.6 / 24.9), less than the host pays for a launch, so that line holds up to
// a row per SM; 300 rows without a readout gain 46.0 / 40.7.
constexpr int kFuseSelectMaxK = 64;

static size_t esize(int dtype) { return dtype == FOVEA_BF16 ? 2 : 4; }
static bool aligned16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }
static size_t align_up(size_t x, size_t a) { return (x + a - 1) / a * a; }

static fovea_status check_dims(const fovea_params* p) {
  if (p == nullptr) return fail(FOVEA_ERR_INVALID_ARG, "params is NULL");
  if (p->dtype != FOVEA_BF16 && p->dtype != FOVEA_FP32)
    return fail(FOVEA_ERR_INVALID_ARG, "dtype %d is neither FOVEA_BF16 nor FOVEA_FP32", p->dtype);
  if (p->d_model <= 0 || p->d_model % 64 != 0)
    return fail(FOVEA_ERR_INVALID_ARG, "d_model %d must be a positive multiple of 64", p->d_model);
  if (p->d_model > FOVEA_MAX_D)
    return fail(FOVEA_ERR_UNSUPPORTED, "d_model %d exceeds %d", p->d_model, FOVEA_MAX_D);
  if (!(p->ln_eps > 0.0f) || !(p->rms_eps > 0.0f))
    return fail(FOVEA_ERR_INVALID_ARG, "ln_eps and rms_eps must be > 0");
  return FOVEA_OK;
}

#define NEED_PTR(ptr, name)                                                             \
  do {                                                                                  \
    if ((ptr) == nullptr) return fail(FOVEA_ERR_INVALID_ARG, "%s is NULL", name);       \
    if (!aligned16(ptr)) return fail(FOVEA_ERR_INVALID_ARG, "%s is not 16-byte aligned", name); \
  } while (0)

static fovea_status check_step_params(const fovea_params* p) {
  fovea_status st = check_dims(p);
  if (st != FOVEA_OK) return st;
  if (p->mlp_hidden <= 0 || p->mlp_hidden % 128 != 0)
    return fail(FOVEA_ERR_INVALID_ARG, "mlp_hidden %d must be a positive multiple of 128",
                p->mlp_hidden);
  if (p->mlp_hidden > FOVEA_MAX_H)
    return fail(FOVEA_ERR_UNSUPPORTED, "mlp_hidden %d exceeds %d", p->mlp_hidden, FOVEA_MAX_H);
  if (p->max_depth < 0) return fail(FOVEA_ERR_INVALID_ARG, "max_depth %d < 0", p->max_depth);
  NEED_PTR(p->ln_h_gamma, "ln_h_gamma");
  NEED_PTR(p->ln_h_beta, "ln_h_beta");
  NEED_PTR(p->E_dep, "E_dep");
  NEED_PTR(p->W_Q, "W_Q");
  NEED_PTR(p->W_f1, "W_f1");
  NEED_PTR(p->b_f1, "b_f1");
  NEED_PTR(p->W_f2, "W_f2");
  NEED_PTR(p->b_f2, "b_f2");
  NEED_PTR(p->W_g1, "W_g1");
  NEED_PTR(p->b_g1, "b_g1");
  NEED_PTR(p->w_g2, "w_g2");
  if (p->b_g2 == nullptr) return fail(FOVEA_ERR_INVALID_ARG, "b_g2 is NULL");
  NEED_PTR(p->rms_gamma, "rms_gamma");
  return FOVEA_OK;
}

// ---------------------------------------------------------------------------
// Device memory.  cudaMalloc and cudaFree cost 30 - 180 us each, ten to twelve of
// them 0.8 ms of a one-image build whose kernels take 0.2 ms, so both kinds of
// memory are kept for the next build, per device:
//   * a handle's buffers lie in one cudaMalloc block (so that they can be exported
//     to other processes and read by peers), rounded up by an eighth at most; a
//     freed handle's block serves later handles on any stream, because free_memory
//     waits for the device first;
//   * a build's temporaries come from a stream-ordered pool, whose reuse the
//     driver orders between streams and threads.  (The pool's own release
//     threshold counts the bytes in use too, so it is off; pool_trim keeps the
//     bound.)
// At most kBlocksKeep + kPoolKeep bytes (2 GiB, under 1 % of the device) are kept
// that nothing uses, and all of it is given back when the device's last handle
// goes: a program that frees each memory before it builds the next allocates anew.
// ---------------------------------------------------------------------------
namespace {
constexpr unsigned long long kBlocksKeep = 1536ull << 20, kPoolKeep = 512ull << 20;
constexpr int kMaxDevices = 64;
struct DeviceMemory {
  cudaMemPool_t pool = nullptr;
  int users = 0;                     // live handles and builds under way
  std::vector<MemoryBlock> unused;   // oldest first
  size_t unused_bytes = 0;
  std::vector<MemoryBlock> parked;   // freed without a wait for the device: not to be used yet
};
std::mutex g_mem_mu;
DeviceMemory g_mem[kMaxDevices];

// One more user of device `dev` and its pool, created at its first use.
cudaError_t mem_enter(int dev, cudaMemPool_t* out) {
  if (dev < 0 || dev >= kMaxDevices) return cudaErrorInvalidDevice;
  std::lock_guard<std::mutex> lk(g_mem_mu);
  DeviceMemory& p = g_mem[dev];
  if (p.pool == nullptr) {
    cudaMemPoolProps props = {};
    props.allocType = cudaMemAllocationTypePinned;
    props.location.type = cudaMemLocationTypeDevice;
    props.location.id = dev;
    cudaMemPool_t pool = nullptr;
    cudaError_t e = cudaMemPoolCreate(&pool, &props);
    if (e != cudaSuccess) return e;
    unsigned long long never = ~0ull;
    e = cudaMemPoolSetAttribute(pool, cudaMemPoolAttrReleaseThreshold, &never);
    if (e != cudaSuccess) {
      cudaMemPoolDestroy(pool);
      return e;
    }
    p.pool = pool;
  }
  ++p.users;
  *out = p.pool;
  return cudaSuccess;
}
// Gives back what the pool holds beyond kPoolKeep unused bytes.
void pool_trim(cudaMemPool_t pool) {
  unsigned long long used = 0, held = 0;
  if (cudaMemPoolGetAttribute(pool, cudaMemPoolAttrUsedMemCurrent, &used) == cudaSuccess &&
      cudaMemPoolGetAttribute(pool, cudaMemPoolAttrReservedMemCurrent, &held) == cudaSuccess &&
      held > used + kPoolKeep)
    cudaMemPoolTrimTo(pool, used + kPoolKeep);
}
// Gives back unused blocks, the oldest first, down to `keep` bytes.  (Nothing on
// the device uses them, so cudaFree's wait is none.)
void blocks_trim(DeviceMemory& p, size_t keep) {
  size_t n = 0;
  while (n < p.unused.size() && p.unused_bytes > keep) {
    if (cudaFree(p.unused[n].ptr) != cudaSuccess) {      // not now (a capture): stays
      cudaGetLastError();
      break;
    }
    p.unused_bytes -= p.unused[n++].bytes;
  }
  p.unused.erase(p.unused.begin(), p.unused.begin() + n);
}
// The block of a handle that goes.  waited: the device has finished all work that
// was enqueued when it was let go (and so with the parked ones); otherwise it is
// kept aside until a wait has succeeded.  One user less; the last one returns
// everything.
void mem_leave(int dev, const MemoryBlock& block, bool waited) {
  std::lock_guard<std::mutex> lk(g_mem_mu);
  DeviceMemory& p = g_mem[dev];
  if (block.ptr != nullptr) p.parked.push_back(block);
  if (waited) {
    for (const MemoryBlock& b : p.parked) {
      p.unused.push_back(b);
      p.unused_bytes += b.bytes;
    }
    p.parked.clear();
  }
  const bool last = --p.users == 0;
  blocks_trim(p, last ? 0 : kBlocksKeep);
  if (last) cudaMemPoolTrimTo(p.pool, 0);
  else pool_trim(p.pool);
}
}  // namespace

static fovea_status alloc_failed(const char* what, size_t bytes, cudaError_t e) {
  cudaGetLastError();
  return fail(FOVEA_ERR_OOM, "allocation of %s (%zu bytes): %s", what, bytes, cudaGetErrorString(e));
}
static bool alloc_fault() {
  const char* fault = getenv("FOVEA_FAULT_ALLOC");
  return fault != nullptr && fault[0] == '1';
}

// A temporary of a build of handle m, from the pool.
static fovea_status alloc_temp(void** ptr, size_t bytes, const char* what, const fovea_memory* m,
                               cudaMemPool_t pool, cudaStream_t s) {
  *ptr = nullptr;
  if (bytes == 0) return FOVEA_OK;
  cudaError_t e = cudaMallocFromPoolAsync(ptr, bytes, pool, s);
  if (e == cudaErrorMemoryAllocation) {                  // make room, once
    cudaGetLastError();
    std::lock_guard<std::mutex> lk(g_mem_mu);
    blocks_trim(g_mem[m->device], 0);
    e = cudaMallocFromPoolAsync(ptr, bytes, pool, s);
  }
  if (e == cudaSuccess) return FOVEA_OK;
  *ptr = nullptr;
  return alloc_failed(what, bytes, e);
}

// The block of handle m: an unused one that it fills to four fifths at least, or a
// new one.
static fovea_status alloc_block(size_t bytes, fovea_memory* m) {
  std::lock_guard<std::mutex> lk(g_mem_mu);
  DeviceMemory& p = g_mem[m->device];
  size_t best = p.unused.size();
  for (size_t i = 0; i < p.unused.size(); ++i)
    if (p.unused[i].bytes >= bytes && p.unused[i].bytes / 5 * 4 <= align_up(bytes, kBlockGrain) &&
        (best == p.unused.size() || p.unused[i].bytes < p.unused[best].bytes))
      best = i;
  MemoryBlock b;
  if (best < p.unused.size()) {
    b = p.unused[best];
    p.unused.erase(p.unused.begin() + best);
    p.unused_bytes -= b.bytes;
  } else {
    size_t grain = kBlockGrain;
    while (grain * 16 < bytes) grain *= 2;
    b.bytes = align_up(bytes, grain);
    cudaError_t e = cudaMalloc(&b.ptr, b.bytes);
    if (e == cudaErrorMemoryAllocation && p.unused_bytes > 0) {   // make room, once
      cudaGetLastError();
      blocks_trim(p, 0);
      cudaMemPoolTrimTo(p.pool, 0);
      e = cudaMalloc(&b.ptr, b.bytes);
    }
    if (e == cudaErrorMemoryAllocation && b.bytes > bytes) {
      cudaGetLastError();
      b.bytes = bytes;
      e = cudaMalloc(&b.ptr, b.bytes);
    }
    if (e != cudaSuccess) return alloc_failed("the handle's buffers", bytes, e);
  }
  m->block = b;
  return FOVEA_OK;
}

// Frees a handle.  Like cudaFree, it waits for the device first, so work still
// enqueued when the caller lets go of the handle finishes on its memory.  Where
// the wait is not allowed (a stream of the device is being captured), the memory
// is set aside until a later wait.
static void free_memory(fovea_memory* m) {
  if (m == nullptr) return;
  int cur = -1;
  cudaGetDevice(&cur);
  if (cur != m->device) cudaSetDevice(m->device);
  const char* fault = getenv("FOVEA_FAULT_WAIT");
  const bool waited = !(fault != nullptr && fault[0] == '1') && cudaDeviceSynchronize() == cudaSuccess;
  if (!waited) cudaGetLastError();
  mem_leave(m->device, m->block, waited);
  if (cur >= 0 && cur != m->device) cudaSetDevice(cur);
  delete m;
}

// The bf16 path runs every GEMM on tcgen05 tensor cores; fp32 runs SIMT.
static cudaError_t run_gemm(int dtype, int epi, const GemmArgs& a, const TmaOperand& A0,
                            const TmaOperand& A1, const TmaOperand& B0, const TmaOperand& B1,
                            int max_m, int max_n, cudaStream_t s) {
  if (dtype == FOVEA_BF16) return launch_gemm_tc(epi, a, A0, A1, B0, B1, max_m, max_n, s);
  return launch_gemm_simt(epi, a, max_m, max_n, s);
}

static void init_args(GemmArgs& a) {
  memset(&a, 0, sizeof(a));
  a.a_split = 0x7fffffff;
  a.a_split2 = 0x7fffffff;
  a.epi_split = 0x7fffffff;
  a.scale = 1.0f;
}

extern "C" {

FOVEA_API const char* fovea_last_error(void) { return g_last_error.c_str(); }

FOVEA_API int fovea_version(void) { return 200; }

FOVEA_API fovea_status fovea_build_memory(const fovea_params* p, const void* v,
                                          const uint8_t* mask, int B, int M_max, void* stream,
                                          fovea_memory** out) {
  g_last_error.clear();
  fovea_status st = check_dims(p);
  if (st != FOVEA_OK) return st;
  if (out == nullptr) return fail(FOVEA_ERR_INVALID_ARG, "out is NULL");
  if (B < 1) return fail(FOVEA_ERR_INVALID_ARG, "B = %d must be >= 1", B);
  if (B > FOVEA_MAX_SEQ) return fail(FOVEA_ERR_UNSUPPORTED, "B = %d exceeds %d", B, FOVEA_MAX_SEQ);
  if (M_max < 0) return fail(FOVEA_ERR_INVALID_ARG, "M_max = %d < 0", M_max);
  if (mask == nullptr && M_max > FOVEA_MAX_ENTRIES)
    return fail(FOVEA_ERR_UNSUPPORTED, "M_max = %d valid entries exceed %d per image", M_max,
                FOVEA_MAX_ENTRIES);
  if ((long long)B * M_max >= (1ll << 31))
    return fail(FOVEA_ERR_UNSUPPORTED, "B * M_max exceeds 2^31 entries");
  if (M_max > 0) NEED_PTR(v, "v");
  NEED_PTR(p->ln_v_gamma, "ln_v_gamma");
  NEED_PTR(p->ln_v_beta, "ln_v_beta");
  NEED_PTR(p->W_K, "W_K");
  NEED_PTR(p->W_U, "W_U");
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  const int d = p->d_model;
  const size_t es = esize(p->dtype);

  if (capturing(s))
    return fail(FOVEA_ERR_CUDA, "fovea_build_memory synchronises: the stream is being captured");
  if (alloc_fault())
    return fail(FOVEA_ERR_OOM, "allocation of build scratch failed (FOVEA_FAULT_ALLOC=1)");
  int dev = 0;
  cudaMemPool_t pool = nullptr;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = mem_enter(dev, &pool);
  if (e != cudaSuccess) {
    cudaGetLastError();
    return fail(FOVEA_ERR_OOM, "device memory pool: %s", cudaGetErrorString(e));
  }

  fovea_memory* m = new fovea_memory();
  m->device = dev;
  m->B = B;
  m->M_max = M_max;
  m->d = d;
  m->dtype = p->dtype;
  // temporaries: error word, valid counts, norms of W_K's rows | LN(v), source
  // rows, marks of the key elements, RMS of the token rows
  void* scratch = nullptr;
  void* temps = nullptr;
  auto run = [&]() -> fovea_status {
    const bool bf = p->dtype == FOVEA_BF16;
    const size_t count_bytes = align_up(B * sizeof(int32_t), 256);
    fovea_status rs = alloc_temp(&scratch, 256 + count_bytes + d * sizeof(float), "build scratch", m, pool, s);
    if (rs != FOVEA_OK) return rs;
    int* errw = static_cast<int*>(scratch);           // error word
    int32_t* d_counts = reinterpret_cast<int32_t*>(static_cast<uint8_t*>(scratch) + 256);
    float* feat_norm = reinterpret_cast<float*>(static_cast<uint8_t*>(scratch) + 256 + count_bytes);
    FOVEA_CUDA(cudaMemsetAsync(scratch, 0, 256, s), "cudaMemsetAsync");
    m->counts.assign(B, M_max);
    cudaError_t err = cudaSuccess;
    if (mask != nullptr && M_max > 0) {
      { KernelTimer t("count_valid", s); err = launch_count_valid(mask, B, M_max, d_counts, s); }
      if (err != cudaSuccess) return cuda_fail(err, "count_valid");
      err = cudaMemcpyAsync(m->counts.data(), d_counts, B * sizeof(int32_t), cudaMemcpyDeviceToHost, s);
      if (err == cudaSuccess) err = cudaStreamSynchronize(s);
      if (err != cudaSuccess) return cuda_fail(err, "reading valid counts");
    }
    m->offsets.assign(B + 1, 0);
    int m_max = 0;
    static thread_local ImageTable itab;
    itab.B = B;
    for (int b = 0; b < B; ++b) {
      if (m->counts[b] > FOVEA_MAX_ENTRIES)
        return fail(FOVEA_ERR_UNSUPPORTED, "image %d has %d valid entries (limit %d)", b,
                    m->counts[b], FOVEA_MAX_ENTRIES);
      itab.off[b] = (int)m->offsets[b];
      itab.m[b] = m->counts[b];
      m_max = std::max(m_max, m->counts[b]);
      m->offsets[b + 1] = m->offsets[b] + m->counts[b];
    }
    m->total = (int)m->offsets[B];
    const int total = m->total;
    if (total == 0) return FOVEA_OK;
    const int H = p->mlp_hidden;
    // bf16 with W_Q given: the folded keys; with the fusion weights given: the
    // projected values and their transpose per image
    const bool fold = bf && p->W_Q != nullptr && aligned16(p->W_Q);
    const bool proj = bf && p->W_f1 != nullptr && p->W_g1 != nullptr && H > 0 && H % 128 == 0 &&
                      H <= FOVEA_MAX_H && aligned16(p->W_f1) && aligned16(p->W_g1);
    const int ld = (m_max + 63) / 64 * 64;
    // bf16: the marks, the RMS of the token rows
    const size_t mark_bytes = align_up((size_t)total * d / 8, 256);
    // the handle's buffers, back to back in one block
    const size_t kv_bytes = align_up((size_t)total * d * es, 256);
    const size_t index_bytes = align_up(total * sizeof(int32_t), 256);
    const size_t fold_bytes = fold ? (size_t)total * 2 * d * 2 : 0;
    const size_t proj_bytes = proj ? align_up((size_t)total * 2 * H * 2, 256) : 0;
    const size_t projT_bytes = proj ? (size_t)B * 2 * H * ld * 2 : 0;
    if ((rs = alloc_block(2 * kv_bytes + index_bytes + fold_bytes + proj_bytes + projT_bytes, m)) != FOVEA_OK ||
        (rs = alloc_temp(&temps, kv_bytes + index_bytes + (bf ? mark_bytes + (size_t)total * 4 : 0),
                         "build temporaries", m, pool, s)) != FOVEA_OK)
      return rs;
    uint8_t* at = static_cast<uint8_t*>(temps);
    auto take = [&](size_t bytes) {
      uint8_t* here = at;
      at += bytes;
      return static_cast<void*>(here);
    };
    void* xv = take(kv_bytes);                      // LN(v)
    int32_t* src_row = static_cast<int32_t*>(take(index_bytes));
    uint32_t* fix = bf ? static_cast<uint32_t*>(take(mark_bytes)) : nullptr;
    float* row_rms = reinterpret_cast<float*>(at);  // bf16
    at = static_cast<uint8_t*>(m->block.ptr);
    m->keys = take(kv_bytes);
    m->values = take(kv_bytes);
    m->orig_index = static_cast<int32_t*>(take(index_bytes));
    if (fold) m->folded = take(fold_bytes);
    if (proj) {
      m->proj = take(proj_bytes);
      m->projT = take(projT_bytes);
    }
    { KernelTimer t("compact", s);
      err = launch_compact(mask, B, M_max, itab, m->orig_index, src_row,
                           RowNorms{p->W_K, d, bf ? feat_norm : nullptr}, s); }
    if (err != cudaSuccess) return cuda_fail(err, "compact");
    { KernelTimer t("ln_v", s);
      err = launch_ln_rows(p->dtype, v, src_row, total, d, p->ln_v_gamma,
                           p->ln_v_beta, p->ln_eps, xv, row_rms, s); }
    if (err != cudaSuccess) return cuda_fail(err, "ln_v");
    if (!bf) {
      static thread_local GemmArgs a;
      init_args(a);
      a.k_total = d;
      a.a_split = d;
      a.b_split = d;
      a.A0 = p->W_K; a.A1 = p->W_U; a.lda0 = d; a.lda1 = d;
      a.B0 = xv; a.B1 = xv; a.ldb0 = d; a.ldb1 = d;
      a.epi_split = d;
      a.out0 = m->keys; a.out1 = m->values; a.ldc = d;
      a.ngroups = 1;
      a.groups[0] = GemmGroup{0, 2 * d, 0, total, 0};
      { KernelTimer t("memory_proj", s);
        err = launch_gemm_simt(kEpiStore, a, 2 * d, total, s); }
      if (err != cudaSuccess) return cuda_fail(err, "memory projection");
    } else {
      PairGemm pg{};
      pg.rows = total;
      pg.err = errw;
      pg.out[0] = m->keys; pg.out[1] = m->values;
      pg.ldc[0] = pg.ldc[1] = d;
      pg.fix_bits = fix;
      pg.row_rms = row_rms;
      pg.feat_norm = feat_norm;
      const TmaOperand none{nullptr, 0, 0, 0}, tokens{xv, total, d, d};
      const TmaOperand kv[3] = {TmaOperand{p->W_K, d, d, d}, TmaOperand{p->W_U, d, d, d}, none};
      { KernelTimer t("memory_proj", s);
        err = launch_pair_gemm(true, pg, kv, tokens, tokens, s); }
      if (err != cudaSuccess) return cuda_fail(err, "memory projection");
      // keys whose fp32 value sat near a bf16 rounding midpoint: exact recompute
      { KernelTimer t("refine_keys", s);
        err = launch_refine_keys(xv, p->W_K, d, pg.fix_bits, total, m->keys, s); }
      if (err != cudaSuccess) return cuda_fail(err, "refine_keys");
      TmaOperand F[3] = {none, none, none};
      if (fold) {
        // kappa_i = W_Q^T k_i, a GEMM of W_Q^T (read along W_Q's rows) with the
        // stored keys, kept as the hi / lo pair of its fp32 accumulator (no bf16
        // rounding of the query map)
        F[0] = TmaOperand{p->W_Q, d, d, d};
        pg.out[0] = m->folded;
        pg.out_lo = static_cast<__nv_bfloat16*>(m->folded) + d;
        pg.ldc[0] = 2 * d;
      }
      if (proj) {
        // p_i = [W_f1 ; W_g1]_r u_i, the first fusion layer's r-half applied to
        // every value once per image
        F[1] = TmaOperand{static_cast<const __nv_bfloat16*>(p->W_f1) + d, H, d, 2 * d};
        F[2] = TmaOperand{static_cast<const __nv_bfloat16*>(p->W_g1) + d, H, d, 2 * d};
        pg.out[1] = m->proj;
        pg.out[2] = static_cast<__nv_bfloat16*>(m->proj) + H;
        pg.ldc[1] = pg.ldc[2] = 2 * H;
      }
      if (fold || proj) {
        KernelTimer t("memory_fold", s);
        err = launch_pair_gemm(false, pg, F, TmaOperand{m->keys, total, d, d},
                               TmaOperand{m->values, total, d, d}, s);
      }
      if (err != cudaSuccess) return cuda_fail(err, "folding the keys and projecting the values");
      if (fold) m->fold_wq = p->W_Q;
      if (proj) {
        { KernelTimer t("memory_proj_transpose", s);
          err = launch_transpose_images(m->proj, 2 * H, ld, itab, m->projT, s); }
        if (err != cudaSuccess) return cuda_fail(err, "transposing the projected values");
        m->proj_ld = ld;
        m->proj_wf1 = p->W_f1;
        m->proj_wg1 = p->W_g1;
        m->proj_h = H;
      }
    }
    int herr = 0;
    err = cudaMemcpyAsync(&herr, errw, sizeof(int), cudaMemcpyDeviceToHost, s);
    if (err == cudaSuccess) err = cudaStreamSynchronize(s);
    if (err != cudaSuccess) return cuda_fail(err, "memory build");
    if (herr & kErrTimeout)
      return fail(FOVEA_ERR_TIMEOUT, "a bounded device wait gave up during the memory build");
    return FOVEA_OK;
  };
  st = run();
  for (void* t : {scratch, temps})
    if (t != nullptr) cudaFreeAsync(t, s);
  cudaStreamSynchronize(s);
  pool_trim(pool);
  if (st != FOVEA_OK) {
    free_memory(m);
    return st;
  }
  *out = m;
  return FOVEA_OK;
}

FOVEA_API void fovea_memory_destroy(fovea_memory* mem) { free_memory(mem); }

FOVEA_API fovea_status fovea_memory_info(const fovea_memory* mem, int* B, int* total_valid,
                                         int32_t* valid_counts) {
  g_last_error.clear();
  if (mem == nullptr) return fail(FOVEA_ERR_INVALID_ARG, "memory is NULL");
  if (B) *B = mem->B;
  if (total_valid) *total_valid = mem->total;
  if (valid_counts) memcpy(valid_counts, mem->counts.data(), mem->B * sizeof(int32_t));
  return FOVEA_OK;
}

FOVEA_API fovea_status fovea_memory_folded_keys(const fovea_memory* mem, const void* W_Q,
                                                const void** folded) {
  g_last_error.clear();
  if (mem == nullptr) return fail(FOVEA_ERR_INVALID_ARG, "memory is NULL");
  if (folded == nullptr) return fail(FOVEA_ERR_INVALID_ARG, "folded is NULL");
  *folded = (mem->folded != nullptr && W_Q != nullptr && mem->fold_wq == W_Q) ? mem->folded : nullptr;
  return FOVEA_OK;
}

FOVEA_API fovea_status fovea_memory_tensors(const fovea_memory* mem, const void** keys,
                                            const void** values, const int32_t** index,
                                            int64_t* offsets) {
  g_last_error.clear();
  if (mem == nullptr) return fail(FOVEA_ERR_INVALID_ARG, "memory is NULL");
  if (keys) *keys = mem->keys;
  if (values) *values = mem->values;
  if (index) *index = mem->orig_index;
  if (offsets) memcpy(offsets, mem->offsets.data(), (mem->B + 1) * sizeof(int64_t));
  return FOVEA_OK;
}

}  // extern "C"

// ---------------------------------------------------------------------------
// Workspace layout (all regions 256-byte aligned)
// ---------------------------------------------------------------------------
namespace {
struct WsLayout {
  size_t err, xh, q, scores, sel_pos, sel_w, sel_cnt, r_lo, act, c, gh, alpha_hi, alpha_lo, total;
};

// LM head workspace: the header, then the candidate keys [N, slots, k_c].
size_t lm_head_ws_bytes(int N, int slots, int k_c) {
  return kWsHeaderBytes + (size_t)N * slots * k_c * sizeof(unsigned long long);
}

int device_sms() {
  static int sms = 0;
  if (sms == 0) {
    int dev = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (sms <= 0) sms = 148;
  }
  return sms;
}

// alpha_ld: entries of a dense weight row (the memory's padded per-image
// count when it keeps the transposed projected values, else 0).
WsLayout ws_layout(int dtype, int d, int H, int N, int k_max, long long score_elems, int alpha_ld) {
  WsLayout L;
  size_t off = 0;
  auto take = [&](size_t bytes) {
    const size_t o = off;
    off = align_up(off + bytes, 256);
    return o;
  };
  const size_t es = esize(dtype);
  L.err = take(kWsHeaderBytes);          // the sticky error word, then reserved words
  L.xh = take((size_t)N * d * es);
  L.q = take((size_t)N * d * es * (dtype == FOVEA_BF16 ? 2 : 1));   // bf16: q_hi | q_lo
  L.scores = take((size_t)score_elems * 4);
  L.sel_pos = take((size_t)N * k_max * 4);
  L.sel_w = take((size_t)N * k_max * 4);
  L.sel_cnt = take((size_t)N * 4);
  L.r_lo = take((size_t)N * d * es);
  L.act = take((size_t)N * 2 * H * es);
  L.c = take((size_t)N * d * 4);
  L.gh = take(dtype == FOVEA_BF16 ? (size_t)N * 2 * H * 4 : 0);   // [W_f1 ; W_g1]_h h, fp32
  L.alpha_hi = take((size_t)N * alpha_ld * 2);                     // dense weights, bf16 hi
  L.alpha_lo = take((size_t)N * alpha_ld * 2);                     // and lo
  L.total = off;
  return L;
}

fovea_status check_rows(const fovea_memory* mem, const int32_t* row_offsets, int* N_out,
                        long long* score_elems, int* max_m, int* max_r, int* ngroups) {
  if (mem == nullptr) return fail(FOVEA_ERR_INVALID_ARG, "memory is NULL");
  if (row_offsets == nullptr) return fail(FOVEA_ERR_INVALID_ARG, "row_offsets is NULL");
  if (row_offsets[0] != 0) return fail(FOVEA_ERR_INVALID_ARG, "row_offsets[0] = %d, expected 0", row_offsets[0]);
  long long se = 0;
  int mm = 0, mr = 0, ng = 0;
  for (int b = 0; b < mem->B; ++b) {
    const int r = row_offsets[b + 1] - row_offsets[b];
    if (r < 0) return fail(FOVEA_ERR_INVALID_ARG, "row_offsets decrease at sequence %d", b);
    se += (long long)r * mem->counts[b];
    if (r > 0 && mem->counts[b] > mm) mm = mem->counts[b];
    if (r > 0 && mem->counts[b] > 0) {
      ++ng;
      if (r > mr) mr = r;
    }
  }
  *N_out = row_offsets[mem->B];
  *score_elems = se;
  *max_m = mm;
  *max_r = mr;
  *ngroups = ng;
  return FOVEA_OK;
}
}  // namespace

extern "C" {

FOVEA_API fovea_status fovea_workspace_size(const fovea_params* p, const fovea_memory* mem,
                                            const int32_t* row_offsets, int k_max,
                                            size_t* bytes) {
  g_last_error.clear();
  fovea_status st = check_dims(p);
  if (st != FOVEA_OK) return st;
  if (bytes == nullptr) return fail(FOVEA_ERR_INVALID_ARG, "bytes is NULL");
  if (p->mlp_hidden <= 0 || p->mlp_hidden % 128 != 0)
    return fail(FOVEA_ERR_INVALID_ARG, "mlp_hidden %d must be a positive multiple of 128",
                p->mlp_hidden);
  if (k_max < 1) return fail(FOVEA_ERR_INVALID_ARG, "k_max = %d < 1", k_max);
  int N, mm, mr, ng;
  long long se;
  if ((st = check_rows(mem, row_offsets, &N, &se, &mm, &mr, &ng)) != FOVEA_OK) return st;
  *bytes = ws_layout(p->dtype, p->d_model, p->mlp_hidden, N, k_max, se,
                     mem->projT != nullptr ? mem->proj_ld : 0).total;
  return FOVEA_OK;
}

FOVEA_API fovea_status fovea_workspace_init(void* workspace, size_t bytes, void* stream) {
  g_last_error.clear();
  if (workspace == nullptr) return fail(FOVEA_ERR_INVALID_ARG, "workspace is NULL");
  if (bytes < kWsHeaderBytes)
    return fail(FOVEA_ERR_INVALID_ARG, "workspace of %zu bytes is too small", bytes);
  FOVEA_CUDA(cudaMemsetAsync(workspace, 0, kWsHeaderBytes, static_cast<cudaStream_t>(stream)),
             "cudaMemsetAsync");
  return FOVEA_OK;
}

FOVEA_API fovea_status fovea_sync_errors(void* workspace, void* stream) {
  g_last_error.clear();
  if (workspace == nullptr) return fail(FOVEA_ERR_INVALID_ARG, "workspace is NULL");
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  int herr = 0;
  FOVEA_CUDA(cudaMemcpyAsync(&herr, workspace, sizeof(int), cudaMemcpyDeviceToHost, s),
             "cudaMemcpyAsync");
  FOVEA_CUDA(cudaStreamSynchronize(s), "cudaStreamSynchronize");
  // clear the whole header: a kernel that gave up may have left other words set
  FOVEA_CUDA(cudaMemsetAsync(workspace, 0, herr ? kWsHeaderBytes : sizeof(int), s),
             "cudaMemsetAsync");
  FOVEA_CUDA(cudaStreamSynchronize(s), "cudaStreamSynchronize");
  if (herr & kErrTimeout)
    return fail(FOVEA_ERR_TIMEOUT, "a bounded device wait gave up (error word 0x%x)", herr);
  if (herr & kErrDepth)
    return fail(FOVEA_ERR_INVALID_ARG, "a draft state had a depth outside [0, max_depth]");
  return FOVEA_OK;
}

FOVEA_API fovea_status fovea_debug_wait_limit(unsigned long long limit_ns) {
  g_last_error.clear();
  set_wait_limit_ns(limit_ns == 0 ? kDefaultWaitLimitNs : limit_ns);
  return FOVEA_OK;
}

FOVEA_API fovea_status fovea_retrieve_fuse(const fovea_params* p, const fovea_memory* mem,
                                           const void* h, const int32_t* depth,
                                           const int32_t* row_offsets, const float* row_scale,
                                           float rho, int k_min, int k_max, int l_max,
                                           void* h_out, int32_t* counts, int32_t* indices,
                                           float* readout, float* gate, void* workspace,
                                           size_t workspace_bytes, void* stream) {
  g_last_error.clear();
  fovea_status st = check_step_params(p);
  if (st != FOVEA_OK) return st;
  if (!(rho > 0.0f && rho <= 1.0f))
    return fail(FOVEA_ERR_INVALID_ARG, "rho = %g must satisfy 0 < rho <= 1", (double)rho);
  if (k_min < 1 || k_min > k_max)
    return fail(FOVEA_ERR_INVALID_ARG, "need 1 <= k_min (%d) <= k_max (%d)", k_min, k_max);
  if (k_max > FOVEA_MAX_K)
    return fail(FOVEA_ERR_UNSUPPORTED, "k_max = %d exceeds %d", k_max, FOVEA_MAX_K);
  if (mem == nullptr) return fail(FOVEA_ERR_INVALID_ARG, "memory is NULL");
  if (mem->d != p->d_model || mem->dtype != p->dtype)
    return fail(FOVEA_ERR_INVALID_ARG, "memory was built with d=%d dtype=%d, params have d=%d dtype=%d",
                mem->d, mem->dtype, p->d_model, p->dtype);
  int N, max_m, max_r, ngroups;
  long long score_elems;
  if ((st = check_rows(mem, row_offsets, &N, &score_elems, &max_m, &max_r, &ngroups)) != FOVEA_OK)
    return st;
  if (N == 0) return FOVEA_OK;
  NEED_PTR(h, "h");
  NEED_PTR(h_out, "h_out");
  if (depth == nullptr) return fail(FOVEA_ERR_INVALID_ARG, "depth is NULL");
  if (readout != nullptr && !aligned16(readout))
    return fail(FOVEA_ERR_INVALID_ARG, "readout is not 16-byte aligned");
  if (workspace == nullptr) return fail(FOVEA_ERR_INVALID_ARG, "workspace is NULL");
  if ((reinterpret_cast<uintptr_t>(workspace) & 255u) != 0)
    return fail(FOVEA_ERR_INVALID_ARG, "workspace is not 256-byte aligned");
  const int d = p->d_model, H = p->mlp_hidden, dt = p->dtype;
  const WsLayout L = ws_layout(dt, d, H, N, k_max, score_elems,
                              mem->projT != nullptr ? mem->proj_ld : 0);
  if (workspace_bytes < L.total)
    return fail(FOVEA_ERR_INVALID_ARG, "workspace has %zu bytes, needs %zu", workspace_bytes, L.total);

  cudaStream_t s = static_cast<cudaStream_t>(stream);
  uint8_t* ws = static_cast<uint8_t*>(workspace);
  int* err = reinterpret_cast<int*>(ws + L.err);
  void* xh = ws + L.xh;
  void* q = ws + L.q;
  float* scores = reinterpret_cast<float*>(ws + L.scores);
  int32_t* sel_pos = reinterpret_cast<int32_t*>(ws + L.sel_pos);
  float* sel_w = reinterpret_cast<float*>(ws + L.sel_w);
  int32_t* sel_cnt = reinterpret_cast<int32_t*>(ws + L.sel_cnt);
  void* r_lo = ws + L.r_lo;
  void* act = ws + L.act;
  float* cbuf = reinterpret_cast<float*>(ws + L.c);
  float* gh = reinterpret_cast<float*>(ws + L.gh);
  // depth gate: rows deeper than l_max are not corrected (their selection is
  // empty and h_hat = h); with l_max >= D every row is corrected and the gate
  // reads nothing
  const DepthGate gate_rows{l_max < p->max_depth ? depth : nullptr, l_max, p->max_depth};

  // Per-sequence table (kernel parameter).
  static thread_local SeqTable tab;
  tab.B = mem->B;
  for (int b = 0; b < mem->B; ++b) {
    tab.row_start[b] = row_offsets[b];
    tab.key_off[b] = (int)mem->offsets[b];
    tab.m[b] = mem->counts[b];
  }
  tab.row_start[mem->B] = row_offsets[mem->B];
  {
    long long so = 0;
    for (int b = 0; b < mem->B; ++b) {
      tab.score_off[b] = so;
      so += (long long)(row_offsets[b + 1] - row_offsets[b]) * mem->counts[b];
    }
  }
  cudaError_t e;

  // (1) x_h = LN_h(h) + E_dep[l]
  { KernelTimer t("ln_query", s);
    e = launch_ln_query(dt, h, N, d, p->ln_h_gamma, p->ln_h_beta, p->ln_eps, p->E_dep, depth,
                        p->max_depth, err, xh, s); }
  if (e != cudaSuccess) return cuda_fail(e, "ln_query");

  static thread_local GemmArgs a;
  // (2) q = W_Q x_h  (bf16 path: stored as q_hi + q_lo).  With the memory's
  // projected values valid for these weights, the same launch computes
  // G_h = [W_f1 ; W_g1]_h h (the h-half of the first fusion layer, fp32):
  // the r-half then reduces to a weighted sum of projected values (4).
  // With the memory's folded keys valid for this W_Q, q is never formed:
  // the scores take x_h against the folded keys, and the launch computes
  // G_h alone (or is skipped without the projected values).
  const bool bf = dt == FOVEA_BF16;
  // The r-half of the first fusion layer from the projected values: either
  // gathered row by row, in the selection kernel or in a kernel after it (rows
  // of <= 2048 entries, k_max <= 256, a batch that fills the GPU in about a
  // wave), or, with the selection weights written as dense rows, one GEMM against the memory's
  // transposed projected values (long rows, large caps, large batches).
  const bool have_proj = bf && mem->proj != nullptr && mem->proj_wf1 == p->W_f1 &&
                         mem->proj_wg1 == p->W_g1 && mem->proj_h == H;
  const bool alpha_path = have_proj && mem->projT != nullptr &&
                          (!select_readout_fits(max_m, k_max) || N > 2 * device_sms());
  const bool use_proj = have_proj && (alpha_path || select_readout_fits(max_m, k_max));
  const bool use_fold = bf && mem->folded != nullptr && mem->fold_wq == p->W_Q;
  // the folded keys are [total, 2d] (hi | lo per entry)
  const long long score_key_bytes = (long long)mem->total * d * 2 * (use_fold ? 2 : 1);
  const void* score_keys = use_fold ? mem->folded : mem->keys;
  // With folded keys and projected values, G_h does not depend on the query:
  // when one sequence's keys serve every row (one score group covering all N
  // rows), the score launch computes it too, as two more feature parts
  // against h.
  int gh_seq = -1;
  if (use_fold && use_proj && ngroups == 1) {
    for (int b = 0; b < mem->B; ++b)
      if (row_offsets[b + 1] - row_offsets[b] == N && mem->counts[b] > 0) gh_seq = b;
  }
  const bool gh_in_scores = gh_seq >= 0;
  // Several score groups: G_h as further groups of the score launch, one per
  // 128 rows, so that its L2-fed tiles run beside the HBM-bound score tiles and
  // a launch is saved: 8 images x 8 rows at d = 1024 29.5 -> 24.5 us a step, 8
  // ragged images x 32 rows 84.3 -> 74.3, 16 x 64 rows 123.3 -> 108.8, 4 x 128
  // rows of 8192 entries 177.8 -> 167.1; of 332 steps drawn over the range 173
  // gain 2 % and more and 20 lose as much (16 images of 1102 entries, 214 rows, d =
  // 4096: 86.7 -> 101.6, whose one launch finds no plan with G_h's accumulators
  // that fits both parts).  Up to one block of narrow rows (d below 512) G_h keeps
  // its own launch, which calls without score groups and with more groups than the
  // table holds need as well; no workload has such rows, and they would gain too (60
  // rows of d = 256: 24.2 -> 20.8).
  const int gh_blocks = (N + 127) / 128;
  const bool gh_groups = use_fold && use_proj && !gh_in_scores && ngroups > 0 &&
                         (N > 128 || d >= 512) && ngroups + gh_blocks <= FOVEA_MAX_SEQ;
  void* q_lo = bf ? static_cast<void*>(static_cast<uint8_t*>(q) + (size_t)N * d * 2) : nullptr;
  init_args(a);
  a.k_total = d; a.b_split = d;
  a.A0 = p->W_Q; a.lda0 = d;
  a.B0 = xh; a.ldb0 = d;
  a.out0 = q; a.out1 = q_lo; a.ldc = d; a.err = err;
  a.ngroups = 1;
  a.groups[0] = GemmGroup{0, d, 0, N, 0};
  if (use_proj) {
    a.a_split = d; a.a_split2 = d + H;
    a.r_by_part = 1;
    a.epi_split = d;
    a.out2 = gh; a.ldc2 = 2 * H;
    a.groups[0] = GemmGroup{0, d + 2 * H, 0, N, 0};
  }
  // entries selected at most: when they are most of the memory, the value
  // rows are prefetched
  long long m_sel = 0;
  for (int b = 0; b < mem->B; ++b)
    m_sel += std::min<long long>(mem->counts[b], (long long)(row_offsets[b + 1] - row_offsets[b]) * k_max);
  if (bf) {
    // the keys when the score GEMM's own loads before its griddepcontrol.wait
    // (its first ring stages) cannot cover them, and the values when most of
    // their rows will be read by the readout
    if (score_key_bytes > (8ll << 20)) {
      a.pf_ptr[a.n_prefetch] = score_keys;
      a.pf_bytes[a.n_prefetch++] = score_key_bytes;
    }
    if (2 * m_sel >= mem->total) {
      if (!use_proj || readout != nullptr) {
        a.pf_ptr[a.n_prefetch] = mem->values;
        a.pf_bytes[a.n_prefetch++] = (long long)mem->total * d * 2;
      }
    }
  }
  if (use_fold && use_proj && !gh_in_scores && !gh_groups) {
    // G_h only: parts W_f1 and W_g1 (h-halves), both against h, fp32 out
    a.A0 = p->W_f1; a.lda0 = 2 * d;
    a.B0 = h;
    a.a_split = H; a.a_split2 = 0x7fffffff;
    a.r_by_part = 0;
    a.epi_split = 0;
    a.out2 = gh; a.ldc2 = 2 * H;
    a.groups[0] = GemmGroup{0, 2 * H, 0, N, 0};
    { KernelTimer t("fusion_h", s);
      e = launch_gemm_tc(kEpiQueryH, a, TmaOperand{p->W_f1, H, d, 2 * d},
                         TmaOperand{p->W_g1, H, d, 2 * d}, TmaOperand{h, N, d, d},
                         TmaOperand{nullptr, 0, 0, 0}, 2 * H, N, s); }
    if (e != cudaSuccess) return cuda_fail(e, "fusion_h");
  } else if (!use_fold) {
    KernelTimer t("query_proj", s);
    if (use_proj)
      e = launch_gemm_tc(kEpiQueryH, a, TmaOperand{p->W_Q, d, d, d}, TmaOperand{p->W_f1, H, d, 2 * d},
                         TmaOperand{xh, N, d, d}, TmaOperand{h, N, d, d}, d + 2 * H, N, s,
                         TmaOperand{p->W_g1, H, d, 2 * d});
    else
      e = run_gemm(dt, bf ? kEpiStoreHiLo : kEpiStore, a, TmaOperand{p->W_Q, d, d, d},
                   TmaOperand{nullptr, 0, 0, 0}, TmaOperand{xh, N, d, d},
                   TmaOperand{nullptr, 0, 0, 0}, d, N, s);
    if (e != cudaSuccess) return cuda_fail(e, "query_proj");
  }

  // (3) s = q k^T / sqrt(d) (* row_scale), per sequence; folded: x_h against
  // kappa_hi and kappa_lo
  if (score_elems > 0) {
    init_args(a);
    a.k_total = d; a.b_split = d;
    a.A0 = score_keys; a.lda0 = use_fold ? 2 * d : d;
    a.B0 = use_fold ? xh : q; a.ldb0 = d;
    a.out0 = scores;
    a.row_scale = row_scale;
    a.scale = (float)(1.0 / sqrt((double)d));
    a.err = err;
    a.f_lo_kb = use_fold ? d / 64 : 0;
    int g = 0;
    if (gh_groups)                               // first: they read more per tile from L2
      for (; g < gh_blocks; ++g)
        a.groups[g] = GemmGroup{-1, 2 * H, 128 * g, std::min(128, N - 128 * g), 0};
    for (int b = 0; b < mem->B; ++b) {
      const int r = row_offsets[b + 1] - row_offsets[b];
      if (r == 0 || mem->counts[b] == 0) continue;
      a.groups[g++] = GemmGroup{(int)mem->offsets[b], mem->counts[b], row_offsets[b], r, tab.score_off[b]};
    }
    a.ngroups = g;
    a.dual_b = bf && !use_fold ? 1 : 0;
    if (use_fold && !use_proj && 2 * m_sel >= mem->total) {
      // no query launch carries the value prefetch on this path
      a.pf_ptr[a.n_prefetch] = mem->values;
      a.pf_bytes[a.n_prefetch++] = (long long)mem->total * d * 2;
    }
    if (bf && !use_proj) {
      // the fusion weights, read after selection and readout (with the
      // projected values the selection kernel prefetches them, and the
      // second correction layer's GEMM loads its weights before its
      // griddepcontrol.wait)
      a.pf_ptr[a.n_prefetch] = p->W_f1;
      a.pf_bytes[a.n_prefetch++] = (long long)H * 2 * d * 2;
      a.pf_ptr[a.n_prefetch] = p->W_g1;
      a.pf_bytes[a.n_prefetch++] = (long long)H * 2 * d * 2;
      if (a.n_prefetch < 4) {
        a.pf_ptr[a.n_prefetch] = p->W_f2;
        a.pf_bytes[a.n_prefetch++] = (long long)d * H * 2;
      }
    }
    const TmaOperand folded_op{mem->folded, mem->total, 2 * d, 2 * d};
    if (gh_in_scores) {
      // one group: the sequence's folded keys (scores, against x_h), then the
      // h-halves of W_f1 and W_g1 (G_h, against h)
      const int M = mem->counts[gh_seq];
      a.groups[0] = GemmGroup{(int)mem->offsets[gh_seq], M + 2 * H, 0, N, 0};
      a.a_split = M; a.a_split2 = M + H;
      a.r_by_part = 1;
      a.epi_split = M;
      a.out2 = gh; a.ldc2 = 2 * H;
      if (readout != nullptr && 2 * m_sel >= mem->total && a.n_prefetch < 4) {
        a.pf_ptr[a.n_prefetch] = mem->values;
        a.pf_bytes[a.n_prefetch++] = (long long)mem->total * d * 2;
      }
      KernelTimer t("score_fusion_h", s);
      e = launch_gemm_tc(kEpiScoresFolded, a, folded_op, TmaOperand{p->W_f1, H, d, 2 * d},
                         TmaOperand{xh, N, d, d}, TmaOperand{h, N, d, d}, M + 2 * H, N, s,
                         TmaOperand{p->W_g1, H, d, 2 * d});
    } else if (gh_groups) {
      a.r_by_part = 1;
      a.gh_cols = H;
      a.out2 = gh; a.ldc2 = 2 * H;
      KernelTimer t("score_fusion_h", s);
      e = launch_gemm_tc(kEpiScoresFolded, a, folded_op, TmaOperand{p->W_f1, H, d, 2 * d},
                         TmaOperand{xh, N, d, d}, TmaOperand{h, N, d, d}, max_m,
                         std::max(max_r, std::min(N, 128)), s, TmaOperand{p->W_g1, H, d, 2 * d});
    } else if (use_fold) {
      KernelTimer t("score_folded", s);
      e = launch_gemm_tc(kEpiScoresFolded, a, folded_op, TmaOperand{nullptr, 0, 0, 0},
                         TmaOperand{xh, N, d, d}, TmaOperand{nullptr, 0, 0, 0}, max_m, max_r, s);
    } else {
      KernelTimer t("score", s);
      e = run_gemm(dt, kEpiScores, a, TmaOperand{mem->keys, mem->total, d, d},
                   TmaOperand{nullptr, 0, 0, 0}, TmaOperand{q, N, d, d},
                   TmaOperand{q_lo, N, d, d}, max_m, max_r, s);
    }
    if (e != cudaSuccess) return cuda_fail(e, "score");
  }

  // (4) softmax, cumulative-mass cardinality, selected set, renormalised weights;
  // (5) r = sum alpha u; with the projected values, also
  // (6) [a_f | a_g] = SiLU(G_h + sum alpha p + [b_f1 | b_g1])
  if (alpha_path) {
    // the selection writes the weights as dense bf16 hi / lo rows; the
    // readout, when asked for, gathers the values row by row
    void* alpha_hi = ws + L.alpha_hi;
    void* alpha_lo = ws + L.alpha_lo;
    { KernelTimer t("select", s);
      e = launch_select(scores, tab, N, mem->orig_index, rho, k_min, k_max, max_m, gate_rows,
                        counts, indices, readout ? sel_pos : nullptr, readout ? sel_w : nullptr,
                        readout ? sel_cnt : nullptr, s, alpha_hi, alpha_lo, mem->proj_ld); }
    if (e != cudaSuccess) return cuda_fail(e, "select");
    if (readout != nullptr) {
      { KernelTimer t("readout", s);
        e = launch_readout(dt, RowGather{sel_cnt, sel_pos, sel_w, k_max, mem->values, d, readout, nullptr},
                           N, s); }
      if (e != cudaSuccess) return cuda_fail(e, "readout");
    }
    // [a_f | a_g] = SiLU(G_h + alpha P + [b_f1 | b_g1]): per image, the
    // weights' hi / lo rows against the image's transposed projected values
    init_args(a);
    a.k_total = mem->proj_ld; a.b_split = mem->proj_ld;
    a.A0 = mem->projT; a.lda0 = mem->proj_ld;
    a.B0 = alpha_hi; a.B1 = alpha_lo; a.ldb0 = mem->proj_ld; a.ldb1 = mem->proj_ld;
    a.epi_split = H;
    a.out0 = act; a.ldc = 2 * H;
    a.bias0 = p->b_f1; a.bias1 = p->b_g1;
    a.add_in = gh; a.ldc2 = 2 * H;
    a.err = err;
    int g = 0, max_rows = 0;
    for (int b = 0; b < mem->B; ++b) {
      const int r = row_offsets[b + 1] - row_offsets[b];
      if (r == 0) continue;
      a.groups[g++] = GemmGroup{b * 2 * H, 2 * H, row_offsets[b], r, 0};
      max_rows = std::max(max_rows, r);
    }
    a.ngroups = g;
    { KernelTimer t("act_gemm", s);
      e = launch_gemm_tc(kEpiAct, a, TmaOperand{mem->projT, (long long)mem->B * 2 * H, mem->proj_ld,
                                                mem->proj_ld},
                         TmaOperand{nullptr, 0, 0, 0}, TmaOperand{alpha_hi, N, mem->proj_ld, mem->proj_ld},
                         TmaOperand{alpha_lo, N, mem->proj_ld, mem->proj_ld}, 2 * H, max_rows, s); }
    if (e != cudaSuccess) return cuda_fail(e, "act_gemm");
  } else if (use_proj && (k_max > kFuseSelectMaxK || (N > device_sms() && readout == nullptr))) {
    { KernelTimer t("select", s);
      e = launch_select(scores, tab, N, mem->orig_index, rho, k_min, k_max, max_m, gate_rows,
                        counts, indices, sel_pos, sel_w, sel_cnt, s); }
    if (e != cudaSuccess) return cuda_fail(e, "select");
    { KernelTimer t("gather_fuse", s);
      e = launch_readout(dt, RowGather{sel_cnt, sel_pos, sel_w, k_max,
                                       readout != nullptr ? mem->values : nullptr, d, readout,
                                       nullptr, mem->proj, H, gh, p->b_f1, p->b_g1, act}, N, s); }
    if (e != cudaSuccess) return cuda_fail(e, "gather_fuse");
  } else if (use_proj) {
    { KernelTimer t("select_fuse", s);
      e = launch_select_gather(dt, scores, tab, N, mem->orig_index, rho, k_min, k_max, max_m,
                               gate_rows, counts, indices, mem->values, d, readout, nullptr,
                               mem->proj, H, gh, p->b_f1, p->b_g1, act, err, s,
                               (long long)mem->total * 2 * H * 2); }
    if (e != cudaSuccess) return cuda_fail(e, "select_fuse");
  } else {
    if (select_readout_fits(max_m, k_max)) {
      { KernelTimer t("select_readout", s);
        e = launch_select_gather(dt, scores, tab, N, mem->orig_index, rho, k_min, k_max, max_m,
                                 gate_rows, counts, indices, mem->values, d, readout, r_lo,
                                 nullptr, H, nullptr, nullptr, nullptr, nullptr, err, s); }
      if (e != cudaSuccess) return cuda_fail(e, "select_readout");
    } else {
      { KernelTimer t("select", s);
        e = launch_select(scores, tab, N, mem->orig_index, rho, k_min, k_max, max_m, gate_rows,
                          counts, indices, sel_pos, sel_w, sel_cnt, s); }
      if (e != cudaSuccess) return cuda_fail(e, "select");
      { KernelTimer t("readout", s);
        e = launch_readout(dt, RowGather{sel_cnt, sel_pos, sel_w, k_max, mem->values, d, readout, r_lo},
                           N, s); }
      if (e != cudaSuccess) return cuda_fail(e, "readout");
    }

    // (6) [a_f | a_g] = SiLU([h; r] [W_f1 | W_g1]^T + [b_f1 | b_g1])
    init_args(a);
    a.k_total = 2 * d;
    a.a_split = H;
    a.b_split = d;
    a.A0 = p->W_f1; a.A1 = p->W_g1; a.lda0 = 2 * d; a.lda1 = 2 * d;
    a.B0 = h; a.B1 = r_lo; a.ldb0 = d; a.ldb1 = d;
    a.epi_split = H;
    a.out0 = act; a.ldc = 2 * H;
    a.bias0 = p->b_f1; a.bias1 = p->b_g1;
    a.err = err;
    a.ngroups = 1;
    a.groups[0] = GemmGroup{0, 2 * H, 0, N, 0};
    { KernelTimer t("fuse_hidden", s);
      e = run_gemm(dt, kEpiBiasSilu, a, TmaOperand{p->W_f1, H, 2 * d, 2 * d},
                   TmaOperand{p->W_g1, H, 2 * d, 2 * d}, TmaOperand{h, N, d, d},
                   TmaOperand{r_lo, N, d, d}, 2 * H, N, s); }
    if (e != cudaSuccess) return cuda_fail(e, "fuse_hidden");
  }

  // (7) c = a_f W_f2^T + b_f2
  init_args(a);
  a.k_total = H; a.b_split = H;
  a.A0 = p->W_f2; a.lda0 = H;
  a.B0 = act; a.ldb0 = 2 * H;
  a.out0 = cbuf; a.ldc = d;
  a.bias0 = p->b_f2;
  a.err = err;
  a.ngroups = 1;
  a.groups[0] = GemmGroup{0, d, 0, N, 0};
  { KernelTimer t("fuse_out", s);
    e = run_gemm(dt, kEpiBiasF32, a, TmaOperand{p->W_f2, d, H, H}, TmaOperand{nullptr, 0, 0, 0},
                 TmaOperand{act, N, H, 2 * H}, TmaOperand{nullptr, 0, 0, 0}, d, N, s); }
  if (e != cudaSuccess) return cuda_fail(e, "fuse_out");

  // (8) g = sigma(a_g w_g2 + b_g2); h_hat = RMSNorm(h + g c); rows past the
  // depth gate: h_hat = h
  { KernelTimer t("finalize", s);
    e = launch_finalize(dt, h, cbuf, act, H, d, p->w_g2, p->b_g2, p->rms_gamma, p->rms_eps, N,
                        gate_rows, h_out, gate, s); }
  if (e != cudaSuccess) return cuda_fail(e, "finalize");
  return FOVEA_OK;
}

FOVEA_API fovea_status fovea_lm_head_topk(const void* W_LM, int vocab, int d_model, int dtype,
                                          const void* h_hat, int N, int k_c, float* logits,
                                          int32_t* top_idx, float* top_val, void* workspace,
                                          size_t workspace_bytes, void* stream) {
  g_last_error.clear();
  if (dtype != FOVEA_BF16 && dtype != FOVEA_FP32)
    return fail(FOVEA_ERR_INVALID_ARG, "dtype %d is neither FOVEA_BF16 nor FOVEA_FP32", dtype);
  if (d_model <= 0 || d_model % 64 != 0 || d_model > FOVEA_MAX_D)
    return fail(FOVEA_ERR_INVALID_ARG, "d_model %d must be a positive multiple of 64 (<= %d)",
                d_model, FOVEA_MAX_D);
  if (N < 0) return fail(FOVEA_ERR_INVALID_ARG, "N = %d < 0", N);
  if (k_c < 1 || k_c > FOVEA_MAX_KC)
    return fail(FOVEA_ERR_INVALID_ARG, "k_c = %d must lie in [1, %d]", k_c, FOVEA_MAX_KC);
  if (vocab < k_c) return fail(FOVEA_ERR_INVALID_ARG, "vocab %d < k_c %d", vocab, k_c);
  NEED_PTR(W_LM, "W_LM");
  NEED_PTR(h_hat, "h_hat");
  if (top_idx == nullptr) return fail(FOVEA_ERR_INVALID_ARG, "top_idx is NULL");
  if (workspace == nullptr || (reinterpret_cast<uintptr_t>(workspace) & 255u) != 0)
    return fail(FOVEA_ERR_INVALID_ARG, "workspace is NULL or not 256-byte aligned");
  if (dtype != FOVEA_BF16)
    return fail(FOVEA_ERR_UNSUPPORTED, "the LM head runs on bf16 weights and states only");
  if (N == 0) return FOVEA_OK;
  const int slots = lm_head_slots(vocab, d_model, N);
  const size_t need = lm_head_ws_bytes(N, slots, k_c);
  if (workspace_bytes < need)
    return fail(FOVEA_ERR_INVALID_ARG, "workspace has %zu bytes, needs %zu "
                "(fovea_lm_head_workspace_size)", workspace_bytes, need);
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  // z = h_hat W_LM^T: W_LM [vocab, d] is the feature operand, streamed once;
  // every column goes to the fp32 logits, and the epilogue keeps each row's
  // k_c largest of every tile as candidates after the header
  unsigned long long* cand = reinterpret_cast<unsigned long long*>(
      static_cast<uint8_t*>(workspace) + kWsHeaderBytes);
  static thread_local GemmArgs a;
  init_args(a);
  a.k_total = d_model; a.b_split = d_model;
  a.epi_split = 0;
  a.out2 = logits; a.ldc2 = vocab;
  a.cand = cand; a.cand_k = k_c; a.cand_ld = (long long)slots * k_c;
  a.err = static_cast<int*>(workspace);
  a.ngroups = 1;
  a.groups[0] = GemmGroup{0, vocab, 0, N, 0};
  cudaError_t e;
  { KernelTimer t("lm_head", s);
    e = launch_gemm_tc(kEpiLogits, a, TmaOperand{W_LM, vocab, d_model, d_model},
                       TmaOperand{nullptr, 0, 0, 0}, TmaOperand{h_hat, N, d_model, d_model},
                       TmaOperand{nullptr, 0, 0, 0}, vocab, N, s); }
  if (e != cudaSuccess) return cuda_fail(e, "lm_head");
  { KernelTimer t("merge_candidates", s);
    e = launch_merge_candidates(cand, N, slots, k_c, top_idx, top_val, s); }
  if (e != cudaSuccess) return cuda_fail(e, "merge_candidates");
  return FOVEA_OK;
}

FOVEA_API fovea_status fovea_lm_head_workspace_size(int vocab, int d_model, int N, int k_c,
                                                    size_t* bytes) {
  g_last_error.clear();
  if (bytes == nullptr) return fail(FOVEA_ERR_INVALID_ARG, "bytes is NULL");
  if (d_model <= 0 || d_model % 64 != 0 || d_model > FOVEA_MAX_D)
    return fail(FOVEA_ERR_INVALID_ARG, "d_model %d must be a positive multiple of 64 (<= %d)",
                d_model, FOVEA_MAX_D);
  if (N < 0) return fail(FOVEA_ERR_INVALID_ARG, "N = %d < 0", N);
  if (k_c < 1 || k_c > FOVEA_MAX_KC)
    return fail(FOVEA_ERR_INVALID_ARG, "k_c = %d must lie in [1, %d]", k_c, FOVEA_MAX_KC);
  if (vocab < k_c) return fail(FOVEA_ERR_INVALID_ARG, "vocab %d < k_c %d", vocab, k_c);
  *bytes = N == 0 ? kWsHeaderBytes : lm_head_ws_bytes(N, lm_head_slots(vocab, d_model, N), k_c);
  return FOVEA_OK;
}

FOVEA_API fovea_status fovea_timing_enable(int enable) {
  std::lock_guard<std::mutex> lk(g_tmu);
  for (auto& r : g_recs) {
    g_free_events.push_back(r.start);
    g_free_events.push_back(r.stop);
  }
  g_recs.clear();
  g_timing = enable != 0;
  return FOVEA_OK;
}

FOVEA_API int fovea_timing_read(const char** names, double* total_ms, int* launches,
                                int capacity) {
  std::lock_guard<std::mutex> lk(g_tmu);
  std::vector<const char*> nm;
  std::vector<double> ms;
  std::vector<int> cnt;
  for (auto& r : g_recs) {
    if (cudaEventSynchronize(r.stop) != cudaSuccess) continue;
    float t = 0.0f;
    if (cudaEventElapsedTime(&t, r.start, r.stop) != cudaSuccess) continue;
    size_t i = 0;
    while (i < nm.size() && strcmp(nm[i], r.name) != 0) ++i;
    if (i == nm.size()) {
      nm.push_back(r.name);
      ms.push_back(0.0);
      cnt.push_back(0);
    }
    ms[i] += t;
    cnt[i] += 1;
  }
  for (size_t i = 0; i < nm.size() && (int)i < capacity; ++i) {
    if (names) names[i] = nm[i];
    if (total_ms) total_ms[i] = ms[i];
    if (launches) launches[i] = cnt[i];
  }
  return (int)nm.size();
}

}  // extern "C"
