// C ABI of the library: cache object, argument checks, launch sequences.
#include <cuda_runtime.h>
#include <math.h>
#include <stdlib.h>
#include <string.h>

#include <atomic>
#include <mutex>
#include <new>
#include <vector>

#include "../../include/gear.h"
#include "gear_call_order.h"
#include "gear_internal.cuh"

using namespace gear;

static std::atomic<unsigned long long> g_launches{0};
static CallOrder g_order;
static CallOrder::Key order_key(cudaStream_t st) {
  CallOrder::Key k = {(uint64_t)(uintptr_t)st, 0, 0, st != cudaStreamPerThread};    // one handle, a stream per thread
  if (st == cudaStreamLegacy) k.stream = 0;
  cudaStreamCaptureStatus capture = cudaStreamCaptureStatusNone;
  unsigned long long id = 0;
  if ((k.stream == 0 && cudaGetDevice(&k.device) != cudaSuccess) || cudaStreamGetCaptureInfo(st, &capture, &id) != cudaSuccess) {
    cudaGetLastError();
    k.ordered = false;
  }
  if (capture == cudaStreamCaptureStatusActive) k.capture = id;
  if (capture == cudaStreamCaptureStatusInvalidated) k.ordered = false;
  return k;
}

void gear::count_launches(int n) { g_launches.fetch_add((unsigned long long)n, std::memory_order_relaxed); }
extern "C" uint64_t gear_kernel_launches(void) { return g_launches.load(std::memory_order_relaxed); }

// Transient workspace of gear_compress comes from one stream-ordered pool per device that keeps its memory between
// calls (the default pool hands it back to the driver at every synchronisation, which costs milliseconds per call).
static std::mutex g_pool_mutex;
static cudaMemPool_t g_pool[64];
static bool g_pool_ready[64];
static cudaMemPool_t workspace_pool(int dev) {
  if (dev < 0 || dev >= 64) return nullptr;
  std::lock_guard<std::mutex> lock(g_pool_mutex);
  if (!g_pool_ready[dev]) {
    cudaMemPoolProps props;
    memset(&props, 0, sizeof(props));
    props.allocType = cudaMemAllocationTypePinned;
    props.handleTypes = cudaMemHandleTypeNone;
    props.location.type = cudaMemLocationTypeDevice;
    props.location.id = dev;
    cudaMemPool_t pool = nullptr;
    if (cudaMemPoolCreate(&pool, &props) != cudaSuccess) { cudaGetLastError(); return nullptr; }
    unsigned long long keep = ~0ull;
    cudaMemPoolSetAttribute(pool, cudaMemPoolAttrReleaseThreshold, &keep);
    g_pool[dev] = pool;
    g_pool_ready[dev] = true;
  }
  return g_pool[dev];
}

// Pinned rows of the host-buffer calls (a ring of kHostSlots slots with an event each).  Pinning costs up to a
// millisecond and waits for the device, so the blocks of freed caches are kept for the next ones: at most kHostPoolBlocks
// blocks and kHostPoolBytes in the process, given back by gear_release_workspace.
constexpr int kHostSlots = 4;
constexpr int kHostPoolBlocks = 64;
constexpr size_t kHostPoolBytes = (size_t)64 << 20;
struct HostBlock {
  unsigned char* mem; size_t bytes; int device;
  cudaEvent_t ev[kHostSlots];
};
static std::mutex g_host_mutex;
static std::vector<HostBlock> g_host_pool;
static size_t g_host_pool_bytes = 0;

static void host_block_destroy(HostBlock& b) {
  if (b.mem) cudaFreeHost(b.mem);
  for (cudaEvent_t& e : b.ev)
    if (e) cudaEventDestroy(e);
  b.mem = nullptr;
}
static bool host_block_get(size_t need, int device, HostBlock* out) {
  {
    std::lock_guard<std::mutex> lock(g_host_mutex);
    for (size_t i = 0; i < g_host_pool.size(); ++i) {
      const HostBlock b = g_host_pool[i];
      if (b.device != device || b.bytes < need || b.bytes > 4 * need + 65536) continue;
      g_host_pool[i] = g_host_pool.back();
      g_host_pool.pop_back();
      g_host_pool_bytes -= b.bytes;
      *out = b;
      return true;
    }
  }
  HostBlock b;
  memset(&b, 0, sizeof(b));
  b.device = device;
  b.bytes = (need + 65535) / 65536 * 65536;
  bool ok = cudaHostAlloc((void**)&b.mem, b.bytes, cudaHostAllocPortable | cudaHostAllocMapped) == cudaSuccess;
  for (cudaEvent_t& e : b.ev) ok = ok && cudaEventCreateWithFlags(&e, cudaEventDisableTiming) == cudaSuccess;
  if (!ok) { cudaGetLastError(); host_block_destroy(b); return false; }
  *out = b;
  return true;
}
static void host_block_put(HostBlock& b) {      // nothing on the device uses it any more
  if (!b.mem) return;
  {
    std::lock_guard<std::mutex> lock(g_host_mutex);
    if ((int)g_host_pool.size() < kHostPoolBlocks && g_host_pool_bytes + b.bytes <= kHostPoolBytes) {
      g_host_pool.push_back(b);
      g_host_pool_bytes += b.bytes;
      b.mem = nullptr;
      return;
    }
  }
  host_block_destroy(b);
}

extern "C" gear_status gear_release_workspace(void) {
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceSynchronize() != cudaSuccess) { cudaGetLastError(); return GEAR_ERR_CUDA; }
  {
    std::lock_guard<std::mutex> lock(g_host_mutex);
    for (size_t i = 0; i < g_host_pool.size();) {
      if (g_host_pool[i].device != dev) { ++i; continue; }
      g_host_pool_bytes -= g_host_pool[i].bytes;
      host_block_destroy(g_host_pool[i]);
      g_host_pool[i] = g_host_pool.back();
      g_host_pool.pop_back();
    }
  }
  std::lock_guard<std::mutex> lock(g_pool_mutex);
  if (dev >= 0 && dev < 64 && g_pool_ready[dev] && cudaMemPoolTrimTo(g_pool[dev], 0) != cudaSuccess) {
    cudaGetLastError();
    return GEAR_ERR_CUDA;
  }
  return GEAR_OK;
}

// Device memory of the caches comes from cudaMalloc unless the caller installed a pair of its own (gear_set_allocator).
static std::mutex g_alloc_mutex;
static gear_alloc_fn g_alloc = nullptr;
static gear_free_fn g_free = nullptr;
static void* g_alloc_ctx = nullptr;

extern "C" gear_status gear_set_allocator(gear_alloc_fn alloc_fn, gear_free_fn free_fn, void* ctx) {
  if ((alloc_fn == nullptr) != (free_fn == nullptr)) return GEAR_ERR_ARG;
  std::lock_guard<std::mutex> lock(g_alloc_mutex);
  g_alloc = alloc_fn; g_free = free_fn; g_alloc_ctx = ctx;
  return GEAR_OK;
}

struct DeviceAllocator {       // the pair a cache was created with (it frees through the same pair)
  gear_alloc_fn alloc; gear_free_fn free; void* ctx;
  void* get(size_t bytes) const {
    if (alloc) return alloc(bytes, ctx);
    void* p = nullptr;
    if (cudaMalloc(&p, bytes) != cudaSuccess) { cudaGetLastError(); return nullptr; }
    return p;
  }
  void put(void* p) const {
    if (!p) return;
    if (free) free(p, ctx); else cudaFree(p);
  }
};

struct gear_cache {
  DeviceAllocator mem;
  gear_config cfg;
  CacheConst cc;
  int device;
  int sm_count;
  int G;                         // query heads per kv head
  int k_k_full;                  // outliers per side for a key group of length g
  // device memory
  unsigned char* arena; size_t arena_bytes; size_t arena_used;
  float* dbg; size_t dbg_bytes; size_t dbg_used;        // fp32 factor copies (GEAR_FLAG_KEEP_FP32_FACTORS)
  SegDesc* table_dev; int table_cap;
  int* blk2seg; int blk_cap;                             // segment index of every compressed block
  void* buf_k; void* buf_v;                              // [BH][n_b][128] fp16
  float* partial; size_t partial_bytes;
  int* tickets; int* status;                             // one block; zeroed on the caller's stream by the first call (scratch_clean)
  bool scratch_clean;
  bool off_default;              // some call went to another stream than the default one
  void* stage_q; float* stage_out; float* stage_b0;      // for the *_host calls: query; result for pageable destinations; B0
  // The *_host calls copy the caller's rows and query into a slot of a pinned ring, from which the push kernel reads them
  // itself: no copy engine and no second stream, hence no event waits between the kernels of a step.  A slot is filled
  // again once the call that used it four calls ago has finished (its event).
  HostBlock host; bool host_used[kHostSlots]; int host_next, host_last;   // host_last: slot of the latest call, -1 = none
  // host state
  std::vector<SegDesc> segs;
  std::vector<long long> dbgA_off, dbgB_off;             // float offsets into dbg (or -1)
  int buf_len;
  long long n_compressed;
  int n_blocks_c;
  // cached launch plan of the decode kernel (depends on the segments' shapes)
  long long plan_key; int plan_occ;
  DecodeArgs plan;
  int test_dead_wait;            // gear_test_dead_wait: the next decode and compress calls wait on a barrier nothing completes
  int max_queries, units_alloc;  // query rows per head the scratch was sized for; units of that size
  CallOrder::Write seg_write, buf_write;   // the last calls that wrote the segments (records, descriptors) and the buffer rows
};

static int outlier_count(float s_pct, int len) {
  const long long s_units = llroundf(s_pct * 10000.0f);
  return (int)((s_units * len + 1999999LL) / 2000000LL);
}

static size_t align_up(size_t x, size_t a) { return (x + a - 1) / a * a; }

static gear_status check_config(const gear_config* c) {
  if (!c) return GEAR_ERR_ARG;
  if (c->batch < 1 || c->n_kv_heads < 1 || c->n_q_heads < 1 || c->max_tokens < 16) return GEAR_ERR_ARG;
  if (c->n_q_heads % c->n_kv_heads) return GEAR_ERR_SHAPE;
  if (c->head_dim != kHeadDim) return GEAR_ERR_SHAPE;
  if (c->bits != 2 && c->bits != 4) return GEAR_ERR_ARG;
  const bool per_vector = c->group == GEAR_GROUP_PER_VECTOR;
  if (!per_vector && c->group != 16 && c->group != 32 && c->group != 64 && c->group != 128) return GEAR_ERR_ARG;
  if (!(c->outlier_pct >= 0.f) || c->outlier_pct > 10.f) return GEAR_ERR_ARG;
  if (c->buffer_cap < 16 || c->buffer_cap % 4 || c->buffer_cap > 1024) return GEAR_ERR_ARG;
  if (per_vector ? c->buffer_cap > 128 : (c->buffer_cap > c->group && c->buffer_cap % c->group)) return GEAR_ERR_SHAPE;
  // a capacity that is not a multiple of 16 (the paper's n_b = 20): the flushed buffer must be a single block
  if (c->buffer_cap % 16 && !per_vector && c->buffer_cap > c->group) return GEAR_ERR_SHAPE;
  if (c->rank_flush < 0 || c->rank_flush > kMaxRank || c->rank_max < 0 || c->rank_max > kMaxRank) return GEAR_ERR_ARG;
  if (c->rank_flush > c->rank_max) return GEAR_ERR_ARG;
  if (c->rank_flush > c->buffer_cap) return GEAR_ERR_SHAPE;
  if (c->max_queries > 64) return GEAR_ERR_ARG;
  if (c->power_iters < 1 || c->power_iters > 64) return GEAR_ERR_ARG;
  const int gv = per_vector || c->group > kHeadDim ? kHeadDim : c->group;
  const int kv = outlier_count(c->outlier_pct, gv);
  if (kv > kMaxOutliers || (kv > 0 && 2 * kv >= gv)) return GEAR_ERR_SHAPE;
  const int tf = per_vector || c->buffer_cap < c->group ? c->buffer_cap : c->group;
  const int kf = outlier_count(c->outlier_pct, tf);
  if (kf > kMaxOutliers || (kf > 0 && 2 * kf >= tf)) return GEAR_ERR_SHAPE;
  return GEAR_OK;
}

static SegDesc shape_segment(const gear_cache* c, int n_c, int rank) {
  SegDesc s;
  memset(&s, 0, sizeof(s));
  s.n_c = n_c;
  s.rank = rank;
  if (c->cfg.group == GEAR_GROUP_PER_VECTOR && n_c > 128) {
    // one key group per channel over the whole segment: 64-token record blocks without outlier slots, the
    // outliers in a list behind the records (csr_base16 is set when the segment is placed)
    s.T = 64;
    s.k_k = 0;
    s.csr_k = 2 * outlier_count(c->cfg.outlier_pct, n_c);
    s.csr_base16 = 1;
  } else {
    s.T = c->cfg.group == GEAR_GROUP_PER_VECTOR || n_c < c->cfg.group ? n_c : c->cfg.group;
    s.k_k = outlier_count(c->cfg.outlier_pct, s.T);
  }
  layout_segment(s, c->cc);
  return s;
}

extern "C" void gear_free(gear_cache* c) {
  if (!c) return;
  // kernels queued by the host-buffer calls still read the ring and write the caller's memory
  if (c->host_last >= 0) cudaEventSynchronize(c->host.ev[c->host_last]);
  const DeviceAllocator& m = c->mem;
  // A pool may hand the memory to work of its own stream at once.  Off the default stream nothing says that this is the stream
  // of the kernels that are still queued here.
  if (m.free && c->off_default && cudaDeviceSynchronize() != cudaSuccess) cudaGetLastError();
  m.put(c->arena); m.put(c->dbg); m.put(c->table_dev); m.put(c->buf_k);
  m.put(c->partial); m.put(c->tickets);
  m.put(c->stage_q); m.put(c->stage_out); m.put(c->stage_b0);
  host_block_put(c->host);
  delete c;
}

// Next slot of the pinned ring: key rows, value rows, query.  The ring is made by the first host-buffer call: a cache that
// lives on device buffers alone does not pay for it.
static size_t host_row_bytes(const gear_cache* c) { return (size_t)c->cc.BH * kHeadDim * 2; }
static size_t host_query_bytes(const gear_cache* c) { return (size_t)c->cfg.batch * c->cfg.n_q_heads * kHeadDim * 2; }
static gear_status host_slot(gear_cache* c, unsigned char** mem, int* slot) {
  const size_t bytes = 2 * host_row_bytes(c) + host_query_bytes(c);       // a multiple of 256
  if (!c->host.mem && !host_block_get(bytes * kHostSlots, c->device, &c->host)) return GEAR_ERR_ALLOC;
  const int i = c->host_next;
  if (c->host_used[i] && cudaEventSynchronize(c->host.ev[i]) != cudaSuccess) { cudaGetLastError(); return GEAR_ERR_CUDA; }
  c->host_used[i] = false;
  c->host_next = (i + 1) % kHostSlots;
  *mem = c->host.mem + (size_t)i * bytes;
  *slot = i;
  return GEAR_OK;
}
static bool host_slot_done(gear_cache* c, int slot, cudaStream_t st) {    // everything that uses the slot has been queued
  if (cudaEventRecord(c->host.ev[slot], st) != cudaSuccess) { cudaGetLastError(); return false; }
  c->host_used[slot] = true;
  c->host_last = slot;
  return true;
}
// A call that fails between taking a slot and queueing its event may have queued a reader of it.
static gear_status host_slot_failed(gear_cache* c, int slot, cudaStream_t st, gear_status s) {
  host_slot_done(c, slot, st);
  return s;
}

static bool note_stream(gear_cache* c, cudaStream_t st) {                 // whether it is another stream than the default one
  const bool off = st != nullptr && st != cudaStreamLegacy;
  c->off_default = c->off_default || off;
  return off;
}

// The merge counters and the status word start at zero on the stream of the first call that writes the cache, so that
// creating one does not wait for the device.  Off the default stream memory of the caller's allocator may still be in use by
// work of the stream that the allocator belongs to: wait for that once.
static bool scratch_zeroed(gear_cache* c, cudaStream_t st) {
  if (c->scratch_clean) return true;
  if (note_stream(c, st) && c->mem.alloc && order_key(st).capture == 0 && cudaDeviceSynchronize() != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  if (cudaMemsetAsync(c->tickets, 0, ((size_t)c->units_alloc + 1) * 4, st) != cudaSuccess) { cudaGetLastError(); return false; }
  c->scratch_clean = true;
  return true;
}

// Query rows per pass over the cache for G rows per kv head and `nb` blocks.  Eight rows share what a block costs once, but a
// block then takes longer and there are half as many: that pays where the CTAs have long ranges and the last pass is more than
// half full.  Blocks per CTA (of 592) when eight rows go together, and the time of fours over that of eights (5 to 32 rows,
// groups of 64 and 128, 2 and 4 bits): below 2 0.48 to 1.04, 6 to 8 0.87 to 1.06, 10 to 12 0.98 to 1.12, above 12 1.03 to 1.15;
// with the last pass half empty 1.02 at most.  16 rows, 2 bits, groups of 64, 4096 tokens, us for fours and eights: 8 heads 18.9 / 27.1, 16
// 28.8 / 32.6, 32 51.7 / 50.5, 128 166.6 / 153.7; 12 rows, 32 heads x 16384 124 / 148.
// Two rows go one at a time through the kernel of one row where the ranges are long: the fours' kernel does most of its work for
// rows that are absent then (us for four and one at a time, blocks per SM: 2 bits, groups of 64 110 85.8 / 61.7, 55 47.9 / 36.8,
// 28 29.4 / 27.0 and 33.2 / 28.4, 14 21.0 / 23.3; groups of 128 55 62.2 / 56.2; 4 bits 110 85.5 / 73.7, 28 32.8 / 35.7; groups
// of 32 110 117.1 / 94.3, but of 16, with eight value scales a token, 126 / 157).
static int rows_per_pass(const gear_cache* c, int G, long long nb) {
  if (G == 2 && c->cc.ngv <= 4 && c->cc.BH * nb >= 40LL * c->sm_count) return 1;
  if (G <= 4) return G == 1 ? 1 : 4;
  if (decode_passes(G, 4) % 2) return 4;
  return c->cc.BH * nb * decode_passes(G, 8) >= 10LL * c->sm_count * kRowsCtasPerSm ? 8 : 4;
}

// Partial results of a launch for G query rows per kv head, hp at a time: slots per unit (a unit's share of the launch's CTAs,
// the first and the last of which may be shared with its neighbours), and the bytes of all slots.
static int partial_slots(const gear_cache* c, int G, int hp) {
  const size_t units = (size_t)c->cc.BH * decode_passes(G, hp);
  const size_t ctas = (size_t)c->sm_count * (hp == 1 ? 32 : kRowsCtasPerSm);
  return (int)(ctas / units + 3);
}
static size_t partial_bytes_for(const gear_cache* c, int G, int hp) {
  return (size_t)c->cc.BH * decode_passes(G, hp) * partial_slots(c, G, hp) * (size_t)hp * kPartRow * 4;
}

#define GEAR_TRY_ALLOC(ptr, bytes)                                                   \
  do {                                                                               \
    *reinterpret_cast<void**>(&(ptr)) = c->mem.get(bytes);                           \
    if ((ptr) == nullptr) {                                                          \
      gear_free(c);                                                                  \
      return GEAR_ERR_ALLOC;                                                         \
    }                                                                                \
  } while (0)

extern "C" gear_status gear_create(gear_cache** out, const gear_config* cfg) {
  if (!out || *out) return GEAR_ERR_ARG;
  gear_status st = check_config(cfg);
  if (st != GEAR_OK) return st;
  gear_cache* c = new (std::nothrow) gear_cache();
  if (!c) return GEAR_ERR_ALLOC;
  c->cfg = *cfg;
  {
    std::lock_guard<std::mutex> lock(g_alloc_mutex);
    c->mem.alloc = g_alloc; c->mem.free = g_free; c->mem.ctx = g_alloc_ctx;
  }
  c->test_dead_wait = 0;
  c->arena = nullptr; c->dbg = nullptr; c->table_dev = nullptr; c->blk2seg = nullptr; c->buf_k = c->buf_v = nullptr;
  c->partial = nullptr; c->tickets = nullptr; c->status = nullptr;
  c->scratch_clean = false;
  c->off_default = false;
  c->stage_q = nullptr; c->stage_out = nullptr; c->stage_b0 = nullptr;
  memset(&c->host, 0, sizeof(c->host));
  for (bool& u : c->host_used) u = false;
  c->host_next = 0; c->host_last = -1;
  c->cc.bits = cfg->bits;
  c->cc.g_v = cfg->group == GEAR_GROUP_PER_VECTOR || cfg->group > kHeadDim ? kHeadDim : cfg->group;
  c->cc.ngv = kHeadDim / c->cc.g_v;
  c->cc.k_v = outlier_count(cfg->outlier_pct, c->cc.g_v);
  c->cc.BH = cfg->batch * cfg->n_kv_heads;
  c->cc.n_b = cfg->buffer_cap;
  c->G = cfg->n_q_heads / cfg->n_kv_heads;
  c->buf_len = 0; c->n_compressed = 0; c->n_blocks_c = 0; c->plan_key = -1;
  if (cudaGetDevice(&c->device) != cudaSuccess ||
      cudaDeviceGetAttribute(&c->sm_count, cudaDevAttrMultiProcessorCount, c->device) != cudaSuccess) {
    delete c;
    return GEAR_ERR_CUDA;
  }
  const size_t BH = c->cc.BH;
  // arena: worst bytes per token over the two segment shapes the cache can see (full groups at rank_max,
  // flushed buffers at rank_flush), plus the per-segment B factors
  const int n_b = cfg->buffer_cap;
  const bool per_vector = cfg->group == GEAR_GROUP_PER_VECTOR;
  SegDesc sp = shape_segment(c, per_vector ? 192 : cfg->group, cfg->rank_max);
  SegDesc sf = shape_segment(c, n_b, cfg->rank_flush);
  const double dens_p = (double)sp.rec_bytes / sp.T, dens_f = (double)sf.rec_bytes / sf.T;
  const double dens = dens_p > dens_f ? dens_p : dens_f;
  const size_t n_flush_max = (size_t)(cfg->max_tokens / n_b) + 1;
  size_t per_bh = (size_t)(dens * (double)cfg->max_tokens) + n_flush_max * sf.bfac_bytes + 8 * (size_t)sp.bfac_bytes +
                  16 * (size_t)(sp.rec_bytes > sf.rec_bytes ? sp.rec_bytes : sf.rec_bytes);
  if (per_vector)      // outlier lists of per-vector key segments: offsets per block, entries per channel (rounded up per segment)
    per_bh += (size_t)(cfg->max_tokens / 64 + 8) * 4 + 64 * 16 +
              (size_t)kHeadDim * 4 * (2 * (size_t)outlier_count(cfg->outlier_pct, (int)cfg->max_tokens) + 2 * 8);
  c->arena_bytes = align_up(per_bh, 256) * BH + 4096;
  c->arena_used = 0;
  GEAR_TRY_ALLOC(c->arena, c->arena_bytes);
  c->table_cap = (int)(cfg->max_tokens / 16 + 8);
  c->blk_cap = c->table_cap;
  GEAR_TRY_ALLOC(c->table_dev, (sizeof(SegDesc) + sizeof(int)) * (size_t)c->table_cap);
  c->blk2seg = reinterpret_cast<int*>(c->table_dev + c->table_cap);
  GEAR_TRY_ALLOC(c->buf_k, 2 * BH * n_b * kHeadDim * 2);
  c->buf_v = reinterpret_cast<__half*>(c->buf_k) + BH * n_b * kHeadDim;
  if (cfg->flags & GEAR_FLAG_KEEP_FP32_FACTORS) {
    const size_t rm = cfg->rank_max > 0 ? cfg->rank_max : 1;
    c->dbg_bytes = (BH * 2 * (size_t)cfg->max_tokens * rm + BH * 2 * kHeadDim * rm * (size_t)c->table_cap) * 4;
    c->dbg_used = 0;
    GEAR_TRY_ALLOC(c->dbg, c->dbg_bytes);
  }
  // decode scratch: one partial per (unit, warp touching it), for every count of query rows that a call may bring and the rows
  // per pass it may take.  The bytes do not grow with the count (more units leave fewer slots to each), so the largest count
  // alone would not do.
  c->max_queries = cfg->max_queries > 1 ? (int)cfg->max_queries : 1;
  c->units_alloc = 0; c->partial_bytes = 0;
  for (int nq = 1; nq <= c->max_queries; ++nq) {
    const int G = c->G * nq;
    for (int hp : {1, 4, 8}) {
      if (hp == 1 ? G > 2 : hp == 4 ? G == 1 : G <= 4) continue;          // what rows_per_pass may return
      const size_t n = partial_bytes_for(c, G, hp);
      if (n > c->partial_bytes) c->partial_bytes = n;
      const int un = (int)(BH * decode_passes(G, hp));
      if (un > c->units_alloc) c->units_alloc = un;
    }
  }
  const size_t units = (size_t)c->units_alloc;
  GEAR_TRY_ALLOC(c->partial, c->partial_bytes);
  GEAR_TRY_ALLOC(c->tickets, (units + 1) * 4);
  c->status = c->tickets + units;
  const size_t q_bytes = host_query_bytes(c);
  GEAR_TRY_ALLOC(c->stage_q, q_bytes);
  GEAR_TRY_ALLOC(c->stage_out, 2 * q_bytes);
  GEAR_TRY_ALLOC(c->stage_b0, BH * 2 * kHeadDim * (size_t)(cfg->rank_flush > 0 ? cfg->rank_flush : 1) * 4);
  *out = c;
  return GEAR_OK;
}

// Append one compressed segment built from K, V [BH][n][128] on the device.
static gear_status compress_segment(gear_cache* c, const void* K, const void* V, int n, int rank, const float* B0,
                                    cudaStream_t st) {
  if ((int)c->segs.size() >= c->table_cap) return GEAR_ERR_CAPACITY;
  if (c->n_compressed + n > c->cfg.max_tokens) return GEAR_ERR_CAPACITY;
  SegDesc sd = shape_segment(c, n, rank);
  if (c->n_blocks_c + sd.nblk > c->blk_cap) return GEAR_ERR_CAPACITY;
  if (sd.k_k > kMaxOutliers || (sd.k_k > 0 && 2 * sd.k_k >= sd.T)) return GEAR_ERR_SHAPE;
  size_t need = align_up((size_t)sd.bh_stride, 16) * c->cc.BH;
  sd.bh_stride = (long long)align_up((size_t)sd.bh_stride, 16);
  const bool per_vector = sd.csr_base16 != 0;
  if (per_vector) {
    if (!kcvt_fits(n) || sd.csr_k >= n || (need >> 4) > 0xFFFFFFFFull) return GEAR_ERR_SHAPE;
    sd.csr_base16 = (unsigned int)(need >> 4);
    need += align_up((size_t)csr_stride_bytes(sd.nblk, sd.csr_k) * c->cc.BH, 16);
  }
  if (c->arena_used + need > c->arena_bytes) return GEAR_ERR_CAPACITY;
  sd.seg_base = (long long)c->arena_used;
  sd.tok_start = (int)c->n_compressed;
  sd.blk_start = c->n_blocks_c;
  sd.dbg_base = -1;
  sd.shape_id = static_shape_id(sd, c->cc);
  float* dbgA = nullptr; float* dbgB = nullptr;
  long long offA = -1, offB = -1;
  if (c->dbg && rank > 0) {
    const size_t nA = (size_t)c->cc.BH * 2 * n * rank, nB = (size_t)c->cc.BH * 2 * kHeadDim * rank;
    if ((c->dbg_used + nA + nB) * 4 > c->dbg_bytes) return GEAR_ERR_CAPACITY;
    offA = (long long)c->dbg_used; offB = offA + (long long)nA;
    dbgA = c->dbg + offA; dbgB = c->dbg + offB;
  }
  CompressJob job;
  job.seg = sd; job.cc = c->cc; job.arena = c->arena;
  job.K = (const __half*)K; job.V = (const __half*)V; job.B0 = B0;
  job.dbgA = dbgA; job.dbgB = dbgB;
  job.seed = c->cfg.seed; job.segment_index = (int)c->segs.size(); job.iters = c->cfg.power_iters;
  job.sms = c->sm_count; job.status = c->status; job.test_dead_wait = c->test_dead_wait;

  const CallOrder::Key key = order_key(st);
  const uint64_t begun = g_order.begin();
  cudaError_t e = cudaSuccess;
  note_stream(c, st);
  if (!scratch_zeroed(c, st)) return GEAR_ERR_CUDA;
  if (sd.T % 16) {     // the last slab of every block is partly empty: its codes, factor rows and scales read as zero
    if (cudaMemsetAsync(c->arena + sd.seg_base, 0, need, st) != cudaSuccess) { cudaGetLastError(); return GEAR_ERR_CUDA; }
    if (!compress_tile_fits(sd.T, sd.n_c, sd.rank)) return GEAR_ERR_SHAPE;
  }
  if (!per_vector && compress_tile_fits(sd.T, sd.n_c, sd.rank)) {
    e = compress_tile(job, c->cc.BH, st);              // short segment: one launch, residual in shared memory
  } else {
    // Bounded transient workspace, (batch, head) pairs processed in ranges.  Flushes of buffers too long for one launch take it
    // from the pool like prompts: held by every cache it was 235 MB for 256 pairs of 256 tokens at rank 4, 7.5 GB for 32 layers.
    // (Kept small by ranges instead, 88 MB, such a flush took 350 us and not 235, of 64 pairs 365 and not 110.)
    const size_t budget = (size_t)3 << 30;
    auto bytes_of = [&](int nbh) { return compress_workspace_bytes(nbh, sd, c->cc, c->sm_count); };
    int ranges = 1, chunk = c->cc.BH;
    while (chunk > 1 && bytes_of(chunk) > budget) chunk = (c->cc.BH + ++ranges - 1) / ranges;      // equal ranges
    unsigned char* ws = nullptr;
    const size_t ws_bytes = bytes_of(chunk);
    cudaMemPool_t pool = workspace_pool(c->device);
    if (pool == nullptr || cudaMallocFromPoolAsync((void**)&ws, ws_bytes, pool, st) != cudaSuccess) {
      cudaGetLastError();
      return GEAR_ERR_ALLOC;
    }
    for (int bh0 = 0; bh0 < c->cc.BH && e == cudaSuccess; bh0 += chunk) {
      const int nbh = bh0 + chunk <= c->cc.BH ? chunk : c->cc.BH - bh0;
      e = compress_range(job, bh0, nbh, ws, st);
    }
    cudaFreeAsync(ws, st);
  }
  if (e != cudaSuccess) { cudaGetLastError(); return GEAR_ERR_CUDA; }
  e = launch_write_desc(c->table_dev, c->blk2seg, (int)c->segs.size(), sd, st);
  if (e != cudaSuccess) { cudaGetLastError(); return GEAR_ERR_CUDA; }
  c->segs.push_back(sd);
  c->dbgA_off.push_back(offA); c->dbgB_off.push_back(offB);
  if (offA >= 0) c->dbg_used += (size_t)c->cc.BH * 2 * n * rank + (size_t)c->cc.BH * 2 * kHeadDim * rank;
  c->arena_used += need;
  c->n_compressed += n;
  c->n_blocks_c += sd.nblk;
  c->plan_key = -1;
  g_order.queued(key, begun);
  c->seg_write = g_order.written(key);
  return GEAR_OK;
}

extern "C" gear_status gear_compress(gear_cache** cache, const gear_config* cfg, const void* K, const void* V,
                                     int64_t n, int32_t rank, const float* B0, void* stream) {
  if (!cache || !K || !V) return GEAR_ERR_ARG;
  if (((uintptr_t)K | (uintptr_t)V) & 15) return GEAR_ERR_ALIGN;
  const gear_config* use = *cache ? &(*cache)->cfg : cfg;
  if (!use) return GEAR_ERR_ARG;
  gear_status st = check_config(use);
  if (st != GEAR_OK) return st;
  if (n < 16 || n % 16 || n > (1 << 30)) return GEAR_ERR_SHAPE;
  if (use->group == GEAR_GROUP_PER_VECTOR ? (n > 128 && n % 64) : (n >= use->group && n % use->group)) return GEAR_ERR_SHAPE;
  if (rank < 0 || rank > use->rank_max || rank > n) return GEAR_ERR_ARG;
  bool created = false;
  if (!*cache) {
    st = gear_create(cache, cfg);
    if (st != GEAR_OK) return st;
    created = true;
  }
  gear_cache* c = *cache;
  if (c->buf_len != 0) return GEAR_ERR_STATE;
  st = compress_segment(c, K, V, (int)n, rank, B0, (cudaStream_t)stream);
  if (st != GEAR_OK && created) { gear_free(c); *cache = nullptr; }
  return st;
}

// Push one token's rows (and bring a query along, q_src != nullptr); compresses the buffer when the push fills it.
static gear_status push_rows(gear_cache* c, const void* k_new, const void* v_new, const void* q_src, bool host_src,
                             const float* B0_flush, cudaStream_t st) {
  const int n_b = c->cfg.buffer_cap;
  if (c->buf_len + 1 == n_b) {     // this push will flush: make sure the segment fits before touching anything
    if (c->n_compressed + n_b > c->cfg.max_tokens || (int)c->segs.size() >= c->table_cap) return GEAR_ERR_CAPACITY;
  }
  note_stream(c, st);
  if (!scratch_zeroed(c, st)) return GEAR_ERR_CUDA;
  PushArgs a;
  a.buf_k = (__half*)c->buf_k; a.buf_v = (__half*)c->buf_v; a.k_new = (const __half*)k_new; a.v_new = (const __half*)v_new;
  a.q_src = (const __half*)q_src; a.q_dst = (__half*)c->stage_q; a.q_pieces = q_src ? (int)(host_query_bytes(c) / 16) : 0;
  a.BH = c->cc.BH; a.n_b = n_b; a.slot = c->buf_len; a.host_src = host_src ? 1 : 0;
  const CallOrder::Key key = order_key(st);
  const uint64_t begun = g_order.begin();
  if (launch_push(a, st) != cudaSuccess) {
    cudaGetLastError();
    return GEAR_ERR_CUDA;
  }
  g_order.queued(key, begun);
  c->buf_write = g_order.written(key);
  c->buf_len += 1;
  if (c->buf_len < n_b) return GEAR_OK;
  gear_status s = compress_segment(c, c->buf_k, c->buf_v, n_b, c->cfg.rank_flush, B0_flush, st);
  if (s != GEAR_OK) { c->buf_len -= 1; return s; }
  c->buf_len = 0;
  return GEAR_FLUSHED;
}

extern "C" gear_status gear_append_buffer(gear_cache* c, const void* k_new, const void* v_new, const float* B0_flush,
                                          void* stream) {
  if (!c || !k_new || !v_new) return GEAR_ERR_ARG;
  if (((uintptr_t)k_new | (uintptr_t)v_new) & 15) return GEAR_ERR_ALIGN;
  return push_rows(c, k_new, v_new, nullptr, false, B0_flush, (cudaStream_t)stream);
}

static gear_status plan_decode(gear_cache* c, int Gq, int hp) {
  // One-head passes: with four warps per scheduler the warps of a scheduler slow one another down by more than
  // the fourth warp adds (measured: 3 warps finish 0.85 blocks per microsecond and scheduler, 4 warps 0.79), so
  // long streams run with twelve resident warps.  Short streams (few blocks per warp) keep sixteen: there the
  // fixed cost per warp and the granularity of the split weigh more.
  int warps_cap = 0;
  if (hp == 1) {
    const long long blocks = (long long)c->cc.BH * Gq * (c->n_blocks_c + (c->buf_len + 15) / 16);
    if (blocks >= 24LL * 16 * c->sm_count) warps_cap = 12;
  }
  // everything else the plan depends on is fixed by the segments: a push that does not flush keeps it (asking the driver
  // for the occupancy again costs a microsecond and a half per decoding step)
  const long long key = (((long long)c->segs.size() * 8192 + Gq) * 2 + (warps_cap ? 1 : 0)) * 16 + hp;
  if (c->plan_key == key) return GEAR_OK;
  int max_k = 0, max_v = 0, max_bfac = 0, max_T = 16;
  for (const SegDesc& s : c->segs) {
    if (s.off_vpart > max_k) max_k = s.off_vpart;
    if (s.rec_bytes - s.off_vpart > max_v) max_v = s.rec_bytes - s.off_vpart;
    if (s.bfac_bytes > max_bfac) max_bfac = s.bfac_bytes;
    if ((s.T + 31) / 32 * 32 > max_T) max_T = (s.T + 31) / 32 * 32;
  }
  if (hp == 1 ? !decode_plan(c->cc.bits, hp, c->cc.ngv, max_k, max_v, max_bfac, max_T, kDecodeSmemBudget, warps_cap, &c->plan)
              : !rows_plan(hp, c->cc.ngv, max_k, max_v, max_bfac, max_T, &c->plan))
    return GEAR_ERR_SHAPE;
  int occ = hp == 1 ? decode_occupancy(c->cc.bits, hp, c->cc.ngv, c->plan.wide, (size_t)c->plan.ws.total)
                    : rows_occupancy(c->plan, c->cc.bits, c->cc.ngv);
  if (hp > 1 && occ > kRowsCtasPerSm) occ = kRowsCtasPerSm;      // what the partial slots are for
  if (occ < 1) return GEAR_ERR_CUDA;
  c->plan_occ = occ;
  c->plan_key = key;
  return GEAR_OK;
}

// Decode attention for Gq query rows per kv head: q, out [B][H][Gq][128] (Gq = G for one query per head).
static gear_status decode_rows(gear_cache* c, const void* q, float* out, int Gq, float softmax_scale, void* stream) {
  if (!c || !q || !out) return GEAR_ERR_ARG;
  if (((uintptr_t)q | (uintptr_t)out) & 15) return GEAR_ERR_ALIGN;
  if (c->n_compressed == 0 && c->buf_len == 0) return GEAR_ERR_STATE;
  note_stream(c, (cudaStream_t)stream);
  const int hp = rows_per_pass(c, Gq, c->n_blocks_c), passes = decode_passes(Gq, hp);
  const int buf_block = hp == 1 ? 16 : kRowsBufBlock;
  const long long nblocks = c->n_blocks_c + (c->buf_len + buf_block - 1) / buf_block;
  gear_status s = plan_decode(c, Gq, hp);
  if (s != GEAR_OK) return s;
  DecodeArgs a = c->plan;
  a.arena = c->arena; a.table = c->table_dev; a.blk2seg = c->blk2seg;
  a.buf_k = (const __half*)c->buf_k; a.buf_v = (const __half*)c->buf_v;
  a.q = (const __half*)q; a.out = out; a.partial = c->partial; a.tickets = c->tickets; a.status = c->status;
  a.cc = c->cc; a.n_blocks_c = c->n_blocks_c; a.buf_len = c->buf_len;
  a.n_kv_heads = c->cfg.n_kv_heads; a.group_heads = Gq;
  const float sc = softmax_scale > 0.f ? softmax_scale : 1.0f / sqrtf((float)kHeadDim);
  a.scale_log2 = sc * 1.4426950408889634f;
  a.test_dead_wait = c->test_dead_wait;
  const CallOrder::Key key = order_key((cudaStream_t)stream);
  const uint64_t begun = g_order.begin();
  a.early_reads = g_order.another_since(key, c->seg_write) ? 1 : 0;
  a.early_buf = c->buf_write.number == 0 || g_order.another_since(key, c->buf_write) ? 1 : 0;
  // never more CTAs than blocks of work
  if ((long long)c->cc.BH * passes > c->units_alloc) return GEAR_ERR_CAPACITY;
  a.max_parts = partial_slots(c, Gq, hp);
  if (partial_bytes_for(c, Gq, hp) > c->partial_bytes) return GEAR_ERR_CAPACITY;
  const long long work = (long long)c->cc.BH * passes * nblocks;
  long long grid = (long long)c->sm_count * c->plan_occ;
  if (grid > work) grid = work;
  // Ranges of one or two blocks: a warp's partial result, its ticket and the merge of up to 64 partials then take as long as
  // the blocks themselves (8 of 15 us for one sequence of 3800 tokens and 32 heads).  Several warps of a unit share a CTA
  // and join in shared memory instead, if that leaves nobody more blocks than one warp per CTA would: the fewest CTAs per
  // unit (one needs no ticket at all), then the fewest warps.  Warps of a CTA wait for one another and for one SM, so with
  // idle SMs about (little work) that has to be worth it.  Where the lines lie (2 bits, groups of 64, rank 4; us without and
  // with):
  //   one CTA per unit       up to ten warps always (8 heads of 10 blocks 7.85 / 7.34), more from 400 blocks of work on
  //                          (8 heads of 14 blocks 7.85 / 8.36, 64 heads 9.81 / 8.70)
  //   several CTAs           of four to eight warps (one head of 66 blocks: 10.55 / 10.5 with 2 or 14, 8.85 with 8); few
  //                          partials only where there is much work, because their merge is short (one head of 26 blocks
  //                          8.36 / 8.50, of 34 8.87 / 8.53, 16 heads of 18 9.20 / 9.01, of 14 8.28 / 9.04); not where a
  //                          few SMs would get a second CTA (32 heads of 34 blocks: 160 CTAs 11.25, 192 10.55)
  if (Gq == 1 && !c->plan.wide) {
    const long long units = c->cc.BH, nb = work / units;
    const long long p1 = grid / units > 1 ? (grid / units < nb ? grid / units : nb) : 1;
    const long long len = (nb + p1 - 1) / p1;
    long long best = 0;
    int best_w = 0;
    if (len <= 2 && nb > 1)
      for (int w = 2; w <= 16 && w <= c->plan_occ; ++w) {
        const long long slots = (long long)c->sm_count * (c->plan_occ / w);
        const long long need = (nb + len * w - 1) / (len * w);            // CTAs per unit for ranges of `len` blocks
        if (need * units > slots || need >= a.max_parts) continue;
        if (need == 1 ? w > 10 && work < 400
                      : w < 4 || w > 8 || (nb <= 32 && work < 200) || (nb <= 16 && work < 400) ||
                            (need * units > c->sm_count && 4 * need * units < 5 * c->sm_count)) continue;
        if (best_w == 0 || need < best) { best = need; best_w = w; }
      }
    if (best_w) { a.cta_warps = best_w; a.unit_ctas = (int)best; grid = best * units; }
  }
  // With few blocks per warp, a warp that runs from one unit into the next pays a second prologue and epilogue and
  // finishes last.  When every unit gets at least six warps, cut each unit into ranges of its own instead: the first
  // units into one range more than the others so that every resident warp has work, and order the CTAs by the length
  // of their range, longest first (the hardware dispatches them in index order, and the oldest warps of an SM
  // finish first).  Otherwise (many blocks per warp) cut the flat space evenly.
  if (a.unit_ctas == 0) {
    const long long units = (long long)c->cc.BH * passes, nb = work / units;
    const long long pb = grid / units, ua = grid - pb * units;         // ua units get pb + 1 ranges
    if (pb >= 6 && pb + 1 <= nb && pb + 1 < a.max_parts) {
      a.aligned = 1;
      a.units_a = (int)ua; a.parts_a = (int)pb + 1; a.parts_b = (int)pb;
      struct Cls { int len, u0, nu, p0, n; } cls[4];
      const int base_a = (int)(nb / (pb + 1)), rem_a = (int)(nb % (pb + 1));
      const int base_b = (int)(nb / pb), rem_b = (int)(nb % pb);
      cls[0] = {base_b + 1, (int)ua, (int)(units - ua), 0, rem_b};
      cls[1] = {base_b, (int)ua, (int)(units - ua), rem_b, (int)pb - rem_b};
      cls[2] = {base_a + 1, 0, (int)ua, 0, rem_a};
      cls[3] = {base_a, 0, (int)ua, rem_a, (int)pb + 1 - rem_a};
      for (int i = 1; i < 4; ++i)                                       // insertion sort, longest first, stable
        for (int j = i; j > 0 && cls[j].len > cls[j - 1].len; --j) { const Cls t = cls[j]; cls[j] = cls[j - 1]; cls[j - 1] = t; }
      int start = 0;
      for (int k = 0; k < 4; ++k) {
        a.cls_start[k] = start; a.cls_u0[k] = cls[k].u0; a.cls_n[k] = cls[k].n > 0 ? cls[k].n : 1; a.cls_p0[k] = cls[k].p0;
        start += cls[k].nu * cls[k].n;
      }
      a.cls_start[4] = start;
      grid = start;                                                     // = units * pb + ua
    }
  }
  if ((hp == 1 ? launch_decode(a, (int)grid, (cudaStream_t)stream) : launch_rows(a, (int)grid, (cudaStream_t)stream)) != cudaSuccess) {
    cudaGetLastError();
    return GEAR_ERR_CUDA;
  }
  g_order.queued(key, begun);
  return GEAR_OK;
}

extern "C" gear_status gear_decode_attn(gear_cache* c, const void* q, float* out, float softmax_scale, void* stream) {
  if (!c) return GEAR_ERR_ARG;
  return decode_rows(c, q, out, c->G, softmax_scale, stream);
}

extern "C" gear_status gear_decode_attn_multi(gear_cache* c, const void* q, float* out, int32_t n_queries,
                                              float softmax_scale, void* stream) {
  if (!c) return GEAR_ERR_ARG;
  if (n_queries < 1 || n_queries > c->max_queries) return GEAR_ERR_ARG;
  // The rows of one kv head -- its G query heads times n_queries positions -- are consecutive in q and out, and every
  // row attends to the whole cache: to the kernel they are G * n_queries query heads of that kv head.
  return decode_rows(c, q, out, c->G * n_queries, softmax_scale, stream);
}

extern "C" gear_status gear_append_buffer_host(gear_cache* c, const void* k_host, const void* v_host,
                                               const float* B0_host, void* stream) {
  if (!c || !k_host || !v_host) return GEAR_ERR_ARG;
  cudaStream_t st = (cudaStream_t)stream;
  const size_t rows = host_row_bytes(c);
  unsigned char* mem = nullptr;
  int slot = 0;
  gear_status s = host_slot(c, &mem, &slot);
  if (s != GEAR_OK) return s;
  memcpy(mem, k_host, rows);
  memcpy(mem + rows, v_host, rows);
  const float* b0 = nullptr;
  const bool with_b0 = B0_host && c->cfg.rank_flush > 0 && c->buf_len + 1 == c->cfg.buffer_cap;
  if (with_b0) {
    if (cudaMemcpyAsync(c->stage_b0, B0_host, (size_t)c->cc.BH * 2 * kHeadDim * c->cfg.rank_flush * 4,
                        cudaMemcpyHostToDevice, st) != cudaSuccess) {
      cudaGetLastError();
      return GEAR_ERR_CUDA;
    }
    b0 = c->stage_b0;
  }
  s = push_rows(c, mem, mem + rows, nullptr, true, b0, st);
  if (s < 0) return host_slot_failed(c, slot, st, s);
  if (!host_slot_done(c, slot, st)) return GEAR_ERR_CUDA;
  // the start vectors are read straight from the caller's memory: only then wait for the copy
  if (with_b0 && cudaStreamSynchronize(st) != cudaSuccess) { cudaGetLastError(); return GEAR_ERR_CUDA; }
  return s;
}

// Attention for the query in stage_q into host memory.  A pinned destination is written by the kernel itself (posted
// writes across the bus); any other goes through the device copy of the result.
static gear_status decode_to_host(gear_cache* c, float* out_host, float softmax_scale, cudaStream_t st) {
  cudaPointerAttributes at;
  float* direct = nullptr;
  if (cudaPointerGetAttributes(&at, out_host) != cudaSuccess) cudaGetLastError();
  else if (at.type == cudaMemoryTypeHost && at.devicePointer && ((uintptr_t)at.devicePointer & 15) == 0)
    direct = reinterpret_cast<float*>(at.devicePointer);
  gear_status s = gear_decode_attn(c, c->stage_q, direct ? direct : c->stage_out, softmax_scale, st);
  if (s != GEAR_OK || direct) return s;
  if (cudaMemcpyAsync(out_host, c->stage_out, 2 * host_query_bytes(c), cudaMemcpyDeviceToHost, st) != cudaSuccess) {
    cudaGetLastError();
    return GEAR_ERR_CUDA;
  }
  return GEAR_OK;
}

static gear_status decode_host(gear_cache* c, const void* q_host, float* out_host, float softmax_scale, void* stream,
                               bool wait) {
  if (!c || !q_host || !out_host) return GEAR_ERR_ARG;
  if (c->n_compressed == 0 && c->buf_len == 0) return GEAR_ERR_STATE;
  cudaStream_t st = (cudaStream_t)stream;
  unsigned char* mem = nullptr;
  int slot = 0;
  gear_status s = host_slot(c, &mem, &slot);
  if (s != GEAR_OK) return s;
  memcpy(mem, q_host, host_query_bytes(c));
  note_stream(c, st);
  PushArgs a;
  memset(&a, 0, sizeof(a));
  a.q_src = (const __half*)mem; a.q_dst = (__half*)c->stage_q; a.q_pieces = (int)(host_query_bytes(c) / 16); a.host_src = 1;
  if (launch_push(a, st) != cudaSuccess) { cudaGetLastError(); return GEAR_ERR_CUDA; }
  s = decode_to_host(c, out_host, softmax_scale, st);
  if (s != GEAR_OK) return host_slot_failed(c, slot, st, s);
  if (!host_slot_done(c, slot, st)) return GEAR_ERR_CUDA;
  return wait ? gear_cache_wait(c) : GEAR_OK;
}

extern "C" gear_status gear_decode_attn_host(gear_cache* c, const void* q_host, float* out_host, float softmax_scale,
                                             void* stream) {
  return decode_host(c, q_host, out_host, softmax_scale, stream, true);
}

extern "C" gear_status gear_decode_attn_host_async(gear_cache* c, const void* q_host, float* out_host,
                                                   float softmax_scale, void* stream) {
  return decode_host(c, q_host, out_host, softmax_scale, stream, false);
}

// One token of one layer through host buffers: push the rows, attend, all queued; two kernels.
extern "C" gear_status gear_step_host(gear_cache* c, const void* k_host, const void* v_host, const void* q_host,
                                      float* out_host, float softmax_scale, void* stream) {
  if (!c || !k_host || !v_host || !q_host || !out_host) return GEAR_ERR_ARG;
  cudaStream_t st = (cudaStream_t)stream;
  const size_t rows = host_row_bytes(c);
  unsigned char* mem = nullptr;
  int slot = 0;
  gear_status s = host_slot(c, &mem, &slot);
  if (s != GEAR_OK) return s;
  memcpy(mem, k_host, rows);
  memcpy(mem + rows, v_host, rows);
  memcpy(mem + 2 * rows, q_host, host_query_bytes(c));
  const gear_status pushed = push_rows(c, mem, mem + rows, mem + 2 * rows, true, nullptr, st);
  if (pushed < 0) return host_slot_failed(c, slot, st, pushed);
  s = decode_to_host(c, out_host, softmax_scale, st);
  if (s != GEAR_OK) return host_slot_failed(c, slot, st, s);
  if (!host_slot_done(c, slot, st)) return GEAR_ERR_CUDA;
  return pushed;
}

extern "C" gear_status gear_cache_wait(gear_cache* c) {
  if (!c) return GEAR_ERR_ARG;
  if (c->host_last >= 0 && cudaEventSynchronize(c->host.ev[c->host_last]) != cudaSuccess) {
    cudaGetLastError();
    return GEAR_ERR_CUDA;
  }
  return GEAR_OK;
}

extern "C" gear_status gear_fp16_decode_attn(const void* K, const void* V, const void* q, float* out, int32_t batch,
                                             int32_t n_q_heads, int32_t n_kv_heads, int32_t head_dim, int64_t n,
                                             int64_t n_alloc, float softmax_scale, void* scratch, size_t scratch_bytes,
                                             void* stream) {
  if (!K || !V || !q || !out || !scratch) return GEAR_ERR_ARG;
  if (batch < 1 || n_kv_heads < 1 || n_q_heads < 1 || n < 1 || n_alloc < n) return GEAR_ERR_ARG;
  if (n_alloc > 0x7fffffffLL) return GEAR_ERR_ARG;                  // token counts travel as 32-bit integers
  if (head_dim != kHeadDim || n_q_heads % n_kv_heads) return GEAR_ERR_SHAPE;
  if (((uintptr_t)K | (uintptr_t)V | (uintptr_t)q | (uintptr_t)out | (uintptr_t)scratch) & 15) return GEAR_ERR_ALIGN;
  if (scratch_bytes < gear_fp16_attn_scratch_bytes(batch, n_q_heads, head_dim)) return GEAR_ERR_CAPACITY;
  const float sc = softmax_scale > 0.f ? softmax_scale : 1.0f / sqrtf((float)kHeadDim);
  if (launch_fp16_attn(K, V, q, out, batch, n_q_heads, n_kv_heads, n, n_alloc, sc, scratch, scratch_bytes,
                       (cudaStream_t)stream) != cudaSuccess) {
    cudaGetLastError();
    return GEAR_ERR_CUDA;
  }
  return GEAR_OK;
}

extern "C" size_t gear_fp16_attn_scratch_bytes(int32_t batch, int32_t n_q_heads, int32_t head_dim) {
  (void)head_dim;
  return fp16_attn_scratch(batch, n_q_heads);
}

// ------------------------------------------------------------------ helpers
static size_t export_elems(const gear_cache* c, const SegDesc& s, int what, size_t* elem_bytes) {
  const size_t BH = c->cc.BH, d = kHeadDim;
  switch (what) {
    case GEAR_EXP_K_CODES: case GEAR_EXP_V_CODES: *elem_bytes = 1; return BH * s.n_c * d;
    case GEAR_EXP_K_SCALE: case GEAR_EXP_K_ZERO: *elem_bytes = 2; return BH * (s.csr_base16 ? 1 : s.nblk) * d;
    case GEAR_EXP_V_SCALE: case GEAR_EXP_V_ZERO: *elem_bytes = 2; return BH * s.n_c * c->cc.ngv;
    case GEAR_EXP_K_OUT_IDX:
      if (s.csr_base16) { *elem_bytes = 4; return BH * d * s.csr_k; }      // token in the segment, 32-bit
      *elem_bytes = 1; return BH * s.nblk * d * 2 * s.k_k;
    case GEAR_EXP_K_OUT_VAL: *elem_bytes = 2; return s.csr_base16 ? BH * d * s.csr_k : BH * s.nblk * d * 2 * s.k_k;
    case GEAR_EXP_V_OUT_IDX: *elem_bytes = 1; return BH * s.n_c * c->cc.ngv * 2 * c->cc.k_v;
    case GEAR_EXP_V_OUT_VAL: *elem_bytes = 2; return BH * s.n_c * c->cc.ngv * 2 * c->cc.k_v;
    case GEAR_EXP_K_A: case GEAR_EXP_V_A: case GEAR_EXP_K_A_FP32: case GEAR_EXP_V_A_FP32:
      *elem_bytes = 4; return BH * s.n_c * s.rank;
    case GEAR_EXP_K_B: case GEAR_EXP_V_B: case GEAR_EXP_K_B_FP32: case GEAR_EXP_V_B_FP32:
      *elem_bytes = 4; return BH * d * s.rank;
    default: *elem_bytes = 0; return 0;
  }
}

extern "C" gear_status gear_export(gear_cache* c, int32_t segment, int32_t what, void* host_dst, size_t bytes) {
  if (!c || (!host_dst && bytes)) return GEAR_ERR_ARG;
  if (what == GEAR_EXP_K_BUFFER || what == GEAR_EXP_V_BUFFER) {
    const size_t row = (size_t)c->buf_len * kHeadDim * 2;
    if (bytes != row * c->cc.BH) return GEAR_ERR_ARG;
    if (row == 0) return GEAR_OK;
    const void* src = what == GEAR_EXP_K_BUFFER ? c->buf_k : c->buf_v;
    if (cudaDeviceSynchronize() != cudaSuccess ||
        cudaMemcpy2D(host_dst, row, src, (size_t)c->cfg.buffer_cap * kHeadDim * 2, row, c->cc.BH,
                     cudaMemcpyDeviceToHost) != cudaSuccess) {
      cudaGetLastError();
      return GEAR_ERR_CUDA;
    }
    return GEAR_OK;
  }
  if (segment < 0 || segment >= (int)c->segs.size()) return GEAR_ERR_ARG;
  const SegDesc& s = c->segs[segment];
  size_t eb = 0;
  const size_t n = export_elems(c, s, what, &eb);
  if (eb == 0) return GEAR_ERR_ARG;
  if (bytes != n * eb) return GEAR_ERR_ARG;
  if (n == 0) return GEAR_OK;
  if (cudaDeviceSynchronize() != cudaSuccess) { cudaGetLastError(); return GEAR_ERR_CUDA; }
  if (what >= GEAR_EXP_K_A_FP32 && what <= GEAR_EXP_V_B_FP32) {
    if (!c->dbg || c->dbgA_off[segment] < 0) return GEAR_ERR_STATE;
    // stored as [BH][2][rows][rank]; gather the side
    const int side = what & 1;
    const bool isA = what == GEAR_EXP_K_A_FP32 || what == GEAR_EXP_V_A_FP32;
    const size_t rows = isA ? (size_t)s.n_c : (size_t)kHeadDim;
    const float* base = c->dbg + (isA ? c->dbgA_off[segment] : c->dbgB_off[segment]);
    const size_t tile = rows * s.rank * 4;
    if (cudaMemcpy2D(host_dst, tile, base + (size_t)side * rows * s.rank, 2 * tile, tile, c->cc.BH,
                     cudaMemcpyDeviceToHost) != cudaSuccess) {
      cudaGetLastError();
      return GEAR_ERR_CUDA;
    }
    return GEAR_OK;
  }
  void* tmp = nullptr;
  if (cudaMalloc(&tmp, bytes) != cudaSuccess) { cudaGetLastError(); return GEAR_ERR_ALLOC; }
  gear_status r = GEAR_OK;
  if (launch_export(c->arena, s, c->cc, what, tmp, n, 0) != cudaSuccess ||
      cudaMemcpy(host_dst, tmp, bytes, cudaMemcpyDeviceToHost) != cudaSuccess) {
    cudaGetLastError();
    r = GEAR_ERR_CUDA;
  }
  cudaFree(tmp);
  return r;
}

extern "C" gear_status gear_cache_info(const gear_cache* c, gear_info* info) {
  if (!c || !info) return GEAR_ERR_ARG;
  info->n_segments = (int)c->segs.size();
  info->buffer_len = c->buf_len;
  info->n_compressed = c->n_compressed;
  return GEAR_OK;
}

extern "C" gear_status gear_segment_info_get(const gear_cache* c, int32_t segment, gear_segment_info* info) {
  if (!c || !info || segment < 0 || segment >= (int)c->segs.size()) return GEAR_ERR_ARG;
  const SegDesc& s = c->segs[segment];
  info->n_c = s.n_c; info->rank = s.rank; info->g_k = s.T; info->g_v = c->cc.g_v; info->k_k = s.k_k; info->k_v = c->cc.k_v;
  if (s.csr_base16 != 0) { info->g_k = s.n_c; info->k_k = s.csr_k / 2; }      // per-vector keys: the whole segment
  return GEAR_OK;
}

extern "C" gear_status gear_cache_bytes(const gear_cache* c, gear_bytes* out) {
  if (!c || !out) return GEAR_ERR_ARG;
  memset(out, 0, sizeof(*out));
  const long long BH = c->cc.BH, d = kHeadDim;
  for (const SegDesc& s : c->segs) {
    out->codes += BH * 2 * (long long)s.n_c * d * c->cc.bits / 8;
    out->scale_zero += BH * ((long long)s.nblk * d * 4 + (long long)s.n_c * c->cc.ngv * 4);
    out->outliers += BH * ((long long)s.nblk * d * 2 * s.k_k * 3 + (long long)s.n_c * c->cc.ngv * 2 * c->cc.k_v * 3);
    out->lowrank_a += BH * 2 * (long long)s.n_c * s.rank * 2;
    out->lowrank_b += BH * 2 * d * s.rank * 2;
    out->stored_total += BH * s.bh_stride;
    if (s.csr_base16 != 0) {     // per-vector keys: the list of the segment's key outliers (the records repeat the scales)
      const long long list = BH * (long long)csr_stride_bytes(s.nblk, s.csr_k);
      out->outliers += list;
      out->stored_total += list;
    }
  }
  out->buffer = BH * 2 * (long long)c->buf_len * d * 2;
  out->stored_total += out->buffer;
  out->alloc_total = (long long)(c->arena_bytes + c->dbg_bytes + c->partial_bytes +
                                 2 * (size_t)BH * c->cfg.buffer_cap * d * 2 + sizeof(SegDesc) * (size_t)c->table_cap);
  return GEAR_OK;
}

extern "C" gear_status gear_last_device_status(gear_cache* c, int32_t* code) {
  if (!c || !code) return GEAR_ERR_ARG;
  int v = 0;
  if (!c->scratch_clean) {                                // nothing that could have set the word has run
    *code = 0;
    if (cudaDeviceSynchronize() != cudaSuccess) { cudaGetLastError(); return GEAR_ERR_CUDA; }
    return GEAR_OK;
  }
  if (cudaDeviceSynchronize() != cudaSuccess || cudaMemcpy(&v, c->status, 4, cudaMemcpyDeviceToHost) != cudaSuccess ||
      cudaMemset(c->status, 0, 4) != cudaSuccess) {
    cudaGetLastError();
    return GEAR_ERR_CUDA;
  }
  if (v != 0) {
    // a warp that gave up left without taking its tickets: start the next call from a clean count
    const size_t units = (size_t)c->units_alloc;
    if (cudaMemset(c->tickets, 0, units * 4) != cudaSuccess) { cudaGetLastError(); return GEAR_ERR_CUDA; }
  }
  *code = v;
  return GEAR_OK;
}

extern "C" gear_status gear_test_dead_wait(gear_cache* c, int32_t on) {
  if (!c) return GEAR_ERR_ARG;
  c->test_dead_wait = on ? 1 : 0;
  return GEAR_OK;
}

extern "C" gear_status gear_fp16_attn_status(void* scratch, int32_t* code) {
  if (!scratch || !code) return GEAR_ERR_ARG;
  int v = 0;
  if (cudaDeviceSynchronize() != cudaSuccess || cudaMemcpy(&v, scratch, 4, cudaMemcpyDeviceToHost) != cudaSuccess ||
      cudaMemset(scratch, 0, 4) != cudaSuccess) {
    cudaGetLastError();
    return GEAR_ERR_CUDA;
  }
  *code = v;
  return GEAR_OK;
}

extern "C" const char* gear_strerror(gear_status s) {
  switch (s) {
    case GEAR_OK: return "ok";
    case GEAR_FLUSHED: return "buffer flushed";
    case GEAR_ERR_ARG: return "invalid argument";
    case GEAR_ERR_SHAPE: return "sizes violate the grouping rules";
    case GEAR_ERR_ALIGN: return "pointer not 16-byte aligned";
    case GEAR_ERR_CAPACITY: return "capacity exhausted";
    case GEAR_ERR_ALLOC: return "device allocation failed";
    case GEAR_ERR_CUDA: return "CUDA runtime error";
    case GEAR_ERR_TIMEOUT: return "bounded device-side wait gave up";
    case GEAR_ERR_STATE: return "call not valid in the cache's current state";
    default: return "unknown status";
  }
}
