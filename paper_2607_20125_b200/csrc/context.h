// The context behind the C ABI of include/headcast.h: device buffers, the state of the cache ring, the cached work
// lists, error reporting and the tensor maps of the cache buffers.  Private to headcast_api.cu (one translation unit).
#pragma once
#include "../../include/headcast.h"

#include <algorithm>
#include <cmath>
#include <cstdarg>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <map>
#include <mutex>
#include <queue>
#include <string>
#include <vector>

#include "attn_kernel.cuh"
#include "copy_kernels.cuh"
#include "move_kernels.cuh"
#include "score_kernels.cuh"
#include "tmap.h"

using namespace hc;

namespace {

enum { STATE_FILLING = 0, STATE_SPLIT = 1 };
enum { MAP_MONO = 0, MAP_SD = 1, MAP_GLOBAL = 2, MAP_SPATIAL = 3, N_MAP_PAIRS = 4 };

// Device memory of the contexts.  A layer's life starts with about thirty allocations, 400 MB at 30 x 52 tokens, and ends
// with giving them back; with cudaMalloc and cudaFree that took half of the 14.8 ms from create to destroy (3.5 us per MB
// and 55 us per small buffer each way), with blocks kept from the context before it takes 0.3 ms.  Per GPU at most
// CACHE_KEEP_BYTES are kept, the blocks given back last; older ones go to the system then and there, all of them and what
// the pool holds unused when an allocation of either kind fails.  A block is kept only if its last use has been waited
// for (see put), so it may serve any stream.
constexpr size_t CACHE_KEEP_BYTES = size_t(384) << 20;
constexpr unsigned long long MONO_KEEP_BYTES = 256ull << 20;  // the same for the monolithic caches, see get_mono

class BlockCache {
 public:
  // The cache of the current device, more exactly of the CUDA context that is current on it: after a device reset, or in
  // another context that a host made through the driver, an older context's memory must not come back.  nullptr: no context.
  static BlockCache* current(int dev) {
    unsigned long long id = 0;
    if (cudaFree(nullptr) != cudaSuccess || !current_context_id(&id)) return nullptr;
    static std::mutex lock;
    static auto& all = *new std::map<std::pair<int, unsigned long long>, BlockCache>;  // never destroyed: a context may outlive static objects
    std::lock_guard<std::mutex> hold(lock);
    return &all[std::make_pair(dev, id)];
  }
  // On the current device, which must be this cache's.  *got: the block's size.  `fresh`: by cudaMalloc, whatever is kept here.
  cudaError_t get(void** ptr, size_t bytes, size_t* got = nullptr, bool fresh = false) {
    const size_t need = round_up(bytes);
    std::lock_guard<std::mutex> hold(lock_);
    size_t at = free_.size();
    for (size_t i = 0; i < free_.size() && !fresh; ++i)
      if (free_[i].bytes >= need && free_[i].bytes <= need + need / 4 && (at == free_.size() || free_[i].bytes < free_[at].bytes)) at = i;
    if (at < free_.size()) {
      *ptr = free_[at].ptr;
      live_[*ptr] = free_[at].bytes;
      if (got) *got = free_[at].bytes;
      kept_ -= free_[at].bytes;
      free_.erase(free_.begin() + at);
      return cudaSuccess;
    }
    cudaError_t e = cudaMalloc(ptr, need);
    if (e == cudaErrorMemoryAllocation) {  // what is kept may be what is missing
      release_all();
      e = cudaMalloc(ptr, need);
    }
    if (e == cudaSuccess) live_[*ptr] = need;
    if (got) *got = need;
    return e;
  }
  // Gives a block back.  idle: since its last use the device has been waited for (wait_idle), or the one stream that orders all
  // its uses.  If not, the block goes through cudaFree, which waits itself, or refuses beside a stream capture: then it is set
  // aside until the device can be waited for.
  void put(void* ptr, bool idle) {
    std::lock_guard<std::mutex> hold(lock_);
    auto it = live_.find(ptr);
    if (it == live_.end()) return;
    const size_t bytes = it->second;
    live_.erase(it);
    if (!idle || bytes > CACHE_KEEP_BYTES) {
      give_up(ptr);
      return;
    }
    shrink(CACHE_KEEP_BYTES - bytes);
    free_.push_back({ptr, bytes});
    kept_ += bytes;
  }
  // The monolithic cache is released in the middle of a stream's work (at the split), so it comes from a stream-ordered pool
  // of its own instead of a block; the pool keeps at most MONO_KEEP_BYTES unused (the default pool keeps nothing: 2.8 ms per
  // 200 MB to map and unmap them again) and hands memory out again only once the work that used it has completed.
  cudaError_t get_mono(void** ptr, size_t bytes, int dev) {
    std::lock_guard<std::mutex> hold(lock_);
    cudaError_t e = pool_ ? cudaSuccess : make_pool(dev);
    if (e != cudaSuccess) return e;
    e = cudaMallocFromPoolAsync(ptr, bytes, pool_, nullptr);
    if (e == cudaErrorMemoryAllocation) {
      release_all();
      e = cudaMallocFromPoolAsync(ptr, bytes, pool_, nullptr);
    }
    return e;
  }
  // The same for memory of get_mono.  Its free is ordered by a stream and does not wait for the others.
  void put_mono(void* ptr, bool idle) {
    if (idle) {
      if (cudaFreeAsync(ptr, nullptr) == cudaSuccess) return;
      cudaGetLastError();
    }
    std::lock_guard<std::mutex> hold(lock_);
    aside_.push_back(ptr);
  }
  // Waits for the device, which must be the current one.  False if the runtime refuses to (it does while any of the device's
  // streams is under capture): work may then be in flight on any stream.
  bool wait_idle() {
    std::vector<void*> aside;  // not what is set aside while this waits
    {
      std::lock_guard<std::mutex> hold(lock_);
      aside.swap(aside_);
    }
    const bool idle = cudaDeviceSynchronize() == cudaSuccess;
    if (!idle) cudaGetLastError();  // (dealt with here and below: no later call is to report it)
    std::lock_guard<std::mutex> hold(lock_);
    if (idle)
      for (void* ptr : aside) give_up(ptr);
    else
      aside_.insert(aside_.end(), aside.begin(), aside.end());
    return idle;
  }
  // Gives back all that is kept.  False if something could not be waited for and stays.
  bool trim() {
    const bool idle = wait_idle();
    std::lock_guard<std::mutex> hold(lock_);
    release_all();
    return idle && aside_.empty();
  }

 private:
  struct Block { void* ptr; size_t bytes; };
  void release_all() {  // all that is kept, of either kind
    cudaGetLastError();
    shrink(0);
    if (pool_) cudaMemPoolTrimTo(pool_, 0);
  }
  cudaError_t make_pool(int dev) {
    cudaMemPoolProps props = {};
    props.allocType = cudaMemAllocationTypePinned;
    props.location.type = cudaMemLocationTypeDevice;
    props.location.id = dev;
    cudaMemPool_t pool;
    cudaError_t e = cudaMemPoolCreate(&pool, &props);
    if (e != cudaSuccess) return e;
    unsigned long long keep = MONO_KEEP_BYTES;
    int off = 0;
    e = cudaMemPoolSetAttribute(pool, cudaMemPoolAttrReleaseThreshold, &keep);
    if (e == cudaSuccess) e = cudaMemPoolSetAttribute(pool, cudaMemPoolReuseFollowEventDependencies, &off);
    if (e == cudaSuccess) e = cudaMemPoolSetAttribute(pool, cudaMemPoolReuseAllowInternalDependencies, &off);
    if (e != cudaSuccess) {
      cudaMemPoolDestroy(pool);
      return e;
    }
    pool_ = pool;
    return cudaSuccess;
  }
  void give_up(void* ptr) {
    if (cudaFree(ptr) == cudaSuccess) return;
    cudaGetLastError();
    aside_.push_back(ptr);
  }
  static size_t round_up(size_t bytes) {
    if (bytes > (size_t(1) << 20)) return (bytes + (size_t(2) << 20) - 1) >> 21 << 21;
    size_t r = 4096;
    while (r < bytes) r *= 2;
    return r;
  }
  void shrink(size_t to) {  // oldest first
    size_t n = 0;
    for (; n < free_.size() && kept_ > to; ++n) {
      give_up(free_[n].ptr);
      kept_ -= free_[n].bytes;
    }
    free_.erase(free_.begin(), free_.begin() + n);
  }
  std::mutex lock_;
  std::vector<Block> free_;
  std::vector<void*> aside_;  // given back while the device could not be waited for: belongs to nobody, handed to nobody
  std::map<void*, size_t> live_;
  size_t kept_ = 0;
  cudaMemPool_t pool_ = nullptr;
};

// `take`, and once more after waiting for the device if memory runs out: what is still on its way back counts then.
template <typename F>
cudaError_t take_or_wait(BlockCache& cache, F take) {
  cudaError_t e = take();
  if (e == cudaErrorMemoryAllocation && cache.wait_idle()) e = take();
  return e;
}

// Where a context's device memory comes from.  Arrays that were outgrown and may still be in use, by work on any stream or by
// a graph, stay until the context goes.
struct ContextMemory {
  BlockCache* cache = nullptr;
  bool captured = false;  // a launch of the context has been captured: a graph may use any of its arrays at any time
  std::vector<void*> outgrown;
  void release(bool idle) {
    for (void* ptr : outgrown) cache->put(ptr, idle);
    outgrown.clear();
  }
};

template <typename T>
struct DevBuf {  // grow-only device array of the context's device
  T* ptr = nullptr;
  size_t cap = 0;
  // The old array stays with the context (small blocks come in powers of two: all of them together are smaller than the new one).
  cudaError_t reserve(ContextMemory& memory, size_t n, cudaStream_t st) {
    return n <= cap ? cudaSuccess : grow(memory, n, st, false);
  }
  // For the large arrays, whose uses all come before this point of `st`: once the stream is waited for, the old array is kept
  // for others.  (A wait for the whole device would be refused beside a capture on whatever stream and destroy that capture.)
  cudaError_t reserve_in_order(ContextMemory& memory, size_t n, cudaStream_t st) {
    return n <= cap ? cudaSuccess : grow(memory, n, st, !memory.captured);
  }
  void retire(ContextMemory& memory) {
    if (ptr) memory.outgrown.push_back(ptr);
    ptr = nullptr;
    cap = 0;
  }
  void release(BlockCache& cache, bool idle) {
    if (ptr) cache.put(ptr, idle);
    ptr = nullptr;
    cap = 0;
  }

 private:
  static bool done(cudaStream_t st) {
    if (cudaStreamSynchronize(st) == cudaSuccess) return true;
    cudaGetLastError();
    return false;
  }
  cudaError_t grow(ContextMemory& memory, size_t n, cudaStream_t st, bool in_order) {
    // while `st` is captured the cache stands aside: cudaMalloc then says whether memory may be taken in this capture mode
    cudaStreamCaptureStatus status = cudaStreamCaptureStatusNone;
    cudaError_t e = cudaStreamIsCapturing(st, &status);
    if (e != cudaSuccess) return e;
    const bool capturing = status != cudaStreamCaptureStatusNone;
    void* bigger = nullptr;
    size_t bytes = 0;
    e = memory.cache->get(&bigger, n * sizeof(T), &bytes, capturing);
    if (e == cudaErrorMemoryAllocation && !memory.captured) {  // what this context does not need any more comes first
      if (ptr && in_order) release(*memory.cache, done(st));
      if (!memory.outgrown.empty() && memory.cache->wait_idle()) memory.release(true);
      e = memory.cache->get(&bigger, n * sizeof(T), &bytes, capturing);
    }
    if (e != cudaSuccess) return e;
    if (ptr && in_order)
      release(*memory.cache, done(st));
    else
      retire(memory);
    ptr = static_cast<T*>(bigger);
    cap = bytes / sizeof(T);
    return cudaSuccess;
  }
};

struct Schedule {
  int key_filled = -1;  // cache fill the lists were built for
  std::vector<WorkItem> items;
  std::vector<int32_t> cta_first;
  std::vector<CombineEntry> combine;  // query tiles to merge; the first n_long are cut into more than COMBINE_LONG_PARTS pieces
  int n_long = 0;
  std::vector<ClsGroup> cls_groups;  // classification only: key ranges of one query pair, merged three ways
  std::vector<ClsPart> cls_parts;
  DevBuf<WorkItem> items_dev;
  DevBuf<int32_t> cta_first_dev;
  DevBuf<CombineEntry> combine_dev;
  DevBuf<ClsGroup> cls_groups_dev;
  DevBuf<ClsPart> cls_parts_dev;
  int n_slots = 0;
  int dyn_first = 0, dyn_end = 0;  // items [dyn_first, dyn_end) form the shared queue the CTAs draw from when their own list is done
  bool uploaded = false;
  double flops = 0.0;
  void release(BlockCache& cache, bool idle) {
    items_dev.release(cache, idle);
    cta_first_dev.release(cache, idle);
    combine_dev.release(cache, idle);
    cls_groups_dev.release(cache, idle);
    cls_parts_dev.release(cache, idle);
  }
};

}  // namespace

struct headcast_ctx {
  headcast_config cfg;
  int H, D, L, T_f, F_b, n_blk, CH, G_h, G_w;
  float scale;
  int radius = 0;  // of the Spatial proxy, at most what reaches every token of a frame: the kernel walks rows and multiplies by it
  int state = STATE_FILLING;
  std::vector<int> slots;  // logical block -> physical ring slot (index 0 = sink block)
  bool have_labels = false;
  std::vector<int32_t> labels;
  int n_cls[4] = {0, 0, 0, 0};
  int sd_slots = 1;   // blocks per head in the Sink-Dummy buffer (2 with sd_mode 1)
  int sd_valid = 0;   // of which hold data
  int dummy_cur = 0;  // slot holding a Dummy head's newest block
  int8_t cls[MAX_HEADS], idx[MAX_HEADS];
  std::vector<int> row_edges, col_edges;
  std::vector<CellGeom> cells;
  std::vector<int> cell_tok_off;  // tokens per frame in earlier cells

  __nv_bfloat16 *mono_k = nullptr, *mono_v = nullptr;
  __nv_bfloat16 *arena_k = nullptr, *arena_v = nullptr;  // zeroed at create; the per-archetype buffers are carved from it
  __nv_bfloat16 *sd_k = nullptr, *sd_v = nullptr, *g_k = nullptr, *g_v = nullptr, *sp_k = nullptr, *sp_v = nullptr;
  int32_t *sp_base = nullptr, *sp_nc = nullptr;
  CellGeom* cells_dev = nullptr;
  CUtensorMap maps[2 * N_MAP_PAIRS];  // host copies; every attention launch carries them as kernel parameters
  // bulk tile movement (move_kernels.cuh): rectangles of the token grid per Spatial cell, their distinct box shapes,
  // and the source tensor maps - of the monolithic cache (built at create) and of recently seen caller blocks
  struct MoveShape { int cw, rows; };
  struct MoveMaps { const void *k = nullptr, *v = nullptr; CUtensorMap rows[2], box[2][MOVE_MAX_SHAPES]; };
  bool move_ok = false;     // false: the geometry does not fit the bulk path (very wide cells, too many cell shapes)
  std::vector<MoveBox> move_boxes;
  std::vector<MoveShape> move_shapes;
  MoveBox* move_boxes_dev = nullptr;
  MoveMaps move_mono;
  MoveMaps move_recent[8];
  int move_next = 0;
  int32_t* status_dev = nullptr;  // followed by the scores and labels of the last classification, see status_words
  int32_t* dyn_counter_dev = nullptr;  // [2]: next queue position, CTAs done (the last one clears both)

  Schedule sched_dense, sched_hc, sched_cls, sched_proxy;
  // headcast_attend_host: the stages of its pipeline, each with its own work list - the first half of the Global
  // heads' rows, the Sink + Dummy heads, the Spatial heads, the second half of the Global heads' rows
  static constexpr int N_HOST_STAGES = 4;
  Schedule sched_stage[N_HOST_STAGES];
  DevBuf<__nv_bfloat16> stage_q, stage_out, stage_k, stage_v;  // device copies of host tensors
  // the last call that used stage_q and stage_out: its stream's number, and what is recorded behind its last copy
  bool stage_used = false;
  unsigned long long stage_stream = 0;
  cudaEvent_t stage_done = nullptr;
  cudaStream_t copy_in = nullptr, copy_out = nullptr;
  cudaEvent_t ev_host[2 + 2 * N_HOST_STAGES] = {};
  DevBuf<float> part_o;
  DevBuf<float2> part_ml;
  DevBuf<float> part_mid;
  // The partial results and the counters of the shared queue: see order_shared_scratch
  bool scratch_used = false;
  unsigned long long scratch_stream = 0;  // of the last call that used them: its number, a handle may name another stream by now
  int stream_changes = 0;
  std::vector<int32_t*> old_counters;  // of streams that were left, see dyn_counter_dev
  cudaEvent_t scratch_done = nullptr;
  DevBuf<float> cls_o, cls_lse, cls_tok;

  int device = 0;
  ContextMemory memory;
  bool attn_configured[2] = {false, false}, move_configured = false;  // dynamic shared memory of the kernels (attention: plain, proxy)
  int n_sm = 148;
  int64_t launches = 0;
  bool tracing = false;  // record per-item start/end times in the attention kernel
  DevBuf<unsigned long long> trace_dev;
  std::vector<WorkItem> trace_items;
  std::vector<int32_t> trace_cta_first;
  bool timing = false;  // record events around the attention kernel of each call
  cudaEvent_t ev_a = nullptr, ev_b = nullptr;
  bool ev_valid = false;
  std::string err;
};

namespace {

int fail(headcast_ctx* c, int code, const char* fmt, ...) {
  if (c) {
    char buf[512];
    va_list ap;
    va_start(ap, fmt);
    vsnprintf(buf, sizeof(buf), fmt, ap);
    va_end(ap);
    c->err = buf;
  }
  return code;
}

#define HC_CUDA(c, expr)                                                                           \
  do {                                                                                             \
    cudaError_t e_ = (expr);                                                                       \
    if (e_ != cudaSuccess) {                                                                       \
      cudaGetLastError(); /* reported here, and by no later call */                                \
      return fail((c), e_ == cudaErrorMemoryAllocation ? HC_ERR_NOMEM : HC_ERR_CUDA, "%s: %s", #expr, \
                  cudaGetErrorString(e_));                                                         \
    }                                                                                              \
  } while (0)

std::vector<int> default_edges(int grid, int cell) {
  const int n = std::max(1, static_cast<int>(std::floor(static_cast<double>(grid) / cell + 0.5)));
  std::vector<int> e(n + 1);
  for (int i = 0; i <= n; ++i) e[i] = static_cast<int>((static_cast<long long>(i) * grid) / n);
  return e;
}

bool edges_ok(const std::vector<int>& e, int grid) {
  if (e.size() < 2 || e.front() != 0 || e.back() != grid) return false;
  for (size_t i = 1; i < e.size(); ++i)
    if (e[i] <= e[i - 1]) return false;
  return true;
}

bool aligned16(const void* p) { return p != nullptr && (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }

size_t cache_elems(const headcast_ctx* c, int heads) {
  return static_cast<size_t>(heads) * c->n_blk * c->L * c->D;
}

// ---------------------------------------------------------------------------------- tensor maps
int build_maps(headcast_ctx* c) {
  CUtensorMap* maps = c->maps;
  std::memset(maps, 0, sizeof(c->maps));
  const uint64_t win_rows = static_cast<uint64_t>(c->n_blk) * c->L;
  bool ok = true;
  if (c->mono_k) {
    ok = ok && make_tmap_bf16_2d(&maps[2 * MAP_MONO], c->mono_k, static_cast<uint64_t>(c->H) * c->D, win_rows,
                                 static_cast<uint64_t>(c->H) * c->D, 128);
    ok = ok && make_tmap_bf16_2d(&maps[2 * MAP_MONO + 1], c->mono_v, static_cast<uint64_t>(c->H) * c->D, win_rows,
                                 static_cast<uint64_t>(c->H) * c->D, 128);
  }
  if (c->sd_k) {
    const uint64_t rows = static_cast<uint64_t>(c->n_cls[CLS_SINK] + c->n_cls[CLS_DUMMY]) * c->sd_slots * c->L;
    ok = ok && make_tmap_bf16_2d(&maps[2 * MAP_SD], c->sd_k, c->D, rows, c->D, 128);
    ok = ok && make_tmap_bf16_2d(&maps[2 * MAP_SD + 1], c->sd_v, c->D, rows, c->D, 128);
  }
  if (c->g_k) {
    const uint64_t rows = c->n_cls[CLS_GLOBAL] * win_rows;
    ok = ok && make_tmap_bf16_2d(&maps[2 * MAP_GLOBAL], c->g_k, c->D, rows, c->D, 128);
    ok = ok && make_tmap_bf16_2d(&maps[2 * MAP_GLOBAL + 1], c->g_v, c->D, rows, c->D, 128);
  }
  if (c->sp_k) {
    const uint64_t rows = c->n_cls[CLS_SPATIAL] * win_rows;
    ok = ok && make_tmap_bf16_2d(&maps[2 * MAP_SPATIAL], c->sp_k, c->D, rows, c->D, 128);
    ok = ok && make_tmap_bf16_2d(&maps[2 * MAP_SPATIAL + 1], c->sp_v, c->D, rows, c->D, 128);
  }
  if (!ok) return fail(c, HC_ERR_CUDA, "cuTensorMapEncodeTiled failed or is unavailable");
  return HC_OK;
}

}  // namespace
