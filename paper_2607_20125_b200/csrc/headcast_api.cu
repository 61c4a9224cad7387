// C ABI of the HeadCast attention path (see include/headcast.h): context, state machine, cache ring,
// tile scheduling, and the launches of the kernels in attn_kernel.cuh / copy_kernels.cuh /
// score_kernels.cuh.  No CPU fallback exists: every step of the path runs in those kernels.
#include "context.h"
#include "noalloc_scratch.h"
#include "schedule.h"

namespace {

// Launches a kernel of this library (every one of them calls pdl_wait before it touches global memory, but for lists whose
// upload was waited for) so that it may become resident while its predecessor on the stream drains.  Since the predecessor may still write while such a kernel
// runs, nothing is read through the non-coherent path (__ldg, ld.global.nc): that path wants data which no one writes for
// as long as the reading kernel lives, and pdl_wait orders ordinary loads only.  Together with the one merge launch instead of two it takes
// the block of 192 tokens and four heads from 86 to 76 us and leaves the large ones where they are (45 x 80: -1 %).
template <typename... P, typename... A>
cudaError_t launch_pdl(void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, A&&... args) {
  cudaLaunchConfig_t lc = {};
  lc.gridDim = grid;
  lc.blockDim = block;
  lc.dynamicSmemBytes = smem;
  lc.stream = st;
  cudaLaunchAttribute attr;
  attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr.val.programmaticStreamSerializationAllowed = 1;
  lc.attrs = &attr;
  lc.numAttrs = 1;
  return cudaLaunchKernelEx(&lc, kernel, static_cast<P>(args)...);
}

int upload_schedule(headcast_ctx* c, Schedule& s, cudaStream_t st) {
  // The partial results are shared by all lists of the context, so every launch makes sure of them and not only the first of
  // its list: another list's growth may have failed in between and left none.
  if (s.n_slots > 0) {
    HC_CUDA(c, c->part_o.reserve_in_order(c->memory, static_cast<size_t>(s.n_slots) * 256 * c->D, st));
    HC_CUDA(c, c->part_ml.reserve_in_order(c->memory, static_cast<size_t>(s.n_slots) * 256, st));
    HC_CUDA(c, c->part_mid.reserve_in_order(c->memory, static_cast<size_t>(s.n_slots) * 256, st));
  }
  if (s.uploaded) return HC_OK;
  HC_CUDA(c, s.items_dev.reserve(c->memory, std::max<size_t>(1, s.items.size()), st));
  HC_CUDA(c, s.cta_first_dev.reserve(c->memory, s.cta_first.size(), st));
  HC_CUDA(c, s.combine_dev.reserve(c->memory, std::max<size_t>(1, s.combine.size()), st));
  if (!s.items.empty())
    HC_CUDA(c, cudaMemcpyAsync(s.items_dev.ptr, s.items.data(), s.items.size() * sizeof(WorkItem),
                               cudaMemcpyHostToDevice, st));
  HC_CUDA(c, cudaMemcpyAsync(s.cta_first_dev.ptr, s.cta_first.data(), s.cta_first.size() * sizeof(int32_t),
                             cudaMemcpyHostToDevice, st));
  if (!s.combine.empty())
    HC_CUDA(c, cudaMemcpyAsync(s.combine_dev.ptr, s.combine.data(), s.combine.size() * sizeof(CombineEntry),
                               cudaMemcpyHostToDevice, st));
  if (!s.cls_groups.empty()) {
    HC_CUDA(c, s.cls_groups_dev.reserve(c->memory, s.cls_groups.size(), st));
    HC_CUDA(c, s.cls_parts_dev.reserve(c->memory, std::max<size_t>(1, s.cls_parts.size()), st));
    HC_CUDA(c, cudaMemcpyAsync(s.cls_groups_dev.ptr, s.cls_groups.data(), s.cls_groups.size() * sizeof(ClsGroup),
                               cudaMemcpyHostToDevice, st));
    HC_CUDA(c, cudaMemcpyAsync(s.cls_parts_dev.ptr, s.cls_parts.data(), s.cls_parts.size() * sizeof(ClsPart),
                               cudaMemcpyHostToDevice, st));
  }
  // The lists are uploaded once per cache fill and reused by later calls, which may come on another stream: wait
  // here, once, so that no later launch can see a half-written list (the host vectors are pageable, so the copies
  // have mostly completed by now anyway).
  HC_CUDA(c, cudaStreamSynchronize(st));
  s.uploaded = true;
  return HC_OK;
}

template <int D, bool PROXY>
int launch_attn_t(headcast_ctx* c, const AttnParams& p, cudaStream_t st) {
  // the attribute belongs to the function in a CUDA context: every headcast_ctx sets it once for itself, whatever GPU it is on
  // and whatever has been reset before
  if (!c->attn_configured[PROXY]) {
    HC_CUDA(c, cudaFuncSetAttribute(attn_kernel<D, PROXY>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                    AttnSmem<D>::DYN_BYTES));
    c->attn_configured[PROXY] = true;
  }
  if (c->timing) HC_CUDA(c, cudaEventRecord(c->ev_a, st));
  HC_CUDA(c, launch_pdl(attn_kernel<D, PROXY>, dim3(c->n_sm), dim3(ATTN_THREADS), AttnSmem<D>::DYN_BYTES, st, p));
  if (c->timing) {
    HC_CUDA(c, cudaEventRecord(c->ev_b, st));
    c->ev_valid = true;
  }
  ++c->launches;
  return HC_OK;
}

// The partial results and the counters of the shared queue are the context's, one set for all its calls, so a call on
// another stream than the last one has to come after it, or use a set of its own.  A caller that moves to another stream once
// or twice gets a new set there; the old one stays with the stream that may still work on it.  One that keeps changing gets
// an event behind every call, and a wait for it when the stream changes.  A single stream is spared both.
constexpr int CHANGES_WITH_NEW_SCRATCH = 3;
int order_shared_scratch(headcast_ctx* c, cudaStream_t st) {
  unsigned long long stream = 0;
  HC_CUDA(c, cudaStreamGetId(st, &stream));
  if (c->scratch_used && c->scratch_stream != stream) {
    if (c->scratch_done) {
      HC_CUDA(c, cudaStreamWaitEvent(st, c->scratch_done, 0));
    } else {
      void* counters = nullptr;
      HC_CUDA(c, c->memory.cache->get(&counters, 2 * sizeof(int32_t)));
      c->old_counters.push_back(c->dyn_counter_dev);
      c->dyn_counter_dev = static_cast<int32_t*>(counters);
      HC_CUDA(c, cudaMemsetAsync(c->dyn_counter_dev, 0, 2 * sizeof(int32_t), st));
      c->part_o.retire(c->memory);
      c->part_ml.retire(c->memory);
      c->part_mid.retire(c->memory);
      if (++c->stream_changes >= CHANGES_WITH_NEW_SCRATCH) HC_CUDA(c, cudaEventCreateWithFlags(&c->scratch_done, cudaEventDisableTiming));
    }
  }
  c->scratch_used = true;
  c->scratch_stream = stream;
  return HC_OK;
}

int run_schedule(headcast_ctx* c, Schedule& s, const void* q, void* out, bool proxy, cudaStream_t st) {
  cudaStreamCaptureStatus status = cudaStreamCaptureStatusNone;
  HC_CUDA(c, cudaStreamIsCapturing(st, &status));
  const bool capturing = status != cudaStreamCaptureStatusNone;
  c->memory.captured = c->memory.captured || capturing;
  // (the launches of a graph are the caller's to order)
  const bool shares_scratch = !capturing && (s.n_slots > 0 || s.dyn_end > s.dyn_first);
  int rc = shares_scratch ? order_shared_scratch(c, st) : HC_OK;
  if (rc == HC_OK) rc = upload_schedule(c, s, st);
  if (rc != HC_OK) return rc;
  if (s.items.empty()) return HC_OK;
  AttnParams p;
  std::memset(&p, 0, sizeof(p));
  p.items = s.items_dev.ptr;
  p.cta_first = s.cta_first_dev.ptr;
  static_assert(sizeof(p.maps) == sizeof(c->maps), "one K and one V map per buffer");
  std::memcpy(p.maps, c->maps, sizeof(p.maps));
  p.cells = c->cells_dev;
  p.q = static_cast<const __nv_bfloat16*>(q);
  p.out = static_cast<__nv_bfloat16*>(out);
  p.part_o = c->part_o.ptr;
  p.part_ml = c->part_ml.ptr;
  p.part_mid = c->part_mid.ptr;
  p.n_heads = c->H;
  p.tokens_per_frame = c->T_f;
  p.grid_w = c->G_w;
  p.block_tokens = c->L;
  p.scale_log2e = c->scale * 1.4426950408889634f;
  p.status = c->status_dev;
  p.dyn_first = s.dyn_first;
  p.dyn_end = s.dyn_end;
  p.dyn_counter = c->dyn_counter_dev;
  p.trace = nullptr;
  if (c->tracing) {
    const size_t trace_words = 2 * s.items.size();
    HC_CUDA(c, c->trace_dev.reserve(c->memory, trace_words, st));
    HC_CUDA(c, cudaMemsetAsync(c->trace_dev.ptr, 0, trace_words * sizeof(unsigned long long), st));
    p.trace = c->trace_dev.ptr;
    c->trace_items = s.items;
    c->trace_cta_first = s.cta_first;
  }
  p.radius = c->radius;
  if (proxy) {
    const int newest = c->slots.back();
    p.mid_seg_lo = c->F_b;
    p.mid_seg_hi = n_filled(c) * c->F_b;
    p.last_seg_lo = newest * c->F_b;
    p.last_seg_hi = (newest + 1) * c->F_b;
  }
  if (c->D == 128)
    rc = proxy ? launch_attn_t<128, true>(c, p, st) : launch_attn_t<128, false>(c, p, st);
  else
    rc = proxy ? launch_attn_t<64, true>(c, p, st) : launch_attn_t<64, false>(c, p, st);
  if (rc != HC_OK) return rc;
  if (!s.cls_groups.empty()) {
    // classification: merge the pieces of every query pair and score its rows (score_kernels.cuh)
    const unsigned blocks = static_cast<unsigned>(s.cls_groups.size()) * 2 * (128 / COMBINE_ROWS);
    const unsigned threads = COMBINE_ROWS * (c->D / 8);
    if (proxy)
      HC_CUDA(c, launch_pdl(c->D == 128 ? proxy_combine_kernel<128> : proxy_combine_kernel<64>, dim3(blocks), dim3(threads), 0, st,
                            s.cls_groups_dev.ptr, s.cls_parts_dev.ptr, c->part_o.ptr, c->part_ml.ptr, c->part_mid.ptr, c->cls_o.ptr,
                            c->cls_lse.ptr, c->cls_tok.ptr, c->H, c->L));
    else
      HC_CUDA(c, launch_pdl(c->D == 128 ? cls_combine_kernel<128> : cls_combine_kernel<64>, dim3(blocks), dim3(threads), 0, st,
                            s.cls_groups_dev.ptr, s.cls_parts_dev.ptr, c->part_o.ptr, c->part_ml.ptr, c->cls_o.ptr, c->cls_lse.ptr,
                            c->cls_tok.ptr, c->H, c->L));
    ++c->launches;
  }
  if (!s.combine.empty()) {
    const unsigned blocks = static_cast<unsigned>(s.combine.size() - s.n_long) * (128 / COMBINE_ROWS) + static_cast<unsigned>(s.n_long) * 128;
    HC_CUDA(c, launch_pdl(c->D == 128 ? combine_kernel<128> : combine_kernel<64>, dim3(blocks), dim3(COMBINE_ROWS * (c->D / 8)), 0, st,
                          s.combine_dev.ptr, s.n_long, c->cells_dev, c->part_o.ptr, c->part_ml.ptr, p.out, c->H, c->T_f, c->G_w, true));
    ++c->launches;
  }
  if (shares_scratch && c->scratch_done) HC_CUDA(c, cudaEventRecord(c->scratch_done, st));
  return HC_OK;
}

// Self-test of the bounded-wait machinery: one CTA waits on an mbarrier that nobody ever arrives on, gives up after
// limit_ns, records `code` in the status word and returns normally (no trap, no fault: the context stays usable).
__global__ void bounded_wait_selftest_kernel(int32_t* status, unsigned long long limit_ns, int code) {
  __shared__ uint64_t bar;
  __shared__ int abort_flag;
  if (threadIdx.x == 0) {
    mbar_init(&bar, 1);
    abort_flag = 0;
    fence_mbar_init();
  }
  __syncthreads();
  volatile int* abortp = &abort_flag;
  mbar_wait_limit(&bar, 0, abortp, status, code, limit_ns);  // every thread waits; the first to expire raises the flag
}

void fill_route(headcast_ctx* c, RouteParams& r) {
  std::memset(&r, 0, sizeof(r));
  r.mono_k = reinterpret_cast<uint4*>(c->mono_k);
  r.mono_v = reinterpret_cast<uint4*>(c->mono_v);
  r.sd_k = reinterpret_cast<uint4*>(c->sd_k);
  r.sd_v = reinterpret_cast<uint4*>(c->sd_v);
  r.g_k = reinterpret_cast<uint4*>(c->g_k);
  r.g_v = reinterpret_cast<uint4*>(c->g_v);
  r.sp_k = reinterpret_cast<uint4*>(c->sp_k);
  r.sp_v = reinterpret_cast<uint4*>(c->sp_v);
  r.sp_base = c->sp_base;
  r.sp_nc = c->sp_nc;
  r.L = c->L;
  r.H = c->H;
  r.chunks = c->CH;
  r.tokens_per_frame = c->T_f;
  r.frames_per_block = c->F_b;
  r.n_blocks = c->n_blk;
  r.n_sink = c->n_cls[CLS_SINK];
  r.sd_slots = c->sd_slots;
  for (int i = 0; i < MAX_BLOCKS; ++i) r.sd_slot_sink[i] = r.sd_slot_dummy[i] = -1;
  for (int h = 0; h < c->H; ++h) {
    r.cls[h] = (c->state == STATE_SPLIT || c->sd_k || c->g_k || c->sp_k) ? c->cls[h] : static_cast<int8_t>(CLS_NONE);
    r.idx[h] = c->idx[h];
  }
}

// Source tensor maps of the bulk path for a [rows][H*d] tensor at k / v.
bool build_move_maps(headcast_ctx* c, headcast_ctx::MoveMaps& m, const void* k, const void* v, uint64_t rows) {
  const uint64_t row_elems = static_cast<uint64_t>(c->H) * c->D;
  const uint32_t tile_rows = MOVE_STAGE_BYTES / (c->D * 2);
  const void* base[2] = {k, v};
  for (int kv = 0; kv < 2; ++kv) {
    if (!make_tmap_bf16_rows(&m.rows[kv], base[kv], row_elems, rows, c->D, tile_rows)) return false;
    for (size_t s = 0; s < c->move_shapes.size(); ++s)
      if (!make_tmap_bf16_grid(&m.box[kv][s], base[kv], row_elems, rows, c->G_w, c->D, c->move_shapes[s].cw, c->move_shapes[s].rows))
        return false;
  }
  m.k = k;
  m.v = v;
  return true;
}

// The same routing as route_block_kernel (RouteParams says which source block feeds which buffer), as bulk tile jobs.
int launch_move(headcast_ctx* c, const RouteParams& r, int n_src, cudaStream_t st) {
  if (!c->move_configured) {
    HC_CUDA(c, cudaFuncSetAttribute(move_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, MOVE_SMEM_BYTES));
    c->move_configured = true;
  }
  MoveParams p;
  std::memset(&p, 0, sizeof(p));
  const headcast_ctx::MoveMaps* maps = nullptr;
  if (r.src_stride != 0) {
    maps = &c->move_mono;
  } else {
    for (auto& m : c->move_recent)
      if (m.k == r.src_k && m.v == r.src_v && m.k) maps = &m;
    if (!maps) {
      headcast_ctx::MoveMaps& m = c->move_recent[c->move_next];
      c->move_next = (c->move_next + 1) % 8;
      m.k = m.v = nullptr;
      if (!build_move_maps(c, m, r.src_k, r.src_v, c->L)) return fail(c, HC_ERR_CUDA, "cuTensorMapEncodeTiled failed for the block to append");
      maps = &m;
    }
  }
  std::memcpy(p.map_rows, maps->rows, sizeof(p.map_rows));
  std::memcpy(p.map_box, maps->box, sizeof(p.map_box));
  p.src_k = reinterpret_cast<const __nv_bfloat16*>(r.src_k);
  p.src_v = reinterpret_cast<const __nv_bfloat16*>(r.src_v);
  p.mono_k = reinterpret_cast<__nv_bfloat16*>(r.mono_k);
  p.mono_v = reinterpret_cast<__nv_bfloat16*>(r.mono_v);
  p.sd_k = reinterpret_cast<__nv_bfloat16*>(r.sd_k);
  p.sd_v = reinterpret_cast<__nv_bfloat16*>(r.sd_v);
  p.g_k = reinterpret_cast<__nv_bfloat16*>(r.g_k);
  p.g_v = reinterpret_cast<__nv_bfloat16*>(r.g_v);
  p.sp_k = reinterpret_cast<__nv_bfloat16*>(r.sp_k);
  p.sp_v = reinterpret_cast<__nv_bfloat16*>(r.sp_v);
  p.boxes = c->move_boxes_dev;
  p.status = c->status_dev;
  p.src_block_rows = r.src_stride ? c->L : 0;
  p.n_boxes = static_cast<int32_t>(c->move_boxes.size());
  p.L = c->L; p.H = c->H; p.D = c->D; p.F_b = c->F_b; p.G_h = c->G_h; p.G_w = c->G_w;
  p.n_blocks = c->n_blk;
  p.n_sink = r.n_sink;
  p.sd_slots = r.sd_slots;
  p.rows_per_tile = MOVE_STAGE_BYTES / (c->D * 2);
  p.tiles_rm = (c->L + p.rows_per_tile - 1) / p.rows_per_tile;
  p.copy_mono = r.copy_mono;
  p.copy_window = r.copy_window;
  const long long block_bytes = static_cast<long long>(c->L) * c->H * c->D * 2;
  p.mono_chunks = r.copy_mono ? static_cast<int32_t>((block_bytes + MOVE_STAGE_BYTES - 1) / MOVE_STAGE_BYTES) : 0;
  p.n_src = n_src;
  for (int h = 0; h < c->H; ++h) {
    p.cls[h] = r.cls[h];
    p.idx[h] = r.idx[h];
    if (r.cls[h] == CLS_SPATIAL && r.copy_window) p.sp[p.n_sp++] = static_cast<int8_t>(h);
  }
  for (int k = 0; k < 4; ++k)
    for (int h = 0; h < c->H; ++h) {
      const int cl = r.cls[h];
      if ((cl == CLS_GLOBAL && r.copy_window) || (cl == CLS_SINK && (k == 0 || k == 2)) || (cl == CLS_DUMMY && (k == 1 || k == 2)))
        p.rm[k][p.n_rm[k]++] = static_cast<int8_t>(h);
    }
  long long jobs = 0;
  for (int i = 0; i < n_src; ++i) {
    p.slots[i] = r.slots[i];
    p.sd_slot_sink[i] = r.sd_slot_sink[i];
    p.sd_slot_dummy[i] = r.sd_slot_dummy[i];
    p.kind[i] = r.kind[i];
    p.job_first[i] = static_cast<int32_t>(jobs);
    jobs += 2ll * (static_cast<long long>(p.n_rm[p.kind[i]]) * p.tiles_rm + static_cast<long long>(p.n_sp) * p.F_b * p.n_boxes + p.mono_chunks);
  }
  p.job_first[n_src] = static_cast<int32_t>(jobs);
  if (jobs == 0) return HC_OK;
  if (jobs >= (1ll << 31)) return fail(c, HC_ERR_UNSUPPORTED, "too many tile jobs");
  const int ctas = static_cast<int>(std::min<long long>(c->n_sm, (jobs + MOVE_ENGINES - 1) / MOVE_ENGINES));
  HC_CUDA(c, launch_pdl(move_kernel, dim3(ctas), dim3(MOVE_ENGINES * 32), MOVE_SMEM_BYTES, st, p));
  ++c->launches;
  return HC_OK;
}

int launch_route(headcast_ctx* c, RouteParams& r, int n_src, cudaStream_t st) {
  // which heads each kind of source row feeds (see RouteParams::kind)
  for (int k = 0; k < 4; ++k) {
    r.n_kept[k] = 0;
    for (int h = 0; h < r.H; ++h) {
      const int cl = r.cls[h];
      const bool keep = r.copy_mono || ((cl == CLS_GLOBAL || cl == CLS_SPATIAL) && r.copy_window) ||
                        (cl == CLS_SINK && (k == 0 || k == 2)) || (cl == CLS_DUMMY && (k == 1 || k == 2));
      if (keep) r.kept[k][r.n_kept[k]++] = static_cast<int8_t>(h);
    }
  }
  int max_kept = 0;
  for (int i = 0; i < n_src; ++i) {
    const bool s = r.sd_slot_sink[i] >= 0, d = r.sd_slot_dummy[i] >= 0;
    r.kind[i] = static_cast<int8_t>(s && d ? 2 : s ? 0 : d ? 1 : 3);
    max_kept = std::max<int>(max_kept, r.n_kept[r.kind[i]]);
  }
  if (max_kept == 0) return HC_OK;  // nothing to move (e.g. an append when every head is a Sink head)
  if (c->move_ok) return launch_move(c, r, n_src, st);
  const int per_token = max_kept * r.chunks;  // <= 64 heads * 16 chunks = 1024
  const int tokens_per_iter = std::max(1, 256 / per_token);
  const int threads = tokens_per_iter * per_token;
  const int resident = std::max(1, 2048 / threads);  // blocks per SM
  const int per_src = std::max(1, (c->n_sm * resident + n_src - 1) / n_src);
  const int needed = (r.L + tokens_per_iter * ROUTE_UNROLL - 1) / (tokens_per_iter * ROUTE_UNROLL);
  route_block_kernel<<<dim3(std::max(1, std::min(needed, per_src)), n_src), threads, 0, st>>>(r);
  HC_CUDA(c, cudaGetLastError());
  ++c->launches;
  return HC_OK;
}

// Words at status_dev: the status, then the scores and the labels of the last classification.
size_t status_words(const headcast_ctx* c) { return 1 + static_cast<size_t>(c->H) * (HC_N_SCORES + 1); }

int report_status(headcast_ctx* c, int32_t status, cudaStream_t st) {
  if (status != 0) {
    cudaMemsetAsync(c->status_dev, 0, sizeof(int32_t), st);
    // a kernel that gave up may have left the queue half drawn
    cudaMemsetAsync(c->dyn_counter_dev, 0, 2 * sizeof(int32_t), st);
    for (int32_t* counter : c->old_counters) cudaMemsetAsync(counter, 0, 2 * sizeof(int32_t), st);  // graphs may hold these
    return fail(c, HC_ERR_TIMEOUT, "a kernel gave up on a bounded wait (site %d)", status);
  }
  return HC_OK;
}

int read_status(headcast_ctx* c, cudaStream_t st) {
  int32_t status = 0;
  HC_CUDA(c, cudaMemcpyAsync(&status, c->status_dev, sizeof(status), cudaMemcpyDeviceToHost, st));
  HC_CUDA(c, cudaStreamSynchronize(st));
  return report_status(c, status, st);
}

void assign_classes(headcast_ctx* c) {
  for (int k = 0; k < 4; ++k) c->n_cls[k] = 0;
  for (int h = 0; h < c->H; ++h) {
    c->cls[h] = static_cast<int8_t>(c->labels[h]);
    c->idx[h] = static_cast<int8_t>(c->n_cls[c->labels[h]]++);
  }
}

}  // namespace

// Host-only half of headcast_create: validates cfg and fills sizes, cell geometry and the cell-major token tables.
static int init_host(headcast_ctx* c, const headcast_config* cfg, std::vector<int32_t>& sp_base, std::vector<int32_t>& sp_nc) {
  if (cfg->n_heads < 1 || cfg->n_heads > MAX_HEADS || (cfg->head_dim != 64 && cfg->head_dim != 128) ||
      cfg->grid_h < 1 || cfg->grid_w < 1 || cfg->frames_per_block < 1 || cfg->n_blocks < 2 ||
      cfg->n_blocks > MAX_BLOCKS || cfg->cell_h < 1 || cfg->cell_w < 1 || cfg->proxy_radius < 0 ||
      !(cfg->softmax_scale >= 0.0f) || cfg->sd_mode < 0 || cfg->sd_mode > 1 || cfg->rule < 0 || cfg->rule > 1 ||
      (cfg->rule == 1 && !(cfg->mass_tau > 0.0f && cfg->mass_tau <= 1.0f)))
    return HC_ERR_INVALID_ARG;
  const long long L = static_cast<long long>(cfg->frames_per_block) * cfg->grid_h * cfg->grid_w;
  if (L * cfg->n_blocks * cfg->n_heads * cfg->head_dim >= (1LL << 40) || L * cfg->n_blocks * cfg->n_heads >= (1LL << 31))
    return HC_ERR_INVALID_ARG;
  c->cfg = *cfg;
  c->H = cfg->n_heads;
  c->D = cfg->head_dim;
  c->G_h = cfg->grid_h;
  c->G_w = cfg->grid_w;
  c->F_b = cfg->frames_per_block;
  c->T_f = cfg->grid_h * cfg->grid_w;
  c->L = static_cast<int>(L);
  c->n_blk = cfg->n_blocks;
  c->CH = c->D / 8;
  c->sd_slots = cfg->sd_mode ? 2 : 1;
  c->radius = std::min(cfg->proxy_radius, std::max(c->G_h, c->G_w));
  c->scale = cfg->softmax_scale > 0.f ? cfg->softmax_scale : 1.0f / std::sqrt(static_cast<float>(c->D));
  c->row_edges = (cfg->row_edges_host && cfg->n_row_edges > 0)
                     ? std::vector<int>(cfg->row_edges_host, cfg->row_edges_host + cfg->n_row_edges)
                     : default_edges(c->G_h, cfg->cell_h);
  c->col_edges = (cfg->col_edges_host && cfg->n_col_edges > 0)
                     ? std::vector<int>(cfg->col_edges_host, cfg->col_edges_host + cfg->n_col_edges)
                     : default_edges(c->G_w, cfg->cell_w);
  c->cfg.row_edges_host = c->cfg.col_edges_host = nullptr;
  if (!edges_ok(c->row_edges, c->G_h) || !edges_ok(c->col_edges, c->G_w)) return HC_ERR_INVALID_ARG;
  c->labels.assign(c->H, HC_GLOBAL);
  for (int h = 0; h < c->H; ++h) {
    c->cls[h] = CLS_NONE;
    c->idx[h] = 0;
  }
  // deployed cells and the cell-major token order of the Spatial buffers
  sp_base.assign(c->T_f, 0);
  sp_nc.assign(c->T_f, 0);
  int tok_off = 0;
  for (size_t i = 0; i + 1 < c->row_edges.size(); ++i)
    for (size_t j = 0; j + 1 < c->col_edges.size(); ++j) {
      CellGeom g = {c->row_edges[i], c->col_edges[j], c->row_edges[i + 1] - c->row_edges[i],
                    c->col_edges[j + 1] - c->col_edges[j]};
      c->cells.push_back(g);
      c->cell_tok_off.push_back(tok_off);
      for (int dy = 0; dy < g.ch; ++dy)
        for (int dx = 0; dx < g.cw; ++dx) {
          const int pos = (g.y0 + dy) * c->G_w + g.x0 + dx;
          sp_base[pos] = c->n_blk * c->F_b * tok_off + dy * g.cw + dx;
          sp_nc[pos] = g.ch * g.cw;
        }
      tok_off += g.ch * g.cw;
    }
  // bulk tile movement: every cell (or, for a cell larger than a stage, every band of its rows) is one rectangle of
  // the token grid; rectangles of equal (width, rows) share a tensor map
  const int stage_tokens = MOVE_STAGE_BYTES / (c->D * 2);
  c->move_ok = true;
  c->move_boxes.clear();
  c->move_shapes.clear();
  for (size_t ci = 0; ci < c->cells.size() && c->move_ok; ++ci) {
    const CellGeom& g = c->cells[ci];
    if (g.cw > stage_tokens || g.cw > 256) {
      c->move_ok = false;
      break;
    }
    const int rb = std::min(std::min(g.ch, 256), std::max(1, stage_tokens / g.cw));
    int shape = -1;
    for (size_t s = 0; s < c->move_shapes.size(); ++s)
      if (c->move_shapes[s].cw == g.cw && c->move_shapes[s].rows == rb) shape = static_cast<int>(s);
    if (shape < 0) {
      if (c->move_shapes.size() == MOVE_MAX_SHAPES) {
        c->move_ok = false;
        break;
      }
      shape = static_cast<int>(c->move_shapes.size());
      c->move_shapes.push_back({g.cw, rb});
    }
    for (int r0 = 0; r0 < g.ch; r0 += rb) {
      MoveBox b;
      b.y0 = g.y0 + r0;
      b.x0 = g.x0;
      b.cw = g.cw;
      b.rows = std::min(rb, g.ch - r0);
      b.shape = shape;
      b.box_tokens = g.cw * rb;
      b.cell_tok_off = c->cell_tok_off[ci];
      b.nc = g.ch * g.cw;
      b.first_tok = r0 * g.cw;
      c->move_boxes.push_back(b);
    }
  }
  return HC_OK;
}

// =====================================================================================================
extern "C" {

void headcast_default_config(headcast_config* cfg) {
  if (!cfg) return;
  std::memset(cfg, 0, sizeof(*cfg));
  cfg->frames_per_block = 3;
  cfg->cell_h = 10;
  cfg->cell_w = 10;
  cfg->proxy_radius = 2;
  cfg->theta_sink = cfg->theta_dummy = cfg->theta_spatial = 0.95f;
  cfg->theta_score = 0.755f;
  cfg->gamma = 5.0f;
  cfg->softmax_scale = 0.0f;
  cfg->rule = HC_RULE_COSINE;
  cfg->mass_tau = 0.9f;
}

int headcast_create(const headcast_config* cfg, headcast_ctx** out) {
  if (!cfg || !out) return HC_ERR_INVALID_ARG;
  *out = nullptr;
  headcast_ctx* c = new (std::nothrow) headcast_ctx();
  if (!c) return HC_ERR_NOMEM;
  std::vector<int32_t> sp_base, sp_nc;
  {
    const int rc = init_host(c, cfg, sp_base, sp_nc);
    if (rc != HC_OK) {
      delete c;
      return rc;
    }
  }
  int major = 0;  // (two attributes: cudaGetDeviceProperties takes 2.5 ms)
  if (cudaGetDevice(&c->device) != cudaSuccess ||
      cudaDeviceGetAttribute(&major, cudaDevAttrComputeCapabilityMajor, c->device) != cudaSuccess ||
      cudaDeviceGetAttribute(&c->n_sm, cudaDevAttrMultiProcessorCount, c->device) != cudaSuccess) {
    delete c;
    return HC_ERR_CUDA;
  }
  if (major != 10) {
    delete c;
    return HC_ERR_UNSUPPORTED;
  }
  const size_t mono_bytes = cache_elems(c, c->H) * sizeof(__nv_bfloat16);
  c->memory.cache = BlockCache::current(c->device);
  if (!c->memory.cache) {
    delete c;
    return HC_ERR_CUDA;
  }
  BlockCache& cache = *c->memory.cache;
  cudaError_t e = cudaSuccess;
  auto step = [&](cudaError_t r) { if (e == cudaSuccess) e = r; };
  auto get = [&](auto** ptr, size_t bytes) {
    void* m = nullptr;
    if (e == cudaSuccess) step(take_or_wait(cache, [&] { return cache.get(&m, bytes); }));
    *ptr = static_cast<std::remove_pointer_t<decltype(ptr)>>(m);
  };
  auto get_mono = [&](__nv_bfloat16** ptr) {
    void* m = nullptr;
    if (e == cudaSuccess) step(take_or_wait(cache, [&] { return cache.get_mono(&m, mono_bytes, c->device); }));
    *ptr = static_cast<__nv_bfloat16*>(m);
  };
  get_mono(&c->mono_k);
  get_mono(&c->mono_v);
  get(&c->arena_k, mono_bytes);
  get(&c->arena_v, mono_bytes);
  get(&c->sp_base, c->T_f * sizeof(int32_t));
  get(&c->sp_nc, c->T_f * sizeof(int32_t));
  get(&c->cells_dev, c->cells.size() * sizeof(CellGeom));
  get(&c->status_dev, status_words(c) * sizeof(int32_t));
  get(&c->dyn_counter_dev, 2 * sizeof(int32_t));
  if (c->move_ok) get(&c->move_boxes_dev, std::max<size_t>(1, c->move_boxes.size()) * sizeof(MoveBox));
  if (e == cudaSuccess) {
    step(cudaMemsetAsync(c->dyn_counter_dev, 0, 2 * sizeof(int32_t), nullptr));
    step(cudaMemsetAsync(c->mono_k, 0, mono_bytes, nullptr));
    step(cudaMemsetAsync(c->mono_v, 0, mono_bytes, nullptr));
    step(cudaMemsetAsync(c->arena_k, 0, mono_bytes, nullptr));
    step(cudaMemsetAsync(c->arena_v, 0, mono_bytes, nullptr));
    step(cudaMemsetAsync(c->status_dev, 0, sizeof(int32_t), nullptr));
    step(cudaMemcpy(c->sp_base, sp_base.data(), c->T_f * sizeof(int32_t), cudaMemcpyHostToDevice));
    step(cudaMemcpy(c->sp_nc, sp_nc.data(), c->T_f * sizeof(int32_t), cudaMemcpyHostToDevice));
    step(cudaMemcpy(c->cells_dev, c->cells.data(), c->cells.size() * sizeof(CellGeom), cudaMemcpyHostToDevice));
    if (c->move_ok && !c->move_boxes.empty())
      step(cudaMemcpy(c->move_boxes_dev, c->move_boxes.data(), c->move_boxes.size() * sizeof(MoveBox), cudaMemcpyHostToDevice));
  }
  if (e == cudaSuccess && c->move_ok &&
      !build_move_maps(c, c->move_mono, c->mono_k, c->mono_v, static_cast<uint64_t>(c->n_blk) * c->L))
    c->move_ok = false;  // the per-thread copy kernel serves every geometry

  int rc = HC_OK;
  if (e != cudaSuccess) rc = (e == cudaErrorMemoryAllocation) ? HC_ERR_NOMEM : HC_ERR_CUDA;
  if (rc == HC_OK) rc = build_maps(c);
  if (rc == HC_OK && !cache.wait_idle()) rc = HC_ERR_CUDA;
  if (rc != HC_OK) {
    cudaGetLastError();
    headcast_destroy(c);
    return rc;
  }
  *out = c;
  return HC_OK;
}

int headcast_destroy(headcast_ctx* c) {
  if (!c) return HC_OK;
  int current = c->device;  // the context's memory belongs to its own device, whichever one is current now
  cudaGetDevice(&current);
  if (current != c->device) cudaSetDevice(c->device);
  BlockCache& cache = *c->memory.cache;
  const bool idle = cache.wait_idle();  // if not, kernels may be at work on any of these: nothing of it is kept for others
  if (c->mono_k) cache.put_mono(c->mono_k, idle);
  if (c->mono_v) cache.put_mono(c->mono_v, idle);
  void* ptrs[] = {c->arena_k, c->arena_v, c->sp_base, c->sp_nc, c->cells_dev, c->status_dev, c->dyn_counter_dev, c->move_boxes_dev};
  for (void* p : ptrs)
    if (p) cache.put(p, idle);
  for (int32_t* counter : c->old_counters) cache.put(counter, idle);
  if (c->ev_a) cudaEventDestroy(c->ev_a);
  if (c->ev_b) cudaEventDestroy(c->ev_b);
  if (c->scratch_done) cudaEventDestroy(c->scratch_done);
  if (c->stage_done) cudaEventDestroy(c->stage_done);
  c->sched_dense.release(cache, idle);
  c->sched_hc.release(cache, idle);
  c->sched_cls.release(cache, idle);
  c->sched_proxy.release(cache, idle);
  for (Schedule& g : c->sched_stage) g.release(cache, idle);
  c->stage_q.release(cache, idle);
  c->stage_out.release(cache, idle);
  c->stage_k.release(cache, idle);
  c->stage_v.release(cache, idle);
  if (c->copy_in) cudaStreamDestroy(c->copy_in);
  if (c->copy_out) cudaStreamDestroy(c->copy_out);
  for (cudaEvent_t e : c->ev_host)
    if (e) cudaEventDestroy(e);
  c->part_o.release(cache, idle);
  c->part_ml.release(cache, idle);
  c->part_mid.release(cache, idle);
  c->trace_dev.release(cache, idle);
  c->cls_o.release(cache, idle);
  c->cls_lse.release(cache, idle);
  c->cls_tok.release(cache, idle);
  c->memory.release(idle);
  if (current != c->device) cudaSetDevice(current);
  delete c;
  return HC_OK;
}

int headcast_release_memory(void) {
  int dev = 0;
  BlockCache* memory = cudaGetDevice(&dev) == cudaSuccess ? BlockCache::current(dev) : nullptr;
  if (memory && memory->trim()) return HC_OK;
  cudaGetLastError();
  return HC_ERR_CUDA;
}

int headcast_append(headcast_ctx* c, const void* k_new, const void* v_new, void* stream) {
  if (!c) return HC_ERR_INVALID_ARG;
  if (!aligned16(k_new) || !aligned16(v_new)) return fail(c, HC_ERR_INVALID_ARG, "k_new/v_new must be 16-byte aligned device pointers");
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  // ring bookkeeping: the sink block never moves; when full, the oldest rolling block's slot is reused
  int slot;
  std::vector<int> next = c->slots;
  if (static_cast<int>(next.size()) < c->n_blk) {
    slot = static_cast<int>(next.size());
    next.push_back(slot);
  } else if (c->n_blk == 1) {
    slot = 0;
  } else {
    slot = next[1];
    next.erase(next.begin() + 1);
    next.push_back(slot);
  }
  const bool split = c->state == STATE_SPLIT;
  const int dummy_next = (c->sd_slots == 2) ? (c->dummy_cur ^ 1) : 0;  // the older of a Dummy head's two blocks is replaced
  RouteParams r;
  fill_route(c, r);
  r.src_k = static_cast<const uint4*>(k_new);
  r.src_v = static_cast<const uint4*>(v_new);
  r.slots[0] = static_cast<int8_t>(slot);
  r.src_stride = 0;
  r.copy_mono = c->mono_k != nullptr;
  r.sd_slot_sink[0] = static_cast<int8_t>((split && c->sd_slots == 2) ? 1 : -1);  // the anchor block stays frozen
  r.sd_slot_dummy[0] = static_cast<int8_t>(split ? dummy_next : -1);
  r.copy_window = split;
  int rc = launch_route(c, r, 1, st);
  if (rc != HC_OK) return rc;
  c->slots.swap(next);
  if (split) {
    c->dummy_cur = dummy_next;
    c->sd_valid = c->sd_slots;
  }
  return HC_OK;
}

int headcast_overwrite_last(headcast_ctx* c, const void* k_new, const void* v_new, void* stream) {
  if (!c) return HC_ERR_INVALID_ARG;
  if (!aligned16(k_new) || !aligned16(v_new)) return fail(c, HC_ERR_INVALID_ARG, "k_new/v_new must be 16-byte aligned device pointers");
  if (c->slots.empty()) return fail(c, HC_ERR_STATE, "the cache is empty");
  const bool split = c->state == STATE_SPLIT;
  RouteParams r;
  fill_route(c, r);
  r.src_k = static_cast<const uint4*>(k_new);
  r.src_v = static_cast<const uint4*>(v_new);
  r.slots[0] = static_cast<int8_t>(c->slots.back());
  r.src_stride = 0;
  r.copy_mono = c->mono_k != nullptr;
  r.sd_slot_sink[0] = static_cast<int8_t>((split && c->sd_slots == 2 && c->sd_valid == 2) ? 1 : -1);
  r.sd_slot_dummy[0] = static_cast<int8_t>(split ? c->dummy_cur : -1);
  r.copy_window = split;
  return launch_route(c, r, 1, static_cast<cudaStream_t>(stream));
}

int headcast_full_attend(headcast_ctx* c, const void* q, void* out, void* stream) {
  if (!c) return HC_ERR_INVALID_ARG;
  if (!aligned16(q) || !aligned16(out)) return fail(c, HC_ERR_INVALID_ARG, "q/out must be 16-byte aligned device pointers");
  if (!c->mono_k) return fail(c, HC_ERR_STATE, "the monolithic cache was released at the split (keep_monolithic = 0)");
  if (c->slots.empty()) return fail(c, HC_ERR_STATE, "the cache is empty");
  if (c->sched_dense.key_filled != n_filled(c)) build_dense_schedule(c, c->sched_dense, OUT_BF16, true);
  return run_schedule(c, c->sched_dense, q, out, false, static_cast<cudaStream_t>(stream));
}

int headcast_set_labels(headcast_ctx* c, const int32_t* labels) {
  if (!c || !labels) return HC_ERR_INVALID_ARG;
  if (c->state != STATE_FILLING) return fail(c, HC_ERR_STATE, "labels are fixed once the cache is split");
  for (int h = 0; h < c->H; ++h)
    if (labels[h] < 0 || labels[h] > 3) return fail(c, HC_ERR_INVALID_ARG, "label %d of head %d is not an archetype", labels[h], h);
  c->labels.assign(labels, labels + c->H);
  c->have_labels = true;
  return HC_OK;
}

int headcast_get_labels(const headcast_ctx* c, int32_t* labels) {
  if (!c || !labels) return HC_ERR_INVALID_ARG;
  if (!c->have_labels) return HC_ERR_STATE;
  std::copy(c->labels.begin(), c->labels.end(), labels);
  return HC_OK;
}

int headcast_classify(headcast_ctx* c, const void* q, int32_t* labels_host, float* scores_host, void* stream) {
  if (!c || !labels_host) return HC_ERR_INVALID_ARG;
  if (!aligned16(q)) return fail(c, HC_ERR_INVALID_ARG, "q must be a 16-byte aligned device pointer");
  if (c->state != STATE_FILLING) return fail(c, HC_ERR_STATE, "classification runs on the monolithic cache, before the split");
  if (n_filled(c) < 2) return fail(c, HC_ERR_STATE, "classification needs at least two cached blocks");
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  const size_t rows = static_cast<size_t>(c->L) * c->H;
  HC_CUDA(c, c->cls_o.reserve(c->memory, rows * c->D, st));  // the reference output (fp32); the proxy outputs never leave registers
  HC_CUDA(c, c->cls_lse.reserve(c->memory, rows, st));
  HC_CUDA(c, c->cls_tok.reserve(c->memory, TOK_N * rows, st));
  const int newest = c->slots.back();
  const int cls_key = n_filled(c) * 64 + newest;  // the work lists depend on the fill and on where the newest block sits
  if (c->sched_cls.key_filled != cls_key) {
    // Reference (Eq. 2), Sink proxy and Dummy proxy from one sweep over the keys: the sweep is cut into the first
    // block, the middle blocks and the newest block (physical ring slots: the middle ones are one or two runs),
    // every piece leaves a partial result and cls_combine_kernel merges them three ways.
    std::vector<Proto> protos;
    Schedule& s = c->sched_cls;
    s.cls_groups.clear();
    const int nf = n_filled(c);
    struct Range { int slot_lo, slot_hi, tag; };
    std::vector<Range> ranges;
    ranges.push_back({0, 1, 0});
    if (newest > 1) ranges.push_back({1, newest, 1});
    if (newest + 1 < nf) ranges.push_back({newest + 1, nf, 1});
    if (newest != 0) ranges.push_back({newest, newest + 1, 2});
    for (int h = 0; h < c->H; ++h)
      for (int q0 = 0; q0 < c->L; q0 += 256) {
        ClsGroup g;
        g.head = h;
        g.q_start = q0;
        g.q_count[0] = std::min(128, c->L - q0);
        g.q_count[1] = std::max(0, std::min(128, c->L - q0 - 128));
        g.first_part = 0;
        g.n_parts = 0;
        const int group = static_cast<int>(s.cls_groups.size());
        s.cls_groups.push_back(g);
        for (const Range& r : ranges) {
          WorkItem w = range_item(h, MAP_MONO, h * c->D, static_cast<long long>(r.slot_lo) * c->L, (r.slot_hi - r.slot_lo) * c->L);
          Proto p;
          p.w = w;
          p.w.q_start[0] = q0;
          p.w.q_start[1] = q0 + 128;
          p.w.q_count[0] = g.q_count[0];
          p.w.q_count[1] = g.q_count[1];
          p.n_tiles = w.tiles_per_seg;
          p.w.tile_begin = 0;
          p.w.tile_end = p.n_tiles;
          p.cls_group = group;
          p.cls_tag = r.tag;
          protos.push_back(p);
        }
      }
    finalize_schedule(c, s, protos, true);
    s.key_filled = cls_key;
  }
  // the reference sweep is on its way before the host builds the proxy's work list
  int rc = run_schedule(c, c->sched_cls, q, nullptr, false, st);
  if (rc != HC_OK) return rc;
  if (c->sched_proxy.key_filled != cls_key) {
    // Spatial proxy: per query-tile pair, the tokens from r rows and r columns before its first query to as many behind
    // its last one, in every cached frame.  A pair that straddles two frames has to sweep whole frames, so frames of more
    // than 256 tokens are dealt into pairs of their own, of equal size (30 x 52 tokens, r = 2: seven pairs of 223 queries
    // and 4 key tiles per frame; with pairs of 256 across the block and whole grid rows it was 5 tiles, and 13 for every
    // sixth pair: 144 us for the sweep, now 113).  Where the bands cannot get shorter - a frame little larger than a pair,
    // rows or a radius that reach over most of it (1 x 300 tokens: 18 tiles per frame against 12) - and for smaller frames,
    // which fit into a tile or two either way, the fewer pairs across the block are the cheaper deal.
    std::vector<Proto> protos;
    c->sched_proxy.cls_groups.clear();
    const long long reach = std::min<long long>(static_cast<long long>(c->radius) * (c->G_w + 1), c->T_f);
    struct Run { int q0, n; };
    auto band_item = [&](const Run& run, int h) {
      const int q0 = run.q0, q1 = run.q0 + run.n - 1;
      int a = 0, b = c->T_f;
      if (q0 / c->T_f == q1 / c->T_f) {
        a = static_cast<int>(std::max<long long>(0, q0 % c->T_f - reach));
        b = static_cast<int>(std::min<long long>(c->T_f, q1 % c->T_f + reach + 1));
      }
      WorkItem w = range_item(h, MAP_MONO, h * c->D, a, b - a);
      w.seg_stride = c->T_f;
      w.q_start[0] = q0;
      w.q_start[1] = q0 + 128;
      w.q_count[0] = std::min(128, run.n);
      w.q_count[1] = std::max(0, run.n - 128);
      return w;
    };
    std::vector<Run> runs, per_frame;
    for (int q0 = 0; q0 < c->L; q0 += 256) runs.push_back({q0, std::min(256, c->L - q0)});
    if (c->T_f > 256) {
      const int n = (c->T_f + 255) / 256, size = (c->T_f + n - 1) / n;
      for (int f = 0; f < c->F_b; ++f)
        for (int i = 0; i < c->T_f; i += size) per_frame.push_back({f * c->T_f + i, std::min(size, c->T_f - i)});
      auto cost = [&](const std::vector<Run>& deal) {
        double sum = 0.0;
        for (const Run& run : deal) {
          const WorkItem w = band_item(run, 0);
          sum += COST_MEASURED.cost(w, w.tiles_per_seg * n_filled(c) * c->F_b, true);
        }
        return sum;
      };
      if (cost(per_frame) < cost(runs)) runs.swap(per_frame);
    }
    for (int h = 0; h < c->H; ++h)
      for (const Run& run : runs) {
        const WorkItem w = band_item(run, h);
        Proto p;
        p.w = w;
        p.n_tiles = w.tiles_per_seg * n_filled(c) * c->F_b;
        p.w.tile_begin = 0;
        p.w.tile_end = p.n_tiles;
        // whole or cut into pieces, a band leaves partial results that proxy_combine_kernel merges and scores
        ClsGroup g;
        g.head = h;
        g.q_start = run.q0;
        g.q_count[0] = p.w.q_count[0];
        g.q_count[1] = p.w.q_count[1];
        g.first_part = 0;
        g.n_parts = 0;
        p.cls_group = static_cast<int>(c->sched_proxy.cls_groups.size());
        p.cls_tag = 0;
        c->sched_proxy.cls_groups.push_back(g);
        protos.push_back(p);
      }
    finalize_schedule(c, c->sched_proxy, protos, true);
    c->sched_proxy.key_filled = cls_key;
  }
  rc = run_schedule(c, c->sched_proxy, q, nullptr, true, st);
  if (rc != HC_OK) return rc;
  {
    DecideParams d;
    d.tok = c->cls_tok.ptr;
    d.scores = reinterpret_cast<float*>(c->status_dev + 1);
    d.labels = c->status_dev + 1 + c->H * HC_N_SCORES;
    d.L = c->L;
    d.H = c->H;
    d.D = c->D;
    const double rank = 0.05 * (c->L - 1);
    d.rank_lo = static_cast<int32_t>(std::floor(rank));
    d.rank_frac = static_cast<float>(rank - std::floor(rank));
    d.theta_sink = c->cfg.theta_sink;
    d.theta_dummy = c->cfg.theta_dummy;
    d.theta_spatial = c->cfg.theta_spatial;
    d.theta_score = c->cfg.theta_score;
    d.gamma = c->cfg.gamma;
    d.rule = c->cfg.rule;
    d.mass_tau = c->cfg.mass_tau;
    HC_CUDA(c, launch_pdl(head_decide_kernel, dim3(c->H), dim3(DECIDE_THREADS), 0, st, d));
    ++c->launches;
  }
  // status word, scores and labels lie together: one copy to the host instead of three that wait for one another
  std::vector<int32_t> result(status_words(c));
  HC_CUDA(c, cudaMemcpyAsync(result.data(), c->status_dev, result.size() * sizeof(int32_t), cudaMemcpyDeviceToHost, st));
  HC_CUDA(c, cudaStreamSynchronize(st));
  rc = report_status(c, result[0], st);
  if (rc != HC_OK) return rc;
  const int32_t* scores = result.data() + 1;
  const int32_t* labels = scores + static_cast<size_t>(c->H) * HC_N_SCORES;
  std::copy(labels, labels + c->H, labels_host);
  if (scores_host) std::memcpy(scores_host, scores, static_cast<size_t>(c->H) * HC_N_SCORES * sizeof(float));
  c->labels.assign(labels_host, labels_host + c->H);
  c->have_labels = true;
  return HC_OK;
}

int headcast_split_cache(headcast_ctx* c, void* stream) {
  if (!c) return HC_ERR_INVALID_ARG;
  if (c->state != STATE_FILLING) return fail(c, HC_ERR_STATE, "the cache is already split");
  if (!c->have_labels) return fail(c, HC_ERR_STATE, "no labels: call headcast_classify or headcast_set_labels first");
  if (c->slots.empty()) return fail(c, HC_ERR_STATE, "the cache is empty");
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  assign_classes(c);
  // carve the three buffers out of the arena reserved (and zeroed) at create: no allocation on this path
  const int n_sd = c->n_cls[CLS_SINK] + c->n_cls[CLS_DUMMY];
  const size_t sd_elems = static_cast<size_t>(n_sd) * c->sd_slots * c->L * c->D;
  const size_t g_elems = cache_elems(c, c->n_cls[CLS_GLOBAL]);
  const size_t sp_elems = cache_elems(c, c->n_cls[CLS_SPATIAL]);
  c->sd_k = sd_elems ? c->arena_k : nullptr;
  c->sd_v = sd_elems ? c->arena_v : nullptr;
  c->g_k = g_elems ? c->arena_k + sd_elems : nullptr;
  c->g_v = g_elems ? c->arena_v + sd_elems : nullptr;
  c->sp_k = sp_elems ? c->arena_k + sd_elems + g_elems : nullptr;
  c->sp_v = sp_elems ? c->arena_v + sd_elems + g_elems : nullptr;
  {
    // one launch: grid row i gathers cached block i (ring slot slots[i]) out of the monolithic cache
    RouteParams r;
    fill_route(c, r);
    r.src_k = reinterpret_cast<const uint4*>(c->mono_k);
    r.src_v = reinterpret_cast<const uint4*>(c->mono_v);
    r.src_stride = static_cast<long long>(c->L) * c->H * c->CH;
    for (size_t i = 0; i < c->slots.size(); ++i) r.slots[i] = static_cast<int8_t>(c->slots[i]);
    r.copy_mono = 0;
    const int n = static_cast<int>(c->slots.size());
    r.sd_slot_sink[0] = 0;  // the first block is the Sink heads' anchor
    if (c->sd_slots == 2 && n >= 2) {
      r.sd_slot_sink[n - 1] = 1;   // anchor + current block
      r.sd_slot_dummy[n - 2] = 0;  // previous + current block
      r.sd_slot_dummy[n - 1] = 1;
      c->dummy_cur = 1;
      c->sd_valid = 2;
    } else {
      r.sd_slot_dummy[n - 1] = 0;
      c->dummy_cur = 0;
      c->sd_valid = 1;
    }
    r.copy_window = 1;
    int rc = launch_route(c, r, static_cast<int>(c->slots.size()), st);
    if (rc != HC_OK) return rc;
  }
  if (!c->cfg.keep_monolithic) {  // released in stream order, after the gather that reads it
    HC_CUDA(c, cudaFreeAsync(c->mono_k, st));
    HC_CUDA(c, cudaFreeAsync(c->mono_v, st));
    c->mono_k = c->mono_v = nullptr;
  }
  c->state = STATE_SPLIT;
  c->sched_hc.key_filled = -1;
  return build_maps(c);
}

int headcast_attend(headcast_ctx* c, const void* q, void* out, void* stream) {
  if (!c) return HC_ERR_INVALID_ARG;
  if (!aligned16(q) || !aligned16(out)) return fail(c, HC_ERR_INVALID_ARG, "q/out must be 16-byte aligned device pointers");
  if (c->state != STATE_SPLIT) return fail(c, HC_ERR_STATE, "head-specific attention needs the split cache");
  if (c->sched_hc.key_filled != n_filled(c) * 4 + c->sd_valid) build_headcast_schedule(c, c->sched_hc);
  return run_schedule(c, c->sched_hc, q, out, false, static_cast<cudaStream_t>(stream));
}

namespace {

int init_host_path(headcast_ctx* c) {
  if (!c->copy_in) HC_CUDA(c, cudaStreamCreateWithFlags(&c->copy_in, cudaStreamNonBlocking));
  if (!c->copy_out) HC_CUDA(c, cudaStreamCreateWithFlags(&c->copy_out, cudaStreamNonBlocking));
  for (cudaEvent_t& e : c->ev_host)
    if (!e) HC_CUDA(c, cudaEventCreateWithFlags(&e, cudaEventDisableTiming));
  return HC_OK;
}

}  // namespace

// What headcast_attend_host cuts a block into.  Its stages hide copies behind attention and copies of the other direction, but
// every run of neighbouring heads of one stage is a strided copy each way, of 5 us of the host (a whole small block: 40 to 60 us), and a
// stage is a launch, a merge and two events.  So a block is copied, attended and copied back as one where there is but one stage, or
// where it is small for the number of copies that the stages would make.  Append + four attends, stages against one: twelve heads of 64
// at 7 x 12 tokens (eight Dummy, four Spatial) 364 us against 204, 32 of 128 at 9 x 15 (all but Global) 1000 against 747; but 16 Global
// heads of 64 at 17 x 28 tokens 827 against 1030, two Spatial and two Global ones of 128 at 21 x 28 801 against 980.  Over 1529 layers of up to
// 4 MiB (2 to 32 heads, every mix of labels) this rule ends at 1.26 times the speed of stages for all of them (slowest twentieth: 0.99;
// one for all of them: 1.25, slowest twentieth 0.89); of 256, 384 and 512 KB per copy 384 comes nearest to the better of the two (1.2 % off).
// Blocks of 4 to 9 MiB stay in stages: as one they were 5 % slower on average.
constexpr size_t HOST_ONE_STAGE_BYTES = 4 << 20, HOST_BYTES_PER_COPY = 384 << 10;

struct HostStage { int group, lo, hi; };  // head group (0 Global, 1 Spatial, 2 Sink + Dummy) and rows [lo, hi)

static int host_group(const headcast_ctx* c, int h) { return c->cls[h] == CLS_GLOBAL ? 0 : c->cls[h] == CLS_SPATIAL ? 1 : 2; }

// Rows of the first of the two stages of the Global heads.
static int host_first_rows(const headcast_ctx* c) { return std::min(c->L, ((c->L / 2 + 255) / 256) * 256); }

static bool host_as_one(const headcast_ctx* c, size_t bytes) {
  if (bytes > HOST_ONE_STAGE_BYTES) return false;
  int stages = 0, copies = 0, runs[3] = {0, 0, 0};
  for (int h = 0; h < c->H; ++h) runs[host_group(c, h)] += h == 0 || host_group(c, h) != host_group(c, h - 1);
  for (int g = 0; g < 3; ++g) {
    const int cut = g == 0 && host_first_rows(c) < c->L ? 2 : 1;
    stages += runs[g] > 0 ? cut : 0;
    copies += runs[g] * cut;
  }
  return stages == 1 || bytes <= (copies - 1) * HOST_BYTES_PER_COPY;
}

int headcast_append_host(headcast_ctx* c, const void* k_host, const void* v_host, void* stream) {
  if (!c || !k_host || !v_host) return HC_ERR_INVALID_ARG;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  const size_t elems = static_cast<size_t>(c->L) * c->H * c->D;
  HC_CUDA(c, c->stage_k.reserve(c->memory, elems, st));
  HC_CUDA(c, c->stage_v.reserve(c->memory, elems, st));
  HC_CUDA(c, cudaMemcpyAsync(c->stage_k.ptr, k_host, elems * sizeof(__nv_bfloat16), cudaMemcpyHostToDevice, st));
  HC_CUDA(c, cudaMemcpyAsync(c->stage_v.ptr, v_host, elems * sizeof(__nv_bfloat16), cudaMemcpyHostToDevice, st));
  return headcast_append(c, c->stage_k.ptr, c->stage_v.ptr, stream);
}

// `done`: recorded once the call's last copy has left the staging buffers (nullptr: not).
static int attend_host(headcast_ctx* c, const void* q_host, void* out_host, cudaStream_t st, cudaEvent_t done) {
  const size_t elems = static_cast<size_t>(c->L) * c->H * c->D, bytes = elems * sizeof(__nv_bfloat16);
  HC_CUDA(c, c->stage_q.reserve(c->memory, elems, st));
  HC_CUDA(c, c->stage_out.reserve(c->memory, elems, st));
  if (host_as_one(c, bytes)) {
    HC_CUDA(c, cudaMemcpyAsync(c->stage_q.ptr, q_host, bytes, cudaMemcpyHostToDevice, st));
    const int rc = headcast_attend(c, c->stage_q.ptr, c->stage_out.ptr, st);
    if (rc != HC_OK) return rc;
    HC_CUDA(c, cudaMemcpyAsync(out_host, c->stage_out.ptr, bytes, cudaMemcpyDeviceToHost, st));
    if (done) HC_CUDA(c, cudaEventRecord(done, st));
    return HC_OK;
  }
  int rc = init_host_path(c);
  if (rc != HC_OK) return rc;
  const int key = n_filled(c) * 4 + c->sd_valid;
  // Stages: a stage's queries are copied in (strided: the rows of [L][H][d] hold all heads), attended and copied out
  // as a unit, so that the next stage's queries arrive and the previous stage's outputs leave while this stage
  // computes.  The Global heads do most of the arithmetic per byte moved, so their query rows are halved (at a
  // multiple of 256 rows: the query-tile pairs stay the same) and the halves go first and last: the kernels start
  // after a small copy, and when they end only a small copy is left; the other heads' copies hide in between.
  const int mid = host_first_rows(c);  // blocks of up to 256 tokens have one stage per group
  const HostStage stages[headcast_ctx::N_HOST_STAGES] = {{0, 0, mid}, {2, 0, c->L}, {1, 0, c->L}, {0, mid, c->L}};
  for (int i = 0; i < headcast_ctx::N_HOST_STAGES; ++i)
    if (c->sched_stage[i].key_filled != key)
      build_headcast_schedule(c, c->sched_stage[i], stages[i].group, stages[i].lo, stages[i].hi);
  const size_t pitch = static_cast<size_t>(c->H) * c->D * sizeof(__nv_bfloat16);
  auto copy_stage = [&](const HostStage& sg, bool in) -> int {
    const int rows = sg.hi - sg.lo;
    if (rows <= 0) return HC_OK;
    for (int h0 = 0; h0 < c->H;) {
      if (host_group(c, h0) != sg.group) {
        ++h0;
        continue;
      }
      int h1 = h0 + 1;
      while (h1 < c->H && host_group(c, h1) == sg.group) ++h1;
      const size_t off = static_cast<size_t>(sg.lo) * c->H * c->D + static_cast<size_t>(h0) * c->D;
      const size_t width = static_cast<size_t>(h1 - h0) * c->D * sizeof(__nv_bfloat16);
      if (in)
        HC_CUDA(c, cudaMemcpy2DAsync(c->stage_q.ptr + off, pitch, static_cast<const __nv_bfloat16*>(q_host) + off, pitch, width,
                                     rows, cudaMemcpyHostToDevice, c->copy_in));
      else
        HC_CUDA(c, cudaMemcpy2DAsync(static_cast<__nv_bfloat16*>(out_host) + off, pitch, c->stage_out.ptr + off, pitch, width,
                                     rows, cudaMemcpyDeviceToHost, c->copy_out));
      h0 = h1;
    }
    return HC_OK;
  };
  // everything enqueued on `stream` before this call (an append, the previous call's copies) comes first
  HC_CUDA(c, cudaEventRecord(c->ev_host[0], st));
  HC_CUDA(c, cudaStreamWaitEvent(c->copy_in, c->ev_host[0], 0));
  HC_CUDA(c, cudaStreamWaitEvent(c->copy_out, c->ev_host[0], 0));
  for (int i = 0; i < headcast_ctx::N_HOST_STAGES; ++i) {
    if (c->sched_stage[i].items.empty()) continue;
    if ((rc = copy_stage(stages[i], true)) != HC_OK) return rc;
    HC_CUDA(c, cudaEventRecord(c->ev_host[2 + 2 * i], c->copy_in));
    HC_CUDA(c, cudaStreamWaitEvent(st, c->ev_host[2 + 2 * i], 0));
    if ((rc = run_schedule(c, c->sched_stage[i], c->stage_q.ptr, c->stage_out.ptr, false, st)) != HC_OK) return rc;
    HC_CUDA(c, cudaEventRecord(c->ev_host[3 + 2 * i], st));
    HC_CUDA(c, cudaStreamWaitEvent(c->copy_out, c->ev_host[3 + 2 * i], 0));
    if ((rc = copy_stage(stages[i], false)) != HC_OK) return rc;
  }
  if (!done) done = c->ev_host[1];
  HC_CUDA(c, cudaEventRecord(done, c->copy_out));
  HC_CUDA(c, cudaStreamWaitEvent(st, done, 0));
  return HC_OK;
}

// All calls go through one pair of staging buffers, so every call leaves an event behind its last copy and a call on another stream
// than the last one waits for it.  (The launches and copies of a graph are the caller's to order; events of a capture mean
// nothing outside it.)
int headcast_attend_host(headcast_ctx* c, const void* q_host, void* out_host, void* stream) {
  if (!c || !q_host || !out_host) return HC_ERR_INVALID_ARG;
  if (c->state != STATE_SPLIT) return fail(c, HC_ERR_STATE, "head-specific attention needs the split cache");
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  cudaStreamCaptureStatus status = cudaStreamCaptureStatusNone;
  HC_CUDA(c, cudaStreamIsCapturing(st, &status));
  if (status != cudaStreamCaptureStatusNone) return attend_host(c, q_host, out_host, st, nullptr);
  unsigned long long id = 0;
  HC_CUDA(c, cudaStreamGetId(st, &id));
  if (!c->stage_done) HC_CUDA(c, cudaEventCreateWithFlags(&c->stage_done, cudaEventDisableTiming));
  if (c->stage_used && c->stage_stream != id) HC_CUDA(c, cudaStreamWaitEvent(st, c->stage_done, 0));
  c->stage_used = true;
  c->stage_stream = id;
  const int rc = attend_host(c, q_host, out_host, st, c->stage_done);
  if (rc != HC_OK) {  // what was enqueued before it failed comes first all the same
    for (cudaStream_t copies : {c->copy_in, c->copy_out})
      if (copies && cudaEventRecord(c->stage_done, copies) == cudaSuccess) cudaStreamWaitEvent(st, c->stage_done, 0);
    cudaEventRecord(c->stage_done, st);
    cudaGetLastError();
  }
  return rc;
}


int headcast_export_cache(headcast_ctx* c, int32_t head, void* k_out, void* v_out, int32_t* n_tokens_host, void* stream) {
  if (!c || head < 0 || head >= c->H) return HC_ERR_INVALID_ARG;
  if ((k_out && !aligned16(k_out)) || (v_out && !aligned16(v_out))) return fail(c, HC_ERR_INVALID_ARG, "outputs must be 16-byte aligned");
  ExportParams e;
  std::memset(&e, 0, sizeof(e));
  e.dst_k = static_cast<uint4*>(k_out);
  e.dst_v = static_cast<uint4*>(v_out);
  e.sp_base = c->sp_base;
  e.sp_nc = c->sp_nc;
  e.L = c->L;
  e.H = c->H;
  e.chunks = c->CH;
  e.tokens_per_frame = c->T_f;
  e.frames_per_block = c->F_b;
  e.n_blocks = c->n_blk;
  e.sd_slots = c->sd_slots;
  const int cl = (c->state == STATE_SPLIT) ? static_cast<int>(c->cls[head]) : static_cast<int>(CLS_NONE);
  if (cl == CLS_NONE) {
    e.layout = 0; e.head = head; e.src_k = reinterpret_cast<const uint4*>(c->mono_k); e.src_v = reinterpret_cast<const uint4*>(c->mono_v);
  } else if (cl == CLS_GLOBAL) {
    e.layout = 1; e.head = c->idx[head]; e.src_k = reinterpret_cast<const uint4*>(c->g_k); e.src_v = reinterpret_cast<const uint4*>(c->g_v);
  } else if (cl == CLS_SPATIAL) {
    e.layout = 2; e.head = c->idx[head]; e.src_k = reinterpret_cast<const uint4*>(c->sp_k); e.src_v = reinterpret_cast<const uint4*>(c->sp_v);
  } else {
    e.layout = 3; e.head = (cl == CLS_SINK) ? c->idx[head] : c->n_cls[CLS_SINK] + c->idx[head];
    e.src_k = reinterpret_cast<const uint4*>(c->sd_k); e.src_v = reinterpret_cast<const uint4*>(c->sd_v);
  }
  if (e.layout == 3) {
    e.n_logical = c->sd_valid;
    if (cl == CLS_SINK) {
      e.slots[0] = 0;
      e.slots[1] = 1;
    } else if (c->sd_valid == 2) {
      e.slots[0] = c->dummy_cur ^ 1;  // previous block first
      e.slots[1] = c->dummy_cur;
    } else {
      e.slots[0] = c->dummy_cur;
    }
  } else {
    e.n_logical = n_filled(c);
    for (int i = 0; i < e.n_logical; ++i) e.slots[i] = c->slots[i];
  }
  if (n_tokens_host) *n_tokens_host = e.n_logical * c->L;
  if (e.n_logical == 0 || (!k_out && !v_out)) return HC_OK;
  const long long total = static_cast<long long>(e.n_logical) * c->L * c->CH;
  const int blocks = static_cast<int>(std::min<long long>((total + 255) / 256, c->n_sm * 16LL));
  export_head_kernel<<<blocks, 256, 0, static_cast<cudaStream_t>(stream)>>>(e);
  HC_CUDA(c, cudaGetLastError());
  ++c->launches;
  return HC_OK;
}

int headcast_n_filled(const headcast_ctx* c) { return c ? n_filled(c) : HC_ERR_INVALID_ARG; }

int64_t headcast_launch_count(const headcast_ctx* c) { return c ? c->launches : 0; }

double headcast_attend_flops(const headcast_ctx* c, int32_t dense) {
  if (!c) return 0.0;
  const int nf = n_filled(c);
  if (dense) return 4.0 * c->H * static_cast<double>(c->L) * nf * c->L * c->D;
  if (!c->have_labels) return 0.0;
  double cell_sq = 0.0;
  for (const CellGeom& g : c->cells) cell_sq += static_cast<double>(g.ch * g.cw) * (g.ch * g.cw);
  double f = 0.0;
  for (int h = 0; h < c->H; ++h) {
    if (c->labels[h] == HC_SINK || c->labels[h] == HC_DUMMY)
      f += 4.0 * c->L * static_cast<double>(c->state == STATE_SPLIT ? c->sd_valid : std::min(c->sd_slots, nf)) * c->L * c->D;
    else if (c->labels[h] == HC_GLOBAL) f += 4.0 * c->L * static_cast<double>(nf) * c->L * c->D;
    else f += 4.0 * c->F_b * static_cast<double>(nf) * c->F_b * cell_sq * c->D;
  }
  return f;
}

int headcast_set_kernel_timing(headcast_ctx* c, int32_t enable) {
  if (!c) return HC_ERR_INVALID_ARG;
  if (enable && !c->ev_a) {
    HC_CUDA(c, cudaEventCreate(&c->ev_a));
    HC_CUDA(c, cudaEventCreate(&c->ev_b));
  }
  c->timing = enable != 0;
  c->ev_valid = false;
  return HC_OK;
}

int headcast_last_attention_kernel_ms(headcast_ctx* c, float* ms_host) {
  if (!c || !ms_host) return HC_ERR_INVALID_ARG;
  if (!c->ev_valid) return fail(c, HC_ERR_STATE, "no attention kernel was timed yet");
  HC_CUDA(c, cudaEventSynchronize(c->ev_b));
  HC_CUDA(c, cudaEventElapsedTime(ms_host, c->ev_a, c->ev_b));
  return HC_OK;
}

int headcast_set_tracing(headcast_ctx* c, int32_t enable) {
  if (!c) return HC_ERR_INVALID_ARG;
  c->tracing = enable != 0;
  return HC_OK;
}

int headcast_read_trace(headcast_ctx* c, int64_t* rows_host, int32_t capacity, int32_t* n_items_host) {
  if (!c || !n_items_host) return HC_ERR_INVALID_ARG;
  const int n = static_cast<int>(c->trace_items.size());
  *n_items_host = n;
  if (!rows_host || n == 0) return HC_OK;
  HC_CUDA(c, cudaDeviceSynchronize());
  std::vector<unsigned long long> t(2 * static_cast<size_t>(n));
  HC_CUDA(c, cudaMemcpy(t.data(), c->trace_dev.ptr, t.size() * sizeof(unsigned long long), cudaMemcpyDeviceToHost));
  int cta = 0;
  for (int i = 0; i < n && i < capacity; ++i) {
    while (cta + 1 < static_cast<int>(c->trace_cta_first.size()) && c->trace_cta_first[cta + 1] <= i) ++cta;
    const WorkItem& w = c->trace_items[i];
    int64_t* r = rows_host + 8 * static_cast<size_t>(i);
    r[0] = cta;
    r[1] = w.head;
    r[2] = w.cell;
    r[3] = w.q_count[0] + w.q_count[1];
    r[4] = w.tile_end - w.tile_begin;
    r[5] = w.out_mode;
    r[6] = static_cast<int64_t>(t[2 * i]);
    r[7] = static_cast<int64_t>(t[2 * i + 1]);
  }
  return HC_OK;
}

int headcast_plan_schedule(const headcast_config* cfg, const int32_t* labels_host, int32_t n_filled, int32_t n_ctas,
                           int32_t dense, int32_t* items_host, int32_t capacity, int32_t* n_items_host,
                           int32_t* cta_first_host) {
  if (!cfg || !n_items_host || n_filled < 1 || n_ctas < 1 || n_ctas > 4096) return HC_ERR_INVALID_ARG;
  headcast_ctx c;
  std::vector<int32_t> sp_base, sp_nc;
  int rc = init_host(&c, cfg, sp_base, sp_nc);
  if (rc != HC_OK) return rc;
  if (n_filled > c.n_blk) return HC_ERR_INVALID_ARG;
  c.n_sm = n_ctas;
  for (int i = 0; i < n_filled; ++i) c.slots.push_back(i);
  Schedule s;
  if (dense) {
    build_dense_schedule(&c, s, OUT_BF16, true);
  } else {
    if (!labels_host) return HC_ERR_INVALID_ARG;
    for (int h = 0; h < c.H; ++h)
      if (labels_host[h] < 0 || labels_host[h] > 3) return HC_ERR_INVALID_ARG;
    c.labels.assign(labels_host, labels_host + c.H);
    assign_classes(&c);
    c.sd_valid = std::min(c.sd_slots, n_filled);
    c.dummy_cur = c.sd_valid - 1;
    build_headcast_schedule(&c, s);
  }
  *n_items_host = static_cast<int32_t>(s.items.size());
  static_assert(sizeof(WorkItem) == 16 * sizeof(int32_t), "work items are exported as 16 int32 each");
  if (items_host)
    std::memcpy(items_host, s.items.data(), std::min<size_t>(s.items.size(), capacity) * sizeof(WorkItem));
  if (cta_first_host) std::copy(s.cta_first.begin(), s.cta_first.end(), cta_first_host);
  return HC_OK;
}

int headcast_selftest_bounded_wait(headcast_ctx* c, int32_t limit_ms, void* stream) {
  if (!c || limit_ms < 1 || limit_ms > 1000) return HC_ERR_INVALID_ARG;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  bounded_wait_selftest_kernel<<<1, 64, 0, st>>>(c->status_dev, static_cast<unsigned long long>(limit_ms) * 1000000ull, 99);
  HC_CUDA(c, cudaGetLastError());
  ++c->launches;
  return read_status(c, st);
}

int headcast_check(headcast_ctx* c, void* stream) {
  if (!c) return HC_ERR_INVALID_ARG;
  return read_status(c, static_cast<cudaStream_t>(stream));
}

const char* headcast_last_error(const headcast_ctx* c) { return c ? c->err.c_str() : "null context"; }

}  // extern "C"

// =====================================================================================================
// Allocation-free dense attention
// =====================================================================================================
// Everything the kernels need in global memory besides the caller's tensors - the work list, the per-CTA ranges, the status
// word, the partial results of key ranges that are cut and what is to be merged - lives in one file-scope device array of
// fixed size (noalloc_scratch.cu; the two tensor maps travel as kernel parameters).  A GPU carries these bytes from its first such call
// until the process exits.
namespace {

constexpr int NOALLOC_MAX_ITEMS = HEADCAST_NOALLOC_MAX_ITEMS;
constexpr int NOALLOC_MAX_CTAS = 1024;
// Of a cut, in key tiles: launch and a first batch of parts, each further part.  Fitted to 1300 timings of equal pieces, merging and
// partial results cost 1.5 + 1.7 times the share of CTAs in use + 0.2 per part at head_dim 64, 1.5 + 2.6 times + 0.2 at 128; with
// the partial result's 1.1 these constants charge a little more where parts are few: no size was slower cut than whole.
constexpr double NOALLOC_MERGE = 3.0, NOALLOC_MERGE_PART = 0.12;

// Query-tile pairs are cut along their keys where whole ones would leave much of the GPU idle, over at most this many CTAs, each
// of which leaves at most two partial results (its first and its last piece).
constexpr int NOALLOC_CUT_CTAS = 148, NOALLOC_SLOTS = 2 * NOALLOC_CUT_CTAS, NOALLOC_MERGES = 2 * NOALLOC_CUT_CTAS;

struct NoAllocScratch {
  WorkItem items[NOALLOC_MAX_ITEMS + NOALLOC_CUT_CTAS];
  CombineEntry merge[NOALLOC_MERGES];  // two per pair that is cut
  int32_t cta_first[NOALLOC_MAX_CTAS + 1];
  int32_t status;
  // of cut pairs alone, behind the lists, which lie on one page that way: an uncut call of 20 us took 0.15 us more with the lists 39 MB into the array
  alignas(256) float part_o[NOALLOC_SLOTS][256 * 128];  // (head_dim 64 uses half of it)
  float2 part_ml[NOALLOC_SLOTS][256];
};

static_assert(sizeof(NoAllocScratch) <= NOALLOC_SCRATCH_BYTES, "the array of noalloc_scratch.cu is too small");

// How the query-tile pairs of one call (all of the same key range) are spread.
struct NoAllocPlan {
  int n_items, n_tiles;  // pairs, key tiles of each
  int n_cta;             // CTAs that get work (cut), or that whole pairs are dealt to
  int cuts;              // 0: whole pairs; > 0: every pair in so many equal pieces, a CTA each; < 0: pairs laid end to end, an equal share of the line to each CTA
  // first key tile of CTA b's share, on the line of all pairs
  __host__ __device__ long long share_begin(int b) const {
    if (cuts > 0) return static_cast<long long>(b / cuts) * n_tiles + static_cast<long long>(b % cuts) * n_tiles / cuts;
    const long long x = static_cast<long long>(n_items) * n_tiles * b / n_cta, in = x % n_tiles;
    return in < MIN_PART_TILES ? x - in : n_tiles - in < MIN_PART_TILES ? x + n_tiles - in : x;  // no piece shorter than that
  }
};

// Whole pairs, equal pieces of each, or equal shares of the line of all of them, whichever the scheduler's cost model expects to
// end first; cutting has to promise 5 %, and merging costs one more launch.  The line is for numbers of pairs that fill the last wave
// badly: its shares are at least two proper pieces long, and beyond eight waves there is too little to gain.  1373 queries, 5492 keys,
// sixteen heads of 64 (a line): 77 -> 61 us; 687 queries, 2748 keys, eight heads of 128 (equal pieces): 46.5 -> 24.8;
// 1785 queries, 12495 keys, four heads of 128: 166 -> 53.
// At head_dim 128 a key tile of a line takes 1.16 times as long as one of whole pairs (the CTAs of whole pairs walk a head's keys in
// step and share them in L2, those of a line stand at different places, and all SMs at work clock lower), so there a line has to end
// earlier by that count too.  Measured on 704 sizes of 1 to 1100 pairs and 8 to 200 key tiles each: without it 130 pairs of 200 key
// tiles took 409 us as a line and 353 whole, 130 of 120 226 and 214, 80 of 16 38.2 and 37.3; with it no line is more than 1.2 % slower
// than whole pairs, and the lines that it refuses were at most 4.5 % faster.  At head_dim 64 and for equal pieces no size was slower cut.
constexpr double NOALLOC_LINE_TILE_128 = 1.16, NOALLOC_LINE_MORE_128 = 10.7, NOALLOC_WHOLE_MORE_128 = 3.5;
NoAllocPlan noalloc_plan(int n_items, int n_keys, int n_sm, int head_dim) {
  NoAllocPlan p = {n_items, (n_keys + 127) / 128, n_sm, 0};
  if (p.n_tiles < 8) return p;  // half of that does not pay for a merge
  const double item = COST_MEASURED.item, piece = COST_MEASURED.item + COST_MEASURED.partial;
  const int waves = (n_items + n_sm - 1) / n_sm;
  double best = 0.95 * waves * (p.n_tiles + item);
  const int n_cta = std::min(n_sm, NOALLOC_CUT_CTAS);
  for (int k = 2; k <= std::min(n_cta / n_items, p.n_tiles); ++k) {
    const double end = (p.n_tiles + k - 1) / k + piece + NOALLOC_MERGE + NOALLOC_MERGE_PART * k;
    if (end < best) {
      best = end;
      p.cuts = k;
      p.n_cta = n_items * k;
    }
  }
  const double share = static_cast<double>(n_items) * p.n_tiles / n_cta;
  if (n_items > n_cta / 4 && n_items < 8 * n_cta && p.n_tiles >= 4 * MIN_PART_TILES && share >= 2 * MIN_PART_TILES) {
    const double end = share + item * n_items / n_cta + 2 * piece - item + NOALLOC_MERGE;
    const bool in_step = head_dim == 128 && waves * (p.n_tiles + NOALLOC_WHOLE_MORE_128) <= NOALLOC_LINE_TILE_128 * share + NOALLOC_LINE_MORE_128;
    if (end < best && !in_step) {
      p.cuts = -1;
      p.n_cta = n_cta;
    }
  }
  return p;
}

// Writes the work list of one call, and what is to be merged: whole pairs (`plan`: their number) over as many blocks as it takes,
// shares of a line in one block with a thread per CTA of the attention kernel (which it scans over).  Built here and not copied from the
// host: three copies from pageable memory made a call take 21 us of host time whatever its size.  For whole pairs it is a kernel without
// shared memory and without the plan among its parameters: with both, the launches of such a call took 7.0 us of the host and not 6.65.
template <typename Plan>
__global__ void __launch_bounds__(std::is_same_v<Plan, int> ? 256 : NOALLOC_MAX_CTAS)
    noalloc_list_kernel(NoAllocScratch* s, Plan plan, int grid, int n_heads, int head_dim, int n_queries, int n_keys) {
  pdl_launch_dependents();
  const int b = blockIdx.x * blockDim.x + threadIdx.x, nt = (n_keys + 127) / 128;
  auto item = [&](int pair, int begin, int end) {
    const int h = pair % n_heads, q0 = pair / n_heads * 256;
    WorkItem w = {};
    w.head = h;
    w.cell = -1;
    w.q_start[0] = q0;
    w.q_start[1] = q0 + 128;
    w.q_count[0] = min(128, n_queries - q0);
    w.q_count[1] = max(0, min(128, n_queries - q0 - 128));
    w.kv_x0 = h * head_dim;
    w.seg_len = n_keys;
    w.tiles_per_seg = nt;
    w.tile_begin = begin;
    w.tile_end = end;
    w.out_mode = OUT_BF16;
    return w;
  };
  if constexpr (std::is_same_v<Plan, int>) {
    const int each = plan / grid, more = plan % grid;  // CTA b owns items b, b + grid, ...: `each`, plus one for the first `more`
    const int at = (b % grid) * each + min(b % grid, more) + b / grid;
    const WorkItem w = item(b, 0, nt);
    pdl_wait();  // the kernel before may still read the list of its own call
    if (b <= grid) s->cta_first[b] = b * each + min(b, more);
    if (b == 0) s->status = 0;  // the array keeps the previous call's contents
    if (b < plan) s->items[at] = w;
  } else {
    __shared__ int32_t warp_sum[3][NOALLOC_MAX_CTAS / 32];
    // CTA b's share [x0, x1) of the line: its pieces, how many of them are partial results, and whether it begins a pair that is cut
    const long long x0 = b < plan.n_cta ? plan.share_begin(b) : 0, x1 = b < plan.n_cta ? plan.share_begin(b + 1) : 0;
    const int p0 = static_cast<int>(x0 / nt), p1 = x1 > x0 ? static_cast<int>((x1 - 1) / nt) : p0 - 1;  // first and last pair
    auto begin_of = [&](int pair) { return pair == p0 ? static_cast<int>(x0 - static_cast<long long>(p0) * nt) : 0; };
    auto end_of = [&](int pair) { return pair == p1 ? static_cast<int>(x1 - static_cast<long long>(p1) * nt) : nt; };
    int n[3] = {p1 - p0 + 1, 0, 0};
    if (n[0] > 0) {
      const bool first_cut = begin_of(p0) > 0 || end_of(p0) < nt;
      n[1] = (first_cut ? 1 : 0) + (p1 > p0 && end_of(p1) < nt ? 1 : 0);
      n[2] = begin_of(p1) == 0 && end_of(p1) < nt ? 1 : 0;
    }
    int before[3];  // the same of all CTAs before this one
#pragma unroll
    for (int q = 0; q < 3; ++q) {
      int upto = n[q];
#pragma unroll
      for (int off = 1; off < 32; off *= 2) {
        const int y = __shfl_up_sync(0xffffffffu, upto, off);
        if ((b & 31) >= off) upto += y;
      }
      if ((b & 31) == 31) warp_sum[q][b >> 5] = upto;
      before[q] = upto - n[q];
    }
    __syncthreads();
#pragma unroll
    for (int q = 0; q < 3; ++q)
      for (int w = 0; w < (b >> 5); ++w) before[q] += warp_sum[q][w];
    pdl_wait();  // the kernel before may still read the list of its own call
    if (b < grid) s->cta_first[b] = before[0];
    if (b == grid - 1) s->cta_first[grid] = before[0] + n[0];
    if (b == 0) s->status = 0;
    int slot = before[1];
    for (int pair = p0; pair <= p1; ++pair) {
      WorkItem w = item(pair, begin_of(pair), end_of(pair));
      if (w.tile_end - w.tile_begin < nt) {
        w.out_mode = OUT_PARTIAL;
        w.out_slot = slot++;
        if (w.tile_begin == 0) {  // this pair's pieces: here and in the CTAs that follow
          int more = 1;
          while (plan.share_begin(b + more + 1) < static_cast<long long>(pair + 1) * nt) ++more;
          for (int t = 0; t < 2; ++t) s->merge[2 * before[2] + t] = {w.head, -1, w.q_start[t], w.q_count[t], w.out_slot, more + 1, t, 0};
        }
      }
      s->items[before[0] + pair - p0] = w;
    }
    // entries that the launch of the merge has blocks for but no pair was cut for
    int n_entries = 0;
    for (int w = 0; w < static_cast<int>(blockDim.x) / 32; ++w) n_entries += 2 * warp_sum[2][w];
    for (int i = n_entries + b; i < NOALLOC_MERGES; i += blockDim.x) s->merge[i].q_count = 0;
  }
}

constexpr int NOALLOC_MAX_DEVICES = 64;
struct NoAllocDevice {
  unsigned long long context = 0;     // the CUDA context that the rest was found in: after a device reset it is another one
  NoAllocScratch* scratch = nullptr;  // the array's address on that GPU
  int n_sm = 0;
};
NoAllocDevice g_noalloc_dev[NOALLOC_MAX_DEVICES];

char g_noalloc_error[256] = "";

int noalloc_fail(int code, const char* msg, cudaError_t e = cudaSuccess) {
  if (e != cudaSuccess) cudaGetLastError();  // reported here, and by no later call
  if (e != cudaSuccess)
    snprintf(g_noalloc_error, sizeof(g_noalloc_error), "%s: %s", msg, cudaGetErrorString(e));
  else
    snprintf(g_noalloc_error, sizeof(g_noalloc_error), "%s", msg);
  return code;
}

// Once per device and CUDA context, with that device current.
int noalloc_setup(int dev) {
  NoAllocDevice& d = g_noalloc_dev[dev];
  unsigned long long context = 0;
  const bool known = current_context_id(&context);
  if (d.scratch && known && d.context == context) return HC_OK;
  cudaDeviceProp prop;
  cudaError_t e = cudaGetDeviceProperties(&prop, dev);
  if (e != cudaSuccess) return noalloc_fail(HC_ERR_CUDA, "cudaGetDeviceProperties", e);
  if (prop.major != 10) return noalloc_fail(HC_ERR_UNSUPPORTED, "this library needs an sm_100 device");
  void* ptr = nullptr;
  e = noalloc_scratch_address(&ptr);
  if (e != cudaSuccess || !ptr) return noalloc_fail(HC_ERR_CUDA, "loading the scratch array", e);
  e = cudaFuncSetAttribute(attn_kernel<128, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, AttnSmem<128>::DYN_BYTES);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(attn_kernel<64, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, AttnSmem<64>::DYN_BYTES);
  if (e != cudaSuccess) return noalloc_fail(HC_ERR_CUDA, "cudaFuncSetAttribute", e);
  // The driver loads a kernel's code when the kernel is first asked for, and may take device memory or wait for the device then:
  // all that any size can need is asked for here, in the first call, whatever its size.
  auto load = [&](auto* kernel) {
    cudaFuncAttributes attributes;
    if (e == cudaSuccess) e = cudaFuncGetAttributes(&attributes, kernel);
  };
  load(noalloc_list_kernel<int>);
  load(noalloc_list_kernel<NoAllocPlan>);
  load(attn_kernel<64, false>);
  load(attn_kernel<128, false>);
  load(combine_kernel<64>);
  load(combine_kernel<128>);
  if (e != cudaSuccess) return noalloc_fail(HC_ERR_CUDA, "cudaFuncGetAttributes", e);
  if (!current_context_id(&d.context)) return noalloc_fail(HC_ERR_CUDA, "cuCtxGetId");
  d.n_sm = std::min(prop.multiProcessorCount, NOALLOC_MAX_CTAS);
  d.scratch = static_cast<NoAllocScratch*>(ptr);
  return HC_OK;
}

}  // namespace

extern "C" {

int headcast_dense_attend_noalloc(const void* q, const void* k, const void* v, void* out, int32_t n_queries,
                                  int32_t n_keys, int32_t n_heads, int32_t head_dim, float softmax_scale, void* stream) {
  if (!aligned16(q) || !aligned16(k) || !aligned16(v) || !aligned16(out))
    return noalloc_fail(HC_ERR_INVALID_ARG, "q, k, v and out must be 16-byte aligned device pointers");
  if (n_queries < 1 || n_keys < 1 || n_heads < 1 || n_heads > MAX_HEADS || (head_dim != 64 && head_dim != 128) ||
      !(softmax_scale >= 0.f))
    return noalloc_fail(HC_ERR_INVALID_ARG, "sizes out of range (head_dim 64 or 128, 1..64 heads)");
  const long long n_items = static_cast<long long>(n_heads) * ((n_queries + 255) / 256);
  if (n_items > NOALLOC_MAX_ITEMS)
    return noalloc_fail(HC_ERR_UNSUPPORTED,
                        "too large for the fixed scratch: n_heads * ceil(n_queries / 256) must not exceed "
                        "HEADCAST_NOALLOC_MAX_ITEMS");
  if (static_cast<long long>(n_keys) * n_heads * head_dim >= (1LL << 40) || static_cast<long long>(n_queries) * n_heads >= (1LL << 31))
    return noalloc_fail(HC_ERR_INVALID_ARG, "sizes out of range");
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return noalloc_fail(HC_ERR_CUDA, "cudaGetDevice", e);
  if (dev < 0 || dev >= NOALLOC_MAX_DEVICES) return noalloc_fail(HC_ERR_UNSUPPORTED, "device index beyond 63");
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  {
    // calls share one scratch array: a graph replayed beside other calls would overwrite their work list, so capturing
    // streams are turned away.  (This query also makes the device's CUDA context current to a thread that is new to it.)
    cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
    e = cudaStreamIsCapturing(st, &cap);
    if (e != cudaSuccess) return noalloc_fail(HC_ERR_CUDA, "cudaStreamIsCapturing", e);
    if (cap != cudaStreamCaptureStatusNone)
      return noalloc_fail(HC_ERR_UNSUPPORTED, "headcast_dense_attend_noalloc cannot be called on a capturing stream");
  }
  int rc = noalloc_setup(dev);
  if (rc != HC_OK) return rc;
  const NoAllocDevice& d = g_noalloc_dev[dev];

  const uint64_t row_elems = static_cast<uint64_t>(n_heads) * head_dim;
  AttnParams p;
  std::memset(&p, 0, sizeof(p));
  if (!make_tmap_bf16_2d(&p.maps[0], k, row_elems, n_keys, row_elems, 128) ||
      !make_tmap_bf16_2d(&p.maps[1], v, row_elems, n_keys, row_elems, 128))
    return noalloc_fail(HC_ERR_CUDA, "cuTensorMapEncodeTiled failed or is unavailable");
  const int n_cta = d.n_sm;
  const NoAllocPlan plan = noalloc_plan(static_cast<int>(n_items), n_keys, n_cta, head_dim);
  const dim3 list_threads(plan.cuts ? (n_cta + 31) / 32 * 32 : 256), list_blocks(plan.cuts ? 1 : (std::max(plan.n_items, n_cta + 1) + 255) / 256);
  e = plan.cuts ? launch_pdl(noalloc_list_kernel<NoAllocPlan>, list_blocks, list_threads, 0, st, d.scratch, plan, n_cta, n_heads, head_dim, n_queries, n_keys)
                : launch_pdl(noalloc_list_kernel<int>, list_blocks, list_threads, 0, st, d.scratch, plan.n_items, n_cta, n_heads, head_dim, n_queries, n_keys);
  if (e != cudaSuccess) return noalloc_fail(HC_ERR_CUDA, "launching the list kernel", e);

  p.items = d.scratch->items;
  p.cta_first = d.scratch->cta_first;
  p.q = static_cast<const __nv_bfloat16*>(q);
  p.out = static_cast<__nv_bfloat16*>(out);
  p.n_heads = n_heads;
  p.tokens_per_frame = n_queries;
  p.grid_w = 1;
  p.block_tokens = n_queries;
  const float scale = softmax_scale > 0.f ? softmax_scale : 1.0f / std::sqrt(static_cast<float>(head_dim));
  p.scale_log2e = scale * 1.4426950408889634f;
  p.status = &d.scratch->status;
  p.part_o = &d.scratch->part_o[0][0];
  p.part_ml = &d.scratch->part_ml[0][0];
  e = launch_pdl(head_dim == 128 ? attn_kernel<128, false> : attn_kernel<64, false>, dim3(n_cta), dim3(ATTN_THREADS),
                 head_dim == 128 ? AttnSmem<128>::DYN_BYTES : AttnSmem<64>::DYN_BYTES, st, p);
  if (e != cudaSuccess) return noalloc_fail(HC_ERR_CUDA, "launching the attention kernel", e);
  if (plan.cuts != 0) {
    // pairs that are cut: with equal pieces all of them, else at most one at every boundary between two shares
    const int entries = 2 * (plan.cuts > 0 ? plan.n_items : std::min(plan.n_items, plan.n_cta - 1));
    const int n_long = plan.cuts > COMBINE_LONG_PARTS ? entries : 0;
    e = launch_pdl(head_dim == 128 ? combine_kernel<128> : combine_kernel<64>, dim3(n_long * 128 + (entries - n_long) * (128 / COMBINE_ROWS)),
                   dim3(COMBINE_ROWS * (head_dim / 8)), 0, st, d.scratch->merge, n_long, nullptr, p.part_o, p.part_ml, p.out, n_heads, n_queries, 1,
                   false);
    if (e != cudaSuccess) return noalloc_fail(HC_ERR_CUDA, "launching the merge kernel", e);
  }
  return HC_OK;
}

int headcast_noalloc_status(void* stream) {
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= NOALLOC_MAX_DEVICES || !g_noalloc_dev[dev].scratch)
    return noalloc_fail(HC_ERR_STATE, "headcast_dense_attend_noalloc has not run on this device");
  int32_t status = 0;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  cudaError_t e = cudaMemcpyAsync(&status, &g_noalloc_dev[dev].scratch->status, sizeof(status), cudaMemcpyDeviceToHost, st);
  if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  if (e != cudaSuccess) return noalloc_fail(HC_ERR_CUDA, "reading the status word", e);
  if (status != 0) return noalloc_fail(HC_ERR_TIMEOUT, "the attention kernel gave up on a bounded wait");
  return HC_OK;
}

const char* headcast_noalloc_last_error(void) { return g_noalloc_error; }

}  // extern "C"
