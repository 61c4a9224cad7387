// A CUDA runtime for tests on the CPU.  Memory is host memory with a settable capacity, kernels are recorded and not run,
// and the failures that matter to the library's host code can be switched on: a device whose work is not finished, a stream
// under capture (what the runtime refuses beside a capture was read off a B200: a device synchronisation in every mode,
// cudaMalloc, cudaFree and cudaFreeAsync in the global mode only), memory that runs out, a device reset.
#include <cuda.h>
#include <cuda_runtime_api.h>

#include <cstdint>
#include <cstdlib>
#include <cstring>
#include <map>
#include <set>
#include <string>
#include <vector>

namespace {

struct Fake {
  long long capacity = 1ll << 40, used = 0, pool_unused = 0;
  std::map<char*, size_t> live;                // cudaMalloc and pool memory in the library's hands
  std::set<char*> from_pool;
  std::multimap<size_t, char*> pool;           // freed to the pool, still reserved
  std::map<char*, size_t> busy;                // memory that work in flight still touches
  long long busy_writes = 0;                   // host-ordered writes into it: somebody was handed memory in use
  long long stray_writes = 0;                  // writes to what is no device memory
  int device = 0;
  int capture = 0;                             // of another or of capture_stream: 0 none, 1 relaxed, 2 global
  cudaStream_t capture_stream = nullptr;
  bool invalidated = false;                    // the capture was destroyed by a refused call
  unsigned long long context_id = 1;
  cudaError_t last_error = cudaSuccess;        // what the next cudaGetLastError reports
  std::map<const void*, std::string> kernels;
  std::map<const void*, int> smem;             // dynamic shared memory that a kernel may be launched with
  std::set<const void*> loaded;                // kernels whose code the driver has been asked for
  // launches, copies to and from the device (with their address there), events, waits and the host's waits for a stream or the
  // device, in order: "L<stream>:<kernel>@<scratch> H<stream>:<to> D<stream>:<from> E<stream>:<event> W<stream>:<event> Y<stream>: S"
  std::string log;
};

Fake& fake() {  // the library registers its kernels before this file's globals would exist
  static Fake state;
  return state;
}

cudaError_t failed(cudaError_t e) {
  fake().last_error = e;
  return e;
}

cudaError_t refused() {
  fake().invalidated = true;
  return failed(cudaErrorStreamCaptureUnsupported);
}

void finish() { fake().busy.clear(); }

bool inside(const std::map<char*, size_t>& blocks, char* c) {
  auto it = blocks.upper_bound(c);
  return it != blocks.begin() && c < (--it)->first + it->second;
}

bool write_to(void* p) {  // by the device
  if (inside(fake().busy, static_cast<char*>(p))) ++fake().busy_writes;
  if (inside(fake().live, static_cast<char*>(p))) return true;
  ++fake().stray_writes;
  return false;
}

cudaError_t take(void** p, size_t bytes) {
  if (fake().used + static_cast<long long>(bytes) > fake().capacity) return failed(cudaErrorMemoryAllocation);
  char* c = static_cast<char*>(std::aligned_alloc(4096, (bytes + 4095) / 4096 * 4096));
  fake().used += bytes;
  fake().live[c] = bytes;
  *p = c;
  return cudaSuccess;
}

void to_pool(char* c) {
  fake().pool.emplace(fake().live[c], c);
  fake().pool_unused += fake().live[c];
  fake().from_pool.erase(c);
  fake().live.erase(c);
}

CUresult encode_tiled(CUtensorMap* m, ...) {
  std::memset(m, 0, sizeof(*m));
  return CUDA_SUCCESS;
}
CUresult context_id(CUcontext, unsigned long long* id) {
  *id = fake().context_id;
  return CUDA_SUCCESS;
}

std::string handle(const void* p) { return std::to_string(reinterpret_cast<uintptr_t>(p)); }

}  // namespace

extern "C" {

const void* fake_saw_launch(const char* name, void** args);

void fake_reset() {
  fake().capacity = 1ll << 40;
  fake().capture = 0;
  fake().capture_stream = nullptr;
  fake().invalidated = false;
  fake().busy.clear();
  fake().busy_writes = fake().stray_writes = 0;
  fake().log.clear();
}
void fake_capacity_left(long long bytes) { fake().capacity = fake().used + bytes; }
long long fake_used() { return fake().used; }
long long fake_pool_unused() { return fake().pool_unused; }
void fake_work_in_flight() { fake().busy = fake().live; }
long long fake_busy() { return static_cast<long long>(fake().busy.size()); }
long long fake_stray_writes() { return fake().stray_writes; }
long long fake_busy_writes() { return fake().busy_writes; }
void fake_capture(int mode, void* stream) {
  fake().capture = mode;
  fake().capture_stream = static_cast<cudaStream_t>(stream);
  fake().invalidated = false;
}
int fake_capture_invalidated() { return fake().invalidated; }
int fake_is_live(void* p) { return fake().live.count(static_cast<char*>(p)) != 0; }
int fake_kernels_loaded() { return static_cast<int>(fake().loaded.size()); }
const char* fake_log() { return fake().log.c_str(); }
void fake_clear_log() { fake().log.clear(); }
void fake_device_reset() {  // every allocation is gone, a new context takes the old one's place
  fake().live.clear();
  fake().from_pool.clear();
  fake().pool.clear();
  fake().busy.clear();
  fake().smem.clear();
  fake().loaded.clear();
  fake().used = fake().pool_unused = 0;
  ++fake().context_id;
}

// ------------------------------------------------------------------------------------------ memory
cudaError_t cudaMalloc(void** p, size_t bytes) { return fake().capture == 2 ? refused() : take(p, bytes); }
cudaError_t cudaFree(void* p) {
  if (!p) return cudaSuccess;
  if (fake().capture == 2) return refused();
  char* c = static_cast<char*>(p);
  if (!fake().live.count(c)) return failed(cudaErrorInvalidValue);
  if (fake().from_pool.count(c)) {
    to_pool(c);
    return cudaSuccess;
  }
  finish();
  fake().used -= fake().live[c];
  fake().live.erase(c);
  std::free(c);
  return cudaSuccess;
}
cudaError_t cudaMemPoolCreate(cudaMemPool_t* pool, const cudaMemPoolProps*) {
  *pool = reinterpret_cast<cudaMemPool_t>(fake().context_id);
  return cudaSuccess;
}
cudaError_t cudaMemPoolDestroy(cudaMemPool_t) { return cudaSuccess; }
cudaError_t cudaMemPoolSetAttribute(cudaMemPool_t, cudaMemPoolAttr, void*) { return cudaSuccess; }
cudaError_t cudaMemPoolTrimTo(cudaMemPool_t pool, size_t) {
  if (reinterpret_cast<unsigned long long>(pool) != fake().context_id) return failed(cudaErrorInvalidValue);
  for (auto& e : fake().pool) {
    fake().used -= e.first;
    std::free(e.second);
  }
  fake().pool.clear();
  fake().pool_unused = 0;
  return cudaSuccess;
}
cudaError_t cudaMallocFromPoolAsync(void** p, size_t bytes, cudaMemPool_t pool, cudaStream_t) {
  if (fake().capture == 2) return refused();
  if (reinterpret_cast<unsigned long long>(pool) != fake().context_id) return failed(cudaErrorInvalidValue);
  auto it = fake().pool.find(bytes);
  if (it != fake().pool.end()) {
    fake().live[it->second] = bytes;
    *p = it->second;
    fake().pool_unused -= bytes;
    fake().pool.erase(it);
  } else {
    cudaError_t e = take(p, bytes);
    if (e != cudaSuccess) return e;
  }
  fake().from_pool.insert(static_cast<char*>(*p));
  return cudaSuccess;
}
cudaError_t cudaFreeAsync(void* p, cudaStream_t) {
  if (fake().capture == 2) return refused();
  if (!fake().from_pool.count(static_cast<char*>(p))) return failed(cudaErrorInvalidValue);
  to_pool(static_cast<char*>(p));
  return cudaSuccess;
}
cudaError_t cudaMemcpy(void* dst, const void* src, size_t n, cudaMemcpyKind kind) {
  if (kind == cudaMemcpyDeviceToHost || write_to(dst)) std::memcpy(dst, src, n);
  return cudaSuccess;
}
static void copied(void* dst, const void* src, cudaMemcpyKind kind, cudaStream_t s) {
  if (kind == cudaMemcpyHostToDevice) fake().log += "H" + handle(s) + ":" + handle(dst) + " ";
  if (kind == cudaMemcpyDeviceToHost) fake().log += "D" + handle(s) + ":" + handle(src) + " ";
}
cudaError_t cudaMemcpyAsync(void* dst, const void* src, size_t n, cudaMemcpyKind kind, cudaStream_t s) {
  copied(dst, src, kind, s);
  return cudaMemcpy(dst, src, n, kind);
}
cudaError_t cudaMemcpy2DAsync(void* dst, size_t, const void* src, size_t, size_t, size_t, cudaMemcpyKind kind, cudaStream_t s) {
  copied(dst, src, kind, s);
  if (kind == cudaMemcpyHostToDevice) write_to(dst);
  return cudaSuccess;
}
cudaError_t cudaMemsetAsync(void* p, int v, size_t n, cudaStream_t) {
  if (write_to(p)) std::memset(p, v, n);
  return cudaSuccess;
}

// ------------------------------------------------------------------------------------------ device, streams, events
cudaError_t cudaGetDevice(int* d) { *d = fake().device; return cudaSuccess; }
cudaError_t cudaSetDevice(int d) { fake().device = d; return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr a, int) {
  *v = a == cudaDevAttrComputeCapabilityMajor ? 10 : 148;
  return cudaSuccess;
}
cudaError_t cudaGetDeviceProperties_v2(cudaDeviceProp* p, int) {
  std::memset(p, 0, sizeof(*p));
  p->major = 10;
  p->multiProcessorCount = 148;
  return cudaSuccess;
}
cudaError_t cudaDeviceSynchronize() {
  if (fake().capture) return refused();
  finish();
  fake().log += "S ";
  return cudaSuccess;
}
cudaError_t cudaStreamIsCapturing(cudaStream_t s, cudaStreamCaptureStatus* st) {
  *st = fake().capture && fake().capture_stream && s == fake().capture_stream ? cudaStreamCaptureStatusActive : cudaStreamCaptureStatusNone;
  return cudaSuccess;
}
cudaError_t cudaStreamSynchronize(cudaStream_t s) {
  if (fake().capture == 2 || (fake().capture && s == fake().capture_stream && s)) return refused();
  fake().log += "Y" + handle(s) + ": ";
  return cudaSuccess;
}
cudaError_t cudaStreamGetId(cudaStream_t s, unsigned long long* id) {
  *id = reinterpret_cast<uintptr_t>(s);
  return cudaSuccess;
}
cudaError_t cudaStreamCreateWithFlags(cudaStream_t* s, unsigned) {
  static uintptr_t n = 1000;
  *s = reinterpret_cast<cudaStream_t>(++n);
  return cudaSuccess;
}
cudaError_t cudaStreamDestroy(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamWaitEvent(cudaStream_t s, cudaEvent_t e, unsigned) {
  fake().log += "W" + handle(s) + ":" + handle(e) + " ";
  return cudaSuccess;
}
cudaError_t cudaEventCreateWithFlags(cudaEvent_t* e, unsigned) {
  static uintptr_t n = 5000;
  *e = reinterpret_cast<cudaEvent_t>(++n);
  return cudaSuccess;
}
cudaError_t cudaEventCreate(cudaEvent_t* e) { return cudaEventCreateWithFlags(e, 0); }
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t e, cudaStream_t s) {
  fake().log += "E" + handle(s) + ":" + handle(e) + " ";
  return cudaSuccess;
}
cudaError_t cudaEventSynchronize(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float* ms, cudaEvent_t, cudaEvent_t) { *ms = 0.f; return cudaSuccess; }
cudaError_t cudaGetLastError() {
  const cudaError_t e = fake().last_error;
  fake().last_error = cudaSuccess;
  return e;
}
const char* cudaGetErrorString(cudaError_t) { return "fake error"; }
cudaError_t cudaGetDriverEntryPoint(const char* name, void** fn, unsigned long long, cudaDriverEntryPointQueryResult* q) {
  *fn = std::strcmp(name, "cuCtxGetId") == 0 ? reinterpret_cast<void*>(context_id) : reinterpret_cast<void*>(encode_tiled);
  *q = cudaDriverEntryPointSuccess;
  return cudaSuccess;
}

// ------------------------------------------------------------------------------------------ kernels
cudaError_t cudaFuncGetAttributes(cudaFuncAttributes* a, const void* fn) {
  std::memset(a, 0, sizeof(*a));
  fake().loaded.insert(fn);
  return cudaSuccess;
}
cudaError_t cudaFuncSetAttribute(const void* fn, cudaFuncAttribute a, int v) {
  fake().loaded.insert(fn);
  if (a == cudaFuncAttributeMaxDynamicSharedMemorySize) fake().smem[fn] = v;
  return cudaSuccess;
}
cudaError_t cudaGetSymbolAddress(void** p, const void*) {
  static char scratch[2][1 << 20];
  *p = scratch[fake().context_id % 2];
  return cudaSuccess;
}
static cudaError_t launched(const void* fn, void** args, size_t smem, cudaStream_t s) {
  if (smem > 48 << 10 && static_cast<int>(smem) > fake().smem[fn]) return failed(cudaErrorInvalidValue);
  fake().loaded.insert(fn);
  const std::string& name = fake().kernels[fn];
  const void* scratch = fake_saw_launch(name.c_str(), args);
  fake().log += "L" + handle(s) + ":" + name + "@" + handle(scratch) + " ";
  return cudaSuccess;
}
cudaError_t cudaLaunchKernel(const void* fn, dim3, dim3, void** args, size_t smem, cudaStream_t s) { return launched(fn, args, smem, s); }
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t* c, const void* fn, void** args) { return launched(fn, args, c->dynamicSmemBytes, c->stream); }
static dim3 pushed_grid, pushed_block;
static size_t pushed_smem;
static void* pushed_stream;
unsigned __cudaPushCallConfiguration(dim3 grid, dim3 block, size_t smem, void* stream) {
  pushed_grid = grid;
  pushed_block = block;
  pushed_smem = smem;
  pushed_stream = stream;
  return 0;
}
cudaError_t __cudaPopCallConfiguration(dim3* grid, dim3* block, size_t* smem, void* stream) {
  *grid = pushed_grid;
  *block = pushed_block;
  *smem = pushed_smem;
  *static_cast<void**>(stream) = pushed_stream;
  return cudaSuccess;
}
void** __cudaRegisterFatBinary(void*) {
  static void* h;
  return &h;
}
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
void __cudaRegisterFunction(void**, const char* host, char*, const char* name, int, void*, void*, void*, void*, int*) { fake().kernels[host] = name; }
void __cudaRegisterVar(void**, char*, char*, const char*, int, size_t, int, int) {}
char __cudaInitModule(void**) { return 1; }

}  // extern "C"
