// A stand-in for the CUDA runtime, linked with the library's own objects in
// place of it: no GPU, no kernel runs.  Device memory is host memory, streams
// are numbers, and every launch is written to a log, so that tests can check
// on any machine which launches the host code makes, in which order, from
// which thread, and under which function attributes.
#include <algorithm>
#include <atomic>
#include <chrono>
#include <cstdlib>
#include <cstring>
#include <map>
#include <mutex>
#include <string>
#include <thread>
#include <vector>

#include <cuda_runtime_api.h>

namespace {

constexpr size_t kStaticLimit = 48 << 10;  // dynamic shared memory a kernel may have without opting in

std::mutex mu;
std::map<const void*, std::string> names;                  // kernels
std::map<std::pair<int, const void*>, size_t> max_smem;    // per (device, kernel)
std::map<std::string, unsigned> delays_us;                 // by a part of the kernel's name
std::map<cudaStream_t, cudaGraph_t> capturing;
std::map<const void*, size_t> allocated;
size_t live_bytes = 0, peak_bytes = 0, stray_copies = 0;
std::string text;
bool logging = true;
void* host_word = nullptr;
std::atomic<uintptr_t> next_handle{0x1000};
std::atomic<int> attr_delay_us{0};

thread_local int device = 0, tag = 0;
thread_local cudaError_t last_error = cudaSuccess;
struct Config {
  dim3 grid, block;
  size_t smem;
  cudaStream_t stream;
};
thread_local std::vector<Config> configs;

cudaError_t fail(cudaError_t e) { return last_error = e; }

template <typename T>
T handle() {
  return reinterpret_cast<T>(next_handle.fetch_add(16));
}

void log_line(const std::string& what, cudaStream_t st, const void* p) {
  if (!logging) return;
  text += std::to_string(tag) + " " + std::to_string(device) + " " + std::to_string((uintptr_t)st) + " " + what + " " +
          std::to_string((uintptr_t)p) + "\n";
}

void pause_us(unsigned us) {
  if (us) std::this_thread::sleep_for(std::chrono::microseconds(us));
}

cudaError_t allocate(void** p, size_t n) {
  *p = nullptr;
  if (posix_memalign(p, 4096, n ? n : 1)) return fail(cudaErrorMemoryAllocation);
  memset(*p, 0, n);
  std::lock_guard<std::mutex> lk(mu);
  allocated[*p] = n;
  live_bytes += n;
  peak_bytes = std::max(peak_bytes, live_bytes);
  return cudaSuccess;
}

cudaError_t release(void* p) {
  {
    std::lock_guard<std::mutex> lk(mu);
    const auto it = allocated.find(p);
    if (p && it == allocated.end()) return fail(cudaErrorInvalidValue);
    if (p) {
      live_bytes -= it->second;
      allocated.erase(it);
    }
  }
  free(p);
  return cudaSuccess;
}

}  // namespace

extern "C" {

// ---- what the tests use ------------------------------------------------------------------

void fake_set_device(int d) { device = d; }
void fake_set_tag(int t) { tag = t; }
void fake_delay(const char* part, unsigned us) {
  std::lock_guard<std::mutex> lk(mu);
  delays_us[part] = us;
}
void fake_capture(void* st, int on) {
  std::lock_guard<std::mutex> lk(mu);
  if (on) capturing[(cudaStream_t)st] = handle<cudaGraph_t>();
  else capturing.erase((cudaStream_t)st);
}
void fake_clear_log() {
  std::lock_guard<std::mutex> lk(mu);
  text.clear();
}
size_t fake_log(char* out, size_t cap) {
  std::lock_guard<std::mutex> lk(mu);
  if (out && cap) {
    const size_t n = std::min(cap - 1, text.size());
    memcpy(out, text.data(), n);
    out[n] = 0;
  }
  return text.size();
}
// From now on a kernel's shared-memory limit is set late in a call of us microseconds if it is below 64 KB, and early
// in one of twice that if it is not.
void fake_slow_attributes(int us) { attr_delay_us = us; }
void* fake_host_word() { return host_word; }
// Copies from addresses that are in no allocation (device memory that has been freed), which were left out.
size_t fake_stray_copies() {
  std::lock_guard<std::mutex> lk(mu);
  return stray_copies;
}
// Most memory allocated at once since the last call, beyond what is allocated now.
size_t fake_peak() {
  std::lock_guard<std::mutex> lk(mu);
  const size_t over = peak_bytes - live_bytes;
  peak_bytes = live_bytes;
  return over;
}

// `episodes` times: sets bit `low` and then bit `high` of the word, as two
// kernels of two sorts would, and waits until the word is 0 again.  Meanwhile
// the calling thread takes the word with take(stream).  Returns in how many
// episodes no take returned `high_status`.
uint64_t fake_status_episodes(int (*take)(void*), void* stream, uint32_t low, uint32_t high, int high_status,
                              uint64_t episodes) {
  uint32_t* word = static_cast<uint32_t*>(host_word);
  std::atomic<uint64_t> done{0};
  {
    std::lock_guard<std::mutex> lk(mu);
    logging = false;  // millions of takes
  }
  std::thread setter([&] {
    uint32_t r = 1;
    for (uint64_t e = 0; e < episodes; ++e) {
      __atomic_fetch_or(word, low, __ATOMIC_ACQ_REL);
      r = r * 1664525u + 1013904223u;
      for (volatile uint32_t k = 0, n = r >> 23; k < n; k = k + 1) {
      }
      __atomic_fetch_or(word, high, __ATOMIC_ACQ_REL);
      for (uint32_t k = 0; __atomic_load_n(word, __ATOMIC_ACQUIRE); ++k)
        if (k > 1000) std::this_thread::yield();
      done.fetch_add(1);
    }
  });
  uint64_t seen = 0;
  for (uint32_t idle = 0; done.load() < episodes;) {
    const int status = take(stream);
    seen += status == high_status ? 1 : 0;
    idle = status ? 0 : idle + 1;
    if (idle > 1000) std::this_thread::yield();
  }
  setter.join();
  return episodes - seen;
}

// ---- the runtime ---------------------------------------------------------------------------

void** __cudaRegisterFatBinary(void*) { return handle<void**>(); }
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
void __cudaRegisterVar(void**, char*, char*, const char*, int, size_t, int, int) {}
void __cudaRegisterFunction(void**, const char* host, char*, const char* name, int, uint3*, uint3*, dim3*, dim3*, int*) {
  std::lock_guard<std::mutex> lk(mu);
  names[host] = name;
}
unsigned __cudaPushCallConfiguration(dim3 grid, dim3 block, size_t smem, struct CUstream_st* st) {
  configs.push_back({grid, block, smem, st});
  return 0;
}
cudaError_t __cudaPopCallConfiguration(dim3* grid, dim3* block, size_t* smem, void* st) {
  const Config c = configs.back();
  configs.pop_back();
  *grid = c.grid;
  *block = c.block;
  *smem = c.smem;
  *static_cast<cudaStream_t*>(st) = c.stream;
  return cudaSuccess;
}
cudaError_t __cudaGetKernel(cudaKernel_t* k, const void* fun) {
  *k = (cudaKernel_t)fun;
  return cudaSuccess;
}
cudaError_t __cudaLaunchKernel(cudaKernel_t k, dim3, dim3, void** args, size_t smem, cudaStream_t st) {
  unsigned us = 0;
  {
    std::lock_guard<std::mutex> lk(mu);
    const void* fun = (const void*)k;
    const std::string& name = names[fun];
    const auto it = max_smem.find({device, fun});
    if (smem > (it == max_smem.end() ? kStaticLimit : it->second)) return fail(cudaErrorInvalidValue);
    const void* first = nullptr;  // the first parameter's leading 8 bytes (a control block's address, for one)
    if (args && args[0]) memcpy(&first, args[0], sizeof(first));
    log_line(name, st, first);
    for (const auto& d : delays_us)
      if (name.find(d.first) != std::string::npos) us = std::max(us, d.second);
  }
  pause_us(us);
  return cudaSuccess;
}

cudaError_t cudaFuncSetAttribute(const void* fun, cudaFuncAttribute, int value) {
  const bool small = value < (64 << 10);
  if (small) pause_us(attr_delay_us);
  {
    std::lock_guard<std::mutex> lk(mu);
    max_smem[{device, fun}] = (size_t)value;
  }
  if (!small) pause_us(2 * attr_delay_us);
  return cudaSuccess;
}
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int* n, const void* fun, int, size_t smem, unsigned) {
  std::lock_guard<std::mutex> lk(mu);
  const auto it = max_smem.find({device, fun});
  *n = smem > (it == max_smem.end() ? kStaticLimit : it->second) ? 0 : 2;
  return cudaSuccess;
}
cudaError_t cudaGetDevice(int* d) {
  *d = device;
  return cudaSuccess;
}
cudaError_t cudaGetDeviceProperties(cudaDeviceProp* p, int) {
  memset(p, 0, sizeof(*p));
  p->major = 10;
  p->minor = 3;
  p->multiProcessorCount = 152;
  return cudaSuccess;
}
cudaError_t cudaGetLastError() {
  const cudaError_t e = last_error;
  last_error = cudaSuccess;
  return e;
}
cudaError_t cudaDeviceGetDefaultMemPool(cudaMemPool_t* p, int) {
  *p = handle<cudaMemPool_t>();
  return cudaSuccess;
}
cudaError_t cudaMemPoolSetAttribute(cudaMemPool_t, cudaMemPoolAttr, void*) { return cudaSuccess; }
cudaError_t cudaMalloc(void** p, size_t n) { return allocate(p, n); }
cudaError_t cudaMallocAsync(void** p, size_t n, cudaStream_t) { return allocate(p, n); }
cudaError_t cudaMallocHost(void** p, size_t n) { return allocate(p, n); }
cudaError_t cudaHostAlloc(void** p, size_t n, unsigned) {
  const cudaError_t e = allocate(p, n);
  host_word = *p;
  return e;
}
cudaError_t cudaHostGetDevicePointer(void** d, void* h, unsigned) {
  *d = h;
  return cudaSuccess;
}
cudaError_t cudaFree(void* p) { return release(p); }
cudaError_t cudaFreeAsync(void* p, cudaStream_t) { return release(p); }
cudaError_t cudaFreeHost(void* p) { return release(p); }
cudaError_t cudaMemcpyAsync(void* d, const void* s, size_t n, cudaMemcpyKind kind, cudaStream_t) {
  std::lock_guard<std::mutex> lk(mu);
  if (kind == cudaMemcpyDeviceToHost) {
    auto it = allocated.upper_bound(s);
    if (it == allocated.begin() || (const char*)s + n > (const char*)(--it)->first + it->second) {
      ++stray_copies;
      return cudaSuccess;
    }
  }
  memmove(d, s, n);
  return cudaSuccess;
}
cudaError_t cudaMemcpyFromSymbol(void* d, const void*, size_t n, size_t, cudaMemcpyKind) {
  memset(d, 0, n);
  return cudaSuccess;
}
cudaError_t cudaMemsetAsync(void* d, int v, size_t n, cudaStream_t) {
  memset(d, v, n);
  return cudaSuccess;
}
cudaError_t cudaGetSymbolAddress(void** p, const void*) {
  static void* scratch = nullptr;
  if (!scratch) allocate(&scratch, 8u << 20);
  *p = scratch;
  return cudaSuccess;
}
cudaError_t cudaPointerGetAttributes(cudaPointerAttributes* a, const void*) {
  memset(a, 0, sizeof(*a));
  return cudaSuccess;
}
cudaError_t cudaEventCreate(cudaEvent_t* e) {
  *e = handle<cudaEvent_t>();
  return cudaSuccess;
}
cudaError_t cudaEventCreateWithFlags(cudaEvent_t* e, unsigned) { return cudaEventCreate(e); }
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float* ms, cudaEvent_t, cudaEvent_t) {
  *ms = 0.f;
  return cudaSuccess;
}
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventSynchronize(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaStreamCreateWithFlags(cudaStream_t* s, unsigned) {
  *s = handle<cudaStream_t>();
  return cudaSuccess;
}
cudaError_t cudaStreamDestroy(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t st) {
  unsigned us;
  {
    std::lock_guard<std::mutex> lk(mu);
    log_line("wait", st, nullptr);
    us = delays_us.count("wait") ? delays_us["wait"] : 0;
  }
  pause_us(us);
  return cudaSuccess;
}
cudaError_t cudaStreamWaitEvent(cudaStream_t, cudaEvent_t, unsigned) { return cudaSuccess; }
cudaError_t cudaStreamIsCapturing(cudaStream_t s, cudaStreamCaptureStatus* c) {
  std::lock_guard<std::mutex> lk(mu);
  *c = capturing.count(s) ? cudaStreamCaptureStatusActive : cudaStreamCaptureStatusNone;
  return cudaSuccess;
}
cudaError_t cudaStreamBeginCapture(cudaStream_t s, cudaStreamCaptureMode) {
  fake_capture(s, 1);
  return cudaSuccess;
}
cudaError_t cudaStreamBeginCaptureToGraph(cudaStream_t s, cudaGraph_t, const cudaGraphNode_t*, const cudaGraphEdgeData*,
                                          size_t, cudaStreamCaptureMode) {
  fake_capture(s, 1);
  return cudaSuccess;
}
cudaError_t cudaStreamEndCapture(cudaStream_t s, cudaGraph_t* g) {
  *g = handle<cudaGraph_t>();
  fake_capture(s, 0);
  return cudaSuccess;
}
cudaError_t cudaStreamGetCaptureInfo(cudaStream_t s, cudaStreamCaptureStatus* c, unsigned long long*, cudaGraph_t* g,
                                     const cudaGraphNode_t** deps, const cudaGraphEdgeData** edges, size_t* n) {
  std::lock_guard<std::mutex> lk(mu);
  const auto it = capturing.find(s);
  *c = it == capturing.end() ? cudaStreamCaptureStatusNone : cudaStreamCaptureStatusActive;
  if (g) *g = it == capturing.end() ? nullptr : it->second;
  if (deps) *deps = nullptr;
  if (edges) *edges = nullptr;
  if (n) *n = 0;
  return cudaSuccess;
}
cudaError_t cudaStreamUpdateCaptureDependencies(cudaStream_t, cudaGraphNode_t*, const cudaGraphEdgeData*, size_t,
                                                unsigned) {
  return cudaSuccess;
}
cudaError_t cudaGraphConditionalHandleCreate(cudaGraphConditionalHandle* h, cudaGraph_t, unsigned, unsigned) {
  *h = next_handle.fetch_add(16);
  return cudaSuccess;
}
cudaError_t cudaGraphAddNode(cudaGraphNode_t* node, cudaGraph_t, const cudaGraphNode_t*, const cudaGraphEdgeData*, size_t,
                             cudaGraphNodeParams* p) {
  *node = handle<cudaGraphNode_t>();
  static thread_local cudaGraph_t body[1];
  body[0] = handle<cudaGraph_t>();
  p->conditional.phGraph_out = body;
  return cudaSuccess;
}
cudaError_t cudaGraphInstantiate(cudaGraphExec_t* e, cudaGraph_t, unsigned long long) {
  *e = handle<cudaGraphExec_t>();
  return cudaSuccess;
}
cudaError_t cudaGraphDestroy(cudaGraph_t) { return cudaSuccess; }
cudaError_t cudaGraphLaunch(cudaGraphExec_t e, cudaStream_t st) {
  std::lock_guard<std::mutex> lk(mu);
  log_line("graph", st, e);
  return cudaSuccess;
}

}  // extern "C"
