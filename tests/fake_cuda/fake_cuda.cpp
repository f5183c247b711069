// A stand-in for the CUDA runtime, linked with the library's own object files so
// that its host side runs without a GPU: memory of a set capacity per device,
// per-device function attributes, and launches that are checked against the
// limits that a real launch has and are otherwise left out.  Copies from the
// (imaginary) device give zeros, which the library reads as success.
#include <cuda.h>
#include <cuda_runtime.h>

#include <cstdlib>
#include <cstring>
#include <map>
#include <mutex>
#include <string>
#include <utility>

namespace {

constexpr int kDevices = 2;
constexpr size_t kDefaultShared = 48 * 1024, kMostShared = 227 * 1024;
const int kSms[kDevices] = {152, 76};

struct Block {
  size_t bytes;
  int dev;
};
struct State {
  std::mutex mu;
  size_t capacity[kDevices] = {}, used[kDevices] = {}, peak[kDevices] = {};
  std::map<uintptr_t, Block> blocks;
  uintptr_t next = uintptr_t(1) << 44;
  std::map<std::pair<const void*, int>, size_t> shared;  // opted-in dynamic shared memory
  std::map<const void*, std::string> names;
  std::map<std::string, long long> counts;
};
State& S() {
  static State* s = new State;
  return *s;
}

thread_local int t_dev = 0;
thread_local cudaError_t t_err = cudaSuccess;
thread_local dim3 t_grid, t_block;
thread_local size_t t_shared;
thread_local cudaStream_t t_stream;

cudaError_t fail(cudaError_t e) {
  t_err = e;
  return e;
}
void count(const std::string& what) {
  std::lock_guard<std::mutex> lk(S().mu);
  ++S().counts[what];
}

cudaError_t launch(const void* f, dim3 g, dim3 b, size_t shared) {
  State& s = S();
  std::lock_guard<std::mutex> lk(s.mu);
  const auto at = s.shared.find({f, t_dev});
  const size_t allowed = at == s.shared.end() ? kDefaultShared : at->second;
  const std::string& name = s.names[f];
  if (shared > allowed || !g.x || !g.y || !g.z || g.x > 0x7fffffffu || g.y > 65535u || g.z > 65535u ||
      b.x * b.y * b.z > 1024u) {
    ++s.counts["refused " + name];
    return fail(cudaErrorInvalidValue);
  }
  ++s.counts["launch " + name];
  return cudaSuccess;
}

void* host_alloc(size_t n) { return std::calloc(1, n ? n : 1); }

CUresult encode(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*, const cuuint64_t*,
                const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle,
                CUtensorMapL2promotion, CUtensorMapFloatOOBfill) {
  return CUDA_SUCCESS;
}

template <class T>
cudaError_t handle(T* p) {
  *p = reinterpret_cast<T>(host_alloc(16));
  return cudaSuccess;
}
template <class T>
cudaError_t drop(T p) {
  std::free(reinterpret_cast<void*>(p));
  return cudaSuccess;
}

}  // namespace

extern "C" {

// ---- for the tests ----
void fake_reset(size_t capacity) {
  State& s = S();
  std::lock_guard<std::mutex> lk(s.mu);
  for (int d = 0; d < kDevices; ++d) {
    s.capacity[d] = capacity;
    s.peak[d] = s.used[d];
  }
  s.counts.clear();
}
long long fake_count(const char* what) {
  std::lock_guard<std::mutex> lk(S().mu);
  long long n = 0;  // of everything whose name begins so
  for (const auto& c : S().counts)
    if (c.first.compare(0, std::strlen(what), what) == 0 || c.first.find(what) != std::string::npos) n += c.second;
  return n;
}
size_t fake_used(int dev) {
  std::lock_guard<std::mutex> lk(S().mu);
  return S().used[dev];
}
size_t fake_peak(int dev) {
  std::lock_guard<std::mutex> lk(S().mu);
  return S().peak[dev];
}

// ---- registration and launches ----
void** __cudaRegisterFatBinary(void*) {
  static void* h;
  return &h;
}
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
void __cudaRegisterVar(void**, char*, char*, const char*, int, size_t, int, int) {}
void __cudaRegisterFunction(void**, const char* f, char*, const char* name, int, uint3*, uint3*, dim3*, dim3*, int*) {
  std::lock_guard<std::mutex> lk(S().mu);
  S().names[f] = name;
}
unsigned __cudaPushCallConfiguration(dim3 g, dim3 b, size_t shared, CUstream_st* s) {
  t_grid = g;
  t_block = b;
  t_shared = shared;
  t_stream = s;
  return 0;
}
cudaError_t __cudaPopCallConfiguration(dim3* g, dim3* b, size_t* shared, void* s) {
  *g = t_grid;
  *b = t_block;
  *shared = t_shared;
  *static_cast<cudaStream_t*>(s) = t_stream;
  return cudaSuccess;
}
cudaError_t __cudaGetKernel(cudaKernel_t* k, const void* f) {
  *k = reinterpret_cast<cudaKernel_t>(const_cast<void*>(f));
  return cudaSuccess;
}
cudaError_t __cudaLaunchKernel(cudaKernel_t k, dim3 g, dim3 b, void**, size_t shared, cudaStream_t) {
  return launch(reinterpret_cast<const void*>(k), g, b, shared);
}
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t* c, const void* f, void**) {
  return launch(f, c->gridDim, c->blockDim, c->dynamicSmemBytes);
}
cudaError_t cudaFuncSetAttribute(const void* f, cudaFuncAttribute a, int v) {
  std::lock_guard<std::mutex> lk(S().mu);
  if (v < 0 || size_t(v) > kMostShared) return fail(cudaErrorInvalidValue);
  if (a == cudaFuncAttributeMaxDynamicSharedMemorySize) {
    size_t& limit = S().shared[{f, t_dev}];
    if (size_t(v) < limit) ++S().counts["lowered " + S().names[f]];
    limit = size_t(v);
  }
  return cudaSuccess;
}
cudaError_t cudaOccupancyMaxActiveClusters(int* n, const void*, const cudaLaunchConfig_t*) {
  *n = kSms[t_dev] / 2;
  return cudaSuccess;
}

// ---- devices and errors ----
cudaError_t cudaGetDeviceCount(int* n) {
  *n = kDevices;
  return cudaSuccess;
}
cudaError_t cudaGetDevice(int* d) {
  *d = t_dev;
  return cudaSuccess;
}
cudaError_t cudaSetDevice(int d) {
  if (d < 0 || d >= kDevices) return fail(cudaErrorInvalidDevice);
  t_dev = d;
  return cudaSuccess;
}
cudaError_t cudaGetDeviceProperties(cudaDeviceProp* p, int d) {
  std::memset(p, 0, sizeof *p);
  p->major = 10;
  p->minor = 3;
  p->multiProcessorCount = kSms[d];
  p->sharedMemPerBlockOptin = kMostShared;
  return cudaSuccess;
}
const char* cudaGetErrorString(cudaError_t) { return "error of the stand-in runtime"; }
cudaError_t cudaGetLastError() {
  const cudaError_t e = t_err;
  t_err = cudaSuccess;
  return e;
}

// ---- memory ----
cudaError_t cudaMalloc(void** p, size_t n) {
  State& s = S();
  std::lock_guard<std::mutex> lk(s.mu);
  *p = nullptr;
  if (s.used[t_dev] + n > s.capacity[t_dev]) {
    ++s.counts["cudaMalloc refused"];
    return fail(cudaErrorMemoryAllocation);
  }
  ++s.counts["cudaMalloc done"];
  s.used[t_dev] += n;
  s.peak[t_dev] = s.used[t_dev] > s.peak[t_dev] ? s.used[t_dev] : s.peak[t_dev];
  *p = reinterpret_cast<void*>(s.next);
  s.blocks[s.next] = {n, t_dev};
  s.next += (n + 0x1fffff) & ~size_t(0x1fffff);
  return cudaSuccess;
}
cudaError_t cudaFree(void* p) {
  if (!p) return cudaSuccess;
  State& s = S();
  std::lock_guard<std::mutex> lk(s.mu);
  const auto at = s.blocks.find(reinterpret_cast<uintptr_t>(p));
  if (at == s.blocks.end()) return fail(cudaErrorInvalidValue);
  ++s.counts["cudaFree"];
  s.used[at->second.dev] -= at->second.bytes;
  s.blocks.erase(at);
  return cudaSuccess;
}
cudaError_t cudaMemGetInfo(size_t* free, size_t* total) {
  State& s = S();
  std::lock_guard<std::mutex> lk(s.mu);
  *free = s.capacity[t_dev] - s.used[t_dev];
  *total = s.capacity[t_dev];
  return cudaSuccess;
}
cudaError_t cudaMallocHost(void** p, size_t n) {
  *p = host_alloc(n);
  return cudaSuccess;
}
cudaError_t cudaHostAlloc(void** p, size_t n, unsigned) { return cudaMallocHost(p, n); }
cudaError_t cudaFreeHost(void* p) { return drop(p); }
static bool on_device(const void* p, int* dev) {
  State& s = S();
  std::lock_guard<std::mutex> lk(s.mu);
  auto at = s.blocks.upper_bound(reinterpret_cast<uintptr_t>(p));
  if (at == s.blocks.begin()) return false;
  --at;
  if (reinterpret_cast<uintptr_t>(p) >= at->first + at->second.bytes) return false;
  *dev = at->second.dev;
  return true;
}
cudaError_t cudaPointerGetAttributes(cudaPointerAttributes* a, const void* p) {
  std::memset(a, 0, sizeof *a);
  a->type = on_device(p, &a->device) ? cudaMemoryTypeDevice : cudaMemoryTypeUnregistered;
  return cudaSuccess;
}
cudaError_t cudaMemcpyAsync(void* dst, const void*, size_t n, cudaMemcpyKind, cudaStream_t) {
  int dev;
  if (n <= (1 << 20) && !on_device(dst, &dev)) std::memset(dst, 0, n);
  return cudaSuccess;
}
cudaError_t cudaMemcpy(void* dst, const void* src, size_t n, cudaMemcpyKind k) {
  return cudaMemcpyAsync(dst, src, n, k, nullptr);
}
cudaError_t cudaMemsetAsync(void*, int, size_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaGetSymbolAddress(void** p, const void* s) {
  *p = const_cast<void*>(s);
  return cudaSuccess;
}

// ---- streams, events, graphs ----
cudaError_t cudaStreamCreateWithFlags(cudaStream_t* s, unsigned) { return handle(s); }
cudaError_t cudaStreamDestroy(cudaStream_t s) { return drop(s); }
cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamWaitEvent(cudaStream_t, cudaEvent_t, unsigned) { return cudaSuccess; }
cudaError_t cudaLaunchHostFunc(cudaStream_t, cudaHostFn_t f, void* p) {
  f(p);
  return cudaSuccess;
}
cudaError_t cudaEventCreate(cudaEvent_t* e) { return handle(e); }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t* e, unsigned) { return handle(e); }
cudaError_t cudaEventDestroy(cudaEvent_t e) { return drop(e); }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float* ms, cudaEvent_t, cudaEvent_t) {
  *ms = 1.0f;
  return cudaSuccess;
}
cudaError_t cudaStreamBeginCapture(cudaStream_t, cudaStreamCaptureMode) { return cudaSuccess; }
cudaError_t cudaStreamEndCapture(cudaStream_t, cudaGraph_t* g) { return handle(g); }
cudaError_t cudaGraphInstantiate(cudaGraphExec_t* x, cudaGraph_t, unsigned long long) {
  count("graph captured");
  return handle(x);
}
cudaError_t cudaGraphDestroy(cudaGraph_t g) { return drop(g); }
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t x) { return drop(x); }
cudaError_t cudaGraphLaunch(cudaGraphExec_t, cudaStream_t) {
  count("graph launched");
  return cudaSuccess;
}
cudaError_t cudaGetDriverEntryPointByVersion(const char* name, void** f, unsigned, unsigned long long,
                                             cudaDriverEntryPointQueryResult* q) {
  const bool known = !std::strcmp(name, "cuTensorMapEncodeTiled");
  *f = known ? reinterpret_cast<void*>(&encode) : nullptr;
  if (q) *q = known ? cudaDriverEntryPointSuccess : cudaDriverEntryPointSymbolNotFound;
  return cudaSuccess;
}

}  // extern "C"
