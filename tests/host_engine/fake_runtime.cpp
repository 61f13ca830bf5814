// A stand-in for the CUDA runtime, to run the host engine (capi.cu) on a CPU: device
// memory is host memory, and an event's time is the sum of the costs that a test set
// for the launches before it.  fake_launchers.cu stands in for the kernels.
#include <cstdint>
#include <cstring>
#include <map>
#include <mutex>
#include <string>

#include <cuda_runtime.h>
#include <sys/mman.h>

namespace {
std::mutex mu, text_mu;
std::string text;
struct Block { size_t bytes; int type, device; };  // type: a cudaMemoryType
std::map<uintptr_t, Block> blocks;
std::map<std::string, int> failing;  // launcher -> error code
std::map<int, double> cost;          // cells per warp -> ms of a fused launch
double now_ms = 0.0;
std::map<uintptr_t, double> event_ms;
uintptr_t next_handle = 16;

void say(const std::string& line) {
  std::lock_guard<std::mutex> lk(text_mu);
  text += line + "\n";
}
std::string num(const char* key, long long v) { return std::string(" ") + key + "=" + std::to_string(v); }

const std::pair<const uintptr_t, Block>* block_of(const void* p) {
  auto it = blocks.upper_bound((uintptr_t)p);
  if (it == blocks.begin()) return nullptr;
  --it;
  return (uintptr_t)p < it->first + it->second.bytes ? &*it : nullptr;
}
int address_range(unsigned long long* base, size_t* size, unsigned long long p) {
  std::lock_guard<std::mutex> lk(mu);
  const auto* b = block_of((const void*)(uintptr_t)p);
  if (!b) return 1;
  *base = b->first;
  *size = b->second.bytes;
  return 0;
}
cudaError_t give(void** p, size_t bytes, int type = cudaMemoryTypeDevice, int device = 0) {
  std::lock_guard<std::mutex> lk(mu);
  const size_t whole = (bytes + 4095) / 4096 * 4096;
  *p = mmap(nullptr, whole ? whole : 4096, PROT_READ | PROT_WRITE, MAP_PRIVATE | MAP_ANONYMOUS | MAP_NORESERVE, -1, 0);
  if (*p == MAP_FAILED) return cudaErrorMemoryAllocation;
  blocks[(uintptr_t)*p] = Block{bytes ? bytes : 1, type, device};
  return cudaSuccess;
}
cudaError_t take(void* p) {
  std::lock_guard<std::mutex> lk(mu);
  auto it = blocks.find((uintptr_t)p);
  if (it == blocks.end()) return cudaErrorInvalidValue;
  munmap(p, (it->second.bytes + 4095) / 4096 * 4096);
  blocks.erase(it);
  return cudaSuccess;
}
}  // namespace

extern "C" {
// ---- for the launchers: a line of the log, what a test wants of a launcher, time ----
void fake_say(const char* line) { say(line); }
int fake_failure(const char* who) { return failing.count(who) ? failing[who] : 0; }
void fake_spend(int cpw) { now_ms += cost.count(cpw) ? cost[cpw] : 1.0; }

// ---- what a test sets and reads ----
const char* fake_log() {
  static std::string out;
  out.swap(text);
  text.clear();
  return out.c_str();
}
void* fake_alloc(size_t bytes, int type, int device) {
  void* p = nullptr;
  give(&p, bytes, type, device);
  return p;
}
void fake_fail(const char* launcher, int code) { failing[launcher] = code; }
void fake_cost(int cpw, double ms) { cost[cpw] = ms; }

// ---- the runtime ----
cudaError_t cudaGetDevice(int* d) { *d = 0; return cudaSuccess; }
cudaError_t cudaSetDevice(int) { return cudaSuccess; }
cudaError_t cudaGetDeviceCount(int* n) { *n = 1; return cudaSuccess; }
cudaError_t cudaGetDeviceProperties(cudaDeviceProp* p, int) {
  std::memset(p, 0, sizeof(*p));
  p->multiProcessorCount = 152;
  return cudaSuccess;
}
cudaError_t cudaMalloc(void** p, size_t n) { return give(p, n); }
cudaError_t cudaMallocAsync(void** p, size_t n, cudaStream_t) { return give(p, n); }
cudaError_t cudaMallocHost(void** p, size_t n) { return give(p, n, cudaMemoryTypeHost); }
cudaError_t cudaFree(void* p) { return take(p); }
cudaError_t cudaFreeAsync(void* p, cudaStream_t) { return take(p); }
cudaError_t cudaMemsetAsync(void* p, int v, size_t n, cudaStream_t) { std::memset(p, v, n); return cudaSuccess; }
cudaError_t cudaMemcpyAsync(void* d, const void* s, size_t n, cudaMemcpyKind kind, cudaStream_t) {
  if (kind == cudaMemcpyDeviceToDevice) {  // the driver's check of both ends
    std::lock_guard<std::mutex> lk(mu);
    for (const void* p : {(const void*)d, s}) {
      const auto* b = block_of(p);
      if (!b || (uintptr_t)p + n > b->first + b->second.bytes) return cudaErrorInvalidValue;
    }
    say("copy" + num("bytes", n));
  } else if (kind == cudaMemcpyDeviceToHost) {
    std::lock_guard<std::mutex> lk(mu);
    say("read" + num("bytes", n));
  }
  std::memcpy(d, s, n);
  return cudaSuccess;
}
cudaError_t cudaPointerGetAttributes(cudaPointerAttributes* a, const void* p) {
  std::lock_guard<std::mutex> lk(mu);
  const auto* b = block_of(p);
  std::memset(a, 0, sizeof(*a));
  a->type = b ? (cudaMemoryType)b->second.type : cudaMemoryTypeUnregistered;
  a->device = b ? b->second.device : -2;
  return cudaSuccess;
}
cudaError_t cudaGetDriverEntryPointByVersion(const char*, void** f, unsigned, unsigned long long,
                                             cudaDriverEntryPointQueryResult* q) {
  *f = (void*)address_range;
  if (q) *q = cudaDriverEntryPointSuccess;
  return cudaSuccess;
}
cudaError_t cudaStreamCreateWithFlags(cudaStream_t* s, unsigned) { *s = (cudaStream_t)next_handle++; return cudaSuccess; }
cudaError_t cudaStreamDestroy(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t) { say("wait"); return cudaSuccess; }
cudaError_t cudaStreamWaitEvent(cudaStream_t, cudaEvent_t, unsigned) { return cudaSuccess; }
cudaError_t cudaStreamBeginCapture(cudaStream_t, cudaStreamCaptureMode) { say("capture"); return cudaSuccess; }
cudaError_t cudaStreamEndCapture(cudaStream_t, cudaGraph_t* g) { *g = (cudaGraph_t)next_handle++; say("end"); return cudaSuccess; }
cudaError_t cudaGraphInstantiate(cudaGraphExec_t* e, cudaGraph_t, unsigned long long) { *e = (cudaGraphExec_t)next_handle++; return cudaSuccess; }
cudaError_t cudaGraphDestroy(cudaGraph_t) { return cudaSuccess; }
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t) { return cudaSuccess; }
cudaError_t cudaGraphLaunch(cudaGraphExec_t, cudaStream_t) { say("graph"); return cudaSuccess; }
cudaError_t cudaEventCreate(cudaEvent_t* e) { *e = (cudaEvent_t)next_handle++; return cudaSuccess; }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t* e, unsigned) { return cudaEventCreate(e); }
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t e, cudaStream_t) { event_ms[(uintptr_t)e] = now_ms; return cudaSuccess; }
cudaError_t cudaEventSynchronize(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float* ms, cudaEvent_t a, cudaEvent_t b) {
  *ms = (float)(event_ms[(uintptr_t)b] - event_ms[(uintptr_t)a]);
  return cudaSuccess;
}
cudaError_t cudaGetLastError() { return cudaSuccess; }
cudaError_t cudaPeekAtLastError() { return cudaSuccess; }
const char* cudaGetErrorString(cudaError_t e) { return e == cudaSuccess ? "no error" : "an error"; }
cudaError_t cudaGetSymbolAddress(void**, const void*) { return cudaErrorInvalidSymbol; }
cudaError_t cudaDeviceGetDefaultMemPool(cudaMemPool_t*, int) { return cudaErrorNotSupported; }
cudaError_t cudaMemPoolSetAttribute(cudaMemPool_t, cudaMemPoolAttr, void*) { return cudaSuccess; }
// what a compiled .cu file of host code asks for when it is loaded
void** __cudaRegisterFatBinary(void*) { static void* h; return &h; }
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
void __cudaRegisterFunction(void**, const char*, char*, const char*, int, uint3*, uint3*, dim3*, dim3*, int*) {}
void __cudaRegisterVar(void**, char*, char*, const char*, int, size_t, int, int) {}
cudaError_t __cudaGetKernel(void** k, const void* f) { *k = const_cast<void*>(f); return cudaSuccess; }
cudaError_t __cudaLaunchKernel(void*, dim3, dim3, void**, size_t, cudaStream_t) { return cudaSuccess; }
cudaError_t __cudaPopCallConfiguration(dim3*, dim3*, size_t*, void*) { return cudaSuccess; }
unsigned __cudaPushCallConfiguration(dim3, dim3, size_t, CUstream_st*) { return 0; }
}
