// Host stand-in for the CUDA runtime calls that the library makes, preloaded
// before libcudart to run the library's host code without a GPU: device
// memory is host memory, copies and memsets act at once, kernels do nothing
// but are counted by name.  Calls can be made to fail, and the current device
// can be changed.  Control functions: fake_*.
#include <cuda_runtime_api.h>

#include <cstdlib>
#include <cstring>
#include <map>
#include <mutex>
#include <string>

namespace {
std::recursive_mutex mu;
using Lock = std::lock_guard<std::recursive_mutex>;
template <typename T>
T& never_destroyed() {  // the library frees and unregisters at exit
  static T* t = new T;
  return *t;
}
auto& names() { return never_destroyed<std::map<const void*, std::string>>(); }      // kernel -> name
auto& launches() { return never_destroyed<std::map<std::string, long long>>(); }     // name -> launches
auto& blocks() { return never_destroyed<std::map<void*, size_t>>(); }                // device allocations
auto& smem_devices() { return never_destroyed<std::map<const void*, unsigned>>(); }  // kernel -> opted-in devices
size_t in_use = 0, peak = 0;
long long fail_malloc = -1;  // allocations until the one that fails
int device = 0, missing_opt_in = 0;
struct Config {
  dim3 grid, block;
  size_t smem;
  cudaStream_t stream;
};
thread_local Config config;

void launched(const void* kernel) {
  Lock l(mu);
  ++launches()[names()[kernel]];
  auto it = smem_devices().find(kernel);
  if (it != smem_devices().end() && !(it->second >> device & 1)) ++missing_opt_in;
}
template <typename T>
T handle() {
  return reinterpret_cast<T>(std::malloc(16));
}
}  // namespace

extern "C" {

void fake_fail_malloc(long long nth) { fail_malloc = nth; }
size_t fake_peak(int reset) {
  const size_t p = peak;
  if (reset) peak = in_use;
  return p;
}
size_t fake_in_use() { return in_use; }
void fake_set_device(int d) { device = d; }
int fake_missing_opt_in() { return missing_opt_in; }  // launches without the device's shared-memory limit raised
long long fake_launches(const char* part) {
  Lock l(mu);
  long long n = 0;
  for (auto& e : launches())
    if (e.first.find(part) != std::string::npos) n += e.second;
  return n;
}

void** __cudaRegisterFatBinary(void*) { return handle<void**>(); }
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
void __cudaRegisterVar(void**, char*, char*, const char*, int, size_t, int, int) {}
void __cudaRegisterFunction(void**, const char* host, char*, const char* name, int, uint3*, uint3*, dim3*, dim3*, int*) {
  Lock l(mu);
  names()[host] = name;
}
unsigned __cudaPushCallConfiguration(dim3 g, dim3 b, size_t s, cudaStream_t st) {
  config = {g, b, s, st};
  return 0;
}
cudaError_t __cudaPopCallConfiguration(dim3* g, dim3* b, size_t* s, void* st) {
  *g = config.grid;
  *b = config.block;
  *s = config.smem;
  *static_cast<cudaStream_t*>(st) = config.stream;
  return cudaSuccess;
}
cudaError_t __cudaGetKernel(cudaKernel_t* k, const void* host) {
  *k = reinterpret_cast<cudaKernel_t>(const_cast<void*>(host));
  return cudaSuccess;
}
cudaError_t __cudaLaunchKernel(cudaKernel_t k, dim3, dim3, void**, size_t, cudaStream_t) {
  launched(reinterpret_cast<const void*>(k));
  return cudaSuccess;
}
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t*, const void* f, void**) {
  launched(f);
  return cudaSuccess;
}
cudaError_t cudaFuncSetAttribute(const void* f, cudaFuncAttribute a, int) {
  Lock l(mu);
  if (a == cudaFuncAttributeMaxDynamicSharedMemorySize) smem_devices()[f] |= 1u << device;
  return cudaSuccess;
}
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int* n, const void*, int, size_t, unsigned) {
  *n = 2;
  return cudaSuccess;
}

cudaError_t cudaGetDevice(int* d) {
  *d = device;
  return cudaSuccess;
}
cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr, int) {
  *v = 152;
  return cudaSuccess;
}
cudaError_t cudaDeviceGetDefaultMemPool(cudaMemPool_t* p, int) {
  *p = nullptr;
  return cudaSuccess;
}
cudaError_t cudaMemPoolSetAttribute(cudaMemPool_t, cudaMemPoolAttr, void*) { return cudaSuccess; }
cudaError_t cudaGetLastError() { return cudaSuccess; }
const char* cudaGetErrorString(cudaError_t) { return "stand-in error"; }
cudaError_t cudaGetSymbolAddress(void** p, const void* symbol) {
  *p = const_cast<void*>(symbol);
  return cudaSuccess;
}

cudaError_t cudaMallocAsync(void** p, size_t n, cudaStream_t) {
  Lock l(mu);
  if (fail_malloc >= 0 && fail_malloc-- == 0) return cudaErrorMemoryAllocation;
  *p = std::calloc(1, n);
  blocks()[*p] = n;
  in_use += n;
  if (in_use > peak) peak = in_use;
  return cudaSuccess;
}
cudaError_t cudaFreeAsync(void* p, cudaStream_t) {
  Lock l(mu);
  auto it = blocks().find(p);
  if (it == blocks().end()) return cudaErrorInvalidValue;
  in_use -= it->second;
  blocks().erase(it);
  std::free(p);
  return cudaSuccess;
}
cudaError_t cudaHostAlloc(void** p, size_t n, unsigned) {
  *p = std::calloc(1, n);
  return cudaSuccess;
}
cudaError_t cudaFreeHost(void* p) {
  std::free(p);
  return cudaSuccess;
}
cudaError_t cudaHostGetDevicePointer(void** d, void* h, unsigned) {
  *d = h;
  return cudaSuccess;
}
cudaError_t cudaMemcpyAsync(void* d, const void* s, size_t n, cudaMemcpyKind, cudaStream_t) {
  std::memmove(d, s, n);
  return cudaSuccess;
}
cudaError_t cudaMemsetAsync(void* d, int v, size_t n, cudaStream_t) {
  std::memset(d, v, n);
  return cudaSuccess;
}

cudaError_t cudaStreamCreateWithFlags(cudaStream_t* s, unsigned) {
  *s = handle<cudaStream_t>();
  return cudaSuccess;
}
cudaError_t cudaStreamDestroy(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamWaitEvent(cudaStream_t, cudaEvent_t, unsigned) { return cudaSuccess; }
cudaError_t cudaStreamBeginCapture(cudaStream_t, cudaStreamCaptureMode) { return cudaSuccess; }
cudaError_t cudaStreamEndCapture(cudaStream_t, cudaGraph_t* g) {
  *g = handle<cudaGraph_t>();
  return cudaSuccess;
}
cudaError_t cudaGraphInstantiate(cudaGraphExec_t* e, cudaGraph_t, unsigned long long) {
  *e = handle<cudaGraphExec_t>();
  return cudaSuccess;
}
cudaError_t cudaGraphLaunch(cudaGraphExec_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaGraphDestroy(cudaGraph_t) { return cudaSuccess; }
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t) { return cudaSuccess; }
cudaError_t cudaEventCreate(cudaEvent_t* e) {
  *e = handle<cudaEvent_t>();
  return cudaSuccess;
}
cudaError_t cudaEventCreateWithFlags(cudaEvent_t* e, unsigned) { return cudaEventCreate(e); }
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventSynchronize(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float* ms, cudaEvent_t, cudaEvent_t) {
  *ms = 1.f;
  return cudaSuccess;
}

}  // extern "C"
