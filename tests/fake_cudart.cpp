// A CUDA runtime without a GPU, for tests of what the library's host code
// launches: two devices, memory from malloc, launches recorded and not run.  A
// kernel's dynamic shared-memory limit belongs to a device, as in the real
// runtime: 48 KB until cudaFuncSetAttribute raises it there, and a launch beyond
// it is refused.
#include <cuda_runtime_api.h>

#include <cstdlib>
#include <cstring>
#include <map>
#include <mutex>
#include <string>
#include <vector>

namespace {
struct Launch {
  std::string name;
  unsigned grid;
  size_t dyn;
  int device;
};
struct Config {
  dim3 grid, block;
  size_t dyn;
  cudaStream_t stream;
};
std::mutex mu;
std::map<const void*, std::string> names;
std::map<std::pair<const void*, int>, size_t> limits;
std::vector<Launch> launches;
thread_local int device = 0;
thread_local std::vector<Config> configs;
thread_local cudaError_t last = cudaSuccess;
bool refuse = false;  // cudaFuncSetAttribute fails

cudaError_t set(cudaError_t e) {
  if (e != cudaSuccess) last = e;
  return e;
}

cudaError_t launch(const void* f, dim3 grid, dim3 block, size_t dyn) {
  std::lock_guard<std::mutex> lock(mu);
  const auto it = limits.find({f, device});
  const size_t limit = it == limits.end() ? (size_t)48 << 10 : it->second;
  // (a limit raised on one device only is taken for a mistake at any size: the
  // kernel's static shared memory, unknown here, counts towards the 48 KB)
  bool elsewhere = false;
  for (int d = 0; d < 2; ++d) elsewhere |= limits.count({f, d}) > 0;
  if (dyn > limit || (dyn > 0 && elsewhere && it == limits.end()) || grid.x == 0 || block.x == 0)
    return set(cudaErrorInvalidValue);
  launches.push_back({names[f], grid.x, dyn, device});
  return cudaSuccess;
}
}  // namespace

extern "C" {
// ------------------------------------------------------------ for the tests --
void fake_reset() {
  std::lock_guard<std::mutex> lock(mu);
  launches.clear();
}
void fake_refuse_limits(int on) { refuse = on != 0; }
long fake_count(const char* part) {
  std::lock_guard<std::mutex> lock(mu);
  long n = 0;
  for (const Launch& l : launches) n += l.name.find(part) != std::string::npos;
  return n;
}
unsigned long fake_max_dyn(const char* part) {
  std::lock_guard<std::mutex> lock(mu);
  size_t n = 0;
  for (const Launch& l : launches)
    if (l.name.find(part) != std::string::npos && l.dyn > n) n = l.dyn;
  return n;
}

// ------------------------------------------------------------- registration --
void** __cudaRegisterFatBinary(void*) { return new void*[1]; }
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void** p) { delete[] p; }
void __cudaRegisterFunction(void**, const char* host, char*, const char* name, int, uint3*, uint3*,
                            dim3*, dim3*, int*) {
  names[host] = name;
}
void __cudaRegisterVar(void**, char*, char*, const char*, int, size_t, int, int) {}

// ------------------------------------------------------------------ launches --
unsigned __cudaPushCallConfiguration(dim3 grid, dim3 block, size_t dyn, cudaStream_t stream) {
  configs.push_back({grid, block, dyn, stream});
  return 0;
}
cudaError_t __cudaPopCallConfiguration(dim3* grid, dim3* block, size_t* dyn, void* stream) {
  const Config c = configs.back();
  configs.pop_back();
  *grid = c.grid;
  *block = c.block;
  *dyn = c.dyn;
  *(cudaStream_t*)stream = c.stream;
  return cudaSuccess;
}
cudaError_t __cudaGetKernel(cudaKernel_t* k, const void* f) {
  *k = (cudaKernel_t)f;
  return cudaSuccess;
}
cudaError_t __cudaLaunchKernel(cudaKernel_t k, dim3 grid, dim3 block, void**, size_t dyn,
                               cudaStream_t) {
  return launch((const void*)k, grid, block, dyn);
}
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t* c, const void* f, void**) {
  return launch(f, c->gridDim, c->blockDim, c->dynamicSmemBytes);
}
cudaError_t cudaFuncSetAttribute(const void* f, cudaFuncAttribute a, int v) {
  if (refuse || a != cudaFuncAttributeMaxDynamicSharedMemorySize || v < 0 || v > (227 << 10))
    return set(cudaErrorInvalidValue);
  std::lock_guard<std::mutex> lock(mu);
  limits[{f, device}] = v;
  return cudaSuccess;
}
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int* n, const void*, int, size_t,
                                                                   unsigned) {
  *n = 2;
  return cudaSuccess;
}

// ------------------------------------------------------- devices and memory --
cudaError_t cudaGetDevice(int* d) {
  *d = device;
  return cudaSuccess;
}
cudaError_t cudaSetDevice(int d) {
  device = d;
  return cudaSuccess;
}
cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr a, int) {
  *v = a == cudaDevAttrMultiProcessorCount ? 152 : 0;
  return cudaSuccess;
}
cudaError_t cudaGetLastError() {
  const cudaError_t e = last;
  last = cudaSuccess;
  return e;
}
const char* cudaGetErrorString(cudaError_t e) { return e == cudaSuccess ? "no error" : "refused"; }
cudaError_t cudaMalloc(void** p, size_t n) {
  *p = aligned_alloc(256, (n + 255) / 256 * 256);
  return *p ? cudaSuccess : set(cudaErrorMemoryAllocation);
}
cudaError_t cudaFree(void* p) {
  free(p);
  return cudaSuccess;
}
cudaError_t cudaHostAlloc(void** p, size_t n, unsigned) { return cudaMalloc(p, n); }
cudaError_t cudaFreeHost(void* p) { return cudaFree(p); }
cudaError_t cudaMemcpy(void* d, const void* s, size_t n, cudaMemcpyKind) {
  memcpy(d, s, n);
  return cudaSuccess;
}
cudaError_t cudaMemcpyAsync(void* d, const void* s, size_t n, cudaMemcpyKind, cudaStream_t) {
  memcpy(d, s, n);
  return cudaSuccess;
}
cudaError_t cudaGetSymbolAddress(void** p, const void*) { return cudaMalloc(p, 256); }

// (streams, events and graphs: not used by the calls under test)
cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamCreateWithFlags(cudaStream_t*, unsigned) { return cudaErrorNotSupported; }
cudaError_t cudaStreamDestroy(cudaStream_t) { return cudaErrorNotSupported; }
cudaError_t cudaStreamWaitEvent(cudaStream_t, cudaEvent_t, unsigned) { return cudaErrorNotSupported; }
cudaError_t cudaStreamBeginCapture(cudaStream_t, cudaStreamCaptureMode) {
  return cudaErrorNotSupported;
}
cudaError_t cudaStreamEndCapture(cudaStream_t, cudaGraph_t*) { return cudaErrorNotSupported; }
cudaError_t cudaEventCreate(cudaEvent_t*) { return cudaErrorNotSupported; }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t*, unsigned) { return cudaErrorNotSupported; }
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaErrorNotSupported; }
cudaError_t cudaEventElapsedTime(float*, cudaEvent_t, cudaEvent_t) { return cudaErrorNotSupported; }
cudaError_t cudaEventQuery(cudaEvent_t) { return cudaErrorNotSupported; }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaErrorNotSupported; }
cudaError_t cudaEventSynchronize(cudaEvent_t) { return cudaErrorNotSupported; }
cudaError_t cudaGraphDestroy(cudaGraph_t) { return cudaErrorNotSupported; }
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t) { return cudaErrorNotSupported; }
cudaError_t cudaGraphInstantiate(cudaGraphExec_t*, cudaGraph_t, unsigned long long) {
  return cudaErrorNotSupported;
}
cudaError_t cudaGraphLaunch(cudaGraphExec_t, cudaStream_t) { return cudaErrorNotSupported; }
}
