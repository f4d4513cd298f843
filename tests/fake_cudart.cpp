// A stand-in for the CUDA runtime, for tests of the library's host side without
// a GPU: device memory is host memory, kernels are recorded and not run, and
// work on the device counts as pending until the host waits for it.  Linked with
// the library's own objects in place of the runtime.
#include <cuda_runtime_api.h>

#include <cstdint>
#include <cstdlib>
#include <cstring>
#include <map>
#include <string>
#include <vector>

namespace {
std::map<const void*, std::string>& names() {
  static std::map<const void*, std::string> n;
  return n;
}
struct Launch {
  std::string kernel;
  dim3 grid, block;
};
std::vector<Launch> launched;  // in order since fake_reset()
std::map<void*, int> pending;          // by stream; nullptr: the default one, which the others do not wait for
struct Config {
  dim3 grid, block;
  size_t smem;
  void* stream;
} config;
}  // namespace

extern "C" {
void fake_reset() {
  launched.clear();
  pending.clear();
}
// Launches, copies and fills that no host wait has covered yet.
int fake_pending() {
  int n = 0;
  for (auto& p : pending) n += p.second;
  return n;
}
int fake_launches() { return int(launched.size()); }
const char* fake_kernel(int i) { return launched[i].kernel.c_str(); }
int fake_grid_x(int i) { return int(launched[i].grid.x); }
int fake_grid_y(int i) { return int(launched[i].grid.y); }
int fake_threads(int i) { return int(launched[i].block.x); }

void** __cudaRegisterFatBinary(void*) {
  static void* handle;
  return &handle;
}
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
void __cudaRegisterVar(void**, char*, char*, const char*, int, size_t, int, int) {}
void __cudaRegisterFunction(void**, const char* host, char*, const char* name, int, uint3*, uint3*, dim3*, dim3*, int*) {
  names()[host] = name;
}
cudaError_t __cudaGetKernel(cudaKernel_t* k, const void* f) {
  *k = reinterpret_cast<cudaKernel_t>(const_cast<void*>(f));
  return cudaSuccess;
}
unsigned __cudaPushCallConfiguration(dim3 grid, dim3 block, size_t smem, void* stream) {
  config = {grid, block, smem, stream};
  return 0;
}
cudaError_t __cudaPopCallConfiguration(dim3* grid, dim3* block, size_t* smem, void* stream) {
  *grid = config.grid;
  *block = config.block;
  *smem = config.smem;
  *static_cast<void**>(stream) = config.stream;
  return cudaSuccess;
}
cudaError_t __cudaLaunchKernel(cudaKernel_t k, dim3 grid, dim3 block, void**, size_t smem, cudaStream_t s) {
  if (grid.x == 0 || grid.y == 0 || grid.y > 65535 || block.x == 0 || block.x > 1024 || smem > 227 * 1024)
    return cudaErrorInvalidConfiguration;
  launched.push_back({names()[reinterpret_cast<const void*>(k)], grid, block});
  ++pending[s];
  return cudaSuccess;
}

cudaError_t cudaDeviceSynchronize() {
  pending.clear();
  return cudaSuccess;
}
cudaError_t cudaMalloc(void** p, size_t n) {
  *p = aligned_alloc(256, (n + 255) & ~size_t(255));
  return *p ? cudaSuccess : cudaErrorMemoryAllocation;
}
cudaError_t cudaFree(void* p) {
  free(p);
  return cudaSuccess;
}
// A copy to the device from pageable memory, or a fill, may still be under way
// on the default stream when the call returns.
cudaError_t cudaMemcpy(void* d, const void* s, size_t n, cudaMemcpyKind kind) {
  memcpy(d, s, n);
  if (kind == cudaMemcpyHostToDevice) ++pending[nullptr];
  return cudaSuccess;
}
cudaError_t cudaMemcpyAsync(void* d, const void* s, size_t n, cudaMemcpyKind, cudaStream_t stream) {
  memcpy(d, s, n);
  ++pending[stream];
  return cudaSuccess;
}
cudaError_t cudaMemset(void*, int, size_t) {
  ++pending[nullptr];
  return cudaSuccess;
}
cudaError_t cudaMemsetAsync(void*, int, size_t, cudaStream_t s) {
  ++pending[s];
  return cudaSuccess;
}
cudaError_t cudaGetDevice(int* d) {
  *d = 0;
  return cudaSuccess;
}
cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr, int) {
  *v = 152;
  return cudaSuccess;
}
cudaError_t cudaGetLastError() { return cudaSuccess; }
cudaError_t cudaFuncSetAttribute(const void*, cudaFuncAttribute, int) { return cudaSuccess; }
cudaError_t cudaGetSymbolAddress(void** p, const void*) {
  *p = nullptr;
  return cudaErrorInvalidSymbol;
}
cudaError_t cudaEventCreate(cudaEvent_t* e) {
  *e = reinterpret_cast<cudaEvent_t>(8);
  return cudaSuccess;
}
cudaError_t cudaEventCreateWithFlags(cudaEvent_t* e, unsigned) { return cudaEventCreate(e); }
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventSynchronize(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float* t, cudaEvent_t, cudaEvent_t) {
  *t = 1.0f;
  return cudaSuccess;
}
cudaError_t cudaStreamCreateWithFlags(cudaStream_t* s, unsigned) {
  *s = reinterpret_cast<cudaStream_t>(8);
  return cudaSuccess;
}
cudaError_t cudaStreamDestroy(cudaStream_t) { return cudaSuccess; }
// A batch's streams are joined to the one that is waited for; none of them waits
// for the default stream.
cudaError_t cudaStreamSynchronize(cudaStream_t s) {
  const int by_default = pending[nullptr];
  if (!s) {
    pending.erase(nullptr);
  } else {
    pending.clear();
    pending[nullptr] = by_default;
  }
  return cudaSuccess;
}
cudaError_t cudaStreamWaitEvent(cudaStream_t, cudaEvent_t, unsigned) { return cudaSuccess; }
cudaError_t cudaStreamBeginCapture(cudaStream_t, cudaStreamCaptureMode) { return cudaSuccess; }
cudaError_t cudaStreamEndCapture(cudaStream_t, cudaGraph_t* g) {
  *g = reinterpret_cast<cudaGraph_t>(8);
  return cudaSuccess;
}
cudaError_t cudaGraphInstantiate(cudaGraphExec_t* e, cudaGraph_t, unsigned long long) {
  *e = reinterpret_cast<cudaGraphExec_t>(8);
  return cudaSuccess;
}
cudaError_t cudaGraphLaunch(cudaGraphExec_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaGraphDestroy(cudaGraph_t) { return cudaSuccess; }
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t) { return cudaSuccess; }
}
