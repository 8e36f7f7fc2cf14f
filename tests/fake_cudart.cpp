// A CUDA runtime of two devices that runs nothing: the library's host objects are
// linked with it, so that what the host code asks of each device can be checked
// without a GPU. Allocations are addresses without memory; a launch fails, as on
// a device, where its shared memory exceeds what its function may have there.
#include <cuda_runtime_api.h>

#include <cstdint>
#include <map>
#include <string>
#include <utility>
#include <vector>

namespace {
constexpr int kDevices = 2;
constexpr int kStatic = 4096, kDefault = 48 * 1024, kOptin = 227 * 1024;
int current = 0;
cudaError_t last = cudaSuccess;
uintptr_t next_address = 0x7000000000ull;
long long allocated = 0;
std::map<std::pair<int, const void*>, int> dynamic_limit;   // (device, function)
std::map<const void*, std::string> names;
struct Launch {
  int device;
  std::string name;
  size_t smem;
  unsigned grid;
};
std::vector<Launch> launches;
struct Config {
  dim3 grid, block;
  size_t smem;
  cudaStream_t stream;
} pushed;

int limit_of(const void* f) {
  auto it = dynamic_limit.find({current, f});
  return it == dynamic_limit.end() ? kDefault - kStatic : it->second;
}
cudaError_t set(cudaError_t e) {
  if (e != cudaSuccess) last = e;
  return e;
}
cudaError_t launch(const void* f, dim3 grid, size_t smem) {
  if (grid.x < 1 || (long long)smem > limit_of(f)) return set(cudaErrorInvalidValue);
  launches.push_back({current, names[f], smem, grid.x});
  return cudaSuccess;
}
}  // namespace

extern "C" {
// what a test reads
long long fake_allocated() { return allocated; }
int fake_launches(int device, const char* part) {
  int n = 0;
  for (const Launch& l : launches) n += l.device == device && l.name.find(part) != std::string::npos;
  return n;
}

void** __cudaRegisterFatBinary(void*) {
  static void* handle;
  return &handle;
}
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
void __cudaRegisterFunction(void**, const char* host, char*, const char* name, int, uint3*, uint3*, dim3*,
                            dim3*, int*) {
  names[host] = name;
}
void __cudaRegisterVar(void**, char*, char*, const char*, int, size_t, int, int) {}
cudaError_t __cudaGetKernel(cudaKernel_t* k, const void* f) {
  *k = (cudaKernel_t)f;
  return cudaSuccess;
}
unsigned __cudaPushCallConfiguration(dim3 grid, dim3 block, size_t smem, cudaStream_t stream) {
  pushed = {grid, block, smem, stream};
  return 0;
}
cudaError_t __cudaPopCallConfiguration(dim3* grid, dim3* block, size_t* smem, void* stream) {
  *grid = pushed.grid;
  *block = pushed.block;
  *smem = pushed.smem;
  *(cudaStream_t*)stream = pushed.stream;
  return cudaSuccess;
}
cudaError_t __cudaLaunchKernel(cudaKernel_t k, dim3 grid, dim3, void**, size_t smem, cudaStream_t) {
  return launch((const void*)k, grid, smem);
}
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t* c, const void* f, void**) {
  return launch(f, c->gridDim, c->dynamicSmemBytes);
}

cudaError_t cudaGetDevice(int* d) {
  *d = current;
  return cudaSuccess;
}
cudaError_t cudaSetDevice(int d) {
  if (d < 0 || d >= kDevices) return set(cudaErrorInvalidDevice);
  current = d;
  return cudaSuccess;
}
cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr a, int) {
  *v = a == cudaDevAttrMultiProcessorCount ? 152 : a == cudaDevAttrMaxSharedMemoryPerBlockOptin ? kOptin : 0;
  return cudaSuccess;
}
cudaError_t cudaFuncGetAttributes(cudaFuncAttributes* a, const void*) {
  *a = cudaFuncAttributes();
  a->sharedSizeBytes = kStatic;
  return cudaSuccess;
}
cudaError_t cudaFuncSetAttribute(const void* f, cudaFuncAttribute a, int v) {
  if (a == cudaFuncAttributeMaxDynamicSharedMemorySize) {
    if (v > kOptin - kStatic) return set(cudaErrorInvalidValue);
    dynamic_limit[{current, f}] = v;
  }
  return cudaSuccess;
}
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int* n, const void* f, int, size_t smem,
                                                                   unsigned) {
  *n = (long long)smem > limit_of(f) ? 0 : 2;
  return cudaSuccess;
}
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessor(int* n, const void* f, int threads, size_t smem) {
  return cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(n, f, threads, smem, 0);
}
cudaError_t cudaMalloc(void** p, size_t bytes) {
  *p = (void*)next_address;
  next_address += (bytes + 511) / 512 * 512;
  allocated += (long long)bytes;
  return cudaSuccess;
}
cudaError_t cudaFree(void*) { return cudaSuccess; }
cudaError_t cudaMemset(void*, int, size_t) { return cudaSuccess; }
cudaError_t cudaMemsetAsync(void*, int, size_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaMemcpy(void*, const void*, size_t, cudaMemcpyKind) { return cudaSuccess; }
cudaError_t cudaMemcpyAsync(void*, const void*, size_t, cudaMemcpyKind, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaGetSymbolAddress(void** p, const void*) {
  *p = (void*)next_address;
  return cudaSuccess;
}
cudaError_t cudaDeviceSynchronize() { return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamIsCapturing(cudaStream_t, cudaStreamCaptureStatus* s) {
  *s = cudaStreamCaptureStatusNone;
  return cudaSuccess;
}
cudaError_t cudaEventCreate(cudaEvent_t* e) {
  *e = (cudaEvent_t)next_address++;
  return cudaSuccess;
}
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventRecordWithFlags(cudaEvent_t, cudaStream_t, unsigned) { return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float* ms, cudaEvent_t, cudaEvent_t) {
  *ms = 0.f;
  return cudaSuccess;
}
cudaError_t cudaGetLastError() {
  cudaError_t e = last;
  last = cudaSuccess;
  return e;
}
const char* cudaGetErrorString(cudaError_t e) { return e == cudaSuccess ? "success" : "error"; }
}
