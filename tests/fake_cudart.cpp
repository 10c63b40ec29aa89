// A stand-in for the CUDA runtime, on the host: the library's objects linked against it run every route's host code
// without a GPU.  Launches are checked against the limits that the runtime checks (grid, dynamic shared memory
// against the attribute of the current device) and recorded; nothing runs on a device.
#include <algorithm>
#include <cstdio>
#include <cstring>
#include <map>
#include <string>
#include <vector>

#include <cuda_runtime_api.h>

namespace {
struct Launch {
  std::string kernel;
  dim3 grid, block;
  size_t smem;
  int coop, device;
};
struct Config {
  dim3 grid, block;
  size_t smem;
  cudaStream_t st;
};
// (the objects register their kernels before this file's own objects are constructed)
std::map<const void*, std::string>& names() {
  static std::map<const void*, std::string> m;
  return m;
}
std::map<std::pair<const void*, int>, size_t> smem_limit;  // by kernel and device
std::vector<Launch> log_;
std::vector<Config> pushed;
int device = 0, devices = 2, refuse_coop = 0;
cudaError_t last = cudaSuccess;

cudaError_t fail(cudaError_t e) { return last = e; }

cudaError_t launch(const void* f, dim3 g, dim3 b, size_t smem, int coop) {
  const unsigned long long threads = (unsigned long long)b.x * b.y * b.z;
  if (!g.x || !g.y || !g.z || g.x > 0x7fffffffu || g.y > 65535 || g.z > 65535 || !threads || threads > 1024)
    return fail(cudaErrorInvalidConfiguration);
  const auto it = smem_limit.find({f, device});
  if (smem > (it == smem_limit.end() ? size_t(48 * 1024) : it->second)) return fail(cudaErrorInvalidValue);
  if (coop && refuse_coop) return fail(cudaError_t(refuse_coop));
  log_.push_back({names()[f], g, b, smem, coop, device});
  return cudaSuccess;
}
}  // namespace

extern "C" {

// ---- what a test reads and sets ----
int fake_count() { return int(log_.size()); }
const char* fake_launch(int i) {
  static std::string s;
  const Launch& l = log_[size_t(i)];
  char t[160];
  std::snprintf(t, sizeof t, " %u %u %u %u %zu %d %d", l.grid.x, l.grid.y, l.grid.z, l.block.x * l.block.y * l.block.z, l.smem, l.coop,
                l.device);
  s = l.kernel + t;
  return s.c_str();
}
void fake_reset() {
  log_.clear();
  last = cudaSuccess;
}
void fake_refuse_cooperative(int error) { refuse_coop = error; }

// ---- what the objects call ----
void** __cudaRegisterFatBinary(void*) {
  static void* handle;
  return &handle;
}
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
void __cudaRegisterFunction(void**, const char* host, char*, const char* name, int, uint3*, uint3*, dim3*, dim3*, int*) { names()[host] = name; }
void __cudaRegisterVar(void**, char*, char*, const char*, int, size_t, int, int) {}
cudaError_t __cudaGetKernel(cudaKernel_t* k, const void* f) {
  *k = reinterpret_cast<cudaKernel_t>(const_cast<void*>(f));
  return cudaSuccess;
}
unsigned __cudaPushCallConfiguration(dim3 g, dim3 b, size_t smem, cudaStream_t st) {
  pushed.push_back({g, b, smem, st});
  return 0;
}
cudaError_t __cudaPopCallConfiguration(dim3* g, dim3* b, size_t* smem, void* st) {
  const Config c = pushed.back();
  pushed.pop_back();
  *g = c.grid;
  *b = c.block;
  *smem = c.smem;
  std::memcpy(st, &c.st, sizeof c.st);
  return cudaSuccess;
}
cudaError_t __cudaLaunchKernel(cudaKernel_t k, dim3 g, dim3 b, void**, size_t smem, cudaStream_t) {
  return launch(reinterpret_cast<const void*>(k), g, b, smem, 0);
}
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t* c, const void* f, void**) {
  return launch(f, c->gridDim, c->blockDim, c->dynamicSmemBytes, 0);
}
cudaError_t cudaLaunchCooperativeKernel(const void* f, dim3 g, dim3 b, void**, size_t smem, cudaStream_t) { return launch(f, g, b, smem, 1); }
cudaError_t cudaFuncSetAttribute(const void* f, cudaFuncAttribute a, int v) {
  if (a == cudaFuncAttributeMaxDynamicSharedMemorySize) smem_limit[{f, device}] = size_t(v);
  return cudaSuccess;
}
// (as if every kernel took 64 registers a thread, those of 4 x 4 cells a thread 128)
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int* n, const void* f, int threads, size_t smem, unsigned) {
  const int regs = names()[f].find("tb2d") != std::string::npos && names()[f].find("ILi2E") == std::string::npos ? 128 : 64;
  *n = 65536 / (regs * threads);
  if (smem) *n = std::min(*n, int(size_t(228 * 1024) / (smem + 1024)));
  return cudaSuccess;
}
cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr a, int) {
  *v = a == cudaDevAttrMultiProcessorCount ? 152 : a == cudaDevAttrMaxSharedMemoryPerBlockOptin ? 227 * 1024 : 1;
  return cudaSuccess;
}
cudaError_t cudaGetDevice(int* d) {
  *d = device;
  return cudaSuccess;
}
cudaError_t cudaSetDevice(int d) {
  if (d < 0 || d >= devices) return fail(cudaErrorInvalidDevice);
  device = d;
  return cudaSuccess;
}
cudaError_t cudaGetLastError() {
  const cudaError_t e = last;
  last = cudaSuccess;
  return e;
}
cudaError_t cudaGetSymbolAddress(void** p, const void*) {
  static char scratch[1 << 10];
  *p = scratch;
  return cudaSuccess;
}
cudaError_t cudaMemsetAsync(void*, int, size_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaMemcpyAsync(void*, const void*, size_t, cudaMemcpyKind, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaMemcpy2DAsync(void*, size_t, const void*, size_t, size_t, size_t, cudaMemcpyKind, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }

}  // extern "C"
