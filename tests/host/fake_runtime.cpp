// Fake of the CUDA runtime for host tests: device memory is host memory, streams do nothing, and
// kernel launches are counted but not run.  Linked with the library's own objects in place of
// the static runtime, it lets a test make an allocation or a launch fail and then look at what the
// next launches are given: every pointer that reaches a step kernel has to be a live allocation.
#include <cuda_runtime_api.h>

#include <cstdint>
#include <cstdlib>
#include <cstring>
#include <map>
#include <string>
#include <vector>

namespace {

struct Block {
  size_t size;
  bool live;
};
std::map<uintptr_t, Block> g_blocks;             // freed blocks stay mapped, marked dead
std::map<const void*, std::string> g_kernels;    // host stub -> mangled kernel name
std::map<std::string, int> g_launches;
std::vector<std::string> g_errors;
int g_fail_alloc = 0;         // the n-th allocation from now fails (-n: and all behind it)
size_t g_largest = SIZE_MAX;  // larger allocations fail
std::string g_fail_launch;   // launches of kernels whose name holds this fail
cudaError_t g_last = cudaSuccess;
float (*g_elapsed)() = nullptr;
float g_adam_correction = 0.f;

void note(const std::string& what) { g_errors.push_back(what); }

// 1: a live allocation, 0: a freed one, -1: host memory
int state_of(const void* p) {
  auto it = g_blocks.upper_bound(reinterpret_cast<uintptr_t>(p));
  if (it == g_blocks.begin()) return -1;
  --it;
  if (reinterpret_cast<uintptr_t>(p) >= it->first + it->second.size) return -1;
  return it->second.live;
}
}  // namespace

void fake_want_live(const void* p, const char* what) {
  if (state_of(p) != 1) note(std::string(what) + (p ? " is a freed pointer" : " is null"));
}
void fake_check_launch(const std::string& name, void** args);  // fake_checks.cu

namespace {

void no_freed(const void* p, const char* what) {
  if (state_of(p) == 0) note(std::string(what) + ": freed memory");
}

bool has(const std::string& name, const char* part) { return name.find(part) != std::string::npos; }

cudaError_t launch(const void* func, void** args) {
  const std::string name = g_kernels.count(func) ? g_kernels[func] : "?";
  if (!g_fail_launch.empty() && has(name, g_fail_launch.c_str())) return g_last = cudaErrorLaunchOutOfResources;
  ++g_launches[name];
  fake_check_launch(name, args);
  if (has(name, "adam_kernel")) g_adam_correction = *static_cast<float*>(args[9]);
  return cudaSuccess;
}

int fake_encode() { return 0; }

}  // namespace

extern "C" {

void fake_fail_allocation(int n) { g_fail_alloc = n; }
void fake_largest_allocation(size_t bytes) { g_largest = bytes; }
void fake_fail_launch(const char* part) { g_fail_launch = part; }
void fake_elapsed(float (*f)()) { g_elapsed = f; }
int fake_live() {
  int n = 0;
  for (const auto& b : g_blocks) n += b.second.live;
  return n;
}
float fake_adam_correction() { return g_adam_correction; }
int fake_launches(const char* part) {
  int n = 0;
  for (const auto& k : g_launches)
    if (has(k.first, part)) n += k.second;
  return n;
}
// the first complaint since the last call, "" if none
const char* fake_errors() {
  static std::string text;
  text.clear();
  for (const std::string& e : g_errors) text += (text.empty() ? "" : "; ") + e;
  g_errors.clear();
  return text.c_str();
}

cudaError_t cudaMallocAsync(void** p, size_t n, cudaStream_t) {
  bool fails = false;
  if (g_fail_alloc > 0) fails = --g_fail_alloc == 0;
  else if (g_fail_alloc == -1) fails = true;
  else if (g_fail_alloc < 0) ++g_fail_alloc;
  if (fails || n > g_largest) return g_last = cudaErrorMemoryAllocation;
  const size_t size = n ? n : 1;
  *p = std::calloc(1, size);
  g_blocks[reinterpret_cast<uintptr_t>(*p)] = Block{size, true};
  return cudaSuccess;
}
cudaError_t cudaFreeAsync(void* p, cudaStream_t) {
  auto it = g_blocks.find(reinterpret_cast<uintptr_t>(p));
  if (it == g_blocks.end() || !it->second.live) note("free of a pointer that is no live allocation");
  else it->second.live = false;  // the memory stays, so its address is not given out again
  return cudaSuccess;
}
cudaError_t cudaMemcpyAsync(void* to, const void* from, size_t n, cudaMemcpyKind, cudaStream_t) {
  no_freed(to, "copy to");
  no_freed(from, "copy from");
  std::memcpy(to, from, n);
  return cudaSuccess;
}
cudaError_t cudaMemcpy2DAsync(void* to, size_t dp, const void* from, size_t sp, size_t w, size_t h, cudaMemcpyKind,
                              cudaStream_t) {
  no_freed(from, "copy from");
  for (size_t r = 0; r < h; ++r) std::memcpy(static_cast<char*>(to) + r * dp, static_cast<const char*>(from) + r * sp, w);
  return cudaSuccess;
}
cudaError_t cudaMemsetAsync(void* p, int v, size_t n, cudaStream_t) {
  fake_want_live(p, "memset target");
  std::memset(p, v, n);
  return cudaSuccess;
}
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t*, const void* func, void** args) { return launch(func, args); }
cudaError_t __cudaLaunchKernel(cudaKernel_t kernel, dim3, dim3, void** args, size_t, cudaStream_t) {
  return launch(reinterpret_cast<const void*>(kernel), args);
}
cudaError_t __cudaGetKernel(cudaKernel_t* k, const void* func) {
  *k = reinterpret_cast<cudaKernel_t>(const_cast<void*>(func));
  return cudaSuccess;
}
unsigned __cudaPushCallConfiguration(dim3, dim3, size_t, struct CUstream_st*) { return 0; }
cudaError_t __cudaPopCallConfiguration(dim3* g, dim3* b, size_t* s, void* stream) {
  *g = *b = dim3(1);
  *s = 0;
  *static_cast<void**>(stream) = nullptr;
  return cudaSuccess;
}
void** __cudaRegisterFatBinary(void*) {
  static void* handle;
  return &handle;
}
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
void __cudaRegisterVar(void**, char*, char*, const char*, int, size_t, int, int) {}
void __cudaRegisterFunction(void**, const char* host, char*, const char* name, int, uint3*, uint3*, dim3*, dim3*, int*) {
  g_kernels[host] = name;
}

cudaError_t cudaGetLastError() {
  const cudaError_t e = g_last;
  g_last = cudaSuccess;
  return e;
}
const char* cudaGetErrorString(cudaError_t e) { return e == cudaErrorMemoryAllocation ? "out of memory" : "error"; }
cudaError_t cudaGetDevice(int* d) { *d = 0; return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr a, int) {
  *v = a == cudaDevAttrMultiProcessorCount ? 152 : a == cudaDevAttrMaxSharedMemoryPerBlockOptin ? 227 * 1024 : 1;
  return cudaSuccess;
}
cudaError_t cudaFuncSetAttribute(const void*, cudaFuncAttribute, int) { return cudaSuccess; }
cudaError_t cudaFuncGetAttributes(cudaFuncAttributes* a, const void*) {
  std::memset(a, 0, sizeof(*a));
  a->numRegs = 96;
  return cudaSuccess;
}
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int* n, const void*, int threads, size_t smem, unsigned) {
  const int by_threads = 640 / threads + 1, by_smem = (int)(228 * 1024 / (smem + 1024));
  *n = by_threads < by_smem ? by_threads : by_smem;
  return cudaSuccess;
}
cudaError_t cudaStreamCreate(cudaStream_t* s) { *s = reinterpret_cast<cudaStream_t>(0x10); return cudaSuccess; }
cudaError_t cudaStreamDestroy(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamBeginCapture(cudaStream_t, cudaStreamCaptureMode) { return cudaSuccess; }
cudaError_t cudaStreamEndCapture(cudaStream_t, cudaGraph_t* g) { *g = nullptr; return cudaSuccess; }
cudaError_t cudaGraphInstantiate(cudaGraphExec_t* e, cudaGraph_t, unsigned long long) {
  *e = reinterpret_cast<cudaGraphExec_t>(0x20);
  return cudaSuccess;
}
cudaError_t cudaGraphLaunch(cudaGraphExec_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaGraphDestroy(cudaGraph_t) { return cudaSuccess; }
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t) { return cudaSuccess; }
cudaError_t cudaEventCreate(cudaEvent_t* e) { *e = nullptr; return cudaSuccess; }
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventSynchronize(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float* ms, cudaEvent_t, cudaEvent_t) {
  *ms = g_elapsed ? g_elapsed() : 1.f;
  return cudaSuccess;
}
cudaError_t cudaGetSymbolAddress(void** p, const void* s) { *p = const_cast<void*>(s); return cudaSuccess; }
cudaError_t cudaGetDriverEntryPointByVersion(const char* name, void** fn, unsigned, unsigned long long,
                                             cudaDriverEntryPointQueryResult* q) {
  *fn = std::strcmp(name, "cuTensorMapEncodeTiled") == 0 ? reinterpret_cast<void*>(&fake_encode) : nullptr;
  *q = *fn ? cudaDriverEntryPointSuccess : cudaDriverEntryPointSymbolNotFound;
  return cudaSuccess;
}

}  // extern "C"
