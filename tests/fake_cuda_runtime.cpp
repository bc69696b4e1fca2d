// Stand-in for the CUDA runtime, so that the host side of the library runs without a GPU: linked with the
// library's objects in place of libcudart, it knows a few devices, keeps the attributes that are set on each
// of them, refuses launches that ask for more dynamic shared memory than was granted there, and records what is
// launched.  Memory calls do nothing (device pointers are never followed on the host).
#include <cuda_runtime_api.h>

#include <cstring>
#include <map>
#include <string>
#include <utility>
#include <vector>

namespace {
struct Launch {
  std::string name;
  int device, grid[3], block;
  size_t smem;
  unsigned long long stream;
};
std::map<const void*, std::string>& names() {  // (filled by the objects' constructors, in whatever order they run)
  static std::map<const void*, std::string> m;
  return m;
}
std::map<std::pair<int, const void*>, int> g_smem_limit;
std::map<unsigned long long, int> g_capturing;
std::vector<Launch> g_launches;
int g_device = 0, g_set_attribute_calls = 0;
void (*g_on_smem_limit)() = nullptr;
cudaError_t g_last = cudaSuccess;
dim3 g_push_grid, g_push_block;
size_t g_push_smem;
cudaStream_t g_push_stream;

unsigned long long id_of(cudaStream_t st) { return reinterpret_cast<unsigned long long>(st); }

cudaError_t record(const void* fn, dim3 g, dim3 b, size_t smem, cudaStream_t st) {
  const auto it = g_smem_limit.find({g_device, fn});
  if (smem > static_cast<size_t>(it == g_smem_limit.end() ? 48 * 1024 : it->second)) return g_last = cudaErrorInvalidValue;
  g_launches.push_back({names()[fn], g_device, {(int)g.x, (int)g.y, (int)g.z}, (int)b.x, smem, id_of(st)});
  return cudaSuccess;
}
int encode_nothing() { return 0; }
}  // namespace

extern "C" {
// ---- for the tests
void fake_reset() {
  g_launches.clear();
  g_set_attribute_calls = 0;
}
void fake_set_device(int d) { g_device = d; }
void fake_set_capturing(unsigned long long stream, int on) { g_capturing[stream] = on; }
// called once, behind the next shared-memory limit that is set: what another thread may do there
void fake_on_smem_limit(void (*fn)()) { g_on_smem_limit = fn; }
int fake_launches() { return static_cast<int>(g_launches.size()); }
int fake_set_attribute_calls() { return g_set_attribute_calls; }
int fake_launch(int i, char* name, int size, int* grid3, long long* smem) {
  const Launch& l = g_launches[i];
  strncpy(name, l.name.c_str(), size - 1);
  name[size - 1] = 0;
  for (int k = 0; k < 3; ++k) grid3[k] = l.grid[k];
  *smem = static_cast<long long>(l.smem);
  return l.device;
}

// ---- what the compiler's host code calls
void** __cudaRegisterFatBinary(void*) {
  static void* handle = nullptr;
  return &handle;
}
char __cudaInitModule(void**) { return 1; }
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
void __cudaRegisterFunction(void**, const char* host, char*, const char* name, int, void*, void*, void*, void*, int*) { names()[host] = name; }
void __cudaRegisterVar(void**, char*, char*, const char*, int, size_t, int, int) {}
unsigned __cudaPushCallConfiguration(dim3 g, dim3 b, size_t smem, cudaStream_t st) {
  g_push_grid = g;
  g_push_block = b;
  g_push_smem = smem;
  g_push_stream = st;
  return 0;
}
cudaError_t __cudaPopCallConfiguration(dim3* g, dim3* b, size_t* smem, void* st) {
  *g = g_push_grid;
  *b = g_push_block;
  *smem = g_push_smem;
  *static_cast<cudaStream_t*>(st) = g_push_stream;
  return cudaSuccess;
}

// ---- the runtime
cudaError_t cudaLaunchKernel(const void* fn, dim3 g, dim3 b, void**, size_t smem, cudaStream_t st) { return record(fn, g, b, smem, st); }
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t* c, const void* fn, void**) {
  return record(fn, c->gridDim, c->blockDim, c->dynamicSmemBytes, c->stream);
}
cudaError_t cudaFuncSetAttribute(const void* fn, cudaFuncAttribute attr, int value) {
  ++g_set_attribute_calls;
  if (attr == cudaFuncAttributeMaxDynamicSharedMemorySize) {
    g_smem_limit[{g_device, fn}] = value;
    if (void (*other)() = g_on_smem_limit) {
      g_on_smem_limit = nullptr;
      other();
    }
  }
  return cudaSuccess;
}
cudaError_t cudaGetDevice(int* d) {
  *d = g_device;
  return cudaSuccess;
}
cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr attr, int) {
  *v = attr == cudaDevAttrComputeCapabilityMajor ? 10 : attr == cudaDevAttrMultiProcessorCount ? 148 : 1;
  return cudaSuccess;
}
cudaError_t cudaGetDriverEntryPoint(const char*, void** fn, unsigned long long, cudaDriverEntryPointQueryResult* q) {
  *fn = reinterpret_cast<void*>(encode_nothing);
  *q = cudaDriverEntryPointSuccess;
  return cudaSuccess;
}
cudaError_t cudaGetSymbolAddress(void** p, const void*) {
  *p = reinterpret_cast<void*>(0x100000);
  return cudaSuccess;
}
cudaError_t cudaOccupancyMaxActiveClusters(int* n, const void*, const cudaLaunchConfig_t*) {
  *n = 16;
  return cudaSuccess;
}
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessor(int* n, const void*, int, size_t) {
  *n = 1;
  return cudaSuccess;
}
cudaError_t cudaStreamIsCapturing(cudaStream_t st, cudaStreamCaptureStatus* s) {
  *s = g_capturing[id_of(st)] ? cudaStreamCaptureStatusActive : cudaStreamCaptureStatusNone;
  return cudaSuccess;
}
cudaError_t cudaStreamGetId(cudaStream_t st, unsigned long long* id) {
  *id = id_of(st);
  return cudaSuccess;
}
cudaError_t cudaGetLastError() {
  const cudaError_t e = g_last;
  g_last = cudaSuccess;
  return e;
}
cudaError_t cudaDeviceSynchronize() { return cudaSuccess; }
cudaError_t cudaMemcpy(void*, const void*, size_t, cudaMemcpyKind) { return cudaSuccess; }
cudaError_t cudaMemcpyAsync(void*, const void*, size_t, cudaMemcpyKind, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaMemset(void*, int, size_t) { return cudaSuccess; }
cudaError_t cudaMemsetAsync(void*, int, size_t, cudaStream_t) { return cudaSuccess; }
}
