// A CUDA runtime for tests of the library's host code on a machine without a
// GPU: memory is host memory with a type, a device and a size, copies check
// their ranges as the driver does, kernel launches do nothing but leave their
// name in a log, and single calls can be made to fail. Two devices, four
// multiprocessors each.
#include <cuda.h>
#include <cuda_runtime.h>

#include <cstdlib>
#include <cstring>
#include <map>
#include <mutex>
#include <string>

namespace {
struct Region {
  size_t bytes;
  int type, device;
};
std::mutex mu;
std::map<char*, Region> regions;
// (the library's static constructors register kernels before those of this file)
std::map<const void*, std::string>& kernels() {
  static std::map<const void*, std::string> k;
  return k;
}
std::string log_text;
int current = 0;
bool refuse_cooperative = false;
thread_local dim3 cfg_grid, cfg_block;
thread_local size_t cfg_smem;
thread_local cudaStream_t cfg_stream;

// the region that p lies in, null for other host memory
std::pair<char* const, Region>* find(const void* p) {
  auto it = regions.upper_bound((char*)p);
  if (it == regions.begin()) return nullptr;
  --it;
  return (char*)p < it->first + it->second.bytes ? &*it : nullptr;
}
bool in_range(const void* p, size_t bytes) {
  auto* r = find(p);
  return !r || (char*)p + bytes <= r->first + r->second.bytes;
}
void note(const std::string& s) { log_text += s + "\n"; }
}  // namespace

extern "C" {

// ---- controls
void fake_region(void* p, size_t bytes, int type, int device) { regions[(char*)p] = {bytes, type, device}; }
void fake_set_device(int dev) { current = dev; }
void fake_refuse_cooperative(int on) { refuse_cooperative = on != 0; }
void fake_clear_log() { log_text.clear(); }
const char* fake_log() { return log_text.c_str(); }

// ---- what nvcc's host code calls
void** __cudaRegisterFatBinary(void*) { static void* h; return &h; }
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
void __cudaRegisterVar(void**, char*, char*, const char*, int, size_t, int, int) {}
void __cudaRegisterFunction(void**, const char* host, char*, const char* name, int, uint3*, uint3*,
                            dim3*, dim3*, int*) {
  kernels()[host] = name;
}
char __cudaInitModule(void**) { return 1; }
unsigned __cudaPushCallConfiguration(dim3 g, dim3 b, size_t m, cudaStream_t s) {
  cfg_grid = g; cfg_block = b; cfg_smem = m; cfg_stream = s;
  return 0;
}
cudaError_t __cudaPopCallConfiguration(dim3* g, dim3* b, size_t* m, void* s) {
  *g = cfg_grid; *b = cfg_block; *m = cfg_smem; *(cudaStream_t*)s = cfg_stream;
  return cudaSuccess;
}
cudaError_t __cudaGetKernel(cudaKernel_t* k, const void* f) { *k = (cudaKernel_t)f; return cudaSuccess; }
cudaError_t __cudaLaunchKernel(cudaKernel_t k, dim3, dim3, void**, size_t, cudaStream_t) {
  std::lock_guard<std::mutex> lk(mu);
  note("launch " + kernels()[(const void*)k]);
  return cudaSuccess;
}

// ---- the runtime
cudaError_t cudaGetDevice(int* d) { *d = current; return cudaSuccess; }
cudaError_t cudaSetDevice(int d) { current = d; return cudaSuccess; }
cudaError_t cudaGetLastError() { return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr a, int) {
  *v = a == cudaDevAttrMultiProcessorCount ? 4 : 1;
  return cudaSuccess;
}
cudaError_t cudaDeviceGetDefaultMemPool(cudaMemPool_t* p, int) { *p = nullptr; return cudaSuccess; }
cudaError_t cudaMemPoolSetAttribute(cudaMemPool_t, cudaMemPoolAttr, void*) { return cudaSuccess; }
cudaError_t cudaMallocAsync(void** p, size_t n, cudaStream_t) {
  *p = std::calloc(1, n + 1);
  std::lock_guard<std::mutex> lk(mu);
  regions[(char*)*p] = {n, cudaMemoryTypeDevice, current};
  return cudaSuccess;
}
cudaError_t cudaFreeAsync(void* p, cudaStream_t) {
  std::lock_guard<std::mutex> lk(mu);
  regions.erase((char*)p);
  std::free(p);
  return cudaSuccess;
}
cudaError_t cudaHostAlloc(void** p, size_t n, unsigned) { *p = std::calloc(1, n); return cudaSuccess; }
cudaError_t cudaFreeHost(void* p) { std::free(p); return cudaSuccess; }
cudaError_t cudaMemGetInfo(size_t* f, size_t* t) { *f = *t = (size_t)1 << 38; return cudaSuccess; }
cudaError_t cudaPointerGetAttributes(cudaPointerAttributes* a, const void* p) {
  std::lock_guard<std::mutex> lk(mu);
  std::memset(a, 0, sizeof(*a));
  auto* r = find(p);
  a->type = r ? (cudaMemoryType)r->second.type : cudaMemoryTypeUnregistered;
  a->device = r ? r->second.device : 0;
  a->devicePointer = (void*)p;
  return cudaSuccess;
}
cudaError_t cudaMemcpyAsync(void* d, const void* s, size_t n, cudaMemcpyKind, cudaStream_t) {
  std::lock_guard<std::mutex> lk(mu);
  if (!in_range(d, n) || !in_range(s, n)) {
    note("copy refused");
    return cudaErrorInvalidValue;
  }
  note("copy " + std::to_string(n));
  std::memmove(d, s, n);
  return cudaSuccess;
}
cudaError_t cudaMemsetAsync(void* d, int v, size_t n, cudaStream_t) { std::memset(d, v, n); return cudaSuccess; }
cudaError_t cudaEventCreate(cudaEvent_t* e) { *e = (cudaEvent_t)1; return cudaSuccess; }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t* e, unsigned) { *e = (cudaEvent_t)1; return cudaSuccess; }
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float* t, cudaEvent_t, cudaEvent_t) { *t = 0; return cudaSuccess; }
cudaError_t cudaStreamCreateWithFlags(cudaStream_t* s, unsigned) { *s = nullptr; return cudaSuccess; }
cudaError_t cudaStreamDestroy(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamWaitEvent(cudaStream_t, cudaEvent_t, unsigned) { return cudaSuccess; }
cudaError_t cudaLaunchHostFunc(cudaStream_t, cudaHostFn_t f, void* p) { f(p); return cudaSuccess; }
cudaError_t cudaFuncSetAttribute(const void*, cudaFuncAttribute, int) { return cudaSuccess; }
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int* b, const void*, int, size_t, unsigned) {
  *b = 2;
  return cudaSuccess;
}
cudaError_t cudaGetSymbolAddress(void** p, const void*) { *p = nullptr; return cudaErrorInvalidValue; }
cudaError_t cudaLaunchCooperativeKernel(const void* f, dim3, dim3, void**, size_t, cudaStream_t) {
  std::lock_guard<std::mutex> lk(mu);
  note((refuse_cooperative ? "refused " : "launch ") + kernels()[f]);
  return refuse_cooperative ? cudaErrorCooperativeLaunchTooLarge : cudaSuccess;
}
static CUresult attributes(unsigned n, CUpointer_attribute* what, void** to, CUdeviceptr p) {
  std::lock_guard<std::mutex> lk(mu);
  auto* r = find((const void*)p);
  for (unsigned i = 0; i < n; ++i) switch (what[i]) {
    case CU_POINTER_ATTRIBUTE_MEMORY_TYPE: *(unsigned*)to[i] = r ? r->second.type : 0; break;
    case CU_POINTER_ATTRIBUTE_IS_MANAGED: *(unsigned*)to[i] = 0; break;
    case CU_POINTER_ATTRIBUTE_DEVICE_ORDINAL: *(int*)to[i] = r ? r->second.device : -2; break;
    case CU_POINTER_ATTRIBUTE_RANGE_START_ADDR: *(CUdeviceptr*)to[i] = r ? (CUdeviceptr)r->first : 0; break;
    case CU_POINTER_ATTRIBUTE_RANGE_SIZE: *(size_t*)to[i] = r ? r->second.bytes : 0; break;
    default: return CUDA_ERROR_INVALID_VALUE;
  }
  return CUDA_SUCCESS;
}
cudaError_t cudaGetDriverEntryPointByVersion(const char* name, void** f, unsigned, unsigned long long,
                                             cudaDriverEntryPointQueryResult* q) {
  const bool known = !std::strcmp(name, "cuPointerGetAttributes");
  *f = known ? (void*)attributes : nullptr;
  if (q) *q = known ? cudaDriverEntryPointSuccess : cudaDriverEntryPointSymbolNotFound;
  return known ? cudaSuccess : cudaErrorInvalidValue;
}

}  // extern "C"
