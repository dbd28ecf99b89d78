// A stand-in for the CUDA runtime, on the host: linked with the library's host
// code and the launchers of fake_launchers.cu, it lets a test make the n-th call
// of a kind fail and see what the handle does then, without a GPU.  "Device"
// memory is host memory.
#include <cuda.h>
#include <cuda_runtime_api.h>

#include <algorithm>
#include <cstdlib>
#include <cstring>
#include <map>

namespace {

enum { MALLOC = 0, MEMCPY_ASYNC = 1, PUSH_COPY = 2, KINDS = 3 };
int g_fail[KINDS];    // the n-th call of the kind from now fails (0: none does)
int g_addressable;    // arrays are device memory (copied by the launch) or unknown to the driver
int g_bad, g_unordered;
cudaError_t g_last = cudaSuccess;
std::map<const char*, size_t>& live() {
  static std::map<const char*, size_t> m;
  return m;
}

bool fails(int kind) { return g_fail[kind] > 0 && --g_fail[kind] == 0; }
cudaError_t error(cudaError_t e) { return g_last = e; }

cudaError_t allocate(void** p, size_t bytes) {
  // nothing reads or writes the rows of a table, so the largest are not there whole
  *p = calloc(1, std::min<size_t>(std::max<size_t>(bytes, 1), (size_t)1 << 26));
  live()[(const char*)*p] = bytes;
  return cudaSuccess;
}
cudaError_t release(void* p) {
  if (p && live().erase((const char*)p) == 0) ++g_bad;  // freed twice, or never allocated
  free(p);
  return cudaSuccess;
}

CUresult pointer_attributes(unsigned int n, CUpointer_attribute*, void** to, CUdeviceptr p) {
  if (n != 6 || !g_addressable) return CUDA_ERROR_INVALID_VALUE;
  *(unsigned int*)to[0] = CU_MEMORYTYPE_DEVICE;
  *(unsigned int*)to[1] = 0;
  *(int*)to[2] = 0;
  *(CUdeviceptr*)to[3] = p;
  *(CUdeviceptr*)to[4] = p;
  *(size_t*)to[5] = (size_t)1 << 40;
  return CUDA_SUCCESS;
}

}  // namespace

extern "C" {

void fake_fail(int kind, int nth) { g_fail[kind] = nth; }
void fake_addressable(int on) { g_addressable = on; }
int fake_bad() { return g_bad; }
int fake_unordered() { return g_unordered; }
long fake_allocations() { return (long)live().size(); }
cudaError_t fake_copy_launch() {
  return fails(PUSH_COPY) ? error(cudaErrorLaunchOutOfResources) : cudaSuccess;
}
void fake_need(const void* p, size_t bytes) {  // [p, p + bytes) lies within one live allocation
  auto it = live().upper_bound((const char*)p);
  if (it != live().begin()) {
    --it;
    if ((const char*)p + bytes <= it->first + it->second) return;
  }
  ++g_bad;
}

cudaError_t cudaMalloc(void** p, size_t n) {
  return fails(MALLOC) ? error(cudaErrorMemoryAllocation) : allocate(p, n);
}
cudaError_t cudaFree(void* p) { return release(p); }
cudaError_t cudaHostAlloc(void** p, size_t n, unsigned int) { return allocate(p, n); }
cudaError_t cudaFreeHost(void* p) { return release(p); }
cudaError_t cudaHostGetDevicePointer(void** d, void* p, unsigned int) { return *d = p, cudaSuccess; }
// these use the default stream, on which the handle's streams do not wait
cudaError_t cudaMemcpy(void* d, const void* s, size_t n, cudaMemcpyKind kind) {
  if (kind != cudaMemcpyDeviceToHost) ++g_unordered;
  return memcpy(d, s, n), cudaSuccess;
}
cudaError_t cudaMemset(void* p, int v, size_t n) {
  ++g_unordered;
  return memset(p, v, n), cudaSuccess;
}
cudaError_t cudaMemcpyAsync(void* d, const void* s, size_t n, cudaMemcpyKind, cudaStream_t) {
  if (fails(MEMCPY_ASYNC)) return error(cudaErrorInvalidValue);
  return memcpy(d, s, n), cudaSuccess;
}
cudaError_t cudaMemsetAsync(void* p, int v, size_t n, cudaStream_t) {
  return memset(p, v, n), cudaSuccess;
}
cudaError_t cudaGetDevice(int* d) { return *d = 0, cudaSuccess; }
cudaError_t cudaSetDevice(int) { return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr, int) { return *v = 152, cudaSuccess; }
cudaError_t cudaStreamCreateWithFlags(cudaStream_t* s, unsigned int) {
  return *s = (cudaStream_t)malloc(1), cudaSuccess;
}
cudaError_t cudaStreamDestroy(cudaStream_t s) { return free(s), cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamWaitEvent(cudaStream_t, cudaEvent_t, unsigned int) { return cudaSuccess; }
cudaError_t cudaEventCreate(cudaEvent_t* e) { return *e = (cudaEvent_t)malloc(1), cudaSuccess; }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t* e, unsigned int) { return cudaEventCreate(e); }
cudaError_t cudaEventDestroy(cudaEvent_t e) { return free(e), cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventSynchronize(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float* ms, cudaEvent_t, cudaEvent_t) { return *ms = 0.f, cudaSuccess; }
cudaError_t cudaGetLastError() {
  const cudaError_t e = g_last;
  g_last = cudaSuccess;
  return e;
}
const char* cudaGetErrorString(cudaError_t) { return "made to fail"; }
cudaError_t cudaGetDriverEntryPointByVersion(const char*, void** f, unsigned int, unsigned long long,
                                             cudaDriverEntryPointQueryResult* found) {
  *f = (void*)pointer_attributes;
  *found = cudaDriverEntryPointSuccess;
  return cudaSuccess;
}
void** __cudaRegisterFatBinary(void*) { return nullptr; }
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}

}  // extern "C"
