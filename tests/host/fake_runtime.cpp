// The CUDA runtime calls of csrc/rgs_api.cu on host memory.
#include <cuda_runtime_api.h>
#include <sys/mman.h>

#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <map>

#include "fake_state.h"

namespace fake {
static std::map<char*, size_t>& blocks() {
  static std::map<char*, size_t> m;
  return m;
}
size_t live = 0, limit = SIZE_MAX, total = 288ull << 30;
bool capturing = false, one_place = false;
const void* wrote_pairs = nullptr;
int stale = 0, unsafe = 0;
unsigned long long visible = 0, cells = 0, pairs = 0, pairs_per_cell = 1;

void check(const void* p, size_t bytes, const char* what) {
  char* c = static_cast<char*>(const_cast<void*>(p));
  auto it = blocks().upper_bound(c);
  if (it != blocks().begin()) {
    --it;
    if (c >= it->first && c + bytes <= it->first + it->second) return;
  }
  ++stale;
  std::printf("not in live memory: %s (%zu bytes)\n", what, bytes);
}
}  // namespace fake

extern "C" {
cudaError_t cudaMalloc(void** p, size_t bytes) {
  fake::unsafe += fake::capturing;
  *p = nullptr;
  if (fake::live + bytes > fake::limit) return cudaErrorMemoryAllocation;
  void* base_ptr = mmap(nullptr, bytes, PROT_READ | PROT_WRITE,
                        MAP_PRIVATE | MAP_ANONYMOUS | MAP_NORESERVE, -1, 0);
  if (base_ptr == MAP_FAILED) return cudaErrorMemoryAllocation;
  char* base = static_cast<char*>(base_ptr);
  fake::blocks()[base] = bytes;
  fake::live += bytes;
  *p = base;
  return cudaSuccess;
}
cudaError_t cudaFree(void* p) {
  fake::unsafe += fake::capturing;
  auto it = fake::blocks().find(static_cast<char*>(p));
  if (it == fake::blocks().end()) return p ? cudaErrorInvalidValue : cudaSuccess;
  fake::live -= it->second;
  munmap(p, it->second);
  fake::blocks().erase(it);
  return cudaSuccess;
}
cudaError_t cudaMemGetInfo(size_t* free_bytes, size_t* total_bytes) {
  const size_t have = fake::limit < fake::total ? fake::limit : fake::total;
  *free_bytes = have - fake::live;
  *total_bytes = fake::total;
  return cudaSuccess;
}
cudaError_t cudaMemsetAsync(void* p, int value, size_t bytes, cudaStream_t) {
  fake::check(p, bytes, "memset");
  if (bytes < (64u << 20)) std::memset(p, value, bytes);
  return cudaSuccess;
}
cudaError_t cudaMemcpyAsync(void* to, const void* from, size_t bytes, cudaMemcpyKind kind,
                            cudaStream_t) {
  if (kind == cudaMemcpyDeviceToHost) fake::check(from, bytes, "copy");
  std::memcpy(to, from, bytes);
  return cudaSuccess;
}
cudaError_t cudaMemcpy(void* to, const void* from, size_t bytes, cudaMemcpyKind) {
  fake::check(from, bytes, "copy");
  fake::check(to, bytes, "copy");
  std::memcpy(to, from, bytes);
  return cudaSuccess;
}
cudaError_t cudaMemcpy2DAsync(void*, size_t, const void*, size_t, size_t, size_t, cudaMemcpyKind,
                              cudaStream_t) { return cudaSuccess; }
cudaError_t cudaHostAlloc(void** p, size_t bytes, unsigned) {
  *p = std::calloc(1, bytes);
  return cudaSuccess;
}
cudaError_t cudaFreeHost(void* p) { std::free(p); return cudaSuccess; }
cudaError_t cudaSetDevice(int) { return cudaSuccess; }
cudaError_t cudaGetDeviceCount(int* n) { *n = 1; return cudaSuccess; }
cudaError_t cudaDeviceSynchronize() {
  fake::unsafe += fake::capturing;
  return cudaSuccess;
}
cudaError_t cudaStreamSynchronize(cudaStream_t) {
  fake::unsafe += fake::capturing;
  return cudaSuccess;
}
cudaError_t cudaStreamWaitEvent(cudaStream_t, cudaEvent_t, unsigned) { return cudaSuccess; }
cudaError_t cudaStreamIsCapturing(cudaStream_t, cudaStreamCaptureStatus* s) {
  *s = fake::capturing ? cudaStreamCaptureStatusActive : cudaStreamCaptureStatusNone;
  return cudaSuccess;
}
cudaError_t cudaEventCreate(cudaEvent_t* e) {
  *e = reinterpret_cast<cudaEvent_t>(16);
  return cudaSuccess;
}
cudaError_t cudaEventCreateWithFlags(cudaEvent_t* e, unsigned) { return cudaEventCreate(e); }
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventRecordWithFlags(cudaEvent_t, cudaStream_t, unsigned) { return cudaSuccess; }
cudaError_t cudaEventSynchronize(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float* ms, cudaEvent_t, cudaEvent_t) {
  *ms = 1.0f;
  return cudaSuccess;
}
cudaError_t cudaGetLastError() { return cudaSuccess; }
const char* cudaGetErrorString(cudaError_t) { return "error"; }
void** __cudaRegisterFatBinary(void*) { static void* h; return &h; }
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
}
