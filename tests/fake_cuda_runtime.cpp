// A stand-in for the CUDA runtime, for tests of the host side on a machine without a GPU: device memory is host
// memory, work is not executed but counted per stream, and events carry what they wait for.  The n-th call that
// enqueues or waits can be made to fail.
#include <cuda_runtime_api.h>
#include <cstdint>
#include <cstdlib>
#include <cstring>
#include <map>

namespace {
struct Clock { long n[2]; };                      // pieces of work seen, per stream: the caller's, the context's second
Clock issued, host_done, stream_at[2];
std::map<cudaEvent_t, Clock> event_at;
long n_calls, fail_at;
int pageable;
const cudaStream_t AUX = (cudaStream_t)(uintptr_t)0x20;

int index_of(cudaStream_t s) { return s == AUX; }
void join(Clock* a, const Clock& b) { for (int i = 0; i < 2; ++i) if (b.n[i] > a->n[i]) a->n[i] = b.n[i]; }
bool fails() { return ++n_calls == fail_at; }
}  // namespace

// One piece of work on a stream (the launchers of host_step_fake.cu call it too).
cudaError_t fake_issue(cudaStream_t s) {
  if (fails()) return cudaErrorUnknown;
  const int i = index_of(s);
  stream_at[i].n[i] = ++issued.n[i];
  return cudaSuccess;
}

extern "C" {
// ---- read and set by the test
void fake_reset(long fail, int host_memory_is_pageable) {
  n_calls = 0; fail_at = fail; pageable = host_memory_is_pageable;
  issued = host_done = stream_at[0] = stream_at[1] = Clock{};
  event_at.clear();
}
long fake_calls() { return n_calls; }
int fake_in_flight() { return issued.n[0] > host_done.n[0] || issued.n[1] > host_done.n[1]; }

// ---- runtime
cudaError_t cudaGetLastError() { return cudaSuccess; }
cudaError_t cudaGetDeviceCount(int* n) { *n = 1; return cudaSuccess; }
cudaError_t cudaSetDevice(int) { return cudaSuccess; }
cudaError_t cudaGetDeviceProperties(cudaDeviceProp* p, int) {
  memset(p, 0, sizeof(*p));
  p->major = 10; p->multiProcessorCount = 148;
  return cudaSuccess;
}
cudaError_t cudaPointerGetAttributes(cudaPointerAttributes* a, const void* p) {
  a->type = pageable ? cudaMemoryTypeUnregistered : cudaMemoryTypeHost;
  a->devicePointer = pageable ? nullptr : (void*)p;
  return cudaSuccess;
}
cudaError_t cudaMalloc(void** p, size_t n) {
  if (posix_memalign(p, 256, n)) return cudaErrorMemoryAllocation;
  memset(*p, 0, n);
  return cudaSuccess;
}
cudaError_t cudaFree(void* p) { free(p); return cudaSuccess; }
cudaError_t cudaHostAlloc(void** p, size_t n, unsigned) { return cudaMalloc(p, n); }
cudaError_t cudaFreeHost(void* p) { return cudaFree(p); }
cudaError_t cudaMemset(void* p, int v, size_t n) { memset(p, v, n); return cudaSuccess; }
cudaError_t cudaStreamCreateWithFlags(cudaStream_t* s, unsigned) { *s = AUX; return cudaSuccess; }
cudaError_t cudaStreamDestroy(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t* e, unsigned) { return cudaMalloc((void**)e, 1); }
cudaError_t cudaEventCreate(cudaEvent_t* e) { return cudaMalloc((void**)e, 1); }
cudaError_t cudaEventDestroy(cudaEvent_t e) { return cudaFree(e); }
cudaError_t cudaEventSynchronize(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float* ms, cudaEvent_t, cudaEvent_t) { *ms = 0; return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t e, cudaStream_t s) {
  if (fails()) return cudaErrorUnknown;
  event_at[e] = stream_at[index_of(s)];
  return cudaSuccess;
}
cudaError_t cudaStreamWaitEvent(cudaStream_t s, cudaEvent_t e, unsigned) {
  if (fails()) return cudaErrorUnknown;
  join(&stream_at[index_of(s)], event_at[e]);
  return cudaSuccess;
}
cudaError_t cudaStreamSynchronize(cudaStream_t s) {
  if (fails()) return cudaErrorUnknown;
  join(&host_done, stream_at[index_of(s)]);
  return cudaSuccess;
}
cudaError_t cudaMemcpyAsync(void*, const void*, size_t, cudaMemcpyKind, cudaStream_t s) { return fake_issue(s); }
cudaError_t cudaMemcpy2DAsync(void*, size_t, const void*, size_t, size_t, size_t, cudaMemcpyKind, cudaStream_t s) { return fake_issue(s); }
cudaError_t cudaMemsetAsync(void* p, int v, size_t n, cudaStream_t s) {
  const cudaError_t e = fake_issue(s);
  if (e == cudaSuccess) memset(p, v, n);
  return e;
}
cudaError_t cudaLaunchKernel(const void*, dim3, dim3, void**, size_t, cudaStream_t s) { return fake_issue(s); }

// ---- what nvcc's host code refers to besides
void** __cudaRegisterFatBinary(void*) { static void* h; return &h; }
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
void __cudaRegisterFunction(void**, const char*, char*, const char*, int, uint3*, uint3*, dim3*, dim3*, int*) {}
unsigned __cudaPushCallConfiguration(dim3, dim3, size_t, struct CUstream_st*) { return 0; }
cudaError_t __cudaPopCallConfiguration(dim3*, dim3*, size_t*, void*) { return cudaSuccess; }
}  // extern "C"
