// A stand-in for the part of the CUDA runtime that kernels are launched through, for tests without a GPU: nothing is
// executed, a kernel's limit on dynamic shared memory is remembered, and a launch beyond it fails as the runtime's does.
// Between two steps of a call another thread may make a whole call of its own: `other`, before a launch that the test names.
#include <cuda.h>
#include <cuda_runtime_api.h>
#include <map>

namespace {
std::map<const void*, size_t> limit;
size_t largest;
int launches, interrupt_at;
int (*interrupt)();
cudaError_t last_error;

CUresult encode(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*, const cuuint64_t*, const cuuint32_t*,
                const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill) {
  return CUDA_SUCCESS;
}
}  // namespace

void fake_limits_reset(int at, int (*other)()) {  // (the limits stay: they are the process's)
  largest = 0; launches = 0; interrupt_at = at; interrupt = other; last_error = cudaSuccess;
}
size_t fake_largest_launch() { return largest; }

extern "C" {
cudaError_t cudaGetLastError() { const cudaError_t e = last_error; last_error = cudaSuccess; return e; }
cudaError_t cudaGetDevice(int* d) { *d = 0; return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaGetDriverEntryPoint(const char*, void** f, unsigned long long, cudaDriverEntryPointQueryResult* r) {
  *f = reinterpret_cast<void*>(&encode);
  *r = cudaDriverEntryPointSuccess;
  return cudaSuccess;
}
cudaError_t cudaFuncSetAttribute(const void* f, cudaFuncAttribute what, int value) {
  if (what == cudaFuncAttributeMaxDynamicSharedMemorySize) limit[f] = (size_t)value;
  return cudaSuccess;
}
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t* cfg, const void* f, void**) {
  if (++launches == interrupt_at) interrupt();
  const size_t bytes = cfg->dynamicSmemBytes, most = limit.count(f) ? limit[f] : 48 * 1024;
  if (bytes > largest) largest = bytes;
  return bytes > most ? last_error = cudaErrorInvalidValue : cudaSuccess;
}
cudaError_t cudaLaunchKernel(const void*, dim3, dim3, void**, size_t, cudaStream_t) { return cudaSuccess; }

// ---- what nvcc's host code refers to besides
void** __cudaRegisterFatBinary(void*) { static void* h; return &h; }
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
void __cudaRegisterFunction(void**, const char*, char*, const char*, int, uint3*, uint3*, dim3*, dim3*, int*) {}
unsigned __cudaPushCallConfiguration(dim3, dim3, size_t, struct CUstream_st*) { return 0; }
cudaError_t __cudaPopCallConfiguration(dim3*, dim3*, size_t*, void*) { return cudaSuccess; }
}  // extern "C"
