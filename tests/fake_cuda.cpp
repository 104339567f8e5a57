// A CUDA runtime that runs nothing: it logs the stream and event calls the joins are
// made of, and fails the launch it is told to (tests/test_join.py).
#include <cuda_runtime_api.h>

#include <cstdio>
#include <cstring>

int g_fail_at = -1;
static int g_launches = 0;
static cudaError_t g_last = cudaSuccess;
static cudaStream_t g_stream;

cudaError_t fake_launch(cudaStream_t st) {
  if (g_launches++ == g_fail_at) return cudaErrorLaunchOutOfResources;
  std::printf("launch %zu\n", (size_t)st);
  return cudaSuccess;
}

extern "C" {
cudaError_t cudaEventRecord(cudaEvent_t ev, cudaStream_t st) {
  std::printf("record %zu %zu\n", (size_t)ev, (size_t)st);
  return cudaSuccess;
}
cudaError_t cudaStreamWaitEvent(cudaStream_t st, cudaEvent_t ev, unsigned) {
  std::printf("wait %zu %zu\n", (size_t)st, (size_t)ev);
  return cudaSuccess;
}
cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventSynchronize(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaGetLastError() {
  const cudaError_t e = g_last;
  g_last = cudaSuccess;
  return e;
}
cudaError_t cudaSetDevice(int) { return cudaSuccess; }
const char* cudaGetErrorString(cudaError_t) { return "failed on purpose"; }
cudaError_t cudaMemsetAsync(void*, int, size_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaFuncSetAttribute(const void*, cudaFuncAttribute, int) { return cudaSuccess; }
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessor(int* n, const void*, int, size_t) {
  *n = 1;
  return cudaSuccess;
}
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int* n, const void*, int, size_t,
                                                                   unsigned) {
  *n = 1;
  return cudaSuccess;
}
void** __cudaRegisterFatBinary(void*) {
  static void* p;
  return &p;
}
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
void __cudaRegisterFunction(void**, const char*, char*, const char*, int, uint3*, uint3*, dim3*, dim3*,
                            int*) {}
void __cudaRegisterVar(void**, char*, char*, const char*, int, size_t, int, int) {}
char __cudaInitModule(void**) { return 0; }
unsigned __cudaPushCallConfiguration(dim3, dim3, size_t, cudaStream_t st) {
  g_stream = st;
  return 0;
}
cudaError_t __cudaPopCallConfiguration(dim3*, dim3*, size_t*, void* st) {
  *(cudaStream_t*)st = g_stream;
  return cudaSuccess;
}
cudaError_t cudaLaunchKernel(const void*, dim3, dim3, void**, size_t, cudaStream_t st) {
  return g_last = fake_launch(st);
}
cudaError_t __cudaGetKernel(cudaKernel_t*, const void*) { return cudaSuccess; }
cudaError_t __cudaLaunchKernel(cudaKernel_t, dim3, dim3, void**, size_t, cudaStream_t st) {
  return g_last = fake_launch(st);
}
// read-backs bring counts of a hundred pairs
cudaError_t cudaMemcpyAsync(void* dst, const void*, size_t bytes, cudaMemcpyKind, cudaStream_t) {
  for (size_t k = 0; k < bytes / 4; ++k) ((int*)dst)[k] = 100;
  return cudaSuccess;
}
}
