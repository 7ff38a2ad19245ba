// A CUDA runtime that launches nothing and notes what it was asked for: with
// fake_kernels.cu, csrc/host.cu linked against it shows, on the CPU, which
// launches a call makes and what it does when one of them is refused
// (test_launches_cpu.py).
#include <cuda_runtime.h>

#include <string>

char kGram, kPrefetchGram, kBulkGram, kLastFirst, kPrefetch, kStream;   // the kernels' addresses

static std::string notes;
static int coop_error = 0;

void note(const char* what) { notes += std::string(what) + " "; }

extern "C" {
const char* fake_notes() { return notes.c_str(); }
void fake_reset(int error) {
  notes.clear();
  coop_error = error;
}

cudaError_t cudaGetDevice(int* d) { *d = 0; return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr, int) { *v = 152; return cudaSuccess; }
cudaError_t cudaFuncSetAttribute(const void*, cudaFuncAttribute, int) { return cudaSuccess; }
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessor(int* n, const void* f, int, size_t) {
  *n = f == &kStream ? 1 : 2;
  return cudaSuccess;
}
cudaError_t cudaGetLastError() { note("cleared"); return cudaSuccess; }
cudaError_t cudaLaunchCooperativeKernel(const void* f, dim3 grid, dim3, void**, size_t, cudaStream_t) {
  note(f == &kStream && grid.x <= 152 ? "stream" : "?");
  return (cudaError_t)coop_error;
}
cudaError_t cudaLaunchKernel(const void* f, dim3, dim3, void**, size_t, cudaStream_t) {
  note(f == &kGram           ? "gram"
       : f == &kPrefetchGram ? "gram-prefetch"
       : f == &kBulkGram     ? "gram-bulk"
       : f == &kLastFirst    ? "combine-last-first"
       : f == &kPrefetch     ? "combine-prefetch"
                             : "?");
  return cudaSuccess;
}
cudaError_t cudaMemsetAsync(void*, int, size_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaMemcpy(void*, const void*, size_t, cudaMemcpyKind) { return cudaSuccess; }
cudaError_t cudaMemcpyAsync(void*, const void*, size_t, cudaMemcpyKind, cudaStream_t) {
  return cudaSuccess;
}
cudaError_t cudaStreamCreateWithFlags(cudaStream_t*, unsigned) { return cudaSuccess; }
cudaError_t cudaStreamDestroy(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamWaitEvent(cudaStream_t, cudaEvent_t, unsigned) { return cudaSuccess; }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t*, unsigned) { return cudaSuccess; }
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { note("event"); return cudaSuccess; }

// what nvcc's start-up code calls
void** __cudaRegisterFatBinary(void*) { return nullptr; }
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
char __cudaInitModule(void**) { return 0; }
}
