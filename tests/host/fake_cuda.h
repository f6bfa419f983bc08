// The CUDA runtime calls of the library's set-up code on host memory, for host
// tests of its decisions (what is allocated, what a failed allocation or a stream
// capture leads to).  Put in front of a library source with -include.  Kernel
// launches fail for want of a device, which cudaGetLastError does not report here:
// what kernels would have written stays zero.
#pragma once

#include <cuda_runtime.h>

#include <cstdlib>
#include <cstring>

struct FakeCuda {
  size_t max_alloc = ~(size_t)0;                   // larger requests fail ...
  cudaError_t alloc_error = cudaErrorMemoryAllocation;   // ... with this
  bool capturing = false;
};
extern FakeCuda fake_cuda;

template <typename T>
inline cudaError_t fake_malloc(T** p, size_t n) {
  if (n > fake_cuda.max_alloc) {
    *p = nullptr;
    return fake_cuda.alloc_error;
  }
  *p = static_cast<T*>(calloc(n + 1, 1));
  return cudaSuccess;
}
inline cudaError_t fake_free(void* p) {
  free(p);
  return cudaSuccess;
}
inline cudaError_t fake_memcpy(void* d, const void* s, size_t n, cudaMemcpyKind, cudaStream_t) {
  memcpy(d, s, n);
  return cudaSuccess;
}
inline cudaError_t fake_memset(void* d, int c, size_t n, cudaStream_t) {
  memset(d, c, n);
  return cudaSuccess;
}
inline cudaError_t fake_success() { return cudaSuccess; }
inline cudaError_t fake_sync(cudaStream_t) { return cudaSuccess; }
inline cudaError_t fake_attribute(int* v, cudaDeviceAttr, int) {
  *v = 152;
  return cudaSuccess;
}
inline cudaError_t fake_capturing(cudaStream_t, cudaStreamCaptureStatus* s) {
  *s = fake_cuda.capturing ? cudaStreamCaptureStatusActive : cudaStreamCaptureStatusNone;
  return cudaSuccess;
}

inline cudaError_t fake_stream(cudaStream_t* s, unsigned) {
  *s = nullptr;
  return cudaSuccess;
}
inline cudaError_t fake_event(cudaEvent_t* e, unsigned) {
  *e = nullptr;
  return cudaSuccess;
}

#define cudaMalloc fake_malloc
#define cudaStreamCreateWithFlags fake_stream
#define cudaEventCreateWithFlags fake_event
#define cudaFree fake_free
#define cudaMemcpyAsync fake_memcpy
#define cudaMemsetAsync fake_memset
#define cudaGetLastError fake_success
#define cudaStreamSynchronize fake_sync
#define cudaDeviceGetAttribute fake_attribute
#define cudaStreamIsCapturing fake_capturing
