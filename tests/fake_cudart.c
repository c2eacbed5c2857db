/* Stand-in for the CUDA runtime calls of libsdg, preloaded by tests.
 *
 * SDG_FAKE_DEVICE: no GPU is used.  Memory is host memory, kernels do nothing,
 * cudaSetDevice chooses among any number of devices.  As on a GPU, a launch
 * that asks for more than 48 KB of dynamic shared memory fails unless that
 * much was allowed for the kernel on the current device.
 * SDG_REFUSE_COOPERATIVE: cooperative launches are refused with the error of a
 * grid that does not fit the SMs; every other call goes where
 * SDG_FAKE_DEVICE says, the real runtime without it. */
#define _GNU_SOURCE
#include <cuda_runtime_api.h>
#include <dlfcn.h>
#include <stdlib.h>
#include <string.h>

enum { kCalls = 4096 };

static int dev_, last_, nallowed;
static struct { const void* f; int dev, smem; } allowed_[kCalls];

static int fake(void) { return getenv("SDG_FAKE_DEVICE") != NULL; }
/* the runtime's own function, unless the device is a fake */
#define FORWARD(name, ...)                                                        \
  do {                                                                            \
    if (!fake()) return ((__typeof__(name)*)dlsym(RTLD_NEXT, #name))(__VA_ARGS__); \
  } while (0)

cudaError_t cudaGetLastError(void) {
  const cudaError_t e = (cudaError_t)last_;
  last_ = 0;
  if (e != cudaSuccess) return e;
  FORWARD(cudaGetLastError);
  return cudaSuccess;
}
cudaError_t cudaFuncSetAttribute(const void* f, enum cudaFuncAttribute attr, int value) {
  FORWARD(cudaFuncSetAttribute, f, attr, value);
  if (attr != cudaFuncAttributeMaxDynamicSharedMemorySize || nallowed == kCalls) return cudaErrorInvalidValue;
  allowed_[nallowed].f = f;
  allowed_[nallowed].dev = dev_;
  allowed_[nallowed++].smem = value;
  return cudaSuccess;
}
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t* c, const void* f, void** args) {
  if (getenv("SDG_REFUSE_COOPERATIVE"))
    for (unsigned i = 0; i < c->numAttrs; ++i)
      if (c->attrs[i].id == cudaLaunchAttributeCooperative && c->attrs[i].val.cooperative)
        return (cudaError_t)(last_ = cudaErrorCooperativeLaunchTooLarge);
  FORWARD(cudaLaunchKernelExC, c, f, args);
  if (c->dynamicSmemBytes <= 48 * 1024) return cudaSuccess;
  for (int i = 0; i < nallowed; ++i)
    if (allowed_[i].f == f && allowed_[i].dev == dev_ && (size_t)allowed_[i].smem >= c->dynamicSmemBytes) return cudaSuccess;
  return (cudaError_t)(last_ = cudaErrorInvalidValue);
}
/* not 0: the <<<...>>> that asks does not call its kernel */
unsigned __cudaPushCallConfiguration(dim3 g, dim3 b, size_t smem, struct CUstream_st* s) {
  FORWARD(__cudaPushCallConfiguration, g, b, smem, s);
  return 1;
}
cudaError_t cudaSetDevice(int d) {
  FORWARD(cudaSetDevice, d);
  dev_ = d;
  return cudaSuccess;
}
cudaError_t cudaGetDevice(int* d) {
  FORWARD(cudaGetDevice, d);
  *d = dev_;
  return cudaSuccess;
}
cudaError_t cudaDeviceGetAttribute(int* v, enum cudaDeviceAttr attr, int d) {
  FORWARD(cudaDeviceGetAttribute, v, attr, d);
  *v = attr == cudaDevAttrMultiProcessorCount ? 152 : 0;
  return cudaSuccess;
}
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int* n, const void* f, int threads, size_t smem,
                                                                   unsigned flags) {
  FORWARD(cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags, n, f, threads, smem, flags);
  *n = 2;
  return cudaSuccess;
}
static cudaError_t host_memory(void** p, size_t n) {
  *p = calloc(1, n);
  return *p ? cudaSuccess : cudaErrorMemoryAllocation;
}
cudaError_t cudaMalloc(void** p, size_t n) {
  FORWARD(cudaMalloc, p, n);
  return host_memory(p, n);
}
cudaError_t cudaHostAlloc(void** p, size_t n, unsigned flags) {
  FORWARD(cudaHostAlloc, p, n, flags);
  return host_memory(p, n);
}
cudaError_t cudaFree(void* p) {
  FORWARD(cudaFree, p);
  free(p);
  return cudaSuccess;
}
cudaError_t cudaFreeHost(void* p) {
  FORWARD(cudaFreeHost, p);
  free(p);
  return cudaSuccess;
}
cudaError_t cudaMemcpy(void* d, const void* s, size_t n, enum cudaMemcpyKind kind) {
  FORWARD(cudaMemcpy, d, s, n, kind);
  memmove(d, s, n);
  return cudaSuccess;
}
cudaError_t cudaMemcpyAsync(void* d, const void* s, size_t n, enum cudaMemcpyKind kind, cudaStream_t st) {
  FORWARD(cudaMemcpyAsync, d, s, n, kind, st);
  memmove(d, s, n);
  return cudaSuccess;
}
cudaError_t cudaMemset(void* d, int v, size_t n) {
  FORWARD(cudaMemset, d, v, n);
  memset(d, v, n);
  return cudaSuccess;
}
cudaError_t cudaMemsetAsync(void* d, int v, size_t n, cudaStream_t st) {
  FORWARD(cudaMemsetAsync, d, v, n, st);
  memset(d, v, n);
  return cudaSuccess;
}
cudaError_t cudaDeviceSynchronize(void) {
  FORWARD(cudaDeviceSynchronize);
  return cudaSuccess;
}
cudaError_t cudaStreamSynchronize(cudaStream_t s) {
  FORWARD(cudaStreamSynchronize, s);
  return cudaSuccess;
}
cudaError_t cudaEventCreate(cudaEvent_t* e) {
  FORWARD(cudaEventCreate, e);
  *e = NULL;
  return cudaSuccess;
}
cudaError_t cudaEventDestroy(cudaEvent_t e) {
  FORWARD(cudaEventDestroy, e);
  return cudaSuccess;
}
