/* A stand-in for the CUDA runtime calls of the library's host code, preloaded
 * by test_plan_memory.py: "device" memory is host memory up to a limit, copies
 * and clears check that they stay inside live allocations, kernels do nothing,
 * and every event interval takes a millisecond. */
#include <cuda_runtime_api.h>
#include <stdlib.h>
#include <string.h>

#define MAX_LIVE 4096
static struct { char* p; size_t n; int device; } live[MAX_LIVE];
static size_t used, limit = (size_t)-1;
static int outside, launches;

void fake_limit(size_t bytes) { limit = bytes; }
size_t fake_used(void) { return used; }
int fake_outside(void) { return outside; }
int fake_launches(void) { return launches; }

static int inside(const void* p, size_t n) {
  for (int i = 0; i < MAX_LIVE; ++i)
    if (live[i].p && (const char*)p >= live[i].p && (const char*)p + n <= live[i].p + live[i].n) return 1;
  return 0;
}
cudaError_t cudaMalloc(void** p, size_t n) {
  if (used + n > limit) return cudaErrorMemoryAllocation;
  for (int i = 0; i < MAX_LIVE; ++i)
    if (!live[i].p) {
      live[i].p = aligned_alloc(256, (n + 256) / 256 * 256);
      memset(live[i].p, 0, n);
      live[i].n = n;
      used += n;
      *p = live[i].p;
      return cudaSuccess;
    }
  return cudaErrorMemoryAllocation;
}
cudaError_t cudaFree(void* p) {
  for (int i = 0; p && i < MAX_LIVE; ++i)
    if (live[i].p == p) {
      used -= live[i].n;
      free(live[i].p);
      live[i].p = 0;
      return cudaSuccess;
    }
  return p ? cudaErrorInvalidValue : cudaSuccess;
}
cudaError_t cudaMemsetAsync(void* p, int v, size_t n, cudaStream_t s) {
  (void)s;
  if (!inside(p, n)) {
    ++outside;
    return cudaErrorInvalidValue;
  }
  memset(p, v, n);
  return cudaSuccess;
}
cudaError_t cudaMemcpyAsync(void* d, const void* s, size_t n, enum cudaMemcpyKind k, cudaStream_t st) {
  (void)st;
  if (((k == cudaMemcpyHostToDevice || k == cudaMemcpyDeviceToDevice) && !inside(d, n)) ||
      ((k == cudaMemcpyDeviceToHost || k == cudaMemcpyDeviceToDevice) && !inside(s, n))) {
    ++outside;
    return cudaErrorInvalidValue;
  }
  memcpy(d, s, n);
  return cudaSuccess;
}
cudaError_t __cudaGetKernel(cudaKernel_t* k, const void* f) { *k = (cudaKernel_t)f; return cudaSuccess; }
cudaError_t __cudaLaunchKernel(cudaKernel_t k, dim3 g, dim3 b, void** a, size_t m, cudaStream_t s) {
  (void)k, (void)g, (void)b, (void)a, (void)m, (void)s;
  ++launches;
  return cudaSuccess;
}
cudaError_t cudaGetLastError(void) { return cudaSuccess; }
cudaError_t cudaGetDevice(int* d) { *d = 0; return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int* v, enum cudaDeviceAttr a, int d) { (void)a, (void)d; *v = 152; return cudaSuccess; }
cudaError_t cudaGetDeviceProperties(struct cudaDeviceProp* p, int d) { (void)d; memset(p, 0, sizeof *p); return cudaSuccess; }
cudaError_t cudaDeviceSynchronize(void) { return cudaSuccess; }
cudaError_t cudaFuncGetAttributes(struct cudaFuncAttributes* a, const void* f) { (void)f; memset(a, 0, sizeof *a); return cudaSuccess; }
cudaError_t cudaFuncSetAttribute(const void* f, enum cudaFuncAttribute a, int v) { (void)f, (void)a, (void)v; return cudaSuccess; }
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessor(int* n, const void* f, int t, size_t m) { (void)f, (void)t, (void)m; *n = 2; return cudaSuccess; }
static int token;
cudaError_t cudaStreamCreateWithFlags(cudaStream_t* s, unsigned f) { (void)f; *s = (cudaStream_t)&token; return cudaSuccess; }
cudaError_t cudaStreamDestroy(cudaStream_t s) { (void)s; return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t s) { (void)s; return cudaSuccess; }
cudaError_t cudaStreamWaitEvent(cudaStream_t s, cudaEvent_t e, unsigned f) { (void)s, (void)e, (void)f; return cudaSuccess; }
cudaError_t cudaStreamBeginCapture(cudaStream_t s, enum cudaStreamCaptureMode m) { (void)s, (void)m; return cudaSuccess; }
cudaError_t cudaStreamEndCapture(cudaStream_t s, cudaGraph_t* g) { (void)s; *g = (cudaGraph_t)&token; return cudaSuccess; }
cudaError_t cudaGraphInstantiate(cudaGraphExec_t* e, cudaGraph_t g, unsigned long long f) { (void)g, (void)f; *e = (cudaGraphExec_t)&token; return cudaSuccess; }
cudaError_t cudaGraphLaunch(cudaGraphExec_t e, cudaStream_t s) { (void)e, (void)s; return cudaSuccess; }
cudaError_t cudaGraphDestroy(cudaGraph_t g) { (void)g; return cudaSuccess; }
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t e) { (void)e; return cudaSuccess; }
cudaError_t cudaEventCreate(cudaEvent_t* e) { *e = (cudaEvent_t)&token; return cudaSuccess; }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t* e, unsigned f) { (void)f; *e = (cudaEvent_t)&token; return cudaSuccess; }
cudaError_t cudaEventDestroy(cudaEvent_t e) { (void)e; return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t e, cudaStream_t s) { (void)e, (void)s; return cudaSuccess; }
cudaError_t cudaEventRecordWithFlags(cudaEvent_t e, cudaStream_t s, unsigned f) { (void)e, (void)s, (void)f; return cudaSuccess; }
cudaError_t cudaEventSynchronize(cudaEvent_t e) { (void)e; return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float* ms, cudaEvent_t a, cudaEvent_t b) { (void)a, (void)b; *ms = 1.0f; return cudaSuccess; }
