/* A CUDA runtime and cuFFT without a device, preloaded in front of the real ones by
 * tests of the library's host side: memory is host memory, launches and transforms do
 * nothing, streams, events and graphs are tokens.  fake_fail_malloc(k) makes the k-th
 * following cudaMalloc fail; fake_captures() counts the graphs instantiated. */
#include <cuda_runtime_api.h>
#include <cufft.h>
#include <stdlib.h>
#include <string.h>

static int fail_at = 0, captures = 0;
static char token;

void fake_fail_malloc(int k) { fail_at = k; }
int fake_captures(void) { return captures; }

cudaError_t cudaMalloc(void **p, size_t n) {
  if (fail_at > 0 && --fail_at == 0) return cudaErrorMemoryAllocation;
  *p = calloc(1, n ? n : 1);
  return cudaSuccess;
}
cudaError_t cudaFree(void *p) { free(p); return cudaSuccess; }
cudaError_t cudaMallocHost(void **p, size_t n) { *p = calloc(1, n ? n : 1); return cudaSuccess; }
cudaError_t cudaFreeHost(void *p) { free(p); return cudaSuccess; }
cudaError_t cudaMemcpy(void *d, const void *s, size_t n, enum cudaMemcpyKind k) { memmove(d, s, n); return cudaSuccess; }
cudaError_t cudaMemcpyAsync(void *d, const void *s, size_t n, enum cudaMemcpyKind k, cudaStream_t t) {
  memmove(d, s, n);
  return cudaSuccess;
}
cudaError_t cudaMemset(void *d, int v, size_t n) { memset(d, v, n); return cudaSuccess; }
cudaError_t cudaMemsetAsync(void *d, int v, size_t n, cudaStream_t t) { memset(d, v, n); return cudaSuccess; }
cudaError_t cudaPointerGetAttributes(struct cudaPointerAttributes *a, const void *p) {
  memset(a, 0, sizeof *a); /* host memory */
  return cudaSuccess;
}

cudaError_t cudaGetDevice(int *d) { *d = 0; return cudaSuccess; }
cudaError_t cudaSetDevice(int d) { return cudaSuccess; }
cudaError_t cudaGetDeviceCount(int *n) { *n = 1; return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int *v, enum cudaDeviceAttr a, int d) {
  *v = a == cudaDevAttrMultiProcessorCount ? 152 : a == cudaDevAttrMaxSharedMemoryPerBlockOptin ? 232448 : 0;
  return cudaSuccess;
}
cudaError_t cudaDeviceSynchronize(void) { return cudaSuccess; }
cudaError_t cudaGetLastError(void) { return cudaSuccess; }
const char *cudaGetErrorString(cudaError_t e) { return "fake"; }
cudaError_t cudaFuncSetAttribute(const void *f, enum cudaFuncAttribute a, int v) { return cudaSuccess; }
cudaError_t cudaFuncGetAttributes(struct cudaFuncAttributes *a, const void *f) {
  memset(a, 0, sizeof *a);
  return cudaSuccess;
}
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int *n, const void *f, int t, size_t s, unsigned g) {
  *n = 2;
  return cudaSuccess;
}
cudaError_t __cudaGetKernel(cudaKernel_t *k, const void *f) { *k = (cudaKernel_t)&token; return cudaSuccess; }
cudaError_t __cudaLaunchKernel(void) { return cudaSuccess; } /* whatever its arguments */

cudaError_t cudaStreamCreateWithFlags(cudaStream_t *s, unsigned f) { *s = (cudaStream_t)&token; return cudaSuccess; }
cudaError_t cudaStreamDestroy(cudaStream_t s) { return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t s) { return cudaSuccess; }
cudaError_t cudaEventCreate(cudaEvent_t *e) { *e = (cudaEvent_t)&token; return cudaSuccess; }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t *e, unsigned f) { *e = (cudaEvent_t)&token; return cudaSuccess; }
cudaError_t cudaEventDestroy(cudaEvent_t e) { return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t e, cudaStream_t s) { return cudaSuccess; }
cudaError_t cudaEventSynchronize(cudaEvent_t e) { return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float *ms, cudaEvent_t a, cudaEvent_t b) { *ms = 1.f; return cudaSuccess; }

cudaError_t cudaStreamBeginCapture(cudaStream_t s, enum cudaStreamCaptureMode m) { return cudaSuccess; }
cudaError_t cudaStreamBeginCaptureToGraph(cudaStream_t s, cudaGraph_t g, const cudaGraphNode_t *d,
                                          const cudaGraphEdgeData *e, size_t n, enum cudaStreamCaptureMode m) {
  return cudaSuccess;
}
cudaError_t cudaStreamEndCapture(cudaStream_t s, cudaGraph_t *g) { *g = (cudaGraph_t)&token; return cudaSuccess; }
cudaError_t cudaStreamIsCapturing(cudaStream_t s, enum cudaStreamCaptureStatus *st) {
  *st = cudaStreamCaptureStatusNone;
  return cudaSuccess;
}
cudaError_t cudaStreamGetCaptureInfo(cudaStream_t s, enum cudaStreamCaptureStatus *st, unsigned long long *id,
                                     cudaGraph_t *g, const cudaGraphNode_t **d, const cudaGraphEdgeData **e, size_t *n) {
  *st = cudaStreamCaptureStatusActive;
  if (id) *id = 1;
  if (g) *g = (cudaGraph_t)&token;
  if (d) *d = NULL;
  if (e) *e = NULL;
  if (n) *n = 0;
  return cudaSuccess;
}
cudaError_t cudaStreamUpdateCaptureDependencies(cudaStream_t s, cudaGraphNode_t *d, const cudaGraphEdgeData *e, size_t n,
                                                unsigned f) {
  return cudaSuccess;
}
cudaError_t cudaGraphConditionalHandleCreate(cudaGraphConditionalHandle *h, cudaGraph_t g, unsigned v, unsigned f) {
  *h = 1;
  return cudaSuccess;
}
cudaError_t cudaGraphAddNode(cudaGraphNode_t *node, cudaGraph_t g, const cudaGraphNode_t *d, const cudaGraphEdgeData *e,
                             size_t n, struct cudaGraphNodeParams *p) {
  static cudaGraph_t body = (cudaGraph_t)&token;
  *node = (cudaGraphNode_t)&token;
  p->conditional.phGraph_out = &body;
  return cudaSuccess;
}
cudaError_t cudaGraphInstantiate(cudaGraphExec_t *x, cudaGraph_t g, unsigned long long f) {
  *x = (cudaGraphExec_t)&token;
  ++captures;
  return cudaSuccess;
}
cudaError_t cudaGraphLaunch(cudaGraphExec_t x, cudaStream_t s) { return cudaSuccess; }
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t x) { return cudaSuccess; }
cudaError_t cudaGraphDestroy(cudaGraph_t g) { return cudaSuccess; }

cufftResult cufftCreate(cufftHandle *h) { *h = 1; return CUFFT_SUCCESS; }
cufftResult cufftDestroy(cufftHandle h) { return CUFFT_SUCCESS; }
cufftResult cufftMakePlanMany(cufftHandle h, int r, int *n, int *ie, int is, int id, int *oe, int os, int od, cufftType t,
                              int b, size_t *w) {
  *w = 16;
  return CUFFT_SUCCESS;
}
cufftResult cufftSetAutoAllocation(cufftHandle h, int a) { return CUFFT_SUCCESS; }
cufftResult cufftSetWorkArea(cufftHandle h, void *w) { return CUFFT_SUCCESS; }
cufftResult cufftSetStream(cufftHandle h, cudaStream_t s) { return CUFFT_SUCCESS; }
cufftResult cufftExecR2C(cufftHandle h, cufftReal *i, cufftComplex *o) { return CUFFT_SUCCESS; }
cufftResult cufftExecC2R(cufftHandle h, cufftComplex *i, cufftReal *o) { return CUFFT_SUCCESS; }
cufftResult cufftExecD2Z(cufftHandle h, cufftDoubleReal *i, cufftDoubleComplex *o) { return CUFFT_SUCCESS; }
cufftResult cufftExecZ2D(cufftHandle h, cufftDoubleComplex *i, cufftDoubleReal *o) { return CUFFT_SUCCESS; }
