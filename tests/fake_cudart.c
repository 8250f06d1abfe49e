/* A CUDA runtime without a GPU, for tests of the library's host code: device memory is host
 * memory, copies are copies, kernels are counted and do nothing, and the n-th launch can be
 * made to fail.  Loaded with LD_PRELOAD before libqcsim.so, whose calls then end here. */
#include <stdio.h>
#include <stdlib.h>
#include <string.h>

#include <cuda_runtime_api.h>

#define API __attribute__((visibility("default")))
enum { kOps = 1 << 20, kNames = 4096 };

/* what the test reads and sets */
API char fake_log[kOps];      /* one letter per operation: L launch, S stream or device wait, W wait for an event
                                * with nothing launched after it, w the same with launches after it */
API int fake_ops = 0;
API int fake_launches = 0;
API int fake_fail_launch = 0; /* this launch (counted from 1) fails */
API long long fake_device_bytes = 0;
API int fake_sms = 2;
API const char* fake_last_kernel = "";
API int fake_count(const char* kernel); /* launches of kernels whose name contains `kernel` */

static const void* entry[kNames];
static const char* name[kNames];
static int launches_of[kNames];
static int names = 0;

static void op(char c) {
  if (fake_ops < kOps - 1) fake_log[fake_ops++] = c;
}
int fake_count(const char* kernel) {
  int n = 0;
  for (int k = 0; k < names; ++k)
    if (strstr(name[k], kernel)) n += launches_of[k];
  return n;
}
static cudaError_t launch(const void* f) {
  op('L');
  if (++fake_launches == fake_fail_launch) return cudaErrorLaunchOutOfResources;
  for (int k = 0; k < names; ++k)
    if (entry[k] == f) {
      ++launches_of[k];
      fake_last_kernel = name[k];
    }
  return cudaSuccess;
}
static cudaError_t last = cudaSuccess;

/* the compiler's registration and launch calls */
API void** __cudaRegisterFatBinary(void* b) { (void)b; static void* h; return &h; }
API void __cudaRegisterFatBinaryEnd(void** h) { (void)h; }
API void __cudaUnregisterFatBinary(void** h) { (void)h; }
API void __cudaRegisterVar(void** h, char* var, char* dev, const char* n, int ext, size_t size, int c, int g) {
  (void)h; (void)var; (void)dev; (void)n; (void)ext; (void)size; (void)c; (void)g;
}
API void __cudaRegisterFunction(void** h, const char* host, char* dev, const char* n, int limit, void* a, void* b, void* c, void* d, int* w) {
  (void)h; (void)dev; (void)limit; (void)a; (void)b; (void)c; (void)d; (void)w;
  if (names < kNames) {
    entry[names] = host;
    name[names++] = strdup(n);
  }
}
API unsigned __cudaPushCallConfiguration(dim3 g, dim3 b, size_t s, void* st) { (void)g; (void)b; (void)s; (void)st; return 0; }
API cudaError_t __cudaPopCallConfiguration(dim3* g, dim3* b, size_t* s, void* st) {
  g->x = g->y = g->z = b->x = b->y = b->z = 1;
  *s = 0;
  *(void**)st = NULL;
  return cudaSuccess;
}
API cudaError_t __cudaGetKernel(cudaKernel_t* k, const void* f) { *k = (cudaKernel_t)f; return cudaSuccess; }
API cudaError_t __cudaLaunchKernel(cudaKernel_t k, dim3 g, dim3 b, void** a, size_t s, cudaStream_t st) {
  (void)g; (void)b; (void)a; (void)s; (void)st;
  const cudaError_t e = launch((const void*)k);
  if (e != cudaSuccess) last = e;
  return e;
}
API cudaError_t cudaLaunchCooperativeKernel(const void* f, dim3 g, dim3 b, void** a, size_t s, cudaStream_t st) {
  (void)g; (void)b; (void)a; (void)s; (void)st;
  return launch(f);
}

/* memory: every device allocation carries its size in front of it */
API cudaError_t cudaMalloc(void** p, size_t n) {
  char* q = (char*)calloc(1, n + 256);
  if (!q) return cudaErrorMemoryAllocation;
  *(size_t*)q = n;
  fake_device_bytes += (long long)n;
  *p = q + 256;
  return cudaSuccess;
}
API cudaError_t cudaFree(void* p) {
  if (!p) return cudaSuccess;
  fake_device_bytes -= (long long)*(size_t*)((char*)p - 256);
  free((char*)p - 256);
  return cudaSuccess;
}
API cudaError_t cudaMallocAsync(void** p, size_t n, cudaStream_t st) { (void)st; return cudaMalloc(p, n); }
API cudaError_t cudaFreeAsync(void* p, cudaStream_t st) { (void)st; return cudaFree(p); }
API cudaError_t cudaHostAlloc(void** p, size_t n, unsigned f) { (void)f; *p = calloc(1, n); return *p ? cudaSuccess : cudaErrorMemoryAllocation; }
API cudaError_t cudaMallocHost(void** p, size_t n) { return cudaHostAlloc(p, n, 0); }
API cudaError_t cudaFreeHost(void* p) { free(p); return cudaSuccess; }
API cudaError_t cudaMemcpy(void* d, const void* s, size_t n, enum cudaMemcpyKind k) { (void)k; memmove(d, s, n); return cudaSuccess; }
API cudaError_t cudaMemcpyAsync(void* d, const void* s, size_t n, enum cudaMemcpyKind k, cudaStream_t st) { (void)st; return cudaMemcpy(d, s, n, k); }
API cudaError_t cudaMemset(void* d, int v, size_t n) { memset(d, v, n); return cudaSuccess; }
API cudaError_t cudaMemsetAsync(void* d, int v, size_t n, cudaStream_t st) { (void)st; return cudaMemset(d, v, n); }
API cudaError_t cudaMemGetInfo(size_t* f, size_t* t) { *f = *t = (size_t)1 << 30; return cudaSuccess; }
API cudaError_t cudaGetSymbolAddress(void** p, const void* s) { (void)s; static char room[16]; *p = room; return cudaSuccess; }

/* devices, streams, events, graphs */
API cudaError_t cudaGetDevice(int* d) { *d = 0; return cudaSuccess; }
API cudaError_t cudaDeviceGetAttribute(int* v, enum cudaDeviceAttr a, int d) { (void)a; (void)d; *v = fake_sms; return cudaSuccess; }
API cudaError_t cudaDeviceSynchronize(void) { op('S'); return cudaSuccess; }
API cudaError_t cudaFuncSetAttribute(const void* f, enum cudaFuncAttribute a, int v) { (void)f; (void)a; (void)v; return cudaSuccess; }
API cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int* n, const void* f, int t, size_t s, unsigned fl) {
  (void)f; (void)t; (void)s; (void)fl;
  *n = 1;
  return cudaSuccess;
}
API cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessor(int* n, const void* f, int t, size_t s) {
  return cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(n, f, t, s, 0);
}
API cudaError_t cudaGetLastError(void) { const cudaError_t e = last; last = cudaSuccess; return e; }
API const char* cudaGetErrorString(cudaError_t e) { (void)e; return "fake"; }
API cudaError_t cudaStreamCreateWithFlags(cudaStream_t* s, unsigned f) { (void)f; *s = (cudaStream_t)malloc(1); return cudaSuccess; }
API cudaError_t cudaStreamDestroy(cudaStream_t s) { free(s); return cudaSuccess; }
API cudaError_t cudaStreamSynchronize(cudaStream_t s) { (void)s; op('S'); return cudaSuccess; }
API cudaError_t cudaStreamWaitEvent(cudaStream_t s, cudaEvent_t e, unsigned f) { (void)s; (void)e; (void)f; return cudaSuccess; }
API cudaError_t cudaStreamBeginCapture(cudaStream_t s, enum cudaStreamCaptureMode m) { (void)s; (void)m; return cudaSuccess; }
API cudaError_t cudaStreamEndCapture(cudaStream_t s, cudaGraph_t* g) { (void)s; *g = (cudaGraph_t)malloc(1); return cudaSuccess; }
API cudaError_t cudaEventCreateWithFlags(cudaEvent_t* e, unsigned f) { (void)f; *e = (cudaEvent_t)calloc(1, sizeof(int)); return cudaSuccess; }
API cudaError_t cudaEventCreate(cudaEvent_t* e) { return cudaEventCreateWithFlags(e, 0); }
API cudaError_t cudaEventDestroy(cudaEvent_t e) { free(e); return cudaSuccess; }
API cudaError_t cudaEventRecord(cudaEvent_t e, cudaStream_t s) { (void)s; *(int*)e = fake_launches; return cudaSuccess; }
API cudaError_t cudaEventSynchronize(cudaEvent_t e) { op(*(int*)e == fake_launches ? 'W' : 'w'); return cudaSuccess; }
API cudaError_t cudaEventElapsedTime(float* ms, cudaEvent_t a, cudaEvent_t b) { (void)a; (void)b; *ms = 1.0f; return cudaSuccess; }
API cudaError_t cudaGraphInstantiate(cudaGraphExec_t* x, cudaGraph_t g, unsigned long long f) { (void)g; (void)f; *x = (cudaGraphExec_t)malloc(1); return cudaSuccess; }
API cudaError_t cudaGraphLaunch(cudaGraphExec_t x, cudaStream_t s) { (void)x; (void)s; return cudaSuccess; }
API cudaError_t cudaGraphDestroy(cudaGraph_t g) { free(g); return cudaSuccess; }
API cudaError_t cudaGraphExecDestroy(cudaGraphExec_t x) { free(x); return cudaSuccess; }
