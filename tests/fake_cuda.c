/* A stand-in for the CUDA runtime and cuSOLVER calls that libxs makes, preloaded by
 * tests of its host side (fake_cuda.py): two devices whose memory is counted and
 * limited, launches that do nothing but fail as real ones do when a kernel asks for
 * more shared memory than was allowed on the current device.  Device memory is zeroed
 * host memory. */
#define _GNU_SOURCE
#include <cuda.h>
#include <cuda_runtime_api.h>
#include <pthread.h>
#include <stdint.h>
#include <stdlib.h>
#include <string.h>
#include <sys/mman.h>

#define MAX_BLOCKS 65536
#define MAX_ATTR 1024

static pthread_mutex_t mu = PTHREAD_MUTEX_INITIALIZER;
static struct { char* p; size_t n; int dev; } blocks[MAX_BLOCKS];
static int nblocks;
static size_t capacity[2] = {(size_t)1 << 40, (size_t)1 << 40}, used[2], peak[2];
static struct { const void* f; size_t n[2]; } attrs[MAX_ATTR];
static int nattrs;
static long long pending;   /* launches since the device was last waited for */
static long long fail_after = -1, fail_times;
static struct { const void* f; const char* name; long long n; } kernels[MAX_ATTR];
static int nkernels;
static __thread int cur;
static __thread cudaError_t last;
static __thread struct { dim3 g, b; size_t smem; void* s; } conf;

/* what the tests look at */
void fake_set_capacity(int dev, size_t bytes) { capacity[dev] = bytes; }
size_t fake_used(int dev) { return used[dev]; }
size_t fake_peak(int dev) { return peak[dev]; }
void fake_reset_peak(int dev) { peak[dev] = used[dev]; }
long long fake_pending(void) { return pending; }
/* after `after` more allocations the next `times` fail */
void fake_fail(long long after, long long times) { fail_after = after; fail_times = times; }
/* launches of the kernels whose names contain `part` */
long long fake_launched(const char* part) {
  long long n = 0;
  for (int i = 0; i < nkernels; ++i)
    if (strstr(kernels[i].name, part)) n += kernels[i].n;
  return n;
}
/* sets every word of the device blocks of n bytes */
void fake_fill(size_t n, int word) {
  for (int i = 0; i < nblocks; ++i)
    if (blocks[i].n == n)
      for (size_t k = 0; k < n / 4; ++k) ((int*)blocks[i].p)[k] = word;
}

static cudaError_t fail(cudaError_t e) { return last = e; }

cudaError_t cudaMalloc(void** p, size_t n) {
  pthread_mutex_lock(&mu);
  cudaError_t e = cudaSuccess;
  int planned = 0;
  if (fail_after == 0 && fail_times > 0) { planned = 1; --fail_times; }
  else if (fail_after > 0) --fail_after;
  if (planned || nblocks == MAX_BLOCKS || used[cur] + n > capacity[cur]) e = cudaErrorMemoryAllocation;
  else {
    char* q = mmap(NULL, n, PROT_READ | PROT_WRITE, MAP_PRIVATE | MAP_ANONYMOUS | MAP_NORESERVE, -1, 0);
    if (q == MAP_FAILED) e = cudaErrorMemoryAllocation;
    else {
      blocks[nblocks].p = q; blocks[nblocks].n = n; blocks[nblocks].dev = cur; ++nblocks;
      used[cur] += n;
      if (used[cur] > peak[cur]) peak[cur] = used[cur];
      *p = q;
    }
  }
  pthread_mutex_unlock(&mu);
  return e ? fail(e) : e;
}
cudaError_t cudaFree(void* p) {
  if (!p) return cudaSuccess;
  pthread_mutex_lock(&mu);
  cudaError_t e = cudaErrorInvalidValue;
  pending = 0;
  for (int i = nblocks - 1; i >= 0; --i)
    if (blocks[i].p == p) {
      munmap(p, blocks[i].n);
      used[blocks[i].dev] -= blocks[i].n;
      blocks[i] = blocks[--nblocks];
      e = cudaSuccess;
      break;
    }
  pthread_mutex_unlock(&mu);
  return e ? fail(e) : e;
}
cudaError_t cudaHostAlloc(void** p, size_t n, unsigned f) { (void)f; *p = calloc(1, n); return *p ? cudaSuccess : fail(cudaErrorMemoryAllocation); }
cudaError_t cudaFreeHost(void* p) { free(p); return cudaSuccess; }
cudaError_t cudaMemGetInfo(size_t* f, size_t* t) {
  *t = capacity[cur];
  *f = capacity[cur] > used[cur] ? capacity[cur] - used[cur] : 0;
  return cudaSuccess;
}
static int find(const void* p) {
  for (int i = 0; i < nblocks; ++i)
    if ((const char*)p >= blocks[i].p && (const char*)p < blocks[i].p + blocks[i].n) return i;
  return -1;
}
cudaError_t cudaPointerGetAttributes(struct cudaPointerAttributes* a, const void* p) {
  memset(a, 0, sizeof(*a));
  pthread_mutex_lock(&mu);
  const int i = find(p);
  a->type = i < 0 ? cudaMemoryTypeUnregistered : cudaMemoryTypeDevice;
  a->device = i < 0 ? 0 : blocks[i].dev;
  pthread_mutex_unlock(&mu);
  return cudaSuccess;
}
static CUresult address_range(CUdeviceptr* base, size_t* n, CUdeviceptr p) {
  pthread_mutex_lock(&mu);
  const int i = find((const void*)(uintptr_t)p);
  if (i >= 0) { *base = (CUdeviceptr)(uintptr_t)blocks[i].p; *n = blocks[i].n; }
  pthread_mutex_unlock(&mu);
  return i < 0 ? CUDA_ERROR_INVALID_VALUE : CUDA_SUCCESS;
}
static CUresult encode_tiled(CUtensorMap* m, CUtensorMapDataType t, cuuint32_t rank, void* p) {
  (void)m; (void)t; (void)rank;
  pthread_mutex_lock(&mu);
  const int i = find(p);
  pthread_mutex_unlock(&mu);
  return i < 0 || blocks[i].dev != cur ? CUDA_ERROR_INVALID_VALUE : CUDA_SUCCESS;
}
cudaError_t cudaGetDriverEntryPointByVersion(const char* s, void** f, unsigned v, unsigned long long fl, enum cudaDriverEntryPointQueryResult* q) {
  (void)v; (void)fl;
  *f = !strcmp(s, "cuMemGetAddressRange") ? (void*)address_range : !strcmp(s, "cuTensorMapEncodeTiled") ? (void*)encode_tiled : NULL;
  *q = *f ? cudaDriverEntryPointSuccess : cudaDriverEntryPointSymbolNotFound;
  return cudaSuccess;
}
cudaError_t cudaMemcpyAsync(void* d, const void* s, size_t n, enum cudaMemcpyKind k, cudaStream_t st) { (void)k; (void)st; memmove(d, s, n); return cudaSuccess; }
cudaError_t cudaMemcpy2DAsync(void* d, size_t dp, const void* s, size_t sp, size_t w, size_t h, enum cudaMemcpyKind k, cudaStream_t st) {
  (void)k; (void)st;
  for (size_t i = 0; i < h; ++i) memmove((char*)d + i * dp, (const char*)s + i * sp, w);
  return cudaSuccess;
}
cudaError_t cudaMemsetAsync(void* d, int v, size_t n, cudaStream_t st) { (void)st; memset(d, v, n); return cudaSuccess; }

cudaError_t cudaGetDeviceCount(int* n) { *n = 2; return cudaSuccess; }
cudaError_t cudaGetDevice(int* d) { *d = cur; return cudaSuccess; }
cudaError_t cudaSetDevice(int d) { if (d < 0 || d > 1) return fail(cudaErrorInvalidDevice); cur = d; return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int* v, enum cudaDeviceAttr a, int d) { (void)d; *v = a == cudaDevAttrMultiProcessorCount ? 152 : 0; return cudaSuccess; }
cudaError_t cudaGetLastError(void) { const cudaError_t e = last; last = cudaSuccess; return e; }
const char* cudaGetErrorString(cudaError_t e) {
  return e == cudaErrorMemoryAllocation ? "out of memory" : e == cudaErrorInvalidValue ? "invalid argument" : "error";
}

cudaError_t cudaFuncSetAttribute(const void* f, enum cudaFuncAttribute a, int v) {
  if (a != cudaFuncAttributeMaxDynamicSharedMemorySize) return cudaSuccess;
  pthread_mutex_lock(&mu);
  int i = 0;
  while (i < nattrs && attrs[i].f != f) ++i;
  if (i == nattrs) { attrs[i].f = f; ++nattrs; }
  attrs[i].n[cur] = (size_t)v;
  pthread_mutex_unlock(&mu);
  return cudaSuccess;
}
static cudaError_t launch(const void* f, size_t smem) {
  size_t allowed = 48 << 10;
  pthread_mutex_lock(&mu);
  for (int i = 0; i < nattrs; ++i)
    if (attrs[i].f == f && attrs[i].n[cur] > allowed) allowed = attrs[i].n[cur];
  ++pending;
  for (int i = 0; i < nkernels; ++i)
    if (kernels[i].f == f) ++kernels[i].n;
  pthread_mutex_unlock(&mu);
  return smem > allowed ? fail(cudaErrorInvalidValue) : cudaSuccess;
}
cudaError_t __cudaGetKernel(cudaKernel_t* k, const void* f) { *k = (cudaKernel_t)f; return cudaSuccess; }
cudaError_t __cudaLaunchKernel(cudaKernel_t k, dim3 g, dim3 b, void** a, size_t smem, cudaStream_t s) {
  (void)g; (void)b; (void)a; (void)s;
  return launch((const void*)k, smem);
}
unsigned __cudaPushCallConfiguration(dim3 g, dim3 b, size_t smem, void* s) { conf.g = g; conf.b = b; conf.smem = smem; conf.s = s; return 0; }
cudaError_t __cudaPopCallConfiguration(dim3* g, dim3* b, size_t* smem, void* s) {
  *g = conf.g; *b = conf.b; *smem = conf.smem; *(void**)s = conf.s;
  return cudaSuccess;
}
void** __cudaRegisterFatBinary(void* f) { (void)f; static void* h; return &h; }
void __cudaRegisterFatBinaryEnd(void** h) { (void)h; }
void __cudaUnregisterFatBinary(void** h) { (void)h; }
void __cudaRegisterFunction(void** h, const char* f, char* d, const char* n, int t, void* a, void* b, void* c, void* e, int* w) {
  (void)h; (void)d; (void)t; (void)a; (void)b; (void)c; (void)e; (void)w;
  if (nkernels < MAX_ATTR) { kernels[nkernels].f = f; kernels[nkernels].name = n; ++nkernels; }
}
void __cudaRegisterVar(void** h, char* v, char* d, const char* n, int e, size_t s, int c, int g) {
  (void)h; (void)v; (void)d; (void)n; (void)e; (void)s; (void)c; (void)g;
}

cudaError_t cudaStreamCreateWithFlags(cudaStream_t* s, unsigned f) { (void)f; static char h; *s = (cudaStream_t)&h; return cudaSuccess; }
cudaError_t cudaStreamDestroy(cudaStream_t s) { (void)s; return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t s) { (void)s; pending = 0; return cudaSuccess; }
cudaError_t cudaStreamIsCapturing(cudaStream_t s, enum cudaStreamCaptureStatus* c) { (void)s; *c = cudaStreamCaptureStatusNone; return cudaSuccess; }
cudaError_t cudaStreamBeginCapture(cudaStream_t s, enum cudaStreamCaptureMode m) { (void)s; (void)m; return cudaSuccess; }
cudaError_t cudaStreamEndCapture(cudaStream_t s, cudaGraph_t* g) { (void)s; static char h; *g = (cudaGraph_t)&h; return cudaSuccess; }
cudaError_t cudaGraphInstantiate(cudaGraphExec_t* e, cudaGraph_t g, unsigned long long f) { (void)g; (void)f; static char h; *e = (cudaGraphExec_t)&h; return cudaSuccess; }
cudaError_t cudaGraphLaunch(cudaGraphExec_t e, cudaStream_t s) { (void)e; (void)s; return cudaSuccess; }
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t e) { (void)e; return cudaSuccess; }
cudaError_t cudaGraphDestroy(cudaGraph_t g) { (void)g; return cudaSuccess; }
cudaError_t cudaEventCreate(cudaEvent_t* e) { static char h; *e = (cudaEvent_t)&h; return cudaSuccess; }
cudaError_t cudaEventDestroy(cudaEvent_t e) { (void)e; return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t e, cudaStream_t s) { (void)e; (void)s; return cudaSuccess; }
cudaError_t cudaEventSynchronize(cudaEvent_t e) { (void)e; pending = 0; return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float* ms, cudaEvent_t a, cudaEvent_t b) { (void)a; (void)b; *ms = 1.0f; return cudaSuccess; }

int cusolverDnCreate(void** h) { static char x; *h = &x; return 0; }
int cusolverDnDestroy(void* h) { (void)h; return 0; }
int cusolverDnSetStream(void* h, void* s) { (void)h; (void)s; return 0; }
int cusolverDnDsyevd_bufferSize(void* h, int j, int u, int n, const double* A, int lda, const double* W, int* l) {
  (void)h; (void)j; (void)u; (void)A; (void)lda; (void)W;
  *l = n;
  return 0;
}
/* eigenvalues 0, 1, 2, ...: a gap between every two orbitals */
int cusolverDnDsyevd(void* h, int j, int u, int n, double* A, int lda, double* W, double* w, int l, int* info) {
  (void)h; (void)j; (void)u; (void)A; (void)lda; (void)w; (void)l;
  for (int i = 0; i < n; ++i) W[i] = i;
  *info = 0;
  return 0;
}
