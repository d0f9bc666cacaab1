/* A CUDA runtime without a GPU, for tests of the library's host code: preloaded before libcudart, it
 * takes every call the library makes.  Device memory is host memory, copies and clears happen at
 * once, kernels do nothing but call the test's hook (name, arguments).  What a stream still has
 * queued is counted until a call waits for that stream, as on a device: a test can ask what a call
 * left behind, and put values where a kernel would have written them.  Tensor maps (what the TMA
 * copies of a kernel may touch) are refused when they leave their allocation or TMA's alignments.
 */
#include <cuda.h>
#include <cuda_runtime_api.h>
#include <stdint.h>
#include <stdlib.h>
#include <string.h>

#define MAX_STREAMS 64
#define MAX_ALLOCS 65536
#define MAX_KERNELS 4096

static char g_streams[MAX_STREAMS];                /* handles: addresses in this array; [0]: the default stream */
static int g_next = 1;
static long g_pending[MAX_STREAMS], g_total[MAX_STREAMS];
static struct { char* p; size_t n; } g_alloc[MAX_ALLOCS];
static int g_nalloc;
static struct { const void* f; const char* name; } g_kernel[MAX_KERNELS];
static int g_nkernel;
static void (*g_hook)(const char*, void**);

static int slot(cudaStream_t s) {
  const char* p = (const char*)s;
  return (p > g_streams && p < g_streams + MAX_STREAMS) ? (int)(p - g_streams) : 0;
}
static cudaError_t queued(cudaStream_t s) {
  ++g_pending[slot(s)];
  ++g_total[slot(s)];
  return cudaSuccess;
}

/* ---- the test's side ---- */
long fake_pending(void* s) { return g_pending[slot((cudaStream_t)s)]; }   /* queued and not waited for */
long fake_total(void* s) { return g_total[slot((cudaStream_t)s)]; }       /* queued ever */
long fake_pending_all(void) {
  long n = 0;
  for (int k = 0; k < MAX_STREAMS; ++k) n += g_pending[k];
  return n;
}
void fake_on_launch(void (*hook)(const char*, void**)) { g_hook = hook; }

/* ---- memory ---- */
cudaError_t cudaMalloc(void** p, size_t n) {
  *p = aligned_alloc(256, (n + 255) / 256 * 256);
  if (!*p || g_nalloc == MAX_ALLOCS) return cudaErrorMemoryAllocation;
  memset(*p, 0, (n + 255) / 256 * 256);
  g_alloc[g_nalloc].p = (char*)*p;
  g_alloc[g_nalloc++].n = n;
  return cudaSuccess;
}
cudaError_t cudaFree(void* p) {
  for (int k = 0; k < g_nalloc; ++k)
    if (g_alloc[k].p == p) g_alloc[k] = g_alloc[--g_nalloc];
  free(p);
  return cudaSuccess;
}
cudaError_t cudaHostAlloc(void** p, size_t n, unsigned flags) {
  (void)flags;
  *p = calloc(1, n);
  return cudaSuccess;
}
cudaError_t cudaFreeHost(void* p) { free(p); return cudaSuccess; }
cudaError_t cudaMemGetInfo(size_t* fr, size_t* tot) { *fr = *tot = (size_t)1 << 30; return cudaSuccess; }
cudaError_t cudaPointerGetAttributes(struct cudaPointerAttributes* a, const void* p) {
  memset(a, 0, sizeof *a);
  a->type = cudaMemoryTypeUnregistered;
  for (int k = 0; k < g_nalloc; ++k)
    if ((const char*)p >= g_alloc[k].p && (const char*)p < g_alloc[k].p + g_alloc[k].n) a->type = cudaMemoryTypeDevice;
  return cudaSuccess;
}
cudaError_t cudaMemsetAsync(void* p, int v, size_t n, cudaStream_t s) { memset(p, v, n); return queued(s); }
cudaError_t cudaMemset(void* p, int v, size_t n) { return cudaMemsetAsync(p, v, n, 0); }
cudaError_t cudaMemcpyAsync(void* d, const void* s, size_t n, enum cudaMemcpyKind k, cudaStream_t st) {
  (void)k;
  memmove(d, s, n);
  return queued(st);
}
/* to the device it returns once the host array has been read; from the device it waits */
cudaError_t cudaMemcpy(void* d, const void* s, size_t n, enum cudaMemcpyKind k) {
  cudaMemcpyAsync(d, s, n, k, 0);
  if (k == cudaMemcpyDeviceToHost) g_pending[0] = 0;
  return cudaSuccess;
}

/* ---- streams, events, graphs ---- */
cudaError_t cudaStreamCreateWithFlags(cudaStream_t* s, unsigned flags) {
  (void)flags;
  *s = (cudaStream_t)(g_streams + g_next++);
  return cudaSuccess;
}
cudaError_t cudaStreamDestroy(cudaStream_t s) { (void)s; return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t s) { g_pending[slot(s)] = 0; return cudaSuccess; }
cudaError_t cudaDeviceSynchronize(void) { memset(g_pending, 0, sizeof g_pending); return cudaSuccess; }
cudaError_t cudaStreamBeginCapture(cudaStream_t s, enum cudaStreamCaptureMode m) {
  (void)s; (void)m;
  return cudaErrorNotSupported;
}
cudaError_t cudaStreamEndCapture(cudaStream_t s, cudaGraph_t* g) { (void)s; *g = 0; return cudaErrorNotSupported; }
cudaError_t cudaGraphDestroy(cudaGraph_t g) { (void)g; return cudaSuccess; }
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t g) { (void)g; return cudaSuccess; }
cudaError_t cudaGraphExecUpdate(cudaGraphExec_t e, cudaGraph_t g, cudaGraphExecUpdateResultInfo* i) {
  (void)e; (void)g; (void)i;
  return cudaErrorNotSupported;
}
cudaError_t cudaGraphInstantiate(cudaGraphExec_t* e, cudaGraph_t g, unsigned long long f) {
  (void)e; (void)g; (void)f;
  return cudaErrorNotSupported;
}
cudaError_t cudaGraphLaunch(cudaGraphExec_t e, cudaStream_t s) { (void)e; (void)s; return cudaErrorNotSupported; }
cudaError_t cudaEventCreate(cudaEvent_t* e) { *e = (cudaEvent_t)g_streams; return cudaSuccess; }
cudaError_t cudaEventDestroy(cudaEvent_t e) { (void)e; return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t e, cudaStream_t s) { (void)e; (void)s; return cudaSuccess; }
cudaError_t cudaEventSynchronize(cudaEvent_t e) { (void)e; return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float* ms, cudaEvent_t a, cudaEvent_t b) { (void)a; (void)b; *ms = 1.0f; return cudaSuccess; }

/* ---- device ---- */
cudaError_t cudaGetDeviceCount(int* n) { *n = 1; return cudaSuccess; }
cudaError_t cudaGetDevice(int* d) { *d = 0; return cudaSuccess; }
cudaError_t cudaSetDevice(int d) { (void)d; return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int* v, enum cudaDeviceAttr a, int d) { (void)a; (void)d; *v = 152; return cudaSuccess; }
cudaError_t cudaGetDeviceProperties(struct cudaDeviceProp* p, int d) {
  (void)d;
  memset(p, 0, sizeof *p);
  p->major = 10;
  p->minor = 3;
  return cudaSuccess;
}
static CUresult encode(CUtensorMap* tm, CUtensorMapDataType type, cuuint32_t rank, void* base, const cuuint64_t* dim,
                       const cuuint64_t* stride, const cuuint32_t* box, const cuuint32_t* step,
                       CUtensorMapInterleave il, CUtensorMapSwizzle sw, CUtensorMapL2promotion l2,
                       CUtensorMapFloatOOBfill fill) {
  (void)step; (void)il; (void)sw; (void)l2; (void)fill;
  const size_t es = type == CU_TENSOR_MAP_DATA_TYPE_UINT8 ? 1 : (type == CU_TENSOR_MAP_DATA_TYPE_BFLOAT16 ? 2 : 4);
  const char* p = (const char*)base;
  memset(tm, 0, sizeof *tm);
  if (rank != 2 || !dim[0] || !dim[1] || dim[0] * es > stride[0] || (uintptr_t)p % 16 || stride[0] % 16 ||
      box[0] * es % 16 || box[0] > 256 || box[1] > 256)
    return CUDA_ERROR_INVALID_VALUE;
  for (int k = 0; k < g_nalloc; ++k)
    if (p >= g_alloc[k].p && p + (dim[1] - 1) * stride[0] + dim[0] * es <= g_alloc[k].p + g_alloc[k].n) return CUDA_SUCCESS;
  return CUDA_ERROR_INVALID_VALUE;
}
cudaError_t cudaGetDriverEntryPointByVersion(const char* n, void** f, unsigned v, unsigned long long fl,
                                             enum cudaDriverEntryPointQueryResult* r) {
  (void)v; (void)fl;
  *f = strcmp(n, "cuTensorMapEncodeTiled") ? 0 : (void*)encode;
  *r = *f ? cudaDriverEntryPointSuccess : cudaDriverEntryPointSymbolNotFound;
  return cudaSuccess;
}
cudaError_t cudaGetSymbolAddress(void** p, const void* s) { (void)p; (void)s; return cudaErrorNotSupported; }
cudaError_t cudaGetLastError(void) { return cudaSuccess; }
const char* cudaGetErrorString(cudaError_t e) { (void)e; return "error"; }

/* ---- kernels ---- */
static cudaError_t run(const void* f, void** args, cudaStream_t s) {
  for (int k = 0; g_hook && k < g_nkernel; ++k)
    if (g_kernel[k].f == f) { g_hook(g_kernel[k].name, args); break; }
  return queued(s);
}
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t* c, const void* f, void** args) { return run(f, args, c->stream); }
cudaError_t cudaFuncSetAttribute(const void* f, enum cudaFuncAttribute a, int v) { (void)f; (void)a; (void)v; return cudaSuccess; }
void** __cudaRegisterFatBinary(void* b) { (void)b; static void* h; return &h; }
void __cudaRegisterFatBinaryEnd(void** h) { (void)h; }
void __cudaUnregisterFatBinary(void** h) { (void)h; }
void __cudaRegisterVar(void** h, char* v, char* a, const char* n, int e, size_t s, int c, int g) {
  (void)h; (void)v; (void)a; (void)n; (void)e; (void)s; (void)c; (void)g;
}
void __cudaRegisterFunction(void** h, const char* f, char* d, const char* name, int t, void* a, void* b, void* c, void* e, int* w) {
  (void)h; (void)d; (void)t; (void)a; (void)b; (void)c; (void)e; (void)w;
  if (g_nkernel < MAX_KERNELS) {
    g_kernel[g_nkernel].f = f;
    g_kernel[g_nkernel++].name = name;
  }
}
static cudaStream_t g_call;
unsigned __cudaPushCallConfiguration(dim3 g, dim3 b, size_t n, void* s) {
  (void)g; (void)b; (void)n;
  g_call = (cudaStream_t)s;
  return 0;
}
cudaError_t __cudaPopCallConfiguration(void* g, void* b, size_t* n, void* s) {
  (void)g; (void)b; (void)n;
  *(cudaStream_t*)s = g_call;
  return cudaSuccess;
}
cudaError_t __cudaGetKernel(cudaKernel_t* k, const void* f) { *k = (cudaKernel_t)f; return cudaSuccess; }
cudaError_t __cudaLaunchKernel(cudaKernel_t k, dim3 g, dim3 b, void** args, size_t n, cudaStream_t s) {
  (void)g; (void)b; (void)n;
  return run((const void*)k, args, s);
}
