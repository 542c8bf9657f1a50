/* A stand-in for the CUDA runtime with two devices and no GPU, for tests of the library's host code: it keeps what the
 * library asks of each device and runs no kernel.  A kernel's limit of dynamic shared memory holds for the device that
 * was current when it was set, as in CUDA; a launch or graph node above it is refused and counted. */
#include <cuda_runtime_api.h>
#include <stdlib.h>
#include <string.h>

#define KERNELS 4096
enum { DEVICES = 2 };
static const int kSms[DEVICES] = {152, 100};
static int device, refused, launched[DEVICES], nlimits, no_limits;
static struct { const void* func; int device, bytes; } limits[KERNELS];

void fake_no_limits(int on) { no_limits = on; }   /* raising a kernel's limit fails from now on */
int fake_refused(void) { return refused; }
int fake_launched(int d) { return launched[d]; }

static cudaError_t launch(const void* func, size_t smem) {
  int limit = 48 << 10;
  for (int i = 0; i < nlimits; ++i)
    if (limits[i].func == func && limits[i].device == device) limit = limits[i].bytes;
  if (smem > (size_t)limit) { ++refused; return cudaErrorInvalidValue; }
  ++launched[device];
  return cudaSuccess;
}

cudaError_t cudaGetDevice(int* d) { *d = device; return cudaSuccess; }
cudaError_t cudaSetDevice(int d) { device = d; return cudaSuccess; }
cudaError_t cudaGetLastError(void) { return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int* v, enum cudaDeviceAttr a, int d) {
  *v = a == cudaDevAttrMultiProcessorCount ? kSms[d] : 0;
  return cudaSuccess;
}
cudaError_t cudaFuncSetAttribute(const void* func, enum cudaFuncAttribute a, int bytes) {
  if (a != cudaFuncAttributeMaxDynamicSharedMemorySize) return cudaSuccess;
  if (no_limits) return cudaErrorInvalidValue;
  for (int i = 0; i < nlimits; ++i)
    if (limits[i].func == func && limits[i].device == device) { limits[i].bytes = bytes; return cudaSuccess; }
  limits[nlimits].func = func; limits[nlimits].device = device; limits[nlimits++].bytes = bytes;
  return cudaSuccess;
}
cudaError_t cudaOccupancyMaxActiveClusters(int* n, const void* func, const cudaLaunchConfig_t* cfg) {
  (void)func; (void)cfg;
  *n = kSms[device] / 16;
  return cudaSuccess;
}
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int* n, const void* func, int threads, size_t smem,
                                                                   unsigned flags) {
  (void)func; (void)threads; (void)smem; (void)flags;
  *n = 1;
  return cudaSuccess;
}
cudaError_t cudaMalloc(void** p, size_t n) { return (*p = malloc(n)) ? cudaSuccess : cudaErrorMemoryAllocation; }
cudaError_t cudaFree(void* p) { free(p); return cudaSuccess; }
cudaError_t cudaMallocAsync(void** p, size_t n, cudaStream_t s) { (void)s; return cudaMalloc(p, n); }
cudaError_t cudaFreeAsync(void* p, cudaStream_t s) { (void)s; return cudaFree(p); }
cudaError_t cudaHostAlloc(void** p, size_t n, unsigned flags) {
  (void)flags;
  return (*p = calloc(1, n)) ? cudaSuccess : cudaErrorMemoryAllocation;
}
cudaError_t cudaFreeHost(void* p) { free(p); return cudaSuccess; }
cudaError_t cudaMemGetInfo(size_t* f, size_t* t) { *f = *t = (size_t)1 << 37; return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float* ms, cudaEvent_t a, cudaEvent_t b) { (void)a; (void)b; *ms = 0.f; return cudaSuccess; }

static int encode(void) { return 0; }
cudaError_t cudaGetDriverEntryPointByVersion(const char* name, void** p, unsigned version, unsigned long long flags,
                                             enum cudaDriverEntryPointQueryResult* q) {
  (void)name; (void)version; (void)flags;
  *p = (void*)encode;
  *q = cudaDriverEntryPointSuccess;
  return cudaSuccess;
}

cudaError_t cudaGetSymbolAddress(void** p, const void* symbol) {
  (void)symbol;
  static char workspace[32 << 20];
  *p = workspace;
  return cudaSuccess;
}

static char handle;
cudaError_t cudaGraphCreate(cudaGraph_t* g, unsigned flags) { (void)flags; *g = (cudaGraph_t)&handle; return cudaSuccess; }
cudaError_t cudaGraphAddNode(cudaGraphNode_t* node, cudaGraph_t g, const cudaGraphNode_t* deps,
                             const cudaGraphEdgeData* edges, size_t n, struct cudaGraphNodeParams* p) {
  (void)g; (void)deps; (void)edges; (void)n;
  static cudaGraph_t bodies[2] = {(cudaGraph_t)&handle, (cudaGraph_t)&handle};
  *node = (cudaGraphNode_t)&handle;
  if (p->type == cudaGraphNodeTypeConditional) p->conditional.phGraph_out = bodies;
  return cudaSuccess;
}
cudaError_t cudaGraphAddKernelNode(cudaGraphNode_t* node, cudaGraph_t g, const cudaGraphNode_t* deps, size_t n,
                                   const struct cudaKernelNodeParams* p) {
  (void)g; (void)deps; (void)n;
  *node = (cudaGraphNode_t)&handle;
  return launch(p->func, p->sharedMemBytes);
}

cudaError_t cudaLaunchKernel(const void* func, dim3 grid, dim3 block, void** args, size_t smem, cudaStream_t s) {
  (void)grid; (void)block; (void)args; (void)s;
  return launch(func, smem);
}
/* what the compiler makes of a launch in angle brackets */
static dim3 grid_, block_;
static size_t smem_;
static void* stream_;
unsigned __cudaPushCallConfiguration(dim3 grid, dim3 block, size_t smem, void* s) {
  grid_ = grid; block_ = block; smem_ = smem; stream_ = s;
  return 0;
}
cudaError_t __cudaPopCallConfiguration(dim3* grid, dim3* block, size_t* smem, void* s) {
  *grid = grid_; *block = block_; *smem = smem_; *(void**)s = stream_;
  return cudaSuccess;
}
cudaError_t __cudaGetKernel(cudaKernel_t* k, const void* func) { *k = (cudaKernel_t)func; return cudaSuccess; }
cudaError_t __cudaLaunchKernel(cudaKernel_t k, dim3 grid, dim3 block, void** args, size_t smem, cudaStream_t s) {
  (void)grid; (void)block; (void)args; (void)s;
  return launch((const void*)k, smem);
}
