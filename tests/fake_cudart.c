/* A stand-in for the CUDA runtime, for tests of the library's host code without
 * a GPU (linked into a copy of the library built with -cudart none): memory is
 * host memory, or for large device arrays an address never read; kernels do not
 * run, their launches are logged and checked against the limits of a grid, and
 * the launch picked by fake_fail returns an error. */
#include <cuda_runtime_api.h>
#include <stdlib.h>
#include <string.h>

#define MAX_KERNELS 256
#define MAX_LOG 65536

static const void* g_fun[MAX_KERNELS];
static const char* g_name[MAX_KERNELS];
static int g_kernels;
static struct {
  const char* name;
  unsigned x, y, z;
} g_log[MAX_LOG];
static int g_launches, g_fail = -1;
static cudaError_t g_last = cudaSuccess;

int fake_launches(void) { return g_launches; }
const char* fake_launch(int k, unsigned grid[3]) {
  grid[0] = g_log[k].x, grid[1] = g_log[k].y, grid[2] = g_log[k].z;
  return g_log[k].name;
}
void fake_reset(void) { g_launches = 0, g_fail = -1, g_last = cudaSuccess; }
void fake_fail(int k) { g_fail = k; } /* the k-th launch from the last reset on */

static cudaError_t launch(const void* fun, dim3 grid) {
  const char* name = "?";
  for (int k = 0; k < g_kernels; ++k)
    if (g_fun[k] == fun) name = g_name[k];
  const int k = g_launches;
  if (k < MAX_LOG) {
    g_log[k].name = name;
    g_log[k].x = grid.x, g_log[k].y = grid.y, g_log[k].z = grid.z;
    ++g_launches;
  }
  cudaError_t e = cudaSuccess;
  if (k == g_fail) e = cudaErrorLaunchOutOfResources;
  if (!grid.x || !grid.y || !grid.z || grid.x > 0x7fffffffu || grid.y > 65535u || grid.z > 65535u)
    e = cudaErrorInvalidConfiguration;
  if (e != cudaSuccess) g_last = e;
  return e;
}

cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t* c, const void* fun, void** args) {
  (void)args;
  return launch(fun, c->gridDim);
}
/* what the stubs of <<<>>> call: a kernel handle is the stub's address */
cudaError_t __cudaGetKernel(cudaKernel_t* k, const void* fun) {
  return *k = (cudaKernel_t)fun, cudaSuccess;
}
cudaError_t __cudaLaunchKernel(cudaKernel_t k, dim3 grid, dim3 block, void** args, size_t smem,
                               cudaStream_t st) {
  (void)block, (void)args, (void)smem, (void)st;
  return launch((const void*)k, grid);
}
static dim3 g_grid, g_block;
static size_t g_smem;
static void* g_stream;
unsigned __cudaPushCallConfiguration(dim3 grid, dim3 block, size_t smem, struct CUstream_st* st) {
  g_grid = grid, g_block = block, g_smem = smem, g_stream = st;
  return 0;
}
cudaError_t __cudaPopCallConfiguration(dim3* grid, dim3* block, size_t* smem, void* st) {
  *grid = g_grid, *block = g_block, *smem = g_smem, *(void**)st = g_stream;
  return cudaSuccess;
}
void** __cudaRegisterFatBinary(void* bin) {
  static void* handle;
  (void)bin;
  return &handle;
}
void __cudaRegisterFatBinaryEnd(void** h) { (void)h; }
void __cudaUnregisterFatBinary(void** h) { (void)h; }
char __cudaInitModule(void** h) { return (void)h, 1; }
void __cudaRegisterFunction(void** h, const char* host, char* dev, const char* name, int limit,
                            void* tid, void* bid, void* bdim, void* gdim, int* wsize) {
  (void)h, (void)dev, (void)limit, (void)tid, (void)bid, (void)bdim, (void)gdim, (void)wsize;
  if (g_kernels < MAX_KERNELS) g_fun[g_kernels] = host, g_name[g_kernels++] = name;
}
void __cudaRegisterVar(void** h, char* host, char* dev, const char* name, int ext, size_t size,
                       int constant, int global) {
  (void)h, (void)host, (void)dev, (void)name, (void)ext, (void)size, (void)constant, (void)global;
}

cudaError_t cudaMalloc(void** p, size_t n) { return (void)n, *p = malloc(256), cudaSuccess; }
cudaError_t cudaFree(void* p) { return free(p), cudaSuccess; }
cudaError_t cudaMallocHost(void** p, size_t n) { return *p = calloc(1, n), cudaSuccess; }
cudaError_t cudaFreeHost(void* p) { return free(p), cudaSuccess; }
cudaError_t cudaMemcpy(void* d, const void* s, size_t n, enum cudaMemcpyKind k) {
  return (void)d, (void)s, (void)n, (void)k, cudaSuccess;
}
cudaError_t cudaMemcpyAsync(void* d, const void* s, size_t n, enum cudaMemcpyKind k,
                            cudaStream_t st) {
  return (void)d, (void)s, (void)n, (void)k, (void)st, cudaSuccess;
}
cudaError_t cudaMemsetAsync(void* d, int v, size_t n, cudaStream_t st) {
  return (void)d, (void)v, (void)n, (void)st, cudaSuccess;
}
cudaError_t cudaStreamCreateWithFlags(cudaStream_t* s, unsigned f) {
  return (void)f, *s = (cudaStream_t)malloc(1), cudaSuccess;
}
cudaError_t cudaStreamDestroy(cudaStream_t s) { return free(s), cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t s) { return (void)s, cudaSuccess; }
cudaError_t cudaStreamWaitEvent(cudaStream_t s, cudaEvent_t e, unsigned f) {
  return (void)s, (void)e, (void)f, cudaSuccess;
}
cudaError_t cudaEventCreate(cudaEvent_t* e) { return *e = (cudaEvent_t)malloc(1), cudaSuccess; }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t* e, unsigned f) {
  return (void)f, cudaEventCreate(e);
}
cudaError_t cudaEventDestroy(cudaEvent_t e) { return free(e), cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t e, cudaStream_t s) { return (void)e, (void)s, cudaSuccess; }
cudaError_t cudaEventSynchronize(cudaEvent_t e) { return (void)e, cudaSuccess; }
cudaError_t cudaEventElapsedTime(float* ms, cudaEvent_t a, cudaEvent_t b) {
  return (void)a, (void)b, *ms = 1.0f, cudaSuccess;
}
cudaError_t cudaGetDevice(int* d) { return *d = 0, cudaSuccess; }
cudaError_t cudaSetDevice(int d) { return (void)d, cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int* v, enum cudaDeviceAttr a, int d) {
  return (void)a, (void)d, *v = 152, cudaSuccess;
}
cudaError_t cudaFuncSetAttribute(const void* f, enum cudaFuncAttribute a, int v) {
  return (void)f, (void)a, (void)v, cudaSuccess;
}
cudaError_t cudaGetSymbolAddress(void** p, const void* s) { return (void)s, *p = malloc(256), cudaSuccess; }
cudaError_t cudaGetDriverEntryPointByVersion(const char* s, void** f, unsigned v,
                                             unsigned long long fl,
                                             enum cudaDriverEntryPointQueryResult* r) {
  return (void)s, (void)v, (void)fl, (void)r, *f = 0, cudaErrorNotSupported;
}
const char* cudaGetErrorString(cudaError_t e) { return e == cudaSuccess ? "no error" : "fake error"; }
cudaError_t cudaGetLastError(void) {
  const cudaError_t e = g_last;
  return g_last = cudaSuccess, e;
}
