/* A CUDA runtime without a GPU, preloaded in front of libcudart by test_host_path_without_gpu.py: device memory is host
 * memory, kernels do not run, and a launch is granted and recorded under the rules that the host path has to keep -- a
 * kernel that asks for more than 48 KB of dynamic shared memory needs its limit raised on the device it is launched on. */
#include <cuda_runtime_api.h>
#include <cuda.h>
#include <stdio.h>
#include <stdlib.h>
#include <string.h>

#define MAX_DEVICES 4
#define MAX_KERNELS 256
#define MAX_LAUNCHES 4096

static int device, sm_count[MAX_DEVICES] = {148, 148, 148, 148}, refuse_limit[MAX_DEVICES];
static cudaError_t last_error;
static struct { const void* func; char name[256]; int limit[MAX_DEVICES]; } kernels[MAX_KERNELS];
static int n_kernels;
static struct { int kernel, device, grid[3]; } launches[MAX_LAUNCHES];
static int n_launches;

static int kernel_of(const void* func) {
  for (int i = 0; i < n_kernels; ++i)
    if (kernels[i].func == func) return i;
  return -1;
}
static cudaError_t fail(cudaError_t e) {
  if (e != cudaSuccess) last_error = e;
  return e;
}

/* what the test calls */
void fake_set_device(int d) { device = d; }
void fake_set_sm_count(int d, int n) { sm_count[d] = n; }
void fake_refuse_limit(int d, int on) { refuse_limit[d] = on; }
int fake_launches(void) { return n_launches; }
const char* fake_launch(int i) {
  static char text[512];
  snprintf(text, sizeof(text), "%d %d %d %d %s", launches[i].device, launches[i].grid[0], launches[i].grid[1], launches[i].grid[2],
           kernels[launches[i].kernel].name);
  return text;
}

/* registration of the library's kernels */
static void* fatbin_handle;
void** __cudaRegisterFatBinary(void* fat) { (void)fat; return &fatbin_handle; }
void __cudaRegisterFatBinaryEnd(void** h) { (void)h; }
void __cudaUnregisterFatBinary(void** h) { (void)h; }
void __cudaRegisterVar(void** h, char* var, char* addr, const char* name, int ext, size_t size, int constant, int global) {
  (void)h; (void)var; (void)addr; (void)name; (void)ext; (void)size; (void)constant; (void)global;
}
void __cudaRegisterFunction(void** h, const char* func, char* fun, const char* name, int limit, void* tid, void* bid, void* bdim,
                            void* gdim, int* wsize) {
  (void)h; (void)fun; (void)limit; (void)tid; (void)bid; (void)bdim; (void)gdim; (void)wsize;
  if (n_kernels == MAX_KERNELS) abort();
  kernels[n_kernels].func = func;
  snprintf(kernels[n_kernels].name, sizeof(kernels[0].name), "%s", name);
  for (int d = 0; d < MAX_DEVICES; ++d) kernels[n_kernels].limit[d] = 48 * 1024;
  ++n_kernels;
}

/* devices and errors */
cudaError_t cudaGetDevice(int* d) { *d = device; return cudaSuccess; }
cudaError_t cudaGetDeviceProperties_v2(struct cudaDeviceProp* p, int d) {
  memset(p, 0, sizeof(*p));
  p->multiProcessorCount = sm_count[d];
  p->major = 10;
  return cudaSuccess;
}
cudaError_t cudaDeviceGetAttribute(int* v, enum cudaDeviceAttr a, int d) {
  if (a != cudaDevAttrMultiProcessorCount) return fail(cudaErrorInvalidValue);
  *v = sm_count[d];
  return cudaSuccess;
}
cudaError_t cudaGetLastError(void) { cudaError_t e = last_error; last_error = cudaSuccess; return e; }
const char* cudaGetErrorString(cudaError_t e) { return e == cudaSuccess ? "no error" : "refused"; }
cudaError_t cudaDeviceSynchronize(void) { return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t s) { (void)s; return cudaSuccess; }

/* memory */
cudaError_t cudaMalloc(void** p, size_t n) { *p = calloc(1, n); return *p ? cudaSuccess : fail(cudaErrorMemoryAllocation); }
cudaError_t cudaFree(void* p) { free(p); return cudaSuccess; }
cudaError_t cudaHostAlloc(void** p, size_t n, unsigned flags) { (void)flags; *p = calloc(1, n); return cudaSuccess; }
cudaError_t cudaFreeHost(void* p) { free(p); return cudaSuccess; }
cudaError_t cudaHostGetDevicePointer(void** d, void* h, unsigned flags) { (void)flags; *d = h; return cudaSuccess; }
cudaError_t cudaMemset(void* p, int v, size_t n) { memset(p, v, n); return cudaSuccess; }
cudaError_t cudaMemcpy(void* d, const void* s, size_t n, enum cudaMemcpyKind k) { (void)k; memcpy(d, s, n); return cudaSuccess; }
cudaError_t cudaMemcpyAsync(void* d, const void* s, size_t n, enum cudaMemcpyKind k, cudaStream_t st) {
  (void)st;
  return cudaMemcpy(d, s, n, k);
}
cudaError_t cudaGetSymbolAddress(void** p, const void* symbol) {
  static char scratch[MAX_DEVICES][1 << 18];
  (void)symbol;
  *p = scratch[device];
  return cudaSuccess;
}

/* events */
cudaError_t cudaEventCreate(cudaEvent_t* e) { *e = (cudaEvent_t)&device; return cudaSuccess; }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t* e, unsigned flags) { (void)flags; return cudaEventCreate(e); }
cudaError_t cudaEventDestroy(cudaEvent_t e) { (void)e; return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t e, cudaStream_t s) { (void)e; (void)s; return cudaSuccess; }
cudaError_t cudaEventQuery(cudaEvent_t e) { (void)e; return cudaSuccess; }
cudaError_t cudaEventSynchronize(cudaEvent_t e) { (void)e; return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float* ms, cudaEvent_t a, cudaEvent_t b) { (void)a; (void)b; *ms = 0.f; return cudaSuccess; }

/* kernels */
cudaError_t cudaFuncSetAttribute(const void* func, enum cudaFuncAttribute a, int v) {
  const int k = kernel_of(func);
  if (k < 0 || refuse_limit[device]) return fail(cudaErrorInvalidValue);
  if (a == cudaFuncAttributeMaxDynamicSharedMemorySize) kernels[k].limit[device] = v;
  return cudaSuccess;
}
cudaError_t cudaOccupancyMaxActiveClusters(int* n, const void* func, const cudaLaunchConfig_t* c) {
  const int k = kernel_of(func);
  if (k < 0 || (int)c->dynamicSmemBytes > kernels[k].limit[device]) return fail(cudaErrorInvalidValue);
  *n = sm_count[device] / 2;
  return cudaSuccess;
}
static cudaError_t launch(const void* func, dim3 grid, size_t smem) {
  const int k = kernel_of(func);
  if (k < 0 || (int)smem > kernels[k].limit[device] || !grid.x || !grid.y || !grid.z || grid.x > 0x7fffffffu)
    return fail(cudaErrorInvalidValue);
  if (n_launches < MAX_LAUNCHES) {
    launches[n_launches].kernel = k;
    launches[n_launches].device = device;
    launches[n_launches].grid[0] = (int)grid.x;
    launches[n_launches].grid[1] = (int)grid.y;
    launches[n_launches].grid[2] = (int)grid.z;
    ++n_launches;
  }
  return cudaSuccess;
}
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t* c, const void* func, void** args) {
  (void)args;
  return launch(func, c->gridDim, c->dynamicSmemBytes);
}
cudaError_t cudaLaunchKernel(const void* func, dim3 grid, dim3 block, void** args, size_t smem, cudaStream_t s) {
  (void)block; (void)args; (void)s;
  return launch(func, grid, smem);
}
unsigned __cudaPopCallConfiguration(dim3* g, dim3* b, size_t* smem, void* s) { (void)g; (void)b; (void)smem; (void)s; return 0; }

/* the driver's tensor-map encoder */
static CUresult encode(CUtensorMap* m) { memset(m, 0, sizeof(*m)); return CUDA_SUCCESS; }
cudaError_t cudaGetDriverEntryPoint(const char* name, void** p, unsigned long long flags, enum cudaDriverEntryPointQueryResult* q) {
  (void)name; (void)flags;
  *p = (void*)encode;
  if (q) *q = cudaDriverEntryPointSuccess;
  return cudaSuccess;
}
