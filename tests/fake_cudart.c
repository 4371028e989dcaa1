/* A CUDA runtime without a device, for tests of the library's host code: "device" memory is host memory, work runs
 * when it is queued, kernels are only recorded.  Preloaded before liblbm.so, whose calls it takes over. */
#include <stddef.h>
#include <stdint.h>
#include <stdio.h>
#include <stdlib.h>
#include <string.h>

#define API __attribute__((visibility("default")))
typedef struct { unsigned x, y, z; } dim3_t;
typedef struct { int type, device; void *devicePointer, *hostPointer; long reserved[8]; } attributes_t;

/* Memory: address ranges with a type (cudaMemoryType: 0 unregistered, 1 host, 2 device, 3 managed) and a device. */
static struct { char *p; size_t n; int type, device; } ranges[1 << 17];
static int n_ranges;
API void fake_range(void* p, size_t n, int type, int device) {
  ranges[n_ranges].p = p;
  ranges[n_ranges].n = n;
  ranges[n_ranges].type = type;
  ranges[n_ranges++].device = device;
}
API int cudaPointerGetAttributes(attributes_t* a, const void* p) {
  memset(a, 0, sizeof *a);
  a->device = -2;
  for (int i = n_ranges - 1; i >= 0; --i)
    if ((char*)p >= ranges[i].p && (char*)p < ranges[i].p + ranges[i].n) {
      a->type = ranges[i].type;
      a->device = ranges[i].device;
      a->devicePointer = a->hostPointer = (void*)p;
      break;
    }
  return 0;
}
static int allocate(void** p, size_t n, int type) {
  *p = aligned_alloc(256, (n + 255) / 256 * 256);
  if (n < 1 << 20) memset(*p, 0xA5, n);   /* (large blocks stay untouched, and so unmapped) */
  fake_range(*p, n, type, 0);
  return 0;
}
API int cudaMalloc(void** p, size_t n) { return allocate(p, n, 2); }
API int cudaMallocAsync(void** p, size_t n, void* st) { return allocate(p, n, 2); }
API int cudaHostAlloc(void** p, size_t n, unsigned flags) { return allocate(p, n, 1); }
API int cudaFree(void* p) {
  free(p);
  return 0;
}
API int cudaFreeAsync(void* p, void* st) { return cudaFree(p); }

/* Copies and launches, in the order in which they were queued. */
struct event { char what[64]; void *a, *b; long long n, smem; };
static struct event events[65536];
static int n_events;
static void record_launch(const char* what, const void* a, const void* b, long long n, long long smem) {
  struct event* e = &events[n_events++ & 65535];
  snprintf(e->what, sizeof e->what, "%s", what);
  e->a = (void*)a;
  e->b = (void*)b;
  e->n = n;
  e->smem = smem;
}
static void record(const char* what, const void* a, const void* b, long long n) { record_launch(what, a, b, n, 0); }
API int fake_events(void) { return n_events; }
API void fake_clear(void) { n_events = 0; }
API const struct event* fake_event(int i) { return &events[i]; }

API int cudaMemcpyAsync(void* d, const void* s, size_t n, int kind, void* st) {
  record("copy", d, s, (long long)n);
  memmove(d, s, n);
  return 0;
}
API int cudaMemcpy2DAsync(void* d, size_t dp, const void* s, size_t sp, size_t w, size_t h, int kind, void* st) {
  record("copy2d", d, s, (long long)(w * h));
  for (size_t y = 0; y < h; ++y) memmove((char*)d + y * dp, (const char*)s + y * sp, w);
  return 0;
}
API int cudaMemsetAsync(void* d, int v, size_t n, void* st) {
  record("set", d, 0, (long long)n);
  if (n < 1 << 20) memset(d, v, n);
  return 0;
}

/* Kernels: the name that was registered with the host stub; a, b: the first two parameters' first words; n: blocks x 1024 +
 * threads; smem: dynamic shared memory. */
static struct { const void* stub; char name[256]; } kernels[1024];
static int n_kernels;
API void __cudaRegisterFunction(void** h, const char* stub, char* dev, const char* name, int lim, void* a, void* b, void* c, void* d,
                                int* e) {
  kernels[n_kernels].stub = stub;
  snprintf(kernels[n_kernels++].name, sizeof kernels[0].name, "%s", name);
}
static int launch(const void* stub, void** args, const dim3_t* g, size_t smem) {
  for (int i = 0; i < n_kernels; ++i)
    if (kernels[i].stub == stub) {
      const char* k = strstr(kernels[i].name, "k_");
      char plain[64];
      size_t n = 0;
      while (k && n < sizeof plain - 1 && (k[n] == '_' || (k[n] >= 'a' && k[n] <= 'z') || (k[n] >= '0' && k[n] <= '9'))) ++n;
      snprintf(plain, sizeof plain, "%.*s", (int)n, k ? k : "");
      record_launch(plain, *(void**)args[0], strcmp(plain, "k_diag") ? *(void**)args[1] : 0, g[0].x * 1024LL + g[1].x, smem);
      return 0;
    }
  return 98;
}
static struct { dim3_t g, b; size_t smem; void* st; } pushed;
API unsigned __cudaPushCallConfiguration(dim3_t g, dim3_t b, size_t smem, void* st) {
  pushed.g = g;
  pushed.b = b;
  pushed.smem = smem;
  pushed.st = st;
  return 0;
}
API int __cudaPopCallConfiguration(dim3_t* g, dim3_t* b, size_t* smem, void** st) {
  *g = pushed.g;
  *b = pushed.b;
  *smem = pushed.smem;
  *st = pushed.st;
  return 0;
}
API int __cudaGetKernel(const void** k, const void* stub) {
  *k = stub;
  return 0;
}
API int __cudaLaunchKernel(const void* k, dim3_t g, dim3_t b, void** args, size_t smem, void* st) {
  const dim3_t gb[2] = {g, b};
  return launch(k, args, gb, smem);
}
API int cudaLaunchKernelExC(const void* cfg, const void* stub, void** args) {
  return launch(stub, args, cfg, *(const size_t*)((const char*)cfg + 24));
}
static void* module;
API void** __cudaRegisterFatBinary(void* bin) { return &module; }
API void __cudaRegisterFatBinaryEnd(void** h) {}
API void __cudaUnregisterFatBinary(void** h) {}
API void __cudaRegisterVar(void** h, char* host, char* dev, const char* name, int ext, size_t n, int c, int g) {}

API int cudaGetDevice(int* d) {
  *d = 0;
  return 0;
}
API int cudaDeviceGetAttribute(int* v, int what, int dev) {
  *v = what == 16 ? 152 : (what == 97 ? 232448 : (what == 111 ? 1024 : 233472));   /* multiprocessors; shared-memory sizes */
  return 0;
}
API int cudaFuncSetAttribute(const void* f, int a, int v) { return 0; }
API int cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int* n, const void* f, int t, size_t s, unsigned fl) {
  *n = 2;
  return 0;
}
API int cudaEventCreateWithFlags(void** e, unsigned f) { return (*e = &module, 0); }
API int cudaEventDestroy(void* e) { return 0; }
API int cudaEventRecord(void* e, void* st) { return 0; }
API int cudaEventSynchronize(void* e) { return 0; }
API int cudaStreamCreateWithFlags(void** s, unsigned f) { return (*s = &module, 0); }
API int cudaStreamDestroy(void* s) { return 0; }
API int cudaStreamSynchronize(void* s) { return 0; }
API int cudaStreamIsCapturing(void* s, int* c) { return (*c = 0, 0); }
API int cudaGetLastError(void) { return 0; }
API const char* cudaGetErrorString(int e) { return e ? "error" : "no error"; }
