/* A CUDA runtime that does nothing, for tests of the library's host side without a device: every call succeeds, copies and launches are
 * not done, and launches are noted by their kernel's name.  Built as libcudart.so.12 and found before the real one.
 * Only names and signatures are those of the CUDA runtime. */
#include <stddef.h>
#include <stdint.h>
#include <stdio.h>
#include <stdlib.h>
#include <string.h>

typedef int err;                                 /* cudaError_t */
typedef struct { unsigned x, y, z; } dim3;
typedef struct { dim3 grid, block; size_t smem; void* stream; void* attrs; unsigned n_attrs; } launch_config;

/* ---- what a test asks and sets ---- */
static char log_[1 << 20];
static size_t log_len;
static const char* refuse_name = "";             /* launches of kernels whose name has this in it ... */
static err refuse_with;                          /* ... return this */
static int unset;                                /* so many calls that set an attribute fail */
static void* host_words;                         /* the last mapped host memory handed out */
static int capturing, asked;                     /* asked: of an event or of a stream's state */
const char* fake_log(void) { return log_; }
void fake_clear(void) { log_len = 0; log_[0] = 0; }
void fake_refuse(const char* name, int with) { refuse_name = strdup(name); refuse_with = with; }
void fake_unset(int calls) { unset = calls; }
void* fake_host_words(void) { return host_words; }
void fake_capture(int on) { capturing = on; }
int fake_asked(void) { const int n = asked; asked = 0; return n; }

/* ---- registration and launches ---- */
static struct { const void* fun; const char* name; } kernels[4096];
static int n_kernels;
void** __cudaRegisterFatBinary(void* f) { (void)f; static void* handle[4]; return handle; }
void __cudaRegisterFatBinaryEnd(void** h) { (void)h; }
void __cudaUnregisterFatBinary(void** h) { (void)h; }
void __cudaRegisterFunction(void** h, const char* fun, char* dev, const char* name, int limit, void* a, void* b, void* c, void* d, int* e) {
  (void)h; (void)dev; (void)limit; (void)a; (void)b; (void)c; (void)d; (void)e;
  if (n_kernels < 4096) { kernels[n_kernels].fun = fun; kernels[n_kernels++].name = strdup(name); }
}
void __cudaRegisterVar(void** h, char* v, char* d, const char* n, int a, size_t s, int b, int c) { (void)h; (void)v; (void)d; (void)n; (void)a; (void)s; (void)b; (void)c; }
err __cudaPopCallConfiguration(dim3* g, dim3* b, size_t* s, void* st) { (void)g; (void)b; (void)s; (void)st; return 1; }
static err last;
static err launch(const void* fun, dim3 grid) {
  if (!grid.x || !grid.y || !grid.z || grid.x > 0x7fffffffu || grid.y > 65535 || grid.z > 65535) return last = 9;      /* cudaErrorInvalidConfiguration */
  const char* name = "?";
  for (int i = 0; i < n_kernels; ++i) if (kernels[i].fun == fun) name = kernels[i].name;
  if (refuse_with && *refuse_name && strstr(name, refuse_name)) { last = refuse_with; return refuse_with; }
  if (log_len + strlen(name) + 2 < sizeof(log_)) log_len += (size_t)sprintf(log_ + log_len, "%s\n", name);
  return 0;
}
err cudaLaunchKernelExC(const launch_config* c, const void* fun, void** args) { (void)args; return launch(fun, c->grid); }
err cudaLaunchKernel(const void* fun, dim3 g, dim3 b, void** args, size_t s, void* st) { (void)b; (void)args; (void)s; (void)st; return launch(fun, g); }

/* ---- the rest ---- */
err cudaGetLastError(void) { const err e = last; last = 0; return e; }
const char* cudaGetErrorString(err e) { return e == 0 ? "no error" : "some error"; }
err cudaGetDevice(int* d) { *d = 0; return 0; }
err cudaDeviceGetAttribute(int* v, int attr, int dev) { (void)attr; (void)dev; *v = 148; return 0; }
err cudaDeviceGetStreamPriorityRange(int* least, int* greatest) { *least = 0; *greatest = -5; return 0; }
err cudaEventCreate(void** e) { *e = malloc(1); return 0; }
err cudaEventCreateWithFlags(void** e, unsigned f) { (void)f; *e = malloc(1); return 0; }
err cudaEventDestroy(void* e) { free(e); return 0; }
err cudaEventElapsedTime(float* ms, void* a, void* b) { (void)a; (void)b; *ms = 0; return 0; }
err cudaEventRecord(void* e, void* s) { (void)e; (void)s; return 0; }
err cudaEventSynchronize(void* e) { (void)e; ++asked; return 0; }
err cudaHostAlloc(void** p, size_t n, unsigned f) { (void)f; host_words = *p = calloc(1, n); return 0; }
err cudaFreeHost(void* p) { free(p); return 0; }
err cudaHostGetDevicePointer(void** d, void* h, unsigned f) { (void)f; *d = h; return 0; }
err cudaFuncSetAttribute(const void* f, int a, int v) { (void)f; (void)a; (void)v; if (unset > 0) { --unset; return last = 1; } return 0; }
static err encode(void) { return 0; }
err cudaGetDriverEntryPoint(const char* name, void** fn, unsigned long long flags, int* found) {
  (void)flags;
  const int map = strstr(name, "TensorMap") != NULL;
  *fn = map ? (void*)encode : NULL;
  if (found) *found = map ? 0 : 1;
  return 0;
}
static char symbol_[4096];
err cudaGetSymbolAddress(void** p, const void* s) { (void)s; *p = symbol_; return 0; }
err cudaMemcpy(void* d, const void* s, size_t n, int k) { (void)s; (void)k; memset(d, 0, n); return 0; }
err cudaMemcpyAsync(void* d, const void* s, size_t n, int k, void* st) { (void)d; (void)s; (void)n; (void)k; (void)st; return 0; }
err cudaMemsetAsync(void* d, int v, size_t n, void* st) { (void)d; (void)v; (void)n; (void)st; return 0; }
err cudaOccupancyMaxActiveClusters(int* n, const void* f, const launch_config* c) { (void)f; (void)c; *n = 7; return 0; }
err cudaPointerGetAttributes(void* a, const void* p) { (void)a; (void)p; last = 1; return 1; }
err cudaStreamCreateWithFlags(void** s, unsigned f) { (void)f; *s = malloc(1); return 0; }
err cudaStreamCreateWithPriority(void** s, unsigned f, int p) { (void)f; (void)p; *s = malloc(1); return 0; }
err cudaStreamDestroy(void* s) { free(s); return 0; }
err cudaStreamIsCapturing(void* s, int* v) { (void)s; *v = capturing; ++asked; return 0; }
err cudaStreamQuery(void* s) { (void)s; ++asked; return 0; }
err cudaStreamSynchronize(void* s) { (void)s; return 0; }
err cudaStreamWaitEvent(void* s, void* e, unsigned f) { (void)s; (void)e; (void)f; return 0; }
