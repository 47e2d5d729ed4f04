/* A CUDA runtime for host-logic tests without a GPU: "device" memory is host
 * memory, copies are made at once, kernels are not run, and every copy,
 * launch and wait is recorded.  fake_mark gives an address range the memory type
 * and device that cudaPointerGetAttributes reports for it. */
#include <stdio.h>
#include <stdlib.h>
#include <string.h>

typedef struct { unsigned x, y, z; } dim3;
typedef struct { int type, device; void* dev; void* host; long reserved[8]; } Attributes;
typedef struct { const char* at; size_t bytes; int type, device; } Range;

static Range ranges[4096];
static int n_ranges, sms = 152, device;
static struct { const void* fun; const char* name; } funs[4096];
static int n_funs;
static char* text;
static size_t text_len, text_cap;
static struct { dim3 grid, block; size_t smem; void* stream; } pushed;

static void record(const char* line) {
  size_t n = strlen(line);
  if (text_len + n + 1 > text_cap) text = realloc(text, text_cap = 2 * (text_len + n + 1));
  memcpy(text + text_len, line, n + 1);
  text_len += n;
}
static void record_launch(const void* fun) {
  char line[4200];
  const char* name = "?";
  for (int i = 0; i < n_funs; ++i)
    if (funs[i].fun == fun) name = funs[i].name;
  snprintf(line, sizeof(line), "launch %.4000s\n", name);
  record(line);
}

void fake_sms(int n) { sms = n; }
void fake_mark(const void* at, size_t bytes, int type, int dev) {
  ranges[n_ranges++] = (Range){at, bytes, type, dev};
}
const char* fake_calls(void) { return text ? text : ""; }
void fake_clear(void) { text_len = 0; if (text) text[0] = 0; }

int cudaMalloc(void** p, size_t n) {
  *p = calloc(n ? n : 1, 1);
  fake_mark(*p, n, 2, device);
  return 0;
}
int cudaFree(void* p) {
  for (int i = 0; i < n_ranges; ++i)
    if (ranges[i].at == p) ranges[i] = ranges[--n_ranges];
  free(p);
  return 0;
}
int cudaMallocHost(void** p, size_t n) { *p = calloc(n, 1); return 0; }
int cudaFreeHost(void* p) { free(p); return 0; }
int cudaPointerGetAttributes(Attributes* a, const void* p) {
  memset(a, 0, sizeof(*a));
  a->device = -1;
  for (int i = n_ranges - 1; i >= 0; --i)
    if ((const char*)p >= ranges[i].at && (const char*)p < ranges[i].at + ranges[i].bytes) {
      a->type = ranges[i].type;
      a->device = ranges[i].device;
      break;
    }
  return 0;
}
int cudaMemcpyAsync(void* d, const void* s, size_t n, int kind, void* stream) {
  char line[96];
  snprintf(line, sizeof(line), "copy %zu %zu %zu\n", (size_t)d, (size_t)s, n);
  record(line);
  memmove(d, s, n);
  return 0;
}
int cudaMemcpy(void* d, const void* s, size_t n, int kind) { memmove(d, s, n); return 0; }
int cudaMemset(void* d, int v, size_t n) { memset(d, v, n); return 0; }
int cudaMemsetAsync(void* d, int v, size_t n, void* stream) { memset(d, v, n); return 0; }
int cudaMemGetInfo(size_t* f, size_t* t) { *f = *t = (size_t)1 << 32; return 0; }
int cudaGetDevice(int* d) { *d = device; return 0; }
int cudaDeviceGetAttribute(int* v, int attr, int dev) { *v = attr == 16 ? sms : 1; return 0; }
int cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int* n, const void* f, int b, size_t s,
                                                           unsigned flags) { *n = 2; return 0; }
int cudaFuncSetAttribute(const void* f, int a, int v) { return 0; }
int cudaGetLastError(void) { return 0; }
const char* cudaGetErrorString(int e) { return "fake"; }
int cudaStreamSynchronize(void* s) { record("wait\n"); return 0; }
int cudaStreamCreateWithFlags(void** s, unsigned f) { *s = (void*)1; return 0; }
int cudaStreamDestroy(void* s) { return 0; }
int cudaStreamIsCapturing(void* s, int* st) { *st = 0; return 0; }
int cudaStreamBeginCapture(void* s, int mode) { return 0; }
int cudaStreamEndCapture(void* s, void** g) { *g = (void*)1; return 0; }
int cudaGraphInstantiate(void** e, void* g, unsigned long long f) { *e = (void*)1; return 0; }
int cudaGraphLaunch(void* e, void* s) { record("graph\n"); return 0; }
int cudaGraphDestroy(void* g) { return 0; }
int cudaGraphExecDestroy(void* e) { return 0; }
int cudaEventCreate(void** e) { *e = (void*)1; return 0; }
int cudaEventDestroy(void* e) { return 0; }
int cudaEventRecord(void* e, void* s) { return 0; }
int cudaEventSynchronize(void* e) { return 0; }
int cudaEventElapsedTime(float* ms, void* a, void* b) { *ms = 0.f; return 0; }
int cudaGetSymbolAddress(void** p, const void* s) { return 1; }
int cudaGetDriverEntryPointByVersion(const char* n, void** p, unsigned v, unsigned long long f,
                                     int* st) { return 1; }
int cudaLaunchKernelExC(const void* cfg, const void* f, void** args) { record_launch(f); return 0; }
int cudaLaunchCooperativeKernel(const void* f, dim3 g, dim3 b, void** args, size_t sm, void* s) {
  record_launch(f);
  return 0;
}

/* what the compiler's launch and registration code calls */
void** __cudaRegisterFatBinary(void* bin) { static void* h; return &h; }
void __cudaRegisterFatBinaryEnd(void** h) {}
void __cudaUnregisterFatBinary(void** h) {}
void __cudaRegisterVar(void** h, char* hv, char* da, const char* name, int ext, size_t size,
                       int constant, int global) {}
void __cudaRegisterFunction(void** h, const char* host, char* dev, const char* name, int limit,
                            void* tid, void* bid, dim3* bd, dim3* gd, int* ws) {
  funs[n_funs].fun = host;
  funs[n_funs++].name = name;
}
unsigned __cudaPushCallConfiguration(dim3 g, dim3 b, size_t sm, void* s) {
  pushed.grid = g;
  pushed.block = b;
  pushed.smem = sm;
  pushed.stream = s;
  return 0;
}
int __cudaPopCallConfiguration(dim3* g, dim3* b, size_t* sm, void* s) {
  *g = pushed.grid;
  *b = pushed.block;
  *sm = pushed.smem;
  *(void**)s = pushed.stream;
  return 0;
}
int __cudaGetKernel(void** k, const void* fun) { *k = (void*)fun; return 0; }
int __cudaLaunchKernel(void* k, dim3 g, dim3 b, void** args, size_t sm, void* s) {
  record_launch(k);
  return 0;
}
