/* A CUDA runtime without a GPU, preloaded in front of the real one: device
   memory is host memory, a launch is a line in a log, and what a launch checks
   (the shared-memory limit of the function on the current device) is checked.
   The N-th launch can be made to fail. */
#include <stdint.h>
#include <stdio.h>
#include <stdlib.h>
#include <string.h>

typedef struct {
  unsigned x, y, z;
} dim3;

enum { DEVICES = 2, FUNCS = 512 };
static struct {
  const void* f;
  char name[256];
  int limit[DEVICES];
} funcs[FUNCS];
static int n_funcs, device, last_error, fail_in;
static char* log_text;
static size_t log_len;

static void note(const char* s) {
  const size_t n = strlen(s);
  log_text = realloc(log_text, log_len + n + 2);
  memcpy(log_text + log_len, s, n);
  log_len += n;
  log_text[log_len++] = '\n';
  log_text[log_len] = 0;
}
static int find(const void* f) {
  for (int i = 0; i < n_funcs; ++i)
    if (funcs[i].f == f) return i;
  return -1;
}

/* for the test */
const char* fake_log(void) { return log_text ? log_text : ""; }
void fake_clear(void) {
  log_len = 0;
  if (log_text) log_text[0] = 0;
}
void fake_fail_launch(int n) { fail_in = n; }

/* registration and launches, as the compiler's host code calls them */
void** __cudaRegisterFatBinary(void* bin) {
  static void* handle;
  (void)bin;
  return &handle;
}
void __cudaRegisterFatBinaryEnd(void** h) { (void)h; }
void __cudaUnregisterFatBinary(void** h) { (void)h; }
void __cudaRegisterVar(void** h, char* v, char* a, const char* n, int e, size_t s, int c, int g) {
  (void)h, (void)v, (void)a, (void)n, (void)e, (void)s, (void)c, (void)g;
}
void __cudaRegisterFunction(void** h, const char* f, char* d, const char* name, int t, void* a, void* b, void* c, void* e,
                            int* w) {
  (void)h, (void)d, (void)t, (void)a, (void)b, (void)c, (void)e, (void)w;
  if (n_funcs == FUNCS) abort();
  funcs[n_funcs].f = f;
  snprintf(funcs[n_funcs].name, sizeof funcs[n_funcs].name, "%s", name);
  for (int i = 0; i < DEVICES; ++i) funcs[n_funcs].limit[i] = 48 * 1024;
  ++n_funcs;
}
static struct {
  dim3 grid, block;
  size_t smem;
  void* stream;
} pushed;
unsigned __cudaPushCallConfiguration(dim3 grid, dim3 block, size_t smem, void* stream) {
  pushed.grid = grid;
  pushed.block = block;
  pushed.smem = smem;
  pushed.stream = stream;
  return 0;
}
int __cudaPopCallConfiguration(dim3* grid, dim3* block, size_t* smem, void* stream) {
  *grid = pushed.grid;
  *block = pushed.block;
  *smem = pushed.smem;
  *(void**)stream = pushed.stream;
  return 0;
}
int __cudaGetKernel(void** kernel, const void* f) {
  *kernel = (void*)f;
  return 0;
}
int cudaLaunchKernel(const void* f, dim3 grid, dim3 block, void** args, size_t smem, void* stream) {
  (void)grid, (void)block, (void)args, (void)stream;
  const int i = find(f);
  if (fail_in > 0 && --fail_in == 0) return last_error = 719;
  if (i < 0 || smem > (size_t)funcs[i].limit[device]) return last_error = 1;
  note(funcs[i].name);
  return 0;
}
int __cudaLaunchKernel(void* k, dim3 grid, dim3 block, void** args, size_t smem, void* stream) {
  return cudaLaunchKernel(k, grid, block, args, smem, stream);
}

/* the runtime's functions the network uses */
int cudaSetDevice(int d) {
  device = d;
  return 0;
}
int cudaGetDevice(int* d) {
  *d = device;
  return 0;
}
int cudaDeviceGetAttribute(int* v, int what, int d) {
  (void)what, (void)d;
  *v = 152;
  return 0;
}
int cudaFuncSetAttribute(const void* f, int what, int v) {
  const int i = find(f);
  if (i < 0) return 1;
  if (what == 8) funcs[i].limit[device] = v; /* cudaFuncAttributeMaxDynamicSharedMemorySize */
  return 0;
}
int cudaMalloc(void** p, size_t n) {
  *p = calloc(1, n);
  return *p ? 0 : 2;
}
int cudaFree(void* p) {
  free(p);
  return 0;
}
int cudaMemcpy(void* d, const void* s, size_t n, int kind) {
  (void)kind;
  memcpy(d, s, n);
  return 0;
}
int cudaMemcpyAsync(void* d, const void* s, size_t n, int kind, void* stream) {
  (void)stream;
  return cudaMemcpy(d, s, n, kind);
}
int cudaMemset(void* d, int v, size_t n) {
  memset(d, v, n);
  return 0;
}
int cudaStreamSynchronize(void* s) {
  (void)s;
  return 0;
}
int cudaGetLastError(void) {
  const int e = last_error;
  last_error = 0;
  return e;
}
static int encode_ok(void) { return 0; }
int cudaGetDriverEntryPointByVersion(const char* name, void** f, unsigned version, unsigned long long flags, int* status) {
  (void)name, (void)version, (void)flags;
  *f = (void*)encode_ok;
  *status = 0;
  return 0;
}
