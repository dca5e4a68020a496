/* A CUDA runtime without a GPU, for tests of libsk's host side: preloaded before libcudart, it answers the calls
 * libsk makes and writes one line per call that enqueues, allocates or frees to the file $FAKE_LOG. Control
 * variables (exported, set by the test through ctypes): */
#include <stdio.h>
#include <stdlib.h>
#include <string.h>

int fake_capturing = 0;              /* every stream is being captured */
unsigned long long fake_max = 0;     /* cudaMalloc of more bytes than this fails (0: none does) */
int fake_busy = 0;                   /* work behind every recorded event is still running */
int fake_kernels = 0, fake_coop = 0, fake_mallocs = 0, fake_frees = 0;
unsigned long long fake_last_malloc = 0;

enum { OK = 0, INVALID = 1, OOM = 2, NOT_READY = 600 };

int cudaGetDevice(int* d) { return *d = 0, OK; }
int cudaDeviceGetAttribute(int* v, int attr, int dev) {
  (void)dev;
  *v = attr == 16 ? 152 : attr == 97 ? 232448 : 0; /* multiprocessors, opt-in shared memory */
  return OK;
}
int cudaFuncSetAttribute(const void* f, int a, int v) { return (void)f, (void)a, (void)v, OK; }
int cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int* n, const void* f, int threads, size_t smem, unsigned fl) {
  (void)f, (void)fl;
  /* 64 registers a thread */
  int by_threads = 1024 / threads, by_smem = smem ? (int)(233472 / (smem + 1024)) : 32;
  *n = by_threads < by_smem ? by_threads : by_smem;
  return OK;
}
int __cudaGetKernel(void** k, const void* f) { return *k = (void*)f, OK; }
int __cudaLaunchKernel(void* k, ...) { return (void)k, ++fake_kernels, OK; }
typedef struct {
  unsigned x, y, z;
} dim3;
unsigned fake_grid = 0; /* CTAs of the last cooperative launch */
int cudaLaunchCooperativeKernel(const void* k, dim3 grid, dim3 block, void** args, size_t smem, void* st) {
  (void)k, (void)block, (void)args, (void)smem, (void)st;
  fake_grid = grid.x;
  return ++fake_coop, OK;
}
int cudaMalloc(void** p, size_t bytes) {
  if (fake_max && bytes > fake_max) return OOM;
  ++fake_mallocs;
  fake_last_malloc = bytes;
  return *p = malloc(64), OK;
}
int cudaFree(void* p) { return ++fake_frees, free(p), OK; }
int fake_memset_fails = 0;
int cudaMemsetAsync(void* p, int v, size_t n, void* st) {
  (void)p, (void)v, (void)st;
  return fake_memset_fails && n > 64 ? INVALID : OK;
}
int cudaMemcpyAsync(void* d, const void* s, size_t n, int kind, void* st) {
  (void)s, (void)st;
  if (kind == 2) memset(d, 0, n); /* device to host */
  return OK;
}
int cudaMemcpy(void* d, const void* s, size_t n, int kind) { return cudaMemcpyAsync(d, s, n, kind, 0); }
int cudaStreamIsCapturing(void* st, int* status) { return (void)st, *status = fake_capturing, OK; }
int cudaStreamGetId(void* st, unsigned long long* id) { return *id = (unsigned long long)(size_t)st, OK; }
int cudaStreamCreateWithFlags(void** st, unsigned fl) { return (void)fl, *st = malloc(8), OK; }
int cudaStreamDestroy(void* st) { return free(st), OK; }
int cudaStreamWaitEvent(void* st, void* e, unsigned fl) { return (void)st, (void)e, (void)fl, OK; }
int cudaThreadExchangeStreamCaptureMode(int* mode) { return (void)mode, OK; }
int cudaEventCreateWithFlags(void** e, unsigned fl) { return (void)fl, *e = malloc(8), OK; }
int cudaEventDestroy(void* e) { return free(e), OK; }
int cudaEventRecord(void* e, void* st) { return (void)e, (void)st, OK; }
int cudaEventQuery(void* e) { return (void)e, fake_busy ? NOT_READY : OK; }
int cudaDeviceSynchronize(void) { return OK; }
int cudaStreamSynchronize(void* st) { return (void)st, OK; }
int cudaGetLastError(void) { return OK; }
static int encode(void* map, ...) { return (void)map, 0; }
int cudaGetDriverEntryPointByVersion(const char* name, void** f, unsigned v, unsigned long long fl, int* q) {
  (void)name, (void)v, (void)fl;
  return *f = (void*)encode, *q = 0, OK;
}
