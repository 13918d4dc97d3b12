/* A stand-in for the CUDA runtime, preloaded into a child process on a machine without a GPU: device memory is host
 * memory that nothing touches, kernels do not run.  Every allocation, release, device-to-device copy,
 * function attribute and launch is written to FAKE_CUDART_LOG; a release of something that is not live is written as "bad-free".  Allocation number
 * FAKE_CUDART_FAIL (from 1) fails. */
#include <stddef.h>
#include <stdint.h>
#include <stdio.h>
#include <stdlib.h>
#include <string.h>

typedef int err_t;
enum { kMax = 4096 };
static uintptr_t live[kMax];
static uintptr_t next_addr = 0x100000000ull;

static void note(const char* what, uintptr_t a, uintptr_t b, size_t n) {
  const char* path = getenv("FAKE_CUDART_LOG");
  FILE* f = path ? fopen(path, "a") : NULL;
  if (!f) return;
  fprintf(f, "%s %llu %llu %llu\n", what, (unsigned long long)a, (unsigned long long)b, (unsigned long long)n);
  fclose(f);
}

err_t cudaGetDeviceCount(int* n) { *n = 1; return 0; }
err_t cudaSetDevice(int d) { (void)d; return 0; }
err_t cudaGetDevice(int* d) { *d = 0; return 0; }
err_t cudaDeviceGetAttribute(int* v, int attr, int d) { (void)d; *v = attr == 97 ? 232448 : 152; return 0; }
err_t cudaDeviceSynchronize(void) { return 0; }
err_t cudaStreamSynchronize(void* s) { (void)s; return 0; }
err_t cudaGetLastError(void) { return 0; }
err_t cudaFuncSetAttribute(const void* f, int a, int v) {
  note("attribute", (uintptr_t)f, (uintptr_t)a, (size_t)v);
  return 0;
}
err_t cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int* n, const void* f, int t, size_t s, unsigned g) {
  (void)f; (void)t; (void)s; (void)g;
  *n = 1;
  return 0;
}
err_t cudaMalloc(void** p, size_t n) {
  static int count;
  const char* fail = getenv("FAKE_CUDART_FAIL");
  *p = NULL;
  if (fail && ++count == atoi(fail)) { note("no-memory", 0, 0, n); return 2; }
  for (int i = 0; i < kMax; i++)
    if (!live[i]) {
      live[i] = next_addr;
      next_addr += (n + 511) / 256 * 256;
      *p = (void*)live[i];
      note("malloc", live[i], 0, n);
      return 0;
    }
  return 2;
}
err_t cudaFree(void* p) {
  if (!p) return 0;
  for (int i = 0; i < kMax; i++)
    if (live[i] == (uintptr_t)p) {
      live[i] = 0;
      note("free", (uintptr_t)p, 0, 0);
      return 0;
    }
  note("bad-free", (uintptr_t)p, 0, 0);
  return 1;
}
err_t cudaMemset(void* p, int v, size_t n) { (void)p; (void)v; (void)n; return 0; }
err_t cudaMemsetAsync(void* p, int v, size_t n, void* s) { (void)p; (void)v; (void)n; (void)s; return 0; }
err_t cudaMemcpyAsync(void* d, const void* s, size_t n, int kind, void* st) {
  (void)kind; (void)st;
  note("copy", (uintptr_t)d, (uintptr_t)s, n);
  return 0;
}
err_t cudaStreamIsCapturing(void* s, int* status) {
  (void)s;
  *status = getenv("FAKE_CUDART_CAPTURING") ? 1 : 0;
  return 0;
}
err_t cudaEventCreate(void** e) { *e = (void*)1; return 0; }
err_t cudaEventDestroy(void* e) { (void)e; return 0; }
err_t cudaEventRecord(void* e, void* s) { (void)e; (void)s; return 0; }
err_t cudaEventSynchronize(void* e) { (void)e; return 0; }
err_t cudaEventElapsedTime(float* ms, void* a, void* b) { /* the times of FAKE_CUDART_MS, a comma-separated list */
  static int turn;
  const char* t = getenv("FAKE_CUDART_MS");
  (void)a; (void)b;
  for (int i = 0; t && i < turn; i++) {
    t = strchr(t, ',');
    if (t) t++;
  }
  turn++;
  *ms = t ? (float)atof(t) : 1.f;
  note("elapsed", 0, 0, (size_t)turn);
  return 0;
}
typedef struct { unsigned x, y, z; } dim3_t;
static dim3_t last_grid, last_block;
static size_t last_smem;
static void* last_stream;
unsigned __cudaPushCallConfiguration(dim3_t grid, dim3_t block, size_t smem, void* stream) {
  last_grid = grid;
  last_block = block;
  last_smem = smem;
  last_stream = stream;
  note("launch", grid.x, block.x, smem);
  return 0;
}
err_t __cudaPopCallConfiguration(dim3_t* grid, dim3_t* block, size_t* smem, void* stream) {
  *grid = last_grid;
  *block = last_block;
  *smem = last_smem;
  *(void**)stream = last_stream;
  return 0;
}
err_t cudaHostAlloc(void** p, size_t n, unsigned flags) { (void)flags; *p = calloc(1, n); return 0; }
err_t cudaFreeHost(void* p) { free(p); return 0; }
err_t cudaStreamCreateWithFlags(void** s, unsigned f) { (void)f; *s = (void*)1; return 0; }
err_t cudaStreamBeginCapture(void* s, int mode) { (void)s; (void)mode; return 0; }
err_t cudaStreamEndCapture(void* s, void** g) { (void)s; *g = (void*)1; return 0; }
err_t cudaGraphInstantiate(void** x, void* g, unsigned long long f) { (void)g; (void)f; *x = (void*)1; return 0; }
err_t cudaGraphLaunch(void* x, void* s) { (void)x; (void)s; return 0; }
err_t cudaGraphDestroy(void* g) { (void)g; return 0; }
err_t cudaGraphExecDestroy(void* x) { (void)x; return 0; }
err_t cudaLaunchKernel(const void* f, ...) { (void)f; return 0; }
err_t __cudaLaunchKernel(const void* f, ...) { (void)f; return 0; }
