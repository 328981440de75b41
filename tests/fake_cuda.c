/* The CUDA runtime calls of the library over host memory, for tests of its host
 * side without a GPU: allocations are counted and can be made to fail, kernels
 * do nothing, copies are copies.  Loaded in front of the runtime (LD_PRELOAD);
 * kernel registration stays the runtime's. */
#include <stddef.h>
#include <stdlib.h>
#include <string.h>

typedef struct { unsigned x, y, z; } dim3_t;
enum { MAXP = 4096 };
static void *live[MAXP];
static size_t size[MAXP];
static int fail_in, bad_frees, launches, query_result, queries, syncs;
static unsigned flags;

int fake_live(void) {
  int n = 0;
  for (int k = 0; k < MAXP; ++k) n += live[k] != NULL;
  return n;
}
long long fake_bytes(void) {
  long long n = 0;
  for (int k = 0; k < MAXP; ++k) n += live[k] ? (long long)size[k] : 0;
  return n;
}
void fake_fail_in(int n) { fail_in = n; } /* the n-th allocation from now on; 0: none */
int fake_pending(void) { return fail_in; }
int fake_bad_frees(void) { return bad_frees; }
int fake_launches(void) { return launches; }
/* what a stream query returns from now on, and the device's flags */
void fake_stream(int rc, unsigned f) { query_result = rc; flags = f; queries = syncs = 0; }
int fake_queries(void) { return queries; }
int fake_syncs(void) { return syncs; }

int cudaMalloc(void **p, size_t n) {
  if (fail_in > 0 && --fail_in == 0) return 2;
  for (int k = 0; k < MAXP; ++k)
    if (!live[k]) {
      size[k] = n;
      *p = live[k] = calloc(n + 256, 1);
      return 0;
    }
  return 2;
}
int cudaFree(void *p) {
  if (!p) return 0;
  for (int k = 0; k < MAXP; ++k)
    if (live[k] == p) {
      live[k] = NULL;
      free(p);
      return 0;
    }
  ++bad_frees;
  return 1;
}
int cudaMallocHost(void **p, size_t n) { return (*p = calloc(n, 1)) ? 0 : 2; }
int cudaFreeHost(void *p) { free(p); return 0; }
int cudaMemcpy(void *d, const void *s, size_t n, int k) { (void)k; memcpy(d, s, n); return 0; }
int cudaMemcpyAsync(void *d, const void *s, size_t n, int k, void *st) {
  (void)k; (void)st; memcpy(d, s, n); return 0;
}
int cudaMemset(void *d, int v, size_t n) { memset(d, v, n); return 0; }
int cudaMemsetAsync(void *d, int v, size_t n, void *st) { (void)st; memset(d, v, n); return 0; }
int cudaStreamSynchronize(void *st) { (void)st; ++syncs; return 0; }
int cudaStreamQuery(void *st) { (void)st; ++queries; return query_result; }
int cudaGetLastError(void) { return 0; }
int cudaPeekAtLastError(void) { return 0; }
int cudaGetDevice(int *d) { *d = 0; return 0; }
int cudaGetDeviceFlags(unsigned *f) { *f = flags; return 0; }
int cudaDeviceGetAttribute(int *v, int a, int d) { (void)a; (void)d; *v = 152; return 0; }
int cudaFuncSetAttribute(const void *f, int a, int v) { (void)f; (void)a; (void)v; return 0; }
int cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int *n, const void *f, int b, size_t s,
                                                          unsigned fl) {
  (void)f; (void)b; (void)s; (void)fl; *n = 2; return 0;
}
int __cudaGetKernel(void **k, const void *entry) { *k = (void *)entry; return 0; }
int __cudaLaunchKernel(void *k, dim3_t g, dim3_t b, void **args, size_t smem, void *st) {
  (void)k; (void)g; (void)b; (void)args; (void)smem; (void)st; ++launches; return 0;
}
int cudaLaunchKernelExC(const void *cfg, const void *f, void **args) {
  (void)cfg; (void)f; (void)args; ++launches; return 0;
}
