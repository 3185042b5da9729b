/* A CUDA runtime for host tests, preloaded before the real one: device memory
 * is host memory with a limit, kernels are not run, graphs are counted. The
 * library's host code (allocation, capture, errors) then runs without a GPU. */
#include <stddef.h>
#include <stdlib.h>
#include <string.h>

enum { kMax = 65536 };
static void* ptr[kMax];
static size_t len[kMax];
static int used_slots;
static size_t in_use, limit = (size_t)-1;
static long mallocs, fail_at = -1, launches, captures, replays;

void fake_set_limit(size_t bytes) { limit = bytes; }
void fake_fail_at(long k) { mallocs = 0; fail_at = k; }   /* the k-th allocation from now (0: the next) */
size_t fake_in_use(void) { return in_use; }
long fake_mallocs(void) { return mallocs; }
long fake_live(void) {
  long v = 0;
  for (int i = 0; i < used_slots; ++i) v += ptr[i] != NULL;
  return v;
}
long fake_launches(void) { return launches; }
long fake_captures(void) { return captures; }
long fake_replays(void) { return replays; }

int cudaMalloc(void** p, size_t n) {
  *p = NULL;
  if (mallocs++ == fail_at || n > limit || in_use > limit - n) return 2;
  int i = 0;
  while (i < used_slots && ptr[i]) ++i;
  if (i == kMax) return 2;
  if (i == used_slots) ++used_slots;
  ptr[i] = calloc(1, n);
  if (!ptr[i]) return 2;
  len[i] = n;
  in_use += n;
  *p = ptr[i];
  return 0;
}

int cudaFree(void* p) {
  for (int i = 0; p && i < used_slots; ++i)
    if (ptr[i] == p) {
      in_use -= len[i];
      free(p);
      ptr[i] = NULL;
      return 0;
    }
  return p ? 1 : 0;
}

int cudaMemGetInfo(size_t* free_bytes, size_t* total) {
  *total = limit;
  *free_bytes = limit > in_use ? limit - in_use : 0;
  return 0;
}

typedef struct { unsigned x, y, z; } dim3_t;
unsigned __cudaPushCallConfiguration(dim3_t g, dim3_t b, size_t s, void* st) {
  (void)g; (void)b; (void)s; (void)st;
  ++launches;
  return 1;   /* the kernel is not called */
}

int cudaMemcpy(void* d, const void* s, size_t n, int k) { (void)k; if (n) memmove(d, s, n); return 0; }
int cudaMemcpyAsync(void* d, const void* s, size_t n, int k, void* st) { (void)st; return cudaMemcpy(d, s, n, k); }
int cudaMemsetAsync(void* d, int v, size_t n, void* st) { (void)st; memset(d, v, n); return 0; }

static int handle;
static int make(void** h) { *h = &handle; return 0; }
int cudaStreamCreateWithFlags(void** s, unsigned f) { (void)f; return make(s); }
int cudaEventCreate(void** e) { return make(e); }
int cudaEventCreateWithFlags(void** e, unsigned f) { (void)f; return make(e); }
int cudaStreamDestroy(void* s) { (void)s; return 0; }
int cudaEventDestroy(void* e) { (void)e; return 0; }
int cudaEventRecord(void* e, void* s) { (void)e; (void)s; return 0; }
int cudaEventQuery(void* e) { (void)e; return 0; }
int cudaStreamWaitEvent(void* s, void* e, unsigned f) { (void)s; (void)e; (void)f; return 0; }
int cudaStreamSynchronize(void* s) { (void)s; return 0; }
int cudaStreamBeginCapture(void* s, int m) { (void)s; (void)m; ++captures; return 0; }
int cudaStreamEndCapture(void* s, void** g) { (void)s; return make(g); }
int cudaGraphInstantiate(void** e, void* g, unsigned long long f) { (void)g; (void)f; return make(e); }
int cudaGraphDestroy(void* g) { (void)g; return 0; }
int cudaGraphExecDestroy(void* e) { (void)e; return 0; }
int cudaGraphLaunch(void* e, void* s) { (void)e; (void)s; ++replays; return 0; }
int cudaHostAlloc(void** p, size_t n, unsigned f) { (void)f; *p = calloc(1, n); return *p ? 0 : 2; }
int cudaFreeHost(void* p) { free(p); return 0; }
int cudaGetLastError(void) { return 0; }
int cudaGetDevice(int* d) { *d = 0; return 0; }
int cudaSetDevice(int d) { (void)d; return 0; }
int cudaDeviceGetAttribute(int* v, int a, int d) {   /* SMs; shared memory a block */
  (void)d;
  *v = a == 16 ? 152 : a == 97 ? 232448 : 0;
  return 0;
}
int cudaFuncSetAttribute(const void* f, int a, int v) { (void)f; (void)a; (void)v; return 0; }
int cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int* n, const void* f, int b, size_t s, unsigned fl) {
  (void)f; (void)b; (void)s; (void)fl;
  *n = 1;
  return 0;
}
