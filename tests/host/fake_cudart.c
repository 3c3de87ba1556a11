/* A CUDA runtime without a GPU, preloaded in front of libcudart by the host-logic tests:
 * device memory is zeroed host memory under a budget, launches are recorded by kernel
 * name and do nothing, and the test decides which launch fails and which leaves bits in
 * the status word that it is given. */
#define _GNU_SOURCE
#include <stdint.h>
#include <stdio.h>
#include <stdlib.h>
#include <string.h>
#include <sys/mman.h>

enum { OK = 0, INVALID = 1, OOM = 2, LAUNCH_OUT_OF_RESOURCES = 701 };
#define NBLOCK 65536
#define NKERNEL 1024

static struct { char *p; size_t n; } block[NBLOCK];
static struct { const void *f; char name[160]; } kernel[NKERNEL];
static int nkernel, last_error;
static size_t total = (size_t)284 << 30, used;
static char log_[1 << 22], fail_name[80], mark_name[80], watch_name[80];
static size_t nlog;
static long long fail_at = -1, malloc_at = -1, mark_left, mark_arg, mark_bits, watch_z;

/* ---- the test's side ---- */
void fake_total(long long n) { total = (size_t)n; }
long long fake_used(void) { return (long long)used; }
/* the n-th launch from now (0: the next) whose kernel's name contains `name` fails */
void fake_fail(const char *name, long long n) { snprintf(fail_name, sizeof fail_name, "%s", name); fail_at = n; }
/* device allocations from the n-th on (0: the next) find no memory; negative: none fails */
void fake_fail_malloc(long long n) { malloc_at = n; }
/* the next n launches of such kernels set `bits` in the int that their argument `arg` points to */
void fake_mark(const char *name, long long n, long long arg, long long bits) {
  snprintf(mark_name, sizeof mark_name, "%s", name);
  mark_left = n, mark_arg = arg, mark_bits = bits;
}
/* the largest gridDim.z of the launches whose kernel's name contains `name`, from now */
void fake_watch(const char *name) { snprintf(watch_name, sizeof watch_name, "%s", name), watch_z = 0; }
long long fake_watched(void) { return watch_z; }
const char *fake_log(void) { return log_; }
void fake_clear(void) { nlog = 0, log_[0] = 0; }
int fake_is_live(const void *p) {
  for (int i = 0; i < NBLOCK; ++i)
    if (block[i].p && (const char *)p >= block[i].p && (const char *)p < block[i].p + block[i].n) return 1;
  return 0;
}

/* ---- memory ---- */
static int set(int e) { if (e) last_error = e; return e; }
int cudaMalloc(void **p, size_t n) {
  *p = NULL;
  if (used + n > total || malloc_at == 0) return set(OOM);
  if (malloc_at > 0) --malloc_at;
  for (int i = 0; i < NBLOCK; ++i)
    if (!block[i].p) {
      void *q = mmap(NULL, n ? n : 1, PROT_READ | PROT_WRITE, MAP_PRIVATE | MAP_ANONYMOUS | MAP_NORESERVE, -1, 0);
      if (q == MAP_FAILED) return set(OOM);
      block[i].p = q, block[i].n = n, used += n, *p = q;
      return OK;
    }
  return set(OOM);
}
int cudaFree(void *p) {
  if (!p) return OK;
  for (int i = 0; i < NBLOCK; ++i)
    if (block[i].p == (char *)p) {
      munmap(p, block[i].n ? block[i].n : 1);
      used -= block[i].n, block[i].p = NULL;
      return OK;
    }
  return set(INVALID);
}
int cudaMemGetInfo(size_t *f, size_t *t) { *f = total - used, *t = total; return OK; }
int cudaHostAlloc(void **p, size_t n, unsigned f) { *p = calloc(1, n ? n : 1); return OK; }
int cudaMallocHost(void **p, size_t n) { *p = calloc(1, n ? n : 1); return OK; }
int cudaFreeHost(void *p) { free(p); return OK; }
int cudaMemPoolCreate(void **p, const void *props) { *p = (void *)1; return OK; }
int cudaMemPoolSetAttribute(void *p, int a, void *v) { return OK; }
int cudaMemPoolTrimTo(void *p, size_t n) { return OK; }
int cudaMallocFromPoolAsync(void **p, size_t n, void *pool, void *st) { return cudaMalloc(p, n); }
int cudaFreeAsync(void *p, void *st) { return cudaFree(p); }
#define BIG ((size_t)64 << 20) /* blocks of this size and more stay untouched zeros */
static void copy(void *d, const void *s, size_t n) { if (n < BIG) memmove(d, s, n); }
int cudaMemcpy(void *d, const void *s, size_t n, int k) { copy(d, s, n); return OK; }
int cudaMemcpyAsync(void *d, const void *s, size_t n, int k, void *st) { copy(d, s, n); return OK; }
int cudaMemset(void *d, int v, size_t n) { if (n < BIG) memset(d, v, n); return OK; }
int cudaMemsetAsync(void *d, int v, size_t n, void *st) { return cudaMemset(d, v, n); }
int cudaMemset2DAsync(void *d, size_t pitch, int v, size_t w, size_t h, void *st) { return OK; }
struct attributes { int type, device; void *dptr, *hptr; long rest[8]; };
int cudaPointerGetAttributes(struct attributes *a, const void *p) {
  a->type = fake_is_live(p) ? 2 : 0;
  return OK;
}

/* ---- launches ---- */
void **__cudaRegisterFatBinary(void *x) { static void *h; return &h; }
void __cudaRegisterFatBinaryEnd(void **h) {}
void __cudaUnregisterFatBinary(void **h) {}
void __cudaRegisterVar(void **h, char *v, char *a, const char *n, int e, size_t s, int c, int g) {}
void __cudaRegisterFunction(void **h, const char *f, char *d, const char *name, int t, void *a, void *b, void *c,
                            void *e, int *w) {
  if (nkernel < NKERNEL) kernel[nkernel].f = f, snprintf(kernel[nkernel++].name, 160, "%s", name);
}
struct dim { uint32_t x, y, z; };
static struct dim config_grid;
static size_t config_smem;
static void *config_stream;
unsigned __cudaPushCallConfiguration(uint64_t gxy, uint32_t gz, uint64_t bxy, uint32_t bz, size_t smem, void *st) {
  config_grid = (struct dim){(uint32_t)gxy, (uint32_t)(gxy >> 32), gz};
  config_smem = smem, config_stream = st;
  return 0;
}
int __cudaPopCallConfiguration(void *g, void *b, size_t *smem, void **st) {
  const uint32_t one[3] = {1, 1, 1};
  memcpy(g, &config_grid, sizeof config_grid), memcpy(b, one, sizeof one);
  *smem = config_smem, *st = config_stream;
  return OK;
}
int __cudaGetKernel(const void **k, const void *f) { *k = f; return OK; }
int __cudaLaunchKernel(const void *k, struct dim g, struct dim b, void **args, size_t smem, void *st) {
  const char *name = "?";
  for (int i = 0; i < nkernel; ++i)
    if (kernel[i].f == k) name = kernel[i].name;
  if (nlog + strlen(name) + 2 < sizeof log_) nlog += (size_t)sprintf(log_ + nlog, "%s\n", name);
  if (watch_name[0] && strstr(name, watch_name) && g.z > watch_z) watch_z = g.z;
  if (fail_at >= 0 && strstr(name, fail_name) && fail_at-- == 0) return set(LAUNCH_OUT_OF_RESOURCES);
  if (mark_left > 0 && strstr(name, mark_name)) --mark_left, **(int **)args[mark_arg] |= (int)mark_bits;
  return OK;
}
int cudaFuncSetAttribute(const void *f, int a, int v) { return OK; }
int cudaGetLastError(void) { const int e = last_error; last_error = OK; return e; }
const char *cudaGetErrorString(int e) { return e == LAUNCH_OUT_OF_RESOURCES ? "too many resources requested" : "fake error"; }
int cudaGetSymbolAddress(void **p, const void *s) { return cudaMalloc(p, (size_t)32 << 20); }
static int encode(void) { return 0; }
int cudaGetDriverEntryPointByVersion(const char *n, void **f, unsigned v, unsigned long long fl, int *q) {
  *f = (void *)encode, *q = 0;
  return OK;
}

/* ---- the rest ---- */
int cudaGetDevice(int *d) { *d = 0; return OK; }
int cudaSetDevice(int d) { return OK; }
int cudaDeviceGetAttribute(int *v, int a, int d) { *v = 152; return OK; }
int cudaEventCreate(void **e) { *e = malloc(1); return OK; }
int cudaEventCreateWithFlags(void **e, unsigned f) { return cudaEventCreate(e); }
int cudaEventDestroy(void *e) { free(e); return OK; }
int cudaEventRecord(void *e, void *s) { return OK; }
int cudaEventSynchronize(void *e) { return OK; }
int cudaEventElapsedTime(float *ms, void *a, void *b) { *ms = 100.f; return OK; }
int cudaStreamCreateWithFlags(void **s, unsigned f) { *s = malloc(1); return OK; }
int cudaStreamDestroy(void *s) { free(s); return OK; }
int cudaStreamSynchronize(void *s) { return OK; }
int cudaStreamWaitEvent(void *s, void *e, unsigned f) { return OK; }
/* a graph remembers nothing; its launch appears in the log */
int cudaStreamBeginCapture(void *s, int m) { return OK; }
int cudaStreamEndCapture(void *s, void **g) { *g = malloc(1); return OK; }
int cudaGraphDestroy(void *g) { free(g); return OK; }
int cudaGraphInstantiate(void **e, void *g, unsigned long long f) { *e = malloc(1); return OK; }
int cudaGraphExecDestroy(void *e) { free(e); return OK; }
int cudaGraphGetNodes(void *g, void *n, size_t *k) { *k = 1; return OK; }
int cudaGraphLaunch(void *e, void *s) {
  if (nlog + 16 < sizeof log_) nlog += (size_t)sprintf(log_ + nlog, "graph launch\n");
  return OK;
}
