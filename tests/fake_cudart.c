/* A CUDA runtime without a GPU, for tests of the library's host logic: device
 * memory is zeroed host memory, copies are carried out at once, kernels are not
 * run, and every call is reported, in order, to a callback.  Loaded before the
 * library, under the name the library asks for. */
#define _GNU_SOURCE
#include <stddef.h>
#include <stdint.h>
#include <string.h>
#include <sys/mman.h>

typedef struct { unsigned x, y, z; } dim3;
typedef struct { dim3 grid, block; size_t smem; void *stream, *attrs; unsigned nattrs; } launch_config;
/* call: name of the runtime function (launches: of the kernel), its stream
 * (NULL: the default stream), a pointer and a size where it has them */
typedef void (*report_fn)(const char *call, void *stream, void *ptr, size_t bytes, const dim3 *grid, void **args);

enum { kOk = 0, kNoMemory = 2, kMaxAllocs = 4096, kMaxKernels = 512 };

static report_fn g_report;
static int g_sms = 152, g_capturing;
static size_t g_fail_at;
static struct { char *p; size_t n; } g_alloc[kMaxAllocs];
static struct { const void *host; const char *name; } g_kernel[kMaxKernels];
static int g_nkernels;
static launch_config g_pushed;

void fake_report(report_fn f) { g_report = f; }
void fake_sms(int n) { g_sms = n; }
void fake_capturing(int on) { g_capturing = on; }
/* Allocations of exactly n bytes fail (0: none does). */
void fake_fail_at(int n) { g_fail_at = (size_t)n; }
/* Bytes from p to the end of its allocation, 0 outside all of them. */
size_t fake_room(const char *p) {
  for (int i = 0; i < kMaxAllocs; ++i)
    if (g_alloc[i].p && p >= g_alloc[i].p && p < g_alloc[i].p + g_alloc[i].n) return g_alloc[i].n - (size_t)(p - g_alloc[i].p);
  return 0;
}

static int say(const char *call, void *stream, void *ptr, size_t n) {
  if (g_report) g_report(call, stream, ptr, n, NULL, NULL);
  return kOk;
}

int cudaMalloc(void **p, size_t n) {
  say("cudaMalloc", NULL, NULL, n);
  if (g_fail_at && n == g_fail_at) return kNoMemory;
  for (int i = 0; i < kMaxAllocs; ++i) {
    if (g_alloc[i].p) continue;
    void *m = mmap(NULL, n ? n : 1, PROT_READ | PROT_WRITE, MAP_PRIVATE | MAP_ANONYMOUS | MAP_NORESERVE, -1, 0);
    if (m == MAP_FAILED) return kNoMemory;
    g_alloc[i].p = m;
    g_alloc[i].n = n ? n : 1;
    *p = m;
    return kOk;
  }
  return kNoMemory;
}
int cudaFree(void *p) {
  if (p == NULL) return kOk;
  say("cudaFree", NULL, p, 0);
  for (int i = 0; i < kMaxAllocs; ++i)
    if (g_alloc[i].p == p) {
      munmap(p, g_alloc[i].n);
      g_alloc[i].p = NULL;
      return kOk;
    }
  return 1;
}
static void fill(void *p, int v, size_t n) {
  if (v != 0 || n <= 65536) memset(p, v, n); /* (large arrays are cleared when they are new) */
}
int cudaMemset(void *p, int v, size_t n) { fill(p, v, n); return say("cudaMemset", NULL, p, n); }
int cudaMemsetAsync(void *p, int v, size_t n, void *st) { fill(p, v, n); return say("cudaMemsetAsync", st, p, n); }
int cudaMemcpy(void *d, const void *s, size_t n, int kind) {
  (void)kind;
  memcpy(d, s, n);
  return say("cudaMemcpy", NULL, d, n);
}
int cudaMemcpyAsync(void *d, const void *s, size_t n, int kind, void *st) {
  (void)kind;
  memcpy(d, s, n);
  return say("cudaMemcpyAsync", st, d, n);
}
int cudaMemcpy2DAsync(void *d, size_t dp, const void *s, size_t sp, size_t w, size_t h, int kind, void *st) {
  (void)kind;
  for (size_t i = 0; i < h; ++i) memcpy((char *)d + i * dp, (const char *)s + i * sp, w);
  return say("cudaMemcpy2DAsync", st, d, w * h);
}

int cudaStreamSynchronize(void *st) { return say("cudaStreamSynchronize", st, NULL, 0); }
int cudaStreamIsCapturing(void *st, int *status) { (void)st; *status = g_capturing; return kOk; }
int cudaStreamCreateWithFlags(void **st, unsigned flags) { static char s[64]; static int n; (void)flags; *st = s + (n++ & 63); return kOk; }
int cudaStreamDestroy(void *st) { (void)st; return kOk; }
int cudaStreamWaitEvent(void *st, void *e, unsigned flags) { (void)flags; return say("cudaStreamWaitEvent", st, e, 0); }
int cudaEventCreateWithFlags(void **e, unsigned flags) { static char s[64]; static int n; (void)flags; *e = s + (n++ & 63); return kOk; }
int cudaEventCreate(void **e) { return cudaEventCreateWithFlags(e, 0); }
int cudaEventDestroy(void *e) { (void)e; return kOk; }
int cudaEventRecord(void *e, void *st) { return say("cudaEventRecord", st, e, 0); }
int cudaEventSynchronize(void *e) { return say("cudaEventSynchronize", NULL, e, 0); }
int cudaEventElapsedTime(float *ms, void *a, void *b) { (void)a; (void)b; *ms = 1.0f; return kOk; }
int cudaGetDevice(int *d) { *d = 0; return kOk; }
int cudaDeviceGetAttribute(int *v, int attr, int dev) { (void)dev; *v = attr == 16 ? g_sms : 0; return kOk; }
int cudaFuncSetAttribute(const void *f, int attr, int v) { (void)attr; return say("cudaFuncSetAttribute", NULL, (void *)f, (size_t)v); }
int cudaGetLastError(void) { return kOk; }
const char *cudaGetErrorString(int e) { return e == kNoMemory ? "out of memory" : "error"; }
int cudaGetSymbolAddress(void **p, const void *sym) { *p = (void *)sym; return kOk; }

/* The two driver functions the library asks for: a descriptor holds the box it
 * was made for, and every pointer counts as pageable memory. */
static int encode_tiled(void *map, int type, unsigned rank, void *base, const uint64_t *dims, const uint64_t *strides,
                        const uint32_t *box) {
  (void)type; (void)base; (void)dims; (void)strides;
  memset(map, 0, 128);
  memcpy(map, box, rank * sizeof(*box));
  return 0;
}
static int pointer_attribute(void *v, int attr, uint64_t p) { (void)v; (void)attr; (void)p; return 1; }
int cudaGetDriverEntryPointByVersion(const char *name, void **fn, unsigned version, unsigned long long flags, int *q) {
  (void)version;
  (void)flags;
  *fn = strcmp(name, "cuTensorMapEncodeTiled") == 0 ? (void *)encode_tiled : (void *)pointer_attribute;
  *q = 0;
  return kOk;
}

static int launch(const void *f, const dim3 *grid, void *st, void **args) {
  const char *name = "?";
  for (int i = 0; i < g_nkernels; ++i)
    if (g_kernel[i].host == f) name = g_kernel[i].name;
  if (g_report) g_report(name, st, NULL, 0, grid, args);
  return grid->y > 65535 || grid->z > 65535 || grid->x > 2147483647u ? 9 : kOk;
}
int cudaLaunchKernelExC(const launch_config *c, const void *f, void **args) { return launch(f, &c->grid, c->stream, args); }
int __cudaGetKernel(const void **k, const void *f) { *k = f; return kOk; }
int __cudaLaunchKernel(const void *k, dim3 grid, dim3 block, void **args, size_t smem, void *st) {
  (void)block;
  (void)smem;
  return launch(k, &grid, st, args);
}
unsigned __cudaPushCallConfiguration(dim3 grid, dim3 block, size_t smem, void *st) {
  const launch_config c = {grid, block, smem, st, NULL, 0};
  g_pushed = c;
  return 0;
}
int __cudaPopCallConfiguration(dim3 *grid, dim3 *block, size_t *smem, void **st) {
  *grid = g_pushed.grid;
  *block = g_pushed.block;
  *smem = g_pushed.smem;
  *st = g_pushed.stream;
  return kOk;
}
void **__cudaRegisterFatBinary(void *bin) { static void *h; (void)bin; return &h; }
void __cudaRegisterFatBinaryEnd(void **h) { (void)h; }
void __cudaUnregisterFatBinary(void **h) { (void)h; }
void __cudaRegisterFunction(void **h, const char *host, char *dev, const char *name, int limit, void *t, void *b, void *bd,
                            void *gd, int *w) {
  (void)h; (void)dev; (void)limit; (void)t; (void)b; (void)bd; (void)gd; (void)w;
  if (g_nkernels < kMaxKernels) {
    g_kernel[g_nkernels].host = host;
    g_kernel[g_nkernels++].name = name;
  }
}
void __cudaRegisterVar(void **h, char *host, char *dev, const char *name, int ext, size_t n, int c, int g) {
  (void)h; (void)host; (void)dev; (void)name; (void)ext; (void)n; (void)c; (void)g;
}
