// A stand-in for the CUDA runtime (preloaded by tests/fakert.py), so that the library's host
// side runs without a GPU: device memory is host memory, launches are logged and compute
// nothing, copies and fills happen at once.  Memory that was freed is kept aside, so a launch
// or a captured graph that still points into it is seen (fake_dead), as is a NULL argument, a
// copy or fill beyond an allocation, and a sum's partials for which there is no room.
// The eigensolver's entries (cuSOLVER) compute nothing either.
// Allocations of a range of sizes can be made to fail, clusters can be made impossible, and
// every timed interval is what the test says.
#define _GNU_SOURCE
#include <cuda_runtime_api.h>
#include <pthread.h>
#include <stdint.h>
#include <stdio.h>
#include <stdlib.h>
#include <string.h>

#define GUARD 65536
typedef struct { char *p; size_t n; int live; } Block;
// two solve lanes launch from two threads
static pthread_mutex_t mu = PTHREAD_RECURSIVE_MUTEX_INITIALIZER_NP;
#define LOCK pthread_mutex_lock(&mu)
#define UNLOCK pthread_mutex_unlock(&mu)

static Block *blocks;
static int nblocks, capblocks;

static size_t fail_lo = 1, fail_hi = 0;  // cudaMalloc of lo <= bytes <= hi fails
static int fail_skip, fail_count;        // after skip of them, count of them
static int clusters = 4;                 // what cudaOccupancyMaxActiveClusters says
static float times[2] = {1.f, 0.f};      // cudaEventElapsedTime: start, step
static int symbol_value;                 // what a read of a device symbol gives
static int dead;
static char dead_what[256];

void fake_fail(size_t lo, size_t hi, int skip, int count) { fail_lo = lo, fail_hi = hi, fail_skip = skip, fail_count = count; }
void fake_clusters(int n) { clusters = n; }
void fake_times(float start, float step) { times[0] = start, times[1] = step; }
void fake_symbol(int v) { symbol_value = v; }
int fake_dead(void) { return dead; }
const char *fake_dead_what(void) { return dead_what; }

static void *get(size_t n) {
  LOCK;
  if (nblocks == capblocks) blocks = realloc(blocks, sizeof(Block) * (capblocks = capblocks ? 2 * capblocks : 256));
  blocks[nblocks].p = calloc(1, n + GUARD);
  blocks[nblocks].n = n;
  blocks[nblocks].live = 1;
  void *p = blocks[nblocks++].p;
  UNLOCK;
  return p;
}
static int state(const void *p) {  // 1 live, 0 freed, -1 not one of ours
  int s = -1;
  LOCK;
  for (int i = 0; i < nblocks; ++i)
    if ((char *)p >= blocks[i].p && (char *)p < blocks[i].p + blocks[i].n) s = blocks[i].live;
  UNLOCK;
  return s;
}

static size_t room(const void *p) {  // bytes from p to its allocation's end; a host pointer: any
  size_t r = (size_t)1 << 62;
  LOCK;
  for (int i = 0; i < nblocks; ++i)
    if ((char *)p >= blocks[i].p && (char *)p < blocks[i].p + blocks[i].n + GUARD)
      r = (char *)p < blocks[i].p + blocks[i].n && blocks[i].live ? blocks[i].p + blocks[i].n - (char *)p : 0;
  UNLOCK;
  return r;
}
static void need(const void *p, size_t n, const char *what) {
  if (room(p) >= n) return;
  ++dead;
  snprintf(dead_what, sizeof dead_what, "%.200s: %zu bytes, room for %zu", what, n, room(p));
}

cudaError_t cudaMalloc(void **p, size_t n) {
  if (n >= fail_lo && n <= fail_hi && fail_skip-- <= 0 && fail_count > 0) {
    --fail_count;
    *p = NULL;
    return cudaErrorMemoryAllocation;
  }
  *p = get(n);
  return cudaSuccess;
}
cudaError_t cudaFree(void *p) {
  LOCK;
  for (int i = 0; i < nblocks; ++i)
    if (blocks[i].p == p) blocks[i].live = 0;
  UNLOCK;
  return cudaSuccess;
}
cudaError_t cudaMallocHost(void **p, size_t n) { *p = calloc(1, n); return cudaSuccess; }
cudaError_t cudaFreeHost(void *p) { free(p); return cudaSuccess; }

// ------------------------------------------------------------- launches
typedef struct { const void *fn; char name[256]; } Kernel;
static Kernel kernels[4096];
static int nkernels;
// the pointer arguments of the kernels whose buffers are watched
typedef struct { const char *name; int arg[6]; } Watch;  // -1 ends
static const Watch watch[] = {  // mangled: length and name
    {"11k_ring_dots", {2, 3, 4, -1}},       {"13k_ring_update", {2, 3, 4, 5, 6, -1}}, {"11k_ring_pass", {2, 3, 4, 5, -1}},
    {"16k_ring64_cluster", {2, 3, 6, 7, -1}}, {"11k_kacz_rows", {2, 3, 4, -1}},     {"12k_kacz_rings", {2, 3, 5, 6, -1}},
    {"10k_restrict", {3, 4, 5, -1}},        {"16k_restrict_lanes", {3, 4, 5, -1}},  {"9k_prolong", {3, 4, 5, -1}},
    {"10k_coarsest", {1, 2, 3, -1}},        {"9k_stencil", {1, 2, 4, -1}},          {"15k_stencil_lanes", {1, 2, 4, -1}},
    {"14k_stencil_tile", {1, 2, 4, -1}},    {"11k_kacz_tile", {2, 3, 4, 5, -1}},    {"11k_kacz_coop", {3, 4, 5, 6, -1}},
    {"12k_kacz_block", {3, 4, 5, 6, -1}},   {NULL, {-1}}};
typedef struct { char name[256]; const void *p[6]; int np, cluster; } Node;
typedef struct { Node *n; int count, cap; } Graph;
static Graph *capturing, last;
static Graph log_;

static void check(const Node *n) {
  LOCK;
  for (int i = 0; i < n->np; ++i)
    if (n->p[i] == NULL || state(n->p[i]) == 0) {
      ++dead;
      snprintf(dead_what, sizeof dead_what, "%.200s, pointer %d: %s", n->name, i, n->p[i] ? "freed" : "NULL");
    }
  UNLOCK;
}
static void add(Graph *g, const Node *n) {
  LOCK;
  if (g->count == g->cap) g->n = realloc(g->n, sizeof(Node) * (g->cap = g->cap ? 2 * g->cap : 64));
  g->n[g->count++] = *n;
  UNLOCK;
}
static cudaError_t launch(const void *fn, void **args, int cluster, unsigned grid) {
  Node n;
  memset(&n, 0, sizeof n);
  n.cluster = cluster;
  for (int i = 0; i < nkernels; ++i)
    if (kernels[i].fn == fn) strcpy(n.name, kernels[i].name);
  for (const Watch *w = watch; w->name; ++w)
    if (strstr(n.name, w->name)) {
      for (int k = 0; w->arg[k] >= 0; ++k) n.p[n.np++] = *(void **)args[w->arg[k]];
      break;
    }
  const char *t = strstr(n.name, "9k_mdot_dfILi"), *u = strstr(n.name, "6k_mdotI");
  if (t) need(*(void **)args[5], 32ul * atoi(t + 13) * grid * *(int *)args[4], "k_mdot_df");
  if (u) need(*(void **)args[5], 16ul * atoi(strstr(u, "Li") + 2) * grid * *(int *)args[4], "k_mdot");
  if (cluster && !clusters) return cudaErrorLaunchOutOfResources;
  if (capturing) {
    add(capturing, &n);
  } else {
    check(&n);
    add(&log_, &n);
  }
  return cudaSuccess;
}
static const char *names(const Graph *g) {
  static char *out;
  size_t len = 1;
  for (int i = 0; i < g->count; ++i) len += strlen(g->n[i].name) + 1;
  out = realloc(out, len);
  *out = 0;
  char *o = out;
  for (int i = 0; i < g->count; ++i) o += sprintf(o, "%s\n", g->n[i].name);
  return out;
}
const char *fake_captured(void) { return names(&last); }  // kernels of the last captured graph
const char *fake_launched(void) { return names(&log_); }  // launched outside graphs since fake_clear
void fake_clear(void) { log_.count = 0; }

void **__cudaRegisterFatBinary(void *b) { static void *h; (void)b; return &h; }
void __cudaRegisterFatBinaryEnd(void **h) { (void)h; }
void __cudaUnregisterFatBinary(void **h) { (void)h; }
void __cudaRegisterFunction(void **h, const char *host, char *dev, const char *name, int tl, uint3 *a, uint3 *b, dim3 *c,
                            dim3 *d, int *e) {
  (void)h, (void)dev, (void)tl, (void)a, (void)b, (void)c, (void)d, (void)e;
  if (nkernels == 4096) abort();
  kernels[nkernels].fn = host;
  snprintf(kernels[nkernels++].name, 256, "%s", name);
}
void __cudaRegisterVar(void **h, char *host, char *dev, const char *name, int ext, size_t n, int c, int g) {
  (void)h, (void)host, (void)dev, (void)name, (void)ext, (void)n, (void)c, (void)g;
}
static __thread struct { dim3 g, b; size_t sm; void *s; } conf[8];
static __thread int nconf;
unsigned __cudaPushCallConfiguration(dim3 g, dim3 b, size_t sm, void *s) {
  conf[nconf].g = g, conf[nconf].b = b, conf[nconf].sm = sm, conf[nconf++].s = s;
  return 0;
}
cudaError_t __cudaPopCallConfiguration(dim3 *g, dim3 *b, size_t *sm, void *s) {
  --nconf;
  *g = conf[nconf].g, *b = conf[nconf].b, *sm = conf[nconf].sm, *(void **)s = conf[nconf].s;
  return cudaSuccess;
}
cudaError_t __cudaGetKernel(cudaKernel_t *k, const void *fn) { *k = (cudaKernel_t)fn; return cudaSuccess; }
cudaError_t __cudaLaunchKernel(cudaKernel_t k, dim3 g, dim3 b, void **args, size_t sm, cudaStream_t s) {
  (void)b, (void)sm, (void)s;
  return launch((const void *)k, args, 0, g.x);
}
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t *c, const void *fn, void **args) {
  int cl = 0;
  for (unsigned i = 0; i < c->numAttrs; ++i) cl |= c->attrs[i].id == cudaLaunchAttributeClusterDimension;
  return launch(fn, args, cl, c->gridDim.x);
}

// ------------------------------------------------------- graphs and streams
cudaError_t cudaStreamBeginCapture(cudaStream_t s, enum cudaStreamCaptureMode m) {
  (void)s, (void)m;
  capturing = calloc(1, sizeof(Graph));
  return cudaSuccess;
}
cudaError_t cudaStreamEndCapture(cudaStream_t s, cudaGraph_t *g) {
  (void)s;
  last = *capturing;
  *g = (cudaGraph_t)capturing;
  capturing = NULL;
  return cudaSuccess;
}
cudaError_t cudaGraphInstantiate(cudaGraphExec_t *e, cudaGraph_t g, unsigned long long f) {
  (void)f;
  *e = (cudaGraphExec_t)g;
  return cudaSuccess;
}
cudaError_t cudaGraphLaunch(cudaGraphExec_t e, cudaStream_t s) {
  (void)s;
  for (int i = 0; i < ((Graph *)e)->count; ++i) check(&((Graph *)e)->n[i]);
  return cudaSuccess;
}
cudaError_t cudaGraphDestroy(cudaGraph_t g) { (void)g; return cudaSuccess; }
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t e) { (void)e; return cudaSuccess; }
cudaError_t cudaStreamCreateWithFlags(cudaStream_t *s, unsigned f) { (void)f; *s = (cudaStream_t)malloc(1); return cudaSuccess; }
cudaError_t cudaStreamDestroy(cudaStream_t s) { free(s); return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t s) { (void)s; return cudaSuccess; }
cudaError_t cudaStreamWaitEvent(cudaStream_t s, cudaEvent_t e, unsigned f) { (void)s, (void)e, (void)f; return cudaSuccess; }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t *e, unsigned f) { (void)f; *e = (cudaEvent_t)malloc(1); return cudaSuccess; }
cudaError_t cudaEventCreate(cudaEvent_t *e) { return cudaEventCreateWithFlags(e, 0); }
cudaError_t cudaEventDestroy(cudaEvent_t e) { free(e); return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t e, cudaStream_t s) { (void)e, (void)s; return cudaSuccess; }
cudaError_t cudaEventSynchronize(cudaEvent_t e) { (void)e; return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float *ms, cudaEvent_t a, cudaEvent_t b) {
  (void)a, (void)b;
  *ms = times[0] += times[1];
  return cudaSuccess;
}

// ------------------------------------------------------------------- copies
cudaError_t cudaMemcpy(void *d, const void *s, size_t n, enum cudaMemcpyKind k) {
  (void)k;
  need(d, n, "copy to"), need(s, n, "copy from");
  memmove(d, s, n);
  return cudaSuccess;
}
cudaError_t cudaMemcpyAsync(void *d, const void *s, size_t n, enum cudaMemcpyKind k, cudaStream_t st) {
  (void)st;
  return capturing ? cudaSuccess : cudaMemcpy(d, s, n, k);
}
cudaError_t cudaMemsetAsync(void *d, int v, size_t n, cudaStream_t s) {
  (void)s;
  need(d, n, "fill");
  if (!capturing) memset(d, v, n);
  return cudaSuccess;
}
cudaError_t cudaMemcpyFromSymbolAsync(void *d, const void *sym, size_t n, size_t o, enum cudaMemcpyKind k, cudaStream_t s) {
  (void)sym, (void)o, (void)k, (void)s;
  memset(d, 0, n);
  if (n == sizeof(int)) memcpy(d, &symbol_value, n);
  return cudaSuccess;
}
cudaError_t cudaMemcpyToSymbolAsync(const void *sym, const void *s, size_t n, size_t o, enum cudaMemcpyKind k, cudaStream_t st) {
  (void)sym, (void)o, (void)k, (void)st;
  if (n == sizeof(int)) memcpy(&symbol_value, s, n);
  return cudaSuccess;
}
cudaError_t cudaGetSymbolAddress(void **p, const void *sym) { (void)sym; *p = get(256); return cudaSuccess; }

// ------------------------------------------------------------------ queries
cudaError_t cudaGetDevice(int *d) { *d = 0; return cudaSuccess; }
cudaError_t cudaSetDevice(int d) { (void)d; return cudaSuccess; }
cudaError_t cudaGetLastError(void) { return cudaSuccess; }
const char *cudaGetErrorString(cudaError_t e) { return e ? "fake error" : "no error"; }
cudaError_t cudaDeviceGetAttribute(int *v, enum cudaDeviceAttr a, int d) {
  (void)d;
  *v = a == cudaDevAttrMultiProcessorCount ? 152 : 1;
  return cudaSuccess;
}
cudaError_t cudaFuncSetAttribute(const void *f, enum cudaFuncAttribute a, int v) { (void)f, (void)a, (void)v; return cudaSuccess; }
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int *n, const void *f, int t, size_t sm, unsigned fl) {
  (void)f, (void)t, (void)sm, (void)fl;
  *n = 2;
  return cudaSuccess;
}
cudaError_t cudaOccupancyMaxActiveClusters(int *n, const void *f, const cudaLaunchConfig_t *c) {
  (void)f, (void)c;
  *n = clusters;
  return cudaSuccess;
}

int cusolverDnCreate(void **h) { *h = get(1); return 0; }
int cusolverDnDestroy(void *h) { (void)h; return 0; }
int cusolverDnSetStream(void *h, cudaStream_t s) { (void)h, (void)s; return 0; }
int cusolverDnZhegvd_bufferSize(void *h, int t, int z, int u, int n, const void *A, int la, const void *B, int lb,
                                const double *W, int *lwork) {
  (void)h, (void)t, (void)z, (void)u, (void)n, (void)A, (void)la, (void)B, (void)lb, (void)W;
  *lwork = 1;
  return 0;
}
int cusolverDnZhegvd(void *h, int t, int z, int u, int n, void *A, int la, void *B, int lb, double *W, void *work, int lwork,
                     int *info) {
  (void)h, (void)t, (void)z, (void)u, (void)n, (void)A, (void)la, (void)B, (void)lb, (void)W, (void)work, (void)lwork;
  *info = 0;
  return 0;
}
