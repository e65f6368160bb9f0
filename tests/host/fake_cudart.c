/* A CUDA runtime without a GPU, preloaded in front of libcudart by tests of the host side of
 * libh4d: two "devices" whose memory is host memory, work done when it is queued, and waits
 * that take a while (so that threads overlap in them).  Kernels do nothing except
 * export_state, which is carried out.  A launch on a stream of another device than the
 * current one is refused, as CUDA does.  A memory pool keeps what is freed to it until the
 * next wait and then, if that is more than its release threshold, gives it back;
 * fake_device_bytes() is what the devices hold.  cudaDeviceReset ends the context: a pool
 * made before it is refused, device variables move and their old memory is gone.  fake_fail_new(k) makes this thread's k-th C++ allocation from then on
 * throw (-1: none), fake_fail_pinned(1) every allocation of pinned memory fail. */
#include <cuda.h>
#include <cuda_runtime_api.h>
#include <stdint.h>
#include <stdlib.h>
#include <string.h>
#include <sys/mman.h>
#include <unistd.h>

static __thread int t_dev;
static __thread cudaError_t t_last;
static __thread struct { dim3 g, b; size_t smem; cudaStream_t s; } t_cfg;

struct stream { int dev; };
static int stream_dev(cudaStream_t s) { return s ? ((struct stream *)s)->dev : t_dev; }

static cudaError_t ret(cudaError_t e) {
  if (e != cudaSuccess) t_last = e;
  return e;
}
static size_t held;
struct pool { size_t idle; unsigned long long keep; int dead; };
static unsigned long long ctx_id = 1;
static void *symbol;  /* the library's device variable */
struct head { size_t n; struct pool *from; char fill[240]; };
static struct pool *pools[16];
static int n_pools;
size_t fake_device_bytes(void) { return held; }
static cudaError_t give(void **p, size_t n, struct pool *from) {
  struct head *h = calloc(1, sizeof *h + n);
  if (!h) return ret(cudaErrorMemoryAllocation);
  h->n = n;
  h->from = from;
  __atomic_add_fetch(&held, n, __ATOMIC_SEQ_CST);
  *p = h + 1;
  return cudaSuccess;
}
static cudaError_t take(void *p) {
  struct head *h = p ? (struct head *)p - 1 : 0;
  if (!h) return cudaSuccess;
  if (h->from) h->from->idle += h->n;
  else __atomic_sub_fetch(&held, h->n, __ATOMIC_SEQ_CST);
  free(h);
  return cudaSuccess;
}
static void trim(struct pool *p, unsigned long long keep) {
  if (p->idle <= keep) return;
  __atomic_sub_fetch(&held, p->idle, __ATOMIC_SEQ_CST);
  p->idle = 0;
}

static __thread int new_left = -1;
static int no_pinned;
void _ZSt17__throw_bad_allocv(void);
void fake_fail_new(int k) { new_left = k; }
void fake_fail_pinned(int on) { no_pinned = on; }
void *_Znwm(size_t n) {
  if (new_left >= 0 && new_left-- == 0) _ZSt17__throw_bad_allocv();
  return malloc(n);
}

/* ---- registration and launches ---- */
static struct { const void *host; char name[256]; } kernels[256];
static int n_kernels;
void **__cudaRegisterFatBinary(void *p) { (void)p; static void *h; return &h; }
void __cudaRegisterFatBinaryEnd(void **h) { (void)h; }
void __cudaUnregisterFatBinary(void **h) { (void)h; }
void __cudaRegisterVar(void **h, char *v, char *d, const char *n, int e, size_t s, int c, int g) {
  (void)h; (void)v; (void)d; (void)n; (void)e; (void)s; (void)c; (void)g;
}
void __cudaRegisterFunction(void **h, const char *host, char *dev, const char *name, int lim, void *t, void *b, void *bd, void *gd, int *w) {
  (void)h; (void)dev; (void)lim; (void)t; (void)b; (void)bd; (void)gd; (void)w;
  if (n_kernels == 256) abort();
  kernels[n_kernels].host = host;
  strncpy(kernels[n_kernels++].name, name, 255);
}
cudaError_t __cudaGetKernel(cudaKernel_t *k, const void *host) {
  for (int i = 0; i < n_kernels; ++i)
    if (kernels[i].host == host) { *k = (cudaKernel_t)kernels[i].name; return cudaSuccess; }
  return ret(cudaErrorInvalidDeviceFunction);
}
unsigned __cudaPushCallConfiguration(dim3 g, dim3 b, size_t smem, cudaStream_t s) {
  t_cfg.g = g; t_cfg.b = b; t_cfg.smem = smem; t_cfg.s = s;
  return 0;
}
cudaError_t __cudaPopCallConfiguration(dim3 *g, dim3 *b, size_t *smem, void *s) {
  *g = t_cfg.g; *b = t_cfg.b; *smem = t_cfg.smem; *(cudaStream_t *)s = t_cfg.s;
  return cudaSuccess;
}
/* the first fields of a replica's table entry */
struct rep { double L; float scale, c_drift; int n_water, nw3, n_pairs, cap_pairs, atom_off, cap_atoms; };
cudaError_t __cudaLaunchKernel(cudaKernel_t k, dim3 g, dim3 b, void **a, size_t smem, cudaStream_t s) {
  (void)g; (void)b; (void)smem;
  if (stream_dev(s) != t_dev) return ret(cudaErrorInvalidResourceHandle);
  if (strstr((const char *)k, "export_state")) {
    const struct rep *r = *(struct rep **)a[0];
    const int n = r->nw3 + *(int *)a[1] * r->n_pairs;
    const uint32_t *pos = *(uint32_t **)a[2];
    const float *hi = *(float **)a[3], *lo = *(float **)a[4];
    char *dst = *(char **)a[5];
    double *x = *(double **)a[6], *v = *(double **)a[7];
    if (x || v) memcpy(dst, r, (size_t)((char *)(x ? x : v) - dst));
    for (int i = 0; i < n; ++i)
      for (int d = 0; d < 3; ++d) {
        const size_t w = ((size_t)r->atom_off + i) * 4 + d;
        if (x) x[3 * i + d] = pos[w] * (r->L / 4294967296.0);
        if (v) v[3 * i + d] = (double)hi[w] + (double)lo[w];
      }
  }
  return cudaSuccess;
}

/* ---- devices, streams, memory ---- */
cudaError_t cudaGetSymbolAddress(void **p, const void *s);
static CUresult ctx_get_id(CUcontext c, unsigned long long *id) { (void)c; *id = ctx_id; return CUDA_SUCCESS; }
cudaError_t cudaGetDriverEntryPointByVersion(const char *name, void **f, unsigned v, unsigned long long fl,
                                             enum cudaDriverEntryPointQueryResult *st) {
  (void)v; (void)fl;
  *f = strcmp(name, "cuCtxGetId") == 0 ? (void *)ctx_get_id : 0;
  if (st) *st = *f ? cudaDriverEntryPointSuccess : cudaDriverEntryPointSymbolNotFound;
  return cudaSuccess;
}
cudaError_t cudaDeviceReset(void) {
  for (int i = 0; i < n_pools; ++i) { trim(pools[i], 0); pools[i]->dead = 1; }
  if (symbol) {
    void *old = symbol;
    cudaGetSymbolAddress((symbol = 0, &symbol), 0); /* at another address */
    munmap(old, 16 << 20);
  }
  ++ctx_id;
  return cudaSuccess;
}
cudaError_t cudaGetDeviceCount(int *n) { *n = 2; return cudaSuccess; }
cudaError_t cudaGetDevice(int *d) { *d = t_dev; return cudaSuccess; }
cudaError_t cudaSetDevice(int d) { t_dev = d; return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int *v, enum cudaDeviceAttr a, int d) {
  (void)d;
  *v = a == cudaDevAttrComputeCapabilityMajor ? 10 : a == cudaDevAttrComputeCapabilityMinor ? 3 : 152;
  return cudaSuccess;
}
cudaError_t cudaGetDeviceProperties(struct cudaDeviceProp *p, int d) {
  (void)d;
  memset(p, 0, sizeof *p);
  p->major = 10; p->minor = 3; p->multiProcessorCount = 152;
  return cudaSuccess;
}
cudaError_t cudaGetLastError(void) { cudaError_t e = t_last; t_last = cudaSuccess; return e; }
cudaError_t cudaStreamCreateWithFlags(cudaStream_t *s, unsigned f) {
  (void)f;
  struct stream *p = malloc(sizeof *p);
  p->dev = t_dev;
  *s = (cudaStream_t)p;
  return cudaSuccess;
}
cudaError_t cudaStreamDestroy(cudaStream_t s) { free(s); return cudaSuccess; }
static void wait_a_while(void) {
  usleep(300);
  for (int i = 0; i < n_pools; ++i) trim(pools[i], pools[i]->keep);
}
cudaError_t cudaStreamSynchronize(cudaStream_t s) { (void)s; wait_a_while(); return cudaSuccess; }
cudaError_t cudaDeviceSynchronize(void) { wait_a_while(); return cudaSuccess; }
cudaError_t cudaMalloc(void **p, size_t n) { return give(p, n, 0); }
cudaError_t cudaFree(void *p) { return take(p); }
cudaError_t cudaMallocHost(void **p, size_t n) {
  return !no_pinned && (*p = calloc(1, n)) ? cudaSuccess : ret(cudaErrorMemoryAllocation);
}
cudaError_t cudaGetSymbolAddress(void **p, const void *s) {
  (void)s;
  if (!symbol) symbol = mmap(0, 16 << 20, PROT_READ | PROT_WRITE, MAP_PRIVATE | MAP_ANONYMOUS, -1, 0);
  *p = symbol;
  return cudaSuccess;
}
cudaError_t cudaFreeHost(void *p) { free(p); return cudaSuccess; }
cudaError_t cudaMemPoolCreate(cudaMemPool_t *p, const struct cudaMemPoolProps *q) {
  (void)q;
  if (n_pools == 16) abort();
  *p = (cudaMemPool_t)(pools[n_pools++] = calloc(1, sizeof(struct pool)));
  return cudaSuccess;
}
cudaError_t cudaMemPoolDestroy(cudaMemPool_t p) { (void)p; return cudaSuccess; }
cudaError_t cudaMemPoolSetAttribute(cudaMemPool_t p, enum cudaMemPoolAttr a, void *v) {
  if (a == cudaMemPoolAttrReleaseThreshold) ((struct pool *)p)->keep = *(unsigned long long *)v;
  return cudaSuccess;
}
cudaError_t cudaMemPoolTrimTo(cudaMemPool_t p, size_t keep) { trim((struct pool *)p, keep); return cudaSuccess; }
cudaError_t cudaMallocFromPoolAsync(void **p, size_t n, cudaMemPool_t from, cudaStream_t s) {
  (void)s;
  if (((struct pool *)from)->dead) return ret(cudaErrorInvalidValue);
  return give(p, n, (struct pool *)from);
}
cudaError_t cudaFreeAsync(void *p, cudaStream_t s) { (void)s; return take(p); }
cudaError_t cudaMemcpy(void *d, const void *s, size_t n, enum cudaMemcpyKind k) { (void)k; memcpy(d, s, n); return cudaSuccess; }
cudaError_t cudaMemcpyAsync(void *d, const void *s, size_t n, enum cudaMemcpyKind k, cudaStream_t t) {
  (void)k; (void)t;
  memcpy(d, s, n);
  return cudaSuccess;
}
cudaError_t cudaMemset(void *d, int v, size_t n) { memset(d, v, n); return cudaSuccess; }
cudaError_t cudaMemsetAsync(void *d, int v, size_t n, cudaStream_t t) { (void)t; memset(d, v, n); return cudaSuccess; }
cudaError_t cudaFuncSetAttribute(const void *f, enum cudaFuncAttribute a, int v) { (void)f; (void)a; (void)v; return cudaSuccess; }
