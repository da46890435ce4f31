// A CUDA runtime that computes nothing: the calls libfpic.so makes, so that its
// host code runs without a device (preloaded before libcudart).  Device memory
// is reserved address space, kernel launches are counted by name, and the next
// allocation of a given size can be made to fail.
#define _GNU_SOURCE
#include <stdint.h>
#include <stdlib.h>
#include <string.h>
#include <sys/mman.h>

typedef struct { unsigned x, y, z; } dim3;
enum { MAXF = 512, MAXB = 4096 };
static struct { const void *f; const char *name; } fn[MAXF];
static int nfn;
static struct { void *p; size_t n; } blk[MAXB];
static int nblk;
static size_t fail_size;
static long long total, launches_of_wanted;
static const char *wanted = "";

void fake_fail_alloc_of(size_t n) { fail_size = n; }
long long fake_bytes(void) { return total; }
void fake_watch(const char *name) { wanted = strdup(name); launches_of_wanted = 0; }
long long fake_launches(void) { return launches_of_wanted; }

static int alloc(void **p, size_t n)
{
    if (n == fail_size) {
        fail_size = 0;
        *p = 0;
        return 2;      // out of memory
    }
    *p = mmap(0, n ? n : 1, PROT_READ | PROT_WRITE, MAP_PRIVATE | MAP_ANONYMOUS | MAP_NORESERVE, -1, 0);
    if (*p == MAP_FAILED || nblk == MAXB) return 2;
    blk[nblk].p = *p;
    blk[nblk++].n = n;
    total += (long long)n;
    return 0;
}

static int release(void *p)
{
    for (int i = 0; i < nblk; ++i)
        if (blk[i].p == p) {
            munmap(p, blk[i].n ? blk[i].n : 1);
            total -= (long long)blk[i].n;
            blk[i] = blk[--nblk];
            return 0;
        }
    return 0;
}

int cudaMalloc(void **p, size_t n) { return alloc(p, n); }
int cudaMallocHost(void **p, size_t n) { return alloc(p, n); }
int cudaHostAlloc(void **p, size_t n, unsigned f) { return alloc(p, n); }
int cudaFree(void *p) { return release(p); }
int cudaFreeHost(void *p) { return release(p); }
int cudaMemset(void *p, int v, size_t n) { return 0; }
int cudaMemsetAsync(void *p, int v, size_t n, void *s) { return 0; }
int cudaMemcpy(void *d, const void *s, size_t n, int k) { if (k == 2) memset(d, 0, n); return 0; }
int cudaMemcpyAsync(void *d, const void *s, size_t n, int k, void *st) { return cudaMemcpy(d, s, n, k); }
int cudaGetDevice(int *d) { *d = 0; return 0; }
int cudaSetDevice(int d) { return 0; }
int cudaDeviceGetAttribute(int *v, int a, int d) { *v = 152; return 0; }
int cudaDeviceSynchronize(void) { return 0; }
int cudaGetLastError(void) { return 0; }
const char *cudaGetErrorString(int e) { return e == 2 ? "out of memory" : "no error"; }
int cudaStreamSynchronize(void *s) { return 0; }
int cudaStreamIsCapturing(void *s, int *c) { *c = 0; return 0; }
int cudaStreamCreateWithFlags(void **s, unsigned f) { *s = (void *)1; return 0; }
int cudaFuncSetAttribute(const void *f, int a, int v) { return 0; }
int cudaEventCreate(void **e) { *e = (void *)1; return 0; }
int cudaEventCreateWithFlags(void **e, unsigned f) { *e = (void *)1; return 0; }
int cudaEventRecord(void *e, void *s) { return 0; }
void **__cudaRegisterFatBinary(void *b) { static void *h; return &h; }
void __cudaRegisterFatBinaryEnd(void **h) {}
void __cudaUnregisterFatBinary(void **h) {}
void __cudaRegisterVar(void **h, char *v, char *a, const char *n, int e, size_t s, int c, int g) {}
void __cudaRegisterFunction(void **h, const char *f, char *df, const char *name, int l, void *t, void *b, void *bd,
                            void *gd, int *w)
{
    if (nfn < MAXF && strstr(name, "fpic")) {       // this library's only
        fn[nfn].f = f;
        fn[nfn++].name = name;
    }
}

static void count(const void *f)
{
    for (int i = 0; i < nfn; ++i)
        if (fn[i].f == f && strstr(fn[i].name, wanted)) {
            ++launches_of_wanted;
            return;
        }
}

int __cudaGetKernel(const void **k, const void *f) { *k = f; return 0; }
unsigned __cudaPushCallConfiguration(dim3 g, dim3 b, size_t sm, void *s) { return 0; }
int __cudaPopCallConfiguration(dim3 *g, dim3 *b, size_t *sm, void **s) { return 0; }
int __cudaLaunchKernel(const void *k, dim3 g, dim3 b, void **a, size_t sm, void *s) { count(k); return 0; }
int cudaLaunchKernelExC(const void *cfg, const void *f, void **a) { count(f); return 0; }
