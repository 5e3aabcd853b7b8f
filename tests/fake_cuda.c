/* Stand-in for the CUDA runtime and cuFFT, preloaded before libpse.so so that
 * its host code runs without a GPU: device memory is zeroed host memory,
 * kernels do nothing but are counted by name, a transform can be made to
 * fail, and event times are the sum of given costs per launch. */
#include <stddef.h>
#include <stdio.h>
#include <stdlib.h>
#include <string.h>

typedef struct { unsigned x, y, z; } dim3;
#define NFUN 2048
#define NCOST 64
static struct { const void *host; const char *name; long launches; } fun[NFUN];
static int nfun;
static struct { char name[64]; double ms; } cost[NCOST];
static int ncost;
static double now_ms;
static long nmalloc, nlive;
static int fail_plans, fail_malloc;
static int slow_n, slow_seen; /* samples of a new context that take slow_ms more */
static double slow_ms;
static char last[128];
static struct { dim3 g, b; size_t smem; void *s; } cfg;

/* ---- what a test sets and reads */
void fake_reset(void) {
    for (int i = 0; i < nfun; ++i) fun[i].launches = 0;
    nmalloc = 0;
}
void fake_fail_plans(int n) { fail_plans = n; }
/* the n-th allocation from now fails (0: none) */
void fake_fail_malloc(int n) { fail_malloc = n; }
long fake_mallocs(void) { return nmalloc; }
long fake_live(void) { return nlive; }
/* launches of the kernels whose (mangled) name contains `part` */
long fake_launches(const char *part) {
    long n = 0;
    for (int i = 0; i < nfun; ++i)
        if (strstr(fun[i].name, part)) n += fun[i].launches;
    return n;
}
/* each launch of a kernel (transform) whose name contains `part` takes ms;
 * the latest matching rule counts */
void fake_cost(const char *part, double ms) {
    snprintf(cost[ncost % NCOST].name, sizeof(cost[0].name), "%s", part);
    cost[ncost++ % NCOST].ms = ms;
}
void fake_slow_start(int n, double ms) { slow_n = n; slow_ms = ms; }
static void spend(const char *name) {
    for (int i = ncost - 1; i >= 0; --i)
        if (strstr(name, cost[i].name)) {
            now_ms += cost[i].ms;
            return;
        }
}

/* ---- registration and launches */
void **__cudaRegisterFatBinary(void *b) { static void *h; (void)b; return &h; }
void __cudaRegisterFatBinaryEnd(void **h) { (void)h; }
void __cudaUnregisterFatBinary(void **h) { (void)h; }
void __cudaRegisterVar(void **h, char *hv, char *da, const char *dn, int ext, size_t size, int c, int g) {
    (void)h; (void)hv; (void)da; (void)dn; (void)ext; (void)size; (void)c; (void)g;
}
void __cudaRegisterFunction(void **h, const char *host, char *dev, const char *name, int lim, void *t, void *b, void *bd,
                            void *gd, int *ws) {
    (void)h; (void)dev; (void)lim; (void)t; (void)b; (void)bd; (void)gd; (void)ws;
    if (nfun == NFUN) abort();
    fun[nfun].host = host;
    fun[nfun++].name = strdup(name);
}
unsigned __cudaPushCallConfiguration(dim3 g, dim3 b, size_t smem, void *s) {
    cfg.g = g; cfg.b = b; cfg.smem = smem; cfg.s = s;
    return 0;
}
int __cudaPopCallConfiguration(dim3 *g, dim3 *b, size_t *smem, void *s) {
    *g = cfg.g; *b = cfg.b; *smem = cfg.smem; *(void **)s = cfg.s;
    return 0;
}
int __cudaGetKernel(void **k, const void *host) { *k = (void *)host; return 0; }
int __cudaLaunchKernel(void *k, dim3 g, dim3 b, void **args, size_t smem, void *s) {
    (void)g; (void)b; (void)args; (void)smem; (void)s;
    for (int i = 0; i < nfun; ++i)
        if (fun[i].host == k) {
            ++fun[i].launches;
            spend(fun[i].name);
            if (strstr(fun[i].name, "k_lz_final") && slow_seen++ < slow_n) now_ms += slow_ms;
            return 0;
        }
    return 98; /* invalid device function */
}
int cudaLaunchKernel(const void *k, dim3 g, dim3 b, void **args, size_t smem, void *s) {
    return __cudaLaunchKernel((void *)k, g, b, args, smem, s);
}
int cudaFuncSetAttribute(const void *f, int a, int v) { (void)f; (void)a; (void)v; return 0; }
int cudaFuncGetAttributes(void *at, const void *f) { (void)f; memset(at, 0, 64); return 0; }
int cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int *n, const void *f, int b, size_t smem, unsigned fl) {
    (void)f; (void)b; (void)smem; (void)fl;
    *n = 2;
    return 0;
}

/* ---- memory */
int cudaMalloc(void **p, size_t n) {
    ++nmalloc;
    *p = NULL;
    if (fail_malloc > 0 && --fail_malloc == 0) return 2; /* cudaErrorMemoryAllocation */
    *p = calloc(n, 1);
    nlive += *p != NULL;
    return *p ? 0 : 2;
}
int cudaFree(void *p) { nlive -= p != NULL; free(p); return 0; }
int cudaMallocHost(void **p, size_t n) { /* once per context */
    slow_seen = 0;
    *p = calloc(n, 1);
    return *p ? 0 : 2;
}
int cudaFreeHost(void *p) { free(p); return 0; }
int cudaMemcpy(void *d, const void *s, size_t n, int k) { (void)k; memcpy(d, s, n); return 0; }
int cudaMemcpyAsync(void *d, const void *s, size_t n, int k, void *st) { (void)k; (void)st; memcpy(d, s, n); return 0; }
int cudaMemset(void *p, int v, size_t n) { (void)p; (void)v; (void)n; return 0; }
int cudaMemsetAsync(void *p, int v, size_t n, void *s) { (void)p; (void)v; (void)n; (void)s; return 0; }
int cudaMemGetInfo(size_t *left, size_t *all) { *left = *all = (size_t)280 << 30; return 0; }

/* ---- device, streams, events */
int cudaGetDevice(int *d) { *d = 0; return 0; }
int cudaSetDevice(int d) { (void)d; return 0; }
int cudaDeviceGetAttribute(int *v, int a, int d) { /* 97: shared memory per block (opt-in); else the SM count */
    (void)d;
    *v = a == 97 ? 232448 : 152;
    return 0;
}
int cudaDeviceGetStreamPriorityRange(int *lo, int *hi) { *lo = 0; *hi = -5; return 0; }
int cudaDeviceSynchronize(void) { return 0; }
int cudaGetLastError(void) { return 0; }
int cudaStreamCreateWithFlags(void **s, unsigned f) { (void)f; *s = malloc(8); return 0; }
int cudaStreamCreateWithPriority(void **s, unsigned f, int p) { (void)f; (void)p; *s = malloc(8); return 0; }
int cudaStreamDestroy(void *s) { free(s); return 0; }
int cudaStreamSynchronize(void *s) { (void)s; return 0; }
int cudaStreamWaitEvent(void *s, void *e, unsigned f) { (void)s; (void)e; (void)f; return 0; }
int cudaEventCreate(void **e) { *e = calloc(1, sizeof(double)); return 0; }
int cudaEventCreateWithFlags(void **e, unsigned f) { (void)f; return cudaEventCreate(e); }
int cudaEventDestroy(void *e) { free(e); return 0; }
int cudaEventRecord(void *e, void *s) { (void)s; *(double *)e = now_ms; return 0; }
int cudaEventSynchronize(void *e) { (void)e; return 0; }
int cudaEventElapsedTime(float *ms, void *a, void *b) { *ms = (float)(*(double *)b - *(double *)a); return 0; }

/* ---- cuFFT: a handle is the grid size */
int cufftPlanMany(int *h, int rank, int *n, int *ie, int is, int id, int *oe, int os, int od, int type, int batch) {
    (void)rank; (void)ie; (void)is; (void)id; (void)oe; (void)os; (void)od; (void)type; (void)batch;
    if (fail_plans > 0) {
        --fail_plans;
        return 2; /* CUFFT_ALLOC_FAILED */
    }
    *h = n[0];
    return 0;
}
int cufftDestroy(int h) { (void)h; return 0; }
int cufftSetStream(int h, void *s) { (void)h; (void)s; return 0; }
static int run(const char *what, int h) {
    snprintf(last, sizeof(last), "%s %d", what, h);
    spend(last);
    return 0;
}
int cufftExecC2R(int h, void *a, void *b) { (void)a; (void)b; return run("C2R", h); }
int cufftExecZ2D(int h, void *a, void *b) { (void)a; (void)b; return run("Z2D", h); }
int cufftExecR2C(int h, void *a, void *b) { (void)a; (void)b; return run("R2C", h); }
int cufftExecD2Z(int h, void *a, void *b) { (void)a; (void)b; return run("D2Z", h); }
