/* A CUDA runtime in host memory for tests of the library's host code: memory is
 * malloc, copies are memcpy, launches are counted and run nothing but the two
 * kernels that set and clear an engine slot's flag.  fake_fail(name, n): the n-th
 * following launch of a kernel whose name contains name, or the n-th following
 * copy for "memcpy", fails with cudaErrorLaunchFailure (719) or
 * cudaErrorInvalidValue (1). */
#include <stdlib.h>
#include <string.h>

typedef struct { unsigned x, y, z; } dim3;
typedef int err;

enum { MAXF = 4096, MAXP = 256 };
static const void* fn_host[MAXF];
static const char* fn_name[MAXF];
static int fn_n;
static int* flags[MAXP];
static int flags_n;
static char fail_name[64];
static int fail_in;
static err last;

void fake_fail(const char* name, int n) {
    strncpy(fail_name, name, sizeof(fail_name) - 1);
    fail_in = n;
}
/* engine slots whose flag is set */
int fake_active(void) {
    int n = 0;
    for (int i = 0; i < flags_n; ++i) n += *flags[i] != 0;
    return n;
}
static err check(const char* name, err e) {
    if (fail_in > 0 && strstr(name, fail_name) && --fail_in == 0) return last = e;
    return 0;
}

void** __cudaRegisterFatBinary(void* p) { static void* h; (void)p; return &h; }
void __cudaRegisterFatBinaryEnd(void** h) { (void)h; }
void __cudaUnregisterFatBinary(void** h) { (void)h; }
void __cudaRegisterVar(void** h, char* a, char* b, const char* c, int d, size_t e, int f, int g) {
    (void)h; (void)a; (void)b; (void)c; (void)d; (void)e; (void)f; (void)g;
}
void __cudaRegisterFunction(void** h, const char* host, char* dev, const char* name, int lim, void* a, void* b, void* c,
                            void* d, int* e) {
    (void)h; (void)dev; (void)lim; (void)a; (void)b; (void)c; (void)d; (void)e;
    if (fn_n < MAXF) { fn_host[fn_n] = host; fn_name[fn_n++] = name; }
}
static dim3 cfg_grid, cfg_block;
static size_t cfg_smem;
static void* cfg_stream;
unsigned __cudaPushCallConfiguration(dim3 g, dim3 b, size_t s, void* st) {
    cfg_grid = g; cfg_block = b; cfg_smem = s; cfg_stream = st;
    return 0;
}
err __cudaPopCallConfiguration(dim3* g, dim3* b, size_t* s, void* st) {
    *g = cfg_grid; *b = cfg_block; *s = cfg_smem; *(void**)st = cfg_stream;
    return 0;
}
err __cudaGetKernel(void** k, const void* f) { *k = (void*)f; return 0; }
static err launch(const void* f, void** args) {
    const char* name = "";
    for (int i = 0; i < fn_n; ++i)
        if (fn_host[i] == f) name = fn_name[i];
    const err e = check(name, 719);
    if (e) return e;
    if (strstr(name, "k_admit")) {
        int* p = *(int**)args[0];
        int i = 0;
        while (i < flags_n && flags[i] != p) ++i;
        if (i == flags_n && flags_n < MAXP) flags[flags_n++] = p;
        *p = 1;
    }
    if (strstr(name, "k_release")) {
        **(int**)args[0] = 0;
        **(unsigned**)args[1] = 0;
    }
    return 0;
}
err __cudaLaunchKernel(void* k, dim3 g, dim3 b, void** args, size_t s, void* st) {
    (void)g; (void)b; (void)s; (void)st;
    return launch(k, args);
}
err cudaLaunchKernelExC(const void* cfg, const void* f, void** args) { (void)cfg; return launch(f, args); }

err cudaMemcpyAsync(void* d, const void* s, size_t n, int kind, void* st) {
    (void)kind; (void)st;
    const err e = check("memcpy", 1);
    if (!e) memcpy(d, s, n);
    return e;
}
err cudaMemsetAsync(void* d, int v, size_t n, void* st) { (void)st; memset(d, v, n); return 0; }
err cudaMalloc(void** p, size_t n) { *p = malloc(n); return *p ? 0 : 2; }
err cudaFree(void* p) { free(p); return 0; }
err cudaHostAlloc(void** p, size_t n, unsigned f) { (void)f; *p = malloc(n); return *p ? 0 : 2; }
err cudaFreeHost(void* p) { free(p); return 0; }
err cudaGetLastError(void) { const err e = last; last = 0; return e; }
err cudaPeekAtLastError(void) { return last; }
err cudaGetDevice(int* d) { *d = 0; return 0; }
err cudaDeviceGetAttribute(int* v, int a, int d) { (void)a; (void)d; *v = 152; return 0; }
err cudaFuncSetAttribute(const void* f, int a, int v) { (void)f; (void)a; (void)v; return 0; }
err cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int* n, const void* f, int t, size_t s, unsigned g) {
    (void)f; (void)t; (void)s; (void)g;
    *n = 1;
    return 0;
}
err cudaOccupancyMaxActiveClusters(int* n, const void* f, const void* c) { (void)f; (void)c; *n = 0; return 0; }
err cudaStreamCreateWithFlags(void** s, unsigned f) { (void)f; *s = malloc(1); return 0; }
err cudaStreamDestroy(void* s) { free(s); return 0; }
err cudaStreamSynchronize(void* s) { (void)s; return 0; }
err cudaStreamWaitEvent(void* s, void* e, unsigned f) { (void)s; (void)e; (void)f; return 0; }
err cudaStreamBeginCapture(void* s, int m) { (void)s; (void)m; return 801; }
err cudaStreamEndCapture(void* s, void** g) { (void)s; *g = 0; return 801; }
err cudaGraphInstantiate(void** x, void* g, unsigned long long f) { (void)g; (void)f; *x = 0; return 801; }
err cudaGraphLaunch(void* x, void* s) { (void)x; (void)s; return 801; }
err cudaGraphExecDestroy(void* x) { (void)x; return 0; }
err cudaGraphDestroy(void* g) { (void)g; return 0; }
err cudaEventCreate(void** e) { *e = malloc(1); return 0; }
err cudaEventCreateWithFlags(void** e, unsigned f) { (void)f; *e = malloc(1); return 0; }
err cudaEventDestroy(void* e) { free(e); return 0; }
err cudaEventRecord(void* e, void* s) { (void)e; (void)s; return 0; }
err cudaEventSynchronize(void* e) { (void)e; return 0; }
err cudaEventElapsedTime(float* t, void* a, void* b) { (void)a; (void)b; *t = 0; return 0; }
err cudaGetSymbolAddress(void** p, const void* s) { (void)s; *p = 0; return 1; }
err cudaGetDriverEntryPointByVersion(const char* n, void** p, unsigned v, unsigned long long f, int* q) {
    (void)n; (void)v; (void)f; (void)q;
    *p = 0;
    return 1;
}
