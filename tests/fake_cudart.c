/* A stand-in for libcudart, preloaded into a child process of the host tests (tests/fakecuda.py): device
 * memory is host memory, kernels do nothing, and chosen calls fail.  Names and signatures are those that
 * liblb.so imports. */
#include <stdlib.h>
#include <string.h>

typedef struct { unsigned x, y, z; } dim3;
typedef struct { dim3 grid, block; size_t smem; void* stream; void* attrs; unsigned num_attrs; } launch_config;
enum { SUCCESS = 0, INVALID_VALUE = 1, NO_MEMORY = 2, INVALID_CONFIG = 9, NO_DEVICE = 100 };

/* ---- what the tests set and read */
static long long capacity = -1, used = 0;      /* bytes of device memory, -1: unlimited */
static char fail_kernel[128] = "";             /* one launch of a kernel whose name holds this is refused */
static int fail_after = 0;                     /* ... after so many that are not */
static int no_device = 0;
static int last_error = SUCCESS;
static struct { const void* fn; char name[512]; int launches; } kernels[4096];
static int nkernels = 0;

void fake_capacity(long long bytes) { capacity = bytes; }
long long fake_used(void) { return used; }
void fake_no_device(int on) { no_device = on; }
void fake_fail_kernel(const char* part, int after) {
    strncpy(fail_kernel, part, sizeof(fail_kernel) - 1);
    fail_after = after;
}
int fake_launches(const char* part) {
    int n = 0;
    for (int k = 0; k < nkernels; ++k)
        if (strstr(kernels[k].name, part)) n += kernels[k].launches;
    return n;
}

static int done(int e) {
    if (e != SUCCESS) last_error = e;
    return e;
}

/* ---- module registration and launches */
void** __cudaRegisterFatBinary(void* bin) { static void* h; (void)bin; return &h; }
void __cudaRegisterFatBinaryEnd(void** h) { (void)h; }
void __cudaUnregisterFatBinary(void** h) { (void)h; }
void __cudaRegisterVar(void) {}
void __cudaRegisterFunction(void** h, const char* host, char* dev, const char* name) {
    (void)h; (void)dev;
    if (nkernels == 4096) abort();
    kernels[nkernels].fn = host;
    strncpy(kernels[nkernels].name, name, sizeof(kernels[0].name) - 1);
    ++nkernels;
}
static int launch(const void* fn) {
    for (int k = 0; k < nkernels; ++k)
        if (kernels[k].fn == fn) {
            if (fail_kernel[0] && strstr(kernels[k].name, fail_kernel) && fail_after-- <= 0) {
                fail_kernel[0] = 0;
                return done(INVALID_CONFIG);
            }
            ++kernels[k].launches;
            return SUCCESS;
        }
    abort();
}
int cudaLaunchKernelExC(const launch_config* c, const void* fn, void** args) { (void)c; (void)args; return launch(fn); }
int __cudaGetKernel(const void** k, const void* fn) { *k = fn; return SUCCESS; }
int __cudaLaunchKernel(const void* k, dim3 g, dim3 b, void** a, size_t s, void* st) {
    (void)g; (void)b; (void)a; (void)s; (void)st;
    return launch(k);
}
static struct { dim3 g, b; size_t s; void* st; } pushed;
unsigned __cudaPushCallConfiguration(dim3 g, dim3 b, size_t s, void* st) {
    pushed.g = g; pushed.b = b; pushed.s = s; pushed.st = st;
    return 0;
}
int __cudaPopCallConfiguration(dim3* g, dim3* b, size_t* s, void** st) {
    *g = pushed.g; *b = pushed.b; *s = pushed.s; *st = pushed.st;
    return SUCCESS;
}

/* ---- memory */
int cudaMalloc(void** p, size_t n) {
    if (no_device) return done(NO_DEVICE);
    if (capacity >= 0 && used + (long long)n > capacity) { *p = 0; return done(NO_MEMORY); }
    size_t* q = calloc(1, n + 256);
    if (!q) return done(NO_MEMORY);
    *q = n;
    used += (long long)n;
    *p = (char*)q + 256;
    return SUCCESS;
}
int cudaFree(void* p) {
    if (p) {
        size_t* q = (size_t*)((char*)p - 256);
        used -= (long long)*q;
        free(q);
    }
    return SUCCESS;
}
int cudaMemcpy(void* d, const void* s, size_t n, int k) { (void)k; if (no_device) return done(NO_DEVICE); memcpy(d, s, n); return SUCCESS; }
int cudaMemcpyAsync(void* d, const void* s, size_t n, int k, void* st) { (void)st; return cudaMemcpy(d, s, n, k); }
int cudaMemsetAsync(void* d, int v, size_t n, void* st) { (void)st; if (no_device) return done(NO_DEVICE); memset(d, v, n); return SUCCESS; }
int cudaGetSymbolAddress(void** p, const void* s) { (void)s; *p = 0; return done(INVALID_VALUE); }

/* ---- device, streams, events, graphs */
int cudaGetDevice(int* d) { if (no_device) return done(NO_DEVICE); *d = 0; return SUCCESS; }
int cudaDeviceGetAttribute(int* v, int a, int d) { (void)a; (void)d; if (no_device) return done(NO_DEVICE); *v = 152; return SUCCESS; }
int cudaDeviceSynchronize(void) { return no_device ? done(NO_DEVICE) : SUCCESS; }
int cudaOccupancyMaxActiveBlocksPerMultiprocessor(int* n, const void* f, int t, size_t s) { (void)f; (void)t; (void)s; *n = 2; return SUCCESS; }
int cudaFuncSetAttribute(const void* f, int a, int v) { (void)f; (void)a; (void)v; return no_device ? done(NO_DEVICE) : SUCCESS; }
int cudaGetLastError(void) { int e = last_error; last_error = SUCCESS; return e; }
const char* cudaGetErrorString(int e) { return e == NO_MEMORY ? "out of memory" : e == NO_DEVICE ? "no device" : "refused"; }
int cudaStreamSynchronize(void* s) { (void)s; return no_device ? done(NO_DEVICE) : SUCCESS; }
int cudaStreamCreateWithFlags(void** s, unsigned f) { (void)f; *s = malloc(1); return SUCCESS; }
int cudaStreamDestroy(void* s) { free(s); return SUCCESS; }
int cudaStreamBeginCapture(void* s, int m) { (void)s; (void)m; return SUCCESS; }
int cudaStreamEndCapture(void* s, void** g) { (void)s; *g = malloc(1); return SUCCESS; }
int cudaGraphInstantiate(void** e, void* g, unsigned long long f) { (void)g; (void)f; *e = malloc(1); return SUCCESS; }
int cudaGraphLaunch(void* e, void* s) { (void)e; (void)s; return SUCCESS; }
int cudaGraphDestroy(void* g) { free(g); return SUCCESS; }
int cudaGraphExecDestroy(void* e) { free(e); return SUCCESS; }
int cudaEventCreate(void** e) { *e = malloc(1); return SUCCESS; }
int cudaEventDestroy(void* e) { free(e); return SUCCESS; }
int cudaEventRecord(void* e, void* s) { (void)e; (void)s; return SUCCESS; }
int cudaEventSynchronize(void* e) { (void)e; return SUCCESS; }
int cudaEventElapsedTime(float* t, void* a, void* b) { (void)a; (void)b; *t = 1.0f; return SUCCESS; }
