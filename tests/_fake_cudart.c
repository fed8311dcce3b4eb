/* A stand-in for the CUDA runtime: the engine's host code linked against it runs
 * without a GPU.  "Device" memory is host memory, kernels do nothing but leave
 * their names in a list, and an allocation can be made to fail.  Only what the
 * engine calls is here, and only the arguments that matter are declared. */
#include <stdlib.h>
#include <string.h>

enum { OK = 0, NO_MEMORY = 2 };

/* ---- the test's side ---- */
static int fail_in = -1; /* allocations until one fails; -1: none does */
static struct { const void *fun; const char *name; } kernels[4096];
static int n_kernels;
static const char *launched[1 << 16];
static int n_launched;

void fake_fail_allocation(int after) { fail_in = after; }
int fake_fail_pending(void) { return fail_in >= 0; }
void fake_clear_launches(void) { n_launched = 0; }
/* launches of kernels whose (mangled) name holds `part` */
int fake_launches(const char *part) {
    int n = 0;
    for (int i = 0; i < n_launched; ++i) n += strstr(launched[i], part) != NULL;
    return n;
}

/* ---- kernels ---- */
static char module;
void **__cudaRegisterFatBinary(void *bin) { (void)bin; return (void **)&module; }
void __cudaRegisterFatBinaryEnd(void **m) { (void)m; }
void __cudaUnregisterFatBinary(void **m) { (void)m; }
void __cudaRegisterFunction(void **m, const char *fun, char *dev, const char *name) {
    (void)m; (void)dev;
    if (n_kernels < 4096) {
        kernels[n_kernels].fun = fun;
        kernels[n_kernels++].name = name;
    }
}
void __cudaRegisterVar(void **m) { (void)m; }
static int record(const void *fun) {
    for (int i = 0; i < n_kernels; ++i)
        if (kernels[i].fun == fun && n_launched < (1 << 16)) {
            launched[n_launched++] = kernels[i].name;
            break;
        }
    return OK;
}
unsigned __cudaPushCallConfiguration(void) { return 0; }
int __cudaPopCallConfiguration(void) { return OK; }
int __cudaGetKernel(const void **k, const void *fun) { *k = fun; return OK; }
int __cudaLaunchKernel(const void *k) { return record(k); }
int cudaLaunchKernelExC(const void *config, const void *fun) { (void)config; return record(fun); }
int cudaLaunchCooperativeKernel(const void *fun) { return record(fun); }
int cudaFuncSetAttribute(void) { return OK; }
int cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int *n) { *n = 3; return OK; }
int cudaOccupancyMaxActiveClusters(int *n) { *n = 50; return OK; }

/* ---- memory ---- */
static int allocate(void **p, size_t n) {
    if (fail_in >= 0 && fail_in-- == 0) { *p = NULL; return NO_MEMORY; }
    *p = calloc(n ? n : 1, 1);
    return *p ? OK : NO_MEMORY;
}
static int release(void *p) { free(p); return OK; }
int cudaMalloc(void **p, size_t n) { return allocate(p, n); }
int cudaMallocAsync(void **p, size_t n) { return allocate(p, n); }
int cudaMallocFromPoolAsync(void **p, size_t n) { return allocate(p, n); }
int cudaMallocHost(void **p, size_t n) { return allocate(p, n); }
int cudaHostAlloc(void **p, size_t n) { return allocate(p, n); }
int cudaFree(void *p) { return release(p); }
int cudaFreeAsync(void *p) { return release(p); }
int cudaFreeHost(void *p) { return release(p); }
int cudaHostGetDevicePointer(void **d, void *h) { *d = h; return OK; }
int cudaMemcpyAsync(void *d, const void *s, size_t n) { memcpy(d, s, n); return OK; }
int cudaMemset(void *d, int v, size_t n) { memset(d, v, n); return OK; }
int cudaMemsetAsync(void *d, int v, size_t n) { memset(d, v, n); return OK; }
static char symbol[1 << 20];
int cudaGetSymbolAddress(void **p) { *p = symbol; return OK; }
int cudaMemPoolCreate(void **p) { *p = &module; return OK; }
int cudaMemPoolSetAttribute(void) { return OK; }
int cudaMemPoolTrimTo(void) { return OK; }
int cudaPointerGetAttributes(void) { return 1; }

/* ---- the rest ---- */
int cudaGetDevice(int *d) { *d = 0; return OK; }
int cudaDeviceGetAttribute(int *v) { *v = 152; return OK; }
int cudaDeviceSynchronize(void) { return OK; }
int cudaGetLastError(void) { return OK; }
int cudaStreamSynchronize(void) { return OK; }
int cudaStreamCreateWithFlags(void **s) { *s = &module; return OK; }
int cudaStreamDestroy(void) { return OK; }
int cudaStreamBeginCapture(void) { return OK; }
int cudaStreamEndCapture(void *s, void **g) { (void)s; *g = &module; return OK; }
int cudaGraphInstantiate(void **e) { *e = &module; return OK; }
int cudaGraphLaunch(void) { return OK; }
int cudaGraphDestroy(void) { return OK; }
int cudaGraphExecDestroy(void) { return OK; }
int cudaEventCreateWithFlags(void **e) { *e = &module; return OK; }
int cudaEventRecord(void) { return OK; }
int cudaEventSynchronize(void) { return OK; }
int cudaEventDestroy(void) { return OK; }
