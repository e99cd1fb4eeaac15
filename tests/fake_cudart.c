/* A CUDA runtime without a GPU, for tests of the host side: device memory is host memory,
 * kernels do nothing, and a host-to-device copy reads its source when it is queued and once
 * more when the stream is waited for, as a copy that is still under way then would.  Sources
 * whose bytes changed in between are counted. */
#include <pthread.h>
#include <stdlib.h>
#include <string.h>

typedef struct { const void* src; void* dst; void* seen; size_t n; } copy_t;
static copy_t pending[4096];
static int npending, ncopies, nstale;
static pthread_mutex_t mu = PTHREAD_MUTEX_INITIALIZER;

int fake_copies(void) { return ncopies; }
int fake_stale(void) { return nstale; }

static int wait_all(void) {
    pthread_mutex_lock(&mu);
    for (int i = 0; i < npending; ++i) {
        copy_t* c = &pending[i];
        if (memcmp(c->src, c->seen, c->n)) ++nstale;
        free(c->seen);
    }
    npending = 0;
    pthread_mutex_unlock(&mu);
    return 0;
}

int cudaMemcpyAsync(void* dst, const void* src, size_t n, int kind, void* st) {
    (void)st;
    if (kind == 1 && n) {
        copy_t c = {src, dst, malloc(n), n};
        memcpy(c.seen, src, n);
        pthread_mutex_lock(&mu);
        if (npending == 4096) abort();
        pending[npending++] = c;
        ++ncopies;
        pthread_mutex_unlock(&mu);
    }
    memmove(dst, src, n);
    return 0;
}
int cudaStreamSynchronize(void* st) { (void)st; return wait_all(); }
int cudaMemsetAsync(void* p, int v, size_t n, void* st) { (void)st; memset(p, v, n); return 0; }
int cudaMallocAsync(void** p, size_t n, void* st) { (void)st; *p = calloc(1, n ? n : 1); return 0; }
int cudaFreeAsync(void* p, void* st) { (void)st; (void)p; return 0; }   /* kept: copies may still write it */
int cudaHostAlloc(void** p, size_t n, unsigned f) { (void)f; *p = calloc(1, n); return 0; }
int cudaHostGetDevicePointer(void** d, void* h, unsigned f) { (void)f; *d = h; return 0; }
int cudaFreeHost(void* p) { free(p); return 0; }

int cudaGetDevice(int* d) { *d = 0; return 0; }
int cudaSetDevice(int d) { (void)d; return 0; }
int cudaDeviceGetAttribute(int* v, int a, int d) { (void)a; (void)d; *v = 152; return 0; }
int cudaMemGetInfo(size_t* f, size_t* t) { *f = *t = (size_t)1 << 38; return 0; }
int cudaGetLastError(void) { return 0; }
const char* cudaGetErrorString(int e) { (void)e; return "fake"; }

static int handle;
int cudaEventCreate(void** e) { *e = &handle; return 0; }
int cudaEventCreateWithFlags(void** e, unsigned f) { (void)f; *e = &handle; return 0; }
int cudaEventDestroy(void* e) { (void)e; return 0; }
int cudaEventRecord(void* e, void* s) { (void)e; (void)s; return 0; }
int cudaEventSynchronize(void* e) { (void)e; return wait_all(); }
int cudaEventElapsedTime(float* ms, void* a, void* b) { (void)a; (void)b; *ms = 1.0f; return 0; }
int cudaStreamCreateWithFlags(void** s, unsigned f) { (void)f; *s = &handle; return 0; }
int cudaStreamDestroy(void* s) { (void)s; return 0; }
int cudaStreamWaitEvent(void* s, void* e, unsigned f) { (void)s; (void)e; (void)f; return 0; }
int cudaStreamBeginCapture(void* s, int m) { (void)s; (void)m; return 0; }
int cudaStreamEndCapture(void* s, void** g) { (void)s; *g = &handle; return 0; }
int cudaGraphInstantiate(void** x, void* g, unsigned long long f) { (void)g; (void)f; *x = &handle; return 0; }
int cudaGraphLaunch(void* x, void* s) { (void)x; (void)s; return 0; }
int cudaGraphExecDestroy(void* x) { (void)x; return 0; }
int cudaGraphDestroy(void* g) { (void)g; return 0; }
int cudaGetSymbolAddress(void** p, const void* s) { *p = (void*)s; return 0; }
int cudaFuncSetAttribute(const void* f, int a, int v) { (void)f; (void)a; (void)v; return 0; }
int cudaOccupancyMaxActiveBlocksPerMultiprocessor(int* n, const void* f, int b, size_t s) {
    (void)f; (void)b; (void)s;
    *n = 1;
    return 0;
}
int cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int* n, const void* f, int b, size_t s, unsigned g) {
    (void)g;
    return cudaOccupancyMaxActiveBlocksPerMultiprocessor(n, f, b, s);
}

/* what the compiled launches call: registration and an empty launch */
void** __cudaRegisterFatBinary(void* b) { (void)b; static void* h; return &h; }
void __cudaRegisterFatBinaryEnd(void** h) { (void)h; }
void __cudaUnregisterFatBinary(void** h) { (void)h; }
void __cudaRegisterFunction(void) {}
void __cudaRegisterVar(void) {}
unsigned __cudaPushCallConfiguration(void) { return 0; }
int __cudaPopCallConfiguration(void) { return 0; }
int __cudaGetKernel(void** k, const void* f) { *k = (void*)f; return 0; }
int __cudaLaunchKernel(void) { return 0; }
