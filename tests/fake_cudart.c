/* A CUDA runtime without a GPU, for host-side tests: linked with the library's objects in the runtime's place.  Device
 * memory is host memory, kernels do nothing, streams and events keep vector clocks of the work enqueued on them.  Any
 * chosen call can be made to fail, and the tests ask which streams' work is not awaited by another stream. */
#include <cuda_runtime_api.h>
#include <pthread.h>
#include <stdlib.h>
#include <string.h>

#define MAX_STREAMS 64

typedef struct {
    long clock[MAX_STREAMS]; /* clock[t]: operations of stream t that come before whatever is enqueued next */
    int used, priority;
    long launches;
} Stream;

typedef struct {
    long clock[MAX_STREAMS];
} Event;

static pthread_mutex_t mu = PTHREAD_MUTEX_INITIALIZER;
static Stream streams[MAX_STREAMS]; /* 0: the legacy default stream */
static long calls, fail_at = -1;
static cudaError_t last = cudaSuccess;
static size_t answer_bytes;
static unsigned char answer[256];

static int id_of(cudaStream_t s) { return s ? (int)((Stream*)s - streams) : 0; }

/* one enqueued operation or other fallible call; 0 where this is the one that fails */
static int passes(void) {
    if (calls++ != fail_at) return 1;
    last = cudaErrorLaunchOutOfResources;
    return 0;
}
static cudaError_t enqueue(cudaStream_t s, int launch) {
    pthread_mutex_lock(&mu);
    const int ok = passes(), k = id_of(s);
    if (ok) {
        streams[k].clock[k]++;
        streams[k].launches += launch;
    }
    pthread_mutex_unlock(&mu);
    return ok ? cudaSuccess : last;
}

/* ---- the tests' side ---- */
void fake_fail_at(long k) { /* the k-th call from now fails (-1: none) */
    pthread_mutex_lock(&mu);
    calls = 0;
    fail_at = k;
    last = cudaSuccess;
    pthread_mutex_unlock(&mu);
}
long fake_calls(void) { return calls; }
void fake_answer(const void* bytes, size_t n) { /* what every device-to-host copy of n bytes reads */
    memcpy(answer, bytes, n);
    answer_bytes = n;
}
/* streams with operations that nothing enqueued on s from now on waits for */
int fake_unjoined(cudaStream_t s) {
    int open = 0;
    pthread_mutex_lock(&mu);
    for (int t = 0; t < MAX_STREAMS; ++t) open += streams[t].clock[t] > streams[id_of(s)].clock[t];
    pthread_mutex_unlock(&mu);
    return open;
}
long fake_launches(int priority) { /* kernels launched so far on streams of this priority */
    long n = 0;
    pthread_mutex_lock(&mu);
    for (int t = 0; t < MAX_STREAMS; ++t) n += streams[t].priority == priority ? streams[t].launches : 0;
    pthread_mutex_unlock(&mu);
    return n;
}

/* ---- streams and events ---- */
cudaError_t cudaStreamCreateWithPriority(cudaStream_t* out, unsigned int flags, int priority) {
    (void)flags;
    pthread_mutex_lock(&mu);
    int k = 1, ok = passes();
    while (k < MAX_STREAMS && streams[k].used) ++k;
    if (ok && k < MAX_STREAMS) {
        streams[k].used = 1;
        streams[k].priority = priority;
        *out = (cudaStream_t)&streams[k];
    }
    pthread_mutex_unlock(&mu);
    return ok && k < MAX_STREAMS ? cudaSuccess : cudaErrorMemoryAllocation;
}
cudaError_t cudaStreamCreateWithFlags(cudaStream_t* out, unsigned int flags) {
    return cudaStreamCreateWithPriority(out, flags, 0);
}
cudaError_t cudaStreamDestroy(cudaStream_t s) { /* its number is not taken again: launches stay counted */
    (void)s;
    return cudaSuccess;
}
cudaError_t cudaStreamGetPriority(cudaStream_t s, int* p) { *p = streams[id_of(s)].priority; return cudaSuccess; }
cudaError_t cudaDeviceGetStreamPriorityRange(int* least, int* greatest) {
    *least = 0;
    *greatest = -5;
    return cudaSuccess;
}
cudaError_t cudaEventCreateWithFlags(cudaEvent_t* e, unsigned int flags) {
    (void)flags;
    *e = (cudaEvent_t)calloc(1, sizeof(Event));
    return cudaSuccess;
}
cudaError_t cudaEventCreate(cudaEvent_t* e) { return cudaEventCreateWithFlags(e, 0); }
cudaError_t cudaEventDestroy(cudaEvent_t e) { free(e); return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t e, cudaStream_t s) {
    pthread_mutex_lock(&mu);
    const int ok = passes();
    if (ok) memcpy(((Event*)e)->clock, streams[id_of(s)].clock, sizeof(((Event*)e)->clock));
    pthread_mutex_unlock(&mu);
    return ok ? cudaSuccess : last;
}
static void join(Stream* s, const long* clock) {
    for (int t = 0; t < MAX_STREAMS; ++t)
        if (clock[t] > s->clock[t]) s->clock[t] = clock[t];
}
cudaError_t cudaStreamWaitEvent(cudaStream_t s, cudaEvent_t e, unsigned int flags) {
    (void)flags;
    pthread_mutex_lock(&mu);
    const int ok = passes();
    if (ok) join(&streams[id_of(s)], ((Event*)e)->clock);
    pthread_mutex_unlock(&mu);
    return ok ? cudaSuccess : last;
}
cudaError_t cudaStreamSynchronize(cudaStream_t s) { /* all that s holds is done: no stream need wait for it */
    pthread_mutex_lock(&mu);
    for (int t = 0; t < MAX_STREAMS; ++t) join(&streams[t], streams[id_of(s)].clock);
    pthread_mutex_unlock(&mu);
    return cudaSuccess;
}
cudaError_t cudaEventSynchronize(cudaEvent_t e) { (void)e; return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float* ms, cudaEvent_t a, cudaEvent_t b) { (void)a; (void)b; *ms = 0; return cudaSuccess; }

/* ---- memory ---- */
cudaError_t cudaMallocAsync(void** p, size_t n, cudaStream_t s) {
    *p = calloc(1, n ? n : 1);
    return enqueue(s, 0);
}
cudaError_t cudaFreeAsync(void* p, cudaStream_t s) { (void)s; free(p); return cudaSuccess; }
cudaError_t cudaMallocHost(void** p, size_t n) { *p = malloc(n); return cudaSuccess; }
cudaError_t cudaFreeHost(void* p) { free(p); return cudaSuccess; }
cudaError_t cudaMemsetAsync(void* p, int v, size_t n, cudaStream_t s) { memset(p, v, n); return enqueue(s, 0); }
cudaError_t cudaMemcpyAsync(void* d, const void* s, size_t n, enum cudaMemcpyKind kind, cudaStream_t stream) {
    if (kind == cudaMemcpyDeviceToHost && answer_bytes && n == answer_bytes) memcpy(d, answer, n);
    else memcpy(d, s, n);
    return enqueue(stream, 0);
}
cudaError_t cudaMemGetInfo(size_t* f, size_t* t) { *f = *t = (size_t)1 << 36; return cudaSuccess; }
cudaError_t cudaDeviceGetDefaultMemPool(cudaMemPool_t* p, int d) { (void)d; *p = 0; return cudaSuccess; }
cudaError_t cudaMemPoolSetAttribute(cudaMemPool_t p, enum cudaMemPoolAttr a, void* v) {
    (void)p; (void)a; (void)v;
    return cudaSuccess;
}
cudaError_t cudaGetSymbolAddress(void** p, const void* symbol) { (void)symbol; *p = 0; return cudaErrorInvalidSymbol; }

/* ---- device, errors, kernels ---- */
cudaError_t cudaGetDevice(int* d) { *d = 0; return cudaSuccess; }
cudaError_t cudaSetDevice(int d) { (void)d; return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int* v, enum cudaDeviceAttr a, int d) { (void)a; (void)d; *v = 152; return cudaSuccess; }
cudaError_t cudaGetLastError(void) { const cudaError_t e = last; last = cudaSuccess; return e; }
const char* cudaGetErrorString(cudaError_t e) { (void)e; return "fake"; }
cudaError_t cudaFuncSetAttribute(const void* f, enum cudaFuncAttribute a, int v) {
    (void)f; (void)a; (void)v;
    pthread_mutex_lock(&mu);
    const int ok = passes();
    pthread_mutex_unlock(&mu);
    return ok ? cudaSuccess : last;
}
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t* c, const void* f, void** args) {
    (void)f; (void)args;
    return enqueue(c->stream, 1);
}
cudaError_t __cudaLaunchKernel(void* k, dim3 g, dim3 b, void** args, size_t smem, cudaStream_t s) {
    (void)k; (void)g; (void)b; (void)args; (void)smem;
    return enqueue(s, 1);
}
cudaError_t __cudaGetKernel(void** k, const void* f) { *k = (void*)f; return cudaSuccess; }
cudaError_t __cudaPopCallConfiguration(dim3* g, dim3* b, size_t* smem, void* s) {
    (void)g; (void)b; (void)smem; (void)s;
    return cudaErrorInvalidValue;
}
void** __cudaRegisterFatBinary(void* p) { (void)p; return (void**)streams; }
void __cudaRegisterFatBinaryEnd(void** h) { (void)h; }
void __cudaUnregisterFatBinary(void** h) { (void)h; }
void __cudaRegisterFunction(void** h, const char* f, char* n, const char* m, int l, void* a, void* b, void* c, void* d, int* w) {
    (void)h; (void)f; (void)n; (void)m; (void)l; (void)a; (void)b; (void)c; (void)d; (void)w;
}
void __cudaRegisterVar(void** h, char* v, char* n, const char* m, int e, size_t s, int c, int g) {
    (void)h; (void)v; (void)n; (void)m; (void)e; (void)s; (void)c; (void)g;
}

/* ---- capture: not offered ---- */
cudaError_t cudaStreamIsCapturing(cudaStream_t s, enum cudaStreamCaptureStatus* c) {
    (void)s;
    *c = cudaStreamCaptureStatusNone;
    return cudaSuccess;
}
cudaError_t cudaStreamBeginCapture(cudaStream_t s, enum cudaStreamCaptureMode m) { (void)s; (void)m; return cudaErrorNotSupported; }
cudaError_t cudaStreamEndCapture(cudaStream_t s, cudaGraph_t* g) { (void)s; (void)g; return cudaErrorNotSupported; }
cudaError_t cudaGraphInstantiate(cudaGraphExec_t* x, cudaGraph_t g, unsigned long long f) {
    (void)x; (void)g; (void)f;
    return cudaErrorNotSupported;
}
cudaError_t cudaGraphLaunch(cudaGraphExec_t x, cudaStream_t s) { (void)x; (void)s; return cudaErrorNotSupported; }
cudaError_t cudaGraphDestroy(cudaGraph_t g) { (void)g; return cudaSuccess; }
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t x) { (void)x; return cudaSuccess; }
