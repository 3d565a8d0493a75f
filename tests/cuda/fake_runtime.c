/* A stand-in for the CUDA runtime, for host logic on a machine without a GPU: linked with the library's own objects in the
 * runtime's place. Nothing runs; every stream keeps the order of what was queued on it, as a vector of how much of every stream
 * comes before its next operation, and one call, by its number, can be made to fail. */
#include <stddef.h>
#include <stdlib.h>
#include <string.h>

enum { kStreams = 512, kFailure = 719 };
typedef struct { int id; long before[kStreams]; } Stream;     /* before[id]: operations queued on this stream */
typedef struct { long before[kStreams]; } Event;
static Stream streams[kStreams];
static int n_streams;
static long calls, fail_at;
static int last_error;

static int step(void) { return ++calls == fail_at ? (last_error = kFailure) : 0; }
static Stream* queue(void* s) { Stream* t = s ? (Stream*)s : &streams[0]; return t; }

void* fake_stream(void) { streams[n_streams].id = n_streams; return &streams[n_streams++]; }
void fake_fail_at(long n) { calls = 0; fail_at = n; last_error = 0; }
long fake_calls(void) { return calls; }
/* 1 if everything queued anywhere comes before what is queued on s next */
int fake_joined(void* s) {
    for (int i = 0; i < n_streams; ++i)
        if (queue(s)->before[i] < streams[i].before[i]) return 0;
    return 1;
}

static int enqueue(void* s) {
    int r = step();
    if (r == 0) { Stream* t = queue(s); ++t->before[t->id]; }
    return r;
}
int cudaStreamCreateWithFlags(void** s, unsigned f) { (void)f; int r = step(); if (r == 0) *s = fake_stream(); return r; }
int cudaStreamDestroy(void* s) { (void)s; return 0; }
int cudaEventCreate(void** e) { int r = step(); if (r == 0) *e = calloc(1, sizeof(Event)); return r; }
int cudaEventCreateWithFlags(void** e, unsigned f) { (void)f; return cudaEventCreate(e); }
int cudaEventDestroy(void* e) { free(e); return 0; }
int cudaEventRecord(void* e, void* s) { int r = step(); if (r == 0) memcpy(((Event*)e)->before, queue(s)->before, sizeof(((Event*)e)->before)); return r; }
int cudaStreamWaitEvent(void* s, void* e, unsigned f) {
    (void)f;
    int r = step();
    if (r == 0)
        for (int i = 0; i < kStreams; ++i)
            if (queue(s)->before[i] < ((Event*)e)->before[i]) queue(s)->before[i] = ((Event*)e)->before[i];
    return r;
}
int cudaStreamSynchronize(void* s) {      /* what was on it is over: nobody has to wait for it any more */
    for (int i = 0; i < n_streams; ++i)
        if (streams[i].before[queue(s)->id] < queue(s)->before[queue(s)->id]) streams[i].before[queue(s)->id] = queue(s)->before[queue(s)->id];
    return 0;
}
typedef struct { unsigned x, y, z; } dim3_t;
typedef struct { int id; char pad[4]; char value[64]; } LaunchAttribute;
typedef struct { dim3_t grid, block; size_t smem; void* stream; LaunchAttribute* attrs; unsigned n; } LaunchConfig;
static int too_large(dim3_t g) { return g.x > 0x7fffffffu || g.y > 65535 || g.z > 65535; }
static int overlapped;             /* whether the last launch was a programmatic dependent */
static unsigned long long capture; /* the capture that is on, on every stream */
int fake_overlapped(void) { return overlapped; }
void fake_capture(unsigned long long id) { capture = id; }
int cudaLaunchKernelExC(const LaunchConfig* c, const void* f, void** a) {
    (void)f; (void)a;
    overlapped = 0;
    if (too_large(c->grid)) return last_error = 9;
    for (unsigned i = 0; i < c->n; ++i) overlapped |= c->attrs[i].id == 6;      /* cudaLaunchAttributeProgrammaticStreamSerialization */
    return enqueue(c->stream);
}
int cudaLaunchKernel(const void* f, dim3_t g, dim3_t b, void** a, size_t m, void* s) {
    (void)f; (void)b; (void)a; (void)m;
    overlapped = 0;
    return too_large(g) ? (last_error = 9) : enqueue(s);
}
int cudaMemsetAsync(void* p, int v, size_t n, void* s) { (void)p; (void)v; (void)n; return enqueue(s); }
int cudaMemcpyAsync(void* d, const void* p, size_t n, int k, void* s) { (void)d; (void)p; (void)n; (void)k; return enqueue(s); }
int cudaMemcpy2DAsync(void* d, size_t dp, const void* p, size_t sp, size_t w, size_t h, int k, void* s) {
    (void)d; (void)dp; (void)p; (void)sp; (void)w; (void)h; (void)k;
    return enqueue(s);
}

/* launches written as kernel<<<...>>>(...) */
static struct { dim3_t g, b; size_t m; void* s; } pushed;
unsigned __cudaPushCallConfiguration(dim3_t g, dim3_t b, size_t m, void* s) { pushed.g = g; pushed.b = b; pushed.m = m; pushed.s = s; return 0; }
int __cudaPopCallConfiguration(dim3_t* g, dim3_t* b, size_t* m, void* s) { *g = pushed.g; *b = pushed.b; *m = pushed.m; *(void**)s = pushed.s; return 0; }
void** __cudaRegisterFatBinary(void* p) { static void* h; (void)p; return &h; }
void __cudaRegisterFatBinaryEnd(void** p) { (void)p; }
void __cudaUnregisterFatBinary(void** p) { (void)p; }
void __cudaRegisterFunction(void) {}
void __cudaRegisterVar(void) {}

static int encode(void) { return 0; }
int cudaGetDriverEntryPoint(const char* name, void** f, unsigned long long flags, int* found) { (void)name; (void)flags; *f = (void*)encode; *found = 0; return 0; }
static long queries;               /* questions about the device */
long fake_queries(void) { long n = queries; queries = 0; return n; }
int cudaGetDevice(int* d) { ++queries; *d = 0; return 0; }
int cudaDeviceGetAttribute(int* v, int a, int d) { (void)a; (void)d; *v = 148; return 0; }
int cudaFuncSetAttribute(const void* f, int a, int v) { ++queries; (void)f; (void)a; (void)v; return 0; }
int cudaGetLastError(void) { int r = last_error; last_error = 0; return r; }
int cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int* n, const void* f, int t, size_t m, unsigned fl) { (void)f; (void)t; (void)m; (void)fl; *n = 1; return 0; }
int cudaOccupancyMaxActiveClusters(int* n, const void* f, const LaunchConfig* c) {      /* as a B200 with one CTA per SM */
    static const int most[17] = {0, 148, 74, 0, 33, 0, 0, 0, 15, 15, 11, 7, 7, 7, 7, 7, 7};
    (void)f;
    ++queries;
    *n = most[*(const unsigned*)c->attrs[0].value];      /* (the cluster's extent is the only attribute) */
    return 0;
}
int cudaStreamIsCapturing(void* s, int* v) { (void)s; *v = capture != 0; return 0; }
int cudaStreamGetCaptureInfo_v2(void* s, int* v, unsigned long long* id, void* g, void* d, void* n) {
    (void)s; (void)g; (void)d; (void)n;
    *v = capture != 0;
    if (id) *id = capture;
    return 0;
}
int cudaStreamBeginCapture(void* s, int m) { (void)s; (void)m; return 900; }
int cudaStreamEndCapture(void* s, void** g) { (void)s; *g = NULL; return 900; }
int cudaGraphInstantiate(void) { return 900; }
int cudaGraphLaunch(void) { return 900; }
int cudaGraphDestroy(void) { return 0; }
int cudaGraphExecDestroy(void) { return 0; }
int cudaEventElapsedTime(float* t, void* a, void* b) { (void)a; (void)b; *t = 0; return 0; }
int cudaEventSynchronize(void* e) { (void)e; return 0; }
int cudaGetSymbolAddress(void** p, const void* s) { *p = (void*)s; return 0; }
int cudaHostAlloc(void** p, size_t n, unsigned f) { (void)f; *p = malloc(n); return 0; }
int cudaFreeHost(void* p) { free(p); return 0; }
