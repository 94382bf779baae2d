/* A CUDA runtime without a device, for the host code's order of work (test_stream_order.py):
   device memory is host memory, copies and fills take place at once, a kernel launch is
   written down and does nothing.  Only the tree kernel's answer, which the host reads, is
   given: levels 0 and 1 with 12 and 48 boxes, done. */
#include <stdarg.h>
#include <stdio.h>
#include <stdlib.h>
#include <string.h>

typedef struct { unsigned x, y, z; } dim3;
typedef struct { dim3 grid, block; size_t smem; void* stream; } launch_config;
static char text[1 << 20];
static size_t used;
static struct { const void* host; const char* name; } kernels[4096];
static int n_kernels;
static launch_config pushed;

static void say(const char* fmt, ...)
{
    va_list a;
    va_start(a, fmt);
    if (used < sizeof text - 512) used += (size_t)vsnprintf(text + used, 512, fmt, a);
    va_end(a);
}
const char* fake_trace(void) { return text; }
void fake_clear(void) { used = 0; text[0] = 0; }

static int launch(const void* host, void** args, void* stream)
{
    const char* name = "?";
    for (int i = 0; i < n_kernels; ++i)
        if (kernels[i].host == host) name = kernels[i].name;
    say("launch %p %s\n", stream, name);
    if (strstr(name, "k_tree_narrow")) {
        long long* levels = *(long long**)args[6];
        levels[0] = 1;
        levels[1] = 1;
        levels[2] = 0;
        levels[3] = 12;
        levels[4] = 60;
    }
    return 0;
}

void** __cudaRegisterFatBinary(void* f) { return (void**)f; }
void __cudaRegisterFatBinaryEnd(void** h) { (void)h; }
void __cudaUnregisterFatBinary(void** h) { (void)h; }
void __cudaRegisterVar(void** h, char* v, char* d, const char* n, int e, size_t s, int c, int g)
{
    (void)h; (void)v; (void)d; (void)n; (void)e; (void)s; (void)c; (void)g;
}
void __cudaRegisterFunction(void** h, const char* host, char* d, const char* name, int t, void* a, void* b, dim3* c, dim3* e, int* w)
{
    (void)h; (void)d; (void)t; (void)a; (void)b; (void)c; (void)e; (void)w;
    if (n_kernels < 4096) { kernels[n_kernels].host = host; kernels[n_kernels++].name = name; }
}
unsigned __cudaPushCallConfiguration(dim3 g, dim3 b, size_t m, void* s)
{
    pushed.grid = g; pushed.block = b; pushed.smem = m; pushed.stream = s;
    return 0;
}
int __cudaPopCallConfiguration(dim3* g, dim3* b, size_t* m, void* s)
{
    *g = pushed.grid; *b = pushed.block; *m = pushed.smem; *(void**)s = pushed.stream;
    return 0;
}
int __cudaGetKernel(void** k, const void* host) { *k = (void*)host; return 0; }
int __cudaLaunchKernel(void* k, dim3 g, dim3 b, void** args, size_t m, void* s) { (void)g; (void)b; (void)m; return launch(k, args, s); }
int cudaLaunchKernelExC(const launch_config* c, const void* f, void** args) { return launch(f, args, c->stream); }

int cudaMalloc(void** p, size_t n) { *p = calloc(1, n); return *p ? 0 : 2; }
int cudaFree(void* p) { free(p); return 0; }
int cudaHostAlloc(void** p, size_t n, unsigned f) { (void)f; return cudaMalloc(p, n); }
int cudaFreeHost(void* p) { free(p); return 0; }
int cudaGetSymbolAddress(void** p, const void* s) { (void)s; return cudaMalloc(p, 1 << 23); }
int cudaMemsetAsync(void* p, int v, size_t n, void* s) { memset(p, v, n); say("memset %p\n", s); return 0; }
int cudaMemcpyAsync(void* d, const void* f, size_t n, int k, void* s) { memcpy(d, f, n); say("copy%d %p\n", k, s); return 0; }
int cudaMemcpy(void* d, const void* f, size_t n, int k) { (void)k; memcpy(d, f, n); say("sync %p\n", (void*)0); return 0; }

static int handle(void** h) { *h = malloc(1); return 0; }
int cudaStreamCreateWithFlags(void** s, unsigned f) { (void)f; return handle(s); }
int cudaStreamDestroy(void* s) { free(s); return 0; }
int cudaStreamSynchronize(void* s) { say("sync %p\n", s); return 0; }
int cudaEventCreate(void** e) { return handle(e); }
int cudaEventCreateWithFlags(void** e, unsigned f) { (void)f; return handle(e); }
int cudaEventDestroy(void* e) { free(e); return 0; }
int cudaEventRecord(void* e, void* s) { say("record %p %p\n", s, e); return 0; }
int cudaStreamWaitEvent(void* s, void* e, unsigned f) { (void)f; say("wait %p %p\n", s, e); return 0; }
int cudaEventSynchronize(void* e) { (void)e; return 0; }
int cudaEventElapsedTime(float* ms, void* a, void* b) { (void)a; (void)b; *ms = 0; return 0; }

int cudaGetLastError(void) { return 0; }
const char* cudaGetErrorString(int e) { (void)e; return "fake"; }
int cudaGetDevice(int* d) { *d = 0; return 0; }
int cudaSetDevice(int d) { (void)d; return 0; }
int cudaDeviceGetAttribute(int* v, int a, int d) { (void)a; (void)d; *v = 152; return 0; }
int cudaFuncSetAttribute(const void* f, int a, int v) { (void)f; (void)a; (void)v; return 0; }

/* graphs are not traced */
int cudaStreamBeginCapture(void) { return 801; }
int cudaStreamEndCapture(void) { return 801; }
int cudaGraphGetNodes(void) { return 801; }
int cudaGraphNodeGetType(void) { return 801; }
int cudaGraphInstantiate(void) { return 801; }
int cudaGraphLaunch(void) { return 801; }
int cudaGraphDestroy(void) { return 801; }
int cudaGraphExecDestroy(void) { return 801; }
