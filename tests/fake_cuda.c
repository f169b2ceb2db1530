/* A stand-in for the CUDA runtime, linked with the library's own object files in place of libcudart: every call that the host
 * code makes is written to a log (which stream, which event, which kernel), nothing runs, and any call can be made to fail.
 * Device pointers are never followed. */
#include <cuda.h>
#include <cuda_runtime_api.h>
#include <stdio.h>
#include <stdlib.h>
#include <string.h>

enum { LAUNCH = 1, RECORD, WAIT, COPY, SET, STREAM_CREATE, EVENT_CREATE, DEVICE_ALLOC };
/* obj: the event, or a launch's dynamic shared memory in bytes */
typedef struct { int kind; long stream, obj, grid; char name[96]; unsigned char arg[256]; } entry;
enum { MAX_LOG = 20000, MAX_KERNELS = 512 };
static entry log_[MAX_LOG];
static int n_log, capturing, fail_kind, fail_after;
static cudaError_t last_error;
static long next_handle = 1;
static struct { const void* f; char name[256]; } kernels[MAX_KERNELS];
static int n_kernels;
static char arg_of[64];
static int arg_bytes;

void fake_reset(void) { n_log = 0; capturing = 0; fail_kind = 0; fail_after = 0; last_error = cudaSuccess; arg_bytes = 0; }
void fake_fail(int kind, int after) { fail_kind = kind; fail_after = after; }      /* the call of that kind after `after` others */
void fake_capturing(int on) { capturing = on; }
/* keep the first `bytes` of the first argument of launches whose kernel's name holds `part` */
void fake_keep_arg(const char* part, int bytes)
{
    snprintf(arg_of, sizeof arg_of, "%s", part);
    arg_bytes = bytes;
}
int fake_count(void) { return n_log; }
const entry* fake_entry(int i) { return &log_[i]; }

static cudaError_t put(int kind, cudaStream_t st, long obj, long grid, const char* name, void** args)
{
    if (kind == fail_kind && fail_after-- == 0) { fail_kind = 0; return last_error = cudaErrorUnknown; }
    if (n_log == MAX_LOG) abort();
    entry* e = &log_[n_log++];
    e->kind = kind; e->stream = (long)st; e->obj = obj; e->grid = grid;
    snprintf(e->name, sizeof e->name, "%s", name ? name : "");
    if (args && arg_bytes && strstr(e->name, arg_of)) memcpy(e->arg, args[0], arg_bytes);
    return cudaSuccess;
}
/* "sinkhorn_tile_kernel" out of a mangled name: the identifier that ends in _kernel and whose length stands in front of it */
static const char* short_name(const char* s, char* out, size_t n)
{
    const char* end = strstr(s, "_kernel");
    snprintf(out, n, "%s", s);
    if (!end) return out;
    end += 7;
    for (const char* b = end - 8; b > s; --b) {
        const char* d = b;
        while (d > s && d[-1] >= '0' && d[-1] <= '9') --d;
        for (; d < b; ++d)
            if (atol(d) == end - b && *d != '0') { snprintf(out, n, "%.*s", (int)(end - b), b); return out; }
    }
    return out;
}
static const char* name_of(const void* f)
{
    for (int i = 0; i < n_kernels; ++i)
        if (kernels[i].f == f) return kernels[i].name;
    return "?";
}

void** __cudaRegisterFatBinary(void* p) { static void* h; (void)p; return &h; }
void __cudaRegisterFatBinaryEnd(void** h) { (void)h; }
void __cudaUnregisterFatBinary(void** h) { (void)h; }
void __cudaRegisterFunction(void** h, const char* host, char* dev, const char* name, int limit, void* a, void* b, void* c, void* d, int* w)
{
    (void)h; (void)dev; (void)limit; (void)a; (void)b; (void)c; (void)d; (void)w;
    if (n_kernels == MAX_KERNELS) abort();
    kernels[n_kernels].f = host;
    short_name(name, kernels[n_kernels].name, sizeof kernels[0].name);
    ++n_kernels;
}
void __cudaRegisterVar(void** h, char* host, char* dev, const char* name, int ext, size_t size, int constant, int global)
{
    (void)h; (void)host; (void)dev; (void)name; (void)ext; (void)size; (void)constant; (void)global;
}
static struct { dim3 grid, block; size_t smem; void* st; } pushed;
unsigned __cudaPushCallConfiguration(dim3 grid, dim3 block, size_t smem, void* st)
{
    pushed.grid = grid; pushed.block = block; pushed.smem = smem; pushed.st = st;
    return 0;
}
cudaError_t __cudaPopCallConfiguration(dim3* grid, dim3* block, size_t* smem, void* st)
{
    *grid = pushed.grid; *block = pushed.block; *smem = pushed.smem; *(void**)st = pushed.st;
    return cudaSuccess;
}
cudaError_t cudaLaunchKernel(const void* f, dim3 grid, dim3 block, void** args, size_t smem, cudaStream_t st)
{
    (void)block;
    return put(LAUNCH, st, (long)smem, (long)grid.x * grid.y * grid.z, name_of(f), args);
}
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t* c, const void* f, void** args)
{
    return put(LAUNCH, c->stream, (long)c->dynamicSmemBytes, (long)c->gridDim.x * c->gridDim.y * c->gridDim.z, name_of(f), args);
}
cudaError_t cudaFuncSetAttribute(const void* f, enum cudaFuncAttribute a, int v) { (void)f; (void)a; (void)v; return cudaSuccess; }
cudaError_t cudaGetLastError(void) { cudaError_t e = last_error; last_error = cudaSuccess; return e; }
cudaError_t cudaGetDevice(int* d) { *d = 0; return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int* v, enum cudaDeviceAttr a, int d) { (void)a; (void)d; *v = 148; return cudaSuccess; }
cudaError_t cudaDeviceSynchronize(void) { return cudaSuccess; }
cudaError_t cudaMalloc(void** p, size_t n)
{
    const cudaError_t e = put(DEVICE_ALLOC, 0, (long)n, 0, "", NULL);
    if (e == cudaSuccess) *p = calloc(1, n ? n : 1);
    return e;
}
cudaError_t cudaFree(void* p) { free(p); return cudaSuccess; }
cudaError_t cudaMemcpy(void* d, const void* s, size_t n, enum cudaMemcpyKind k) { (void)k; memcpy(d, s, n); return cudaSuccess; }
cudaError_t cudaMemset(void* d, int v, size_t n) { memset(d, v, n); return cudaSuccess; }
cudaError_t cudaMemcpyAsync(void* d, const void* s, size_t n, enum cudaMemcpyKind k, cudaStream_t st)
{
    (void)d; (void)s;
    return put(COPY, st, (long)n, 0, k == cudaMemcpyHostToDevice ? "in" : "out", NULL);
}
cudaError_t cudaMemsetAsync(void* d, int v, size_t n, cudaStream_t st) { (void)d; (void)v; return put(SET, st, (long)n, 0, "", NULL); }
cudaError_t cudaStreamCreateWithFlags(cudaStream_t* s, unsigned f)
{
    (void)f;
    const long h = 0x1000 + next_handle++;
    const cudaError_t e = put(STREAM_CREATE, (cudaStream_t)h, h, 0, "", NULL);
    if (e == cudaSuccess) *s = (cudaStream_t)h;
    return e;
}
cudaError_t cudaStreamDestroy(cudaStream_t s) { (void)s; return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t s) { (void)s; return cudaSuccess; }
cudaError_t cudaStreamIsCapturing(cudaStream_t s, enum cudaStreamCaptureStatus* out)
{
    (void)s;
    *out = capturing ? cudaStreamCaptureStatusActive : cudaStreamCaptureStatusNone;
    return cudaSuccess;
}
cudaError_t cudaStreamWaitEvent(cudaStream_t s, cudaEvent_t e, unsigned f) { (void)f; return put(WAIT, s, (long)e, 0, "", NULL); }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t* e, unsigned f)
{
    (void)f;
    const long h = 0x100000 + next_handle++;
    const cudaError_t r = put(EVENT_CREATE, 0, h, 0, "", NULL);
    if (r == cudaSuccess) *e = (cudaEvent_t)h;
    return r;
}
cudaError_t cudaEventCreate(cudaEvent_t* e) { return cudaEventCreateWithFlags(e, 0); }
cudaError_t cudaEventRecord(cudaEvent_t e, cudaStream_t s) { return put(RECORD, s, (long)e, 0, "", NULL); }
cudaError_t cudaEventDestroy(cudaEvent_t e) { (void)e; return cudaSuccess; }
cudaError_t cudaEventSynchronize(cudaEvent_t e) { (void)e; return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float* ms, cudaEvent_t a, cudaEvent_t b) { (void)a; (void)b; *ms = 0.0f; return cudaSuccess; }
cudaError_t cudaGetSymbolAddress(void** p, const void* s) { (void)s; *p = (void*)0x100000000; return cudaSuccess; }
static int encode_ok(void) { return 0; }
cudaError_t cudaGetDriverEntryPoint(const char* name, void** f, unsigned long long flags, enum cudaDriverEntryPointQueryResult* q)
{
    (void)name; (void)flags;
    *f = (void*)encode_ok;
    if (q) *q = cudaDriverEntryPointSuccess;
    return cudaSuccess;
}
