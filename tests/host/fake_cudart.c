/* A stand-in for the CUDA runtime, preloaded before libisc.so so that its host code runs without a GPU: device memory
 * is host memory, kernels do nothing, and a launch is refused as the real runtime refuses it when its dynamic shared
 * memory exceeds what cudaFuncSetAttribute granted on the current device.  Every launch is recorded. */
#include <cuda_runtime_api.h>
#include <pthread.h>
#include <stdlib.h>
#include <string.h>
#include <unistd.h>

#define MAX_FUNCS 64
#define MAX_DEVICES 4
#define MAX_LAUNCHES 65536

typedef struct { const void *host; const char *name; int smem[MAX_DEVICES]; } Func;
typedef struct { const char *name; int device, stream_device, priority, ok, watched; unsigned long long words[20]; } Launch;
struct CUstream_st { int priority, device; };

static Func funcs[MAX_FUNCS];
static int n_funcs, n_launches, set_attribute_delay_us;
static Launch launches[MAX_LAUNCHES];
static size_t allocated, largest = (size_t)-1;
static int refused;
static const void *watched;
static pthread_mutex_t lock = PTHREAD_MUTEX_INITIALIZER;
static __thread int device;
static __thread cudaError_t last;
static __thread struct { dim3 grid, block; size_t smem; void *stream; } pending;

/* what the tests ask and set */
void fake_set_device(int d) { device = d; }
void fake_set_attribute_delay(int us) { set_attribute_delay_us = us; }
void fake_reset(void) { n_launches = 0; }
int fake_launches(void) { return n_launches; }
const char *fake_launch_name(int i) { return launches[i].name; }
int fake_launch_device(int i) { return launches[i].device; }
int fake_launch_priority(int i) { return launches[i].priority; }
int fake_launch_stream_device(int i) { return launches[i].stream_device; }
int fake_launch_ok(int i) { return launches[i].ok; }
/* 1: the word `watch` stands in the launch's first argument */
void fake_watch(const void *word) { watched = word; }
int fake_launch_watched(int i) { return launches[i].watched; }
/* word `k` of the first twenty of k_line's parameters */
unsigned long long fake_launch_word(int i, int k) { return launches[i].words[k]; }
size_t fake_allocated(void) { return allocated; }
/* larger allocations are refused from now on; how many were */
void fake_set_largest(size_t bytes) { largest = bytes; refused = 0; }
int fake_refused(void) { return refused; }

static Func *find(const void *host)
{
    for (int i = 0; i < n_funcs; ++i)
        if (funcs[i].host == host) return &funcs[i];
    return NULL;
}

/* registration, as compiled CUDA code calls it when it is loaded */
void **__cudaRegisterFatBinary(void *image) { static void *handle; (void)image; return &handle; }
void __cudaRegisterFatBinaryEnd(void **h) { (void)h; }
void __cudaUnregisterFatBinary(void **h) { (void)h; }
void __cudaRegisterVar(void **h, char *host, char *dev, const char *name, int ext, size_t size, int constant, int global)
{
    (void)h; (void)host; (void)dev; (void)name; (void)ext; (void)size; (void)constant; (void)global;
}
void __cudaRegisterFunction(void **h, const char *host, char *dev, const char *name, int limit, uint3 *t, uint3 *b, dim3 *bd, dim3 *gd, int *w)
{
    (void)h; (void)dev; (void)limit; (void)t; (void)b; (void)bd; (void)gd; (void)w;
    if (n_funcs < MAX_FUNCS) funcs[n_funcs++] = (Func){host, name, {0}};
}
unsigned __cudaPushCallConfiguration(dim3 grid, dim3 block, size_t smem, void *stream)
{
    pending.grid = grid; pending.block = block; pending.smem = smem; pending.stream = stream;
    return 0;
}
cudaError_t __cudaPopCallConfiguration(dim3 *grid, dim3 *block, size_t *smem, void *stream)
{
    *grid = pending.grid; *block = pending.block; *smem = pending.smem; *(void **)stream = pending.stream;
    return cudaSuccess;
}

cudaError_t cudaLaunchKernel(const void *func, dim3 grid, dim3 block, void **args, size_t smem, cudaStream_t st)
{
    (void)grid; (void)block;
    pthread_mutex_lock(&lock);
    Func *f = find(func);
    const int ok = f && (smem <= 48 * 1024 || smem <= (size_t)f->smem[device]);
    if (f && n_launches < MAX_LAUNCHES) {
        int seen = 0;
        /* the first argument of the kernels in question is a structure of more than 256 bytes */
        if (watched && (strstr(f->name, "k_stem") || strstr(f->name, "k_line")))
            for (int i = 0; i < 256 / 8; ++i) seen |= ((const void **)args[0])[i] == watched;
        launches[n_launches++] = (Launch){f->name, device, st ? st->device : device, st ? st->priority : 0, ok, seen, {0}};
        if (strstr(f->name, "k_line")) memcpy(launches[n_launches - 1].words, args[0], sizeof(launches[0].words));
    }
    pthread_mutex_unlock(&lock);
    if (!ok) last = cudaErrorInvalidValue;
    return ok ? cudaSuccess : cudaErrorInvalidValue;
}
cudaError_t cudaFuncSetAttribute(const void *func, enum cudaFuncAttribute attr, int value)
{
    if (set_attribute_delay_us) usleep((useconds_t)set_attribute_delay_us);
    pthread_mutex_lock(&lock);
    Func *f = find(func);
    if (f && attr == cudaFuncAttributeMaxDynamicSharedMemorySize) f->smem[device] = value;
    pthread_mutex_unlock(&lock);
    return f ? cudaSuccess : cudaErrorInvalidDeviceFunction;
}

cudaError_t cudaGetLastError(void) { const cudaError_t e = last; last = cudaSuccess; return e; }
const char *cudaGetErrorString(cudaError_t e) { return e == cudaSuccess ? "no error" : "fake error"; }
cudaError_t cudaGetDevice(int *d) { *d = device; return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int *value, enum cudaDeviceAttr attr, int d)
{
    (void)d;
    *value = attr == cudaDevAttrMultiProcessorCount ? 148 : 0;
    return cudaSuccess;
}
cudaError_t cudaGetDeviceProperties(struct cudaDeviceProp *p, int d)
{
    (void)d;
    memset(p, 0, sizeof(*p));
    p->major = 10; p->multiProcessorCount = 148; p->sharedMemPerBlockOptin = 227 * 1024;
    return cudaSuccess;
}
cudaError_t cudaGetDriverEntryPoint(const char *symbol, void **fn, unsigned long long flags, enum cudaDriverEntryPointQueryResult *r)
{
    (void)symbol; (void)flags;
    *fn = NULL;
    *r = cudaDriverEntryPointSymbolNotFound;
    return cudaSuccess;
}
cudaError_t cudaGetSymbolAddress(void **p, const void *symbol)
{
    static unsigned char scratch[MAX_DEVICES][40 << 20] __attribute__((aligned(256)));
    (void)symbol;
    *p = scratch[device];
    return cudaSuccess;
}

cudaError_t cudaMalloc(void **p, size_t bytes)
{
    pthread_mutex_lock(&lock);
    const int fits = bytes <= largest;
    if (fits) allocated += bytes; else refused += 1;
    pthread_mutex_unlock(&lock);
    if (!fits) return last = cudaErrorMemoryAllocation;
    return posix_memalign(p, 256, bytes) ? cudaErrorMemoryAllocation : cudaSuccess;
}
cudaError_t cudaFree(void *p) { free(p); return cudaSuccess; }
cudaError_t cudaHostAlloc(void **p, size_t bytes, unsigned flags) { (void)flags; return posix_memalign(p, 4096, bytes) ? cudaErrorMemoryAllocation : cudaSuccess; }
cudaError_t cudaFreeHost(void *p) { free(p); return cudaSuccess; }
cudaError_t cudaMemcpy(void *d, const void *s, size_t n, enum cudaMemcpyKind k) { (void)k; memcpy(d, s, n); return cudaSuccess; }
cudaError_t cudaMemcpyAsync(void *d, const void *s, size_t n, enum cudaMemcpyKind k, cudaStream_t st) { (void)k; (void)st; memcpy(d, s, n); return cudaSuccess; }
cudaError_t cudaMemset(void *d, int v, size_t n) { memset(d, v, n); return cudaSuccess; }
cudaError_t cudaMemsetAsync(void *d, int v, size_t n, cudaStream_t st) { (void)st; memset(d, v, n); return cudaSuccess; }

cudaError_t cudaStreamCreateWithPriority(cudaStream_t *st, unsigned flags, int priority)
{
    (void)flags;
    *st = malloc(sizeof(**st));
    (*st)->priority = priority;
    (*st)->device = device;
    return cudaSuccess;
}
cudaError_t cudaStreamCreateWithFlags(cudaStream_t *st, unsigned flags) { return cudaStreamCreateWithPriority(st, flags, 0); }
cudaError_t cudaStreamGetPriority(cudaStream_t st, int *priority) { *priority = st ? st->priority : 0; return cudaSuccess; }
cudaError_t cudaStreamDestroy(cudaStream_t st) { free(st); return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t st) { (void)st; return cudaSuccess; }
cudaError_t cudaStreamWaitEvent(cudaStream_t st, cudaEvent_t e, unsigned flags) { (void)st; (void)e; (void)flags; return cudaSuccess; }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t *e, unsigned flags) { (void)flags; *e = malloc(1); return cudaSuccess; }
cudaError_t cudaEventDestroy(cudaEvent_t e) { free(e); return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t e, cudaStream_t st) { (void)e; (void)st; return cudaSuccess; }
cudaError_t cudaEventSynchronize(cudaEvent_t e) { (void)e; return cudaSuccess; }
