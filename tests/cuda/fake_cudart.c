/* A stand-in for the CUDA runtime, preloaded ahead of libcudart: libmc.so's host code runs without a GPU.  Kernels are
 * not executed: every launch is logged by name, with whether it may start before its predecessor has ended
 * (programmatic serialisation).  "Device" memory is host memory that the test allocates; copies and fills are
 * real.  Streams know whether they are being captured, graphs hold the launches captured into them.
 * fake_* functions are for the tests. */
#include <cuda_runtime_api.h>
#include <stdio.h>
#include <stdlib.h>
#include <string.h>

#define MAXK 512
#define LOGLEN (1 << 22)
#define GRAPHLEN (1 << 20)

struct graph {
    char text[GRAPHLEN];
    size_t len;
};
struct stream {
    int capturing; /* 1: of its own, 2: joined another stream's through an event */
    struct graph *g;
};
struct event {
    int captured;
};

static struct {
    const void *host;
    char name[256];
} kernels[MAXK];
static int n_kernels;
static char log_text[LOGLEN];
static size_t log_len;
static struct stream null_stream;
static cudaError_t last_error;
static int fail_after = -1, regs = 128, clusters = 19;
static struct {
    dim3 grid, block;
    size_t smem;
    cudaStream_t s;
} pushed;

const char *fake_log(void) { return log_text; }
void fake_clear(void) { log_text[log_len = 0] = 0; }
/* the n-th launch from now on (0 = the next) fails, once; -1: none */
void fake_fail_launch(int n) { fail_after = n; }
void fake_set_regs(int n) { regs = n; }
/* clusters that fit the device at once (0: a cluster cannot be placed) */
void fake_set_clusters(int n) { clusters = n; }

static cudaError_t result(cudaError_t e)
{
    if (e != cudaSuccess)
        last_error = e;
    return e;
}
static struct stream *of(cudaStream_t s) { return s ? (struct stream *)s : &null_stream; }
static void put(const char *text)
{
    const size_t n = strlen(text);
    if (log_len + n + 1 < LOGLEN) {
        memcpy(log_text + log_len, text, n + 1);
        log_len += n;
    }
}
static cudaError_t launch(const void *host, dim3 grid, dim3 block, int programmatic, cudaStream_t st)
{
    if (fail_after >= 0 && fail_after-- == 0)
        return result(cudaErrorLaunchOutOfResources);
    const char *name = "?";
    for (int i = 0; i < n_kernels; ++i)
        if (kernels[i].host == host)
            name = kernels[i].name;
    char line[400];
    snprintf(line, sizeof line, "%s %u %u %s\n", name, grid.x, block.x, programmatic ? "programmatic" : "plain");
    struct stream *s = of(st);
    if (s->g) {
        const size_t n = strlen(line);
        if (s->g->len + n + 1 < GRAPHLEN) {
            memcpy(s->g->text + s->g->len, line, n + 1);
            s->g->len += n;
        }
    } else {
        put(line);
    }
    return cudaSuccess;
}

/* ---- kernels */
void **__cudaRegisterFatBinary(void *p)
{
    (void)p;
    static void *handle;
    return &handle;
}
void __cudaRegisterFatBinaryEnd(void **h) { (void)h; }
void __cudaUnregisterFatBinary(void **h) { (void)h; }
void __cudaRegisterFunction(void **h, const char *host, char *dev, const char *name, int limit, void *tid, void *bid, void *bd,
                            void *gd, int *ws)
{
    (void)h, (void)dev, (void)limit, (void)tid, (void)bid, (void)bd, (void)gd, (void)ws;
    if (n_kernels < MAXK) {
        kernels[n_kernels].host = host;
        snprintf(kernels[n_kernels++].name, sizeof kernels[0].name, "%s", name);
    }
}
void __cudaRegisterVar(void **h, char *host, char *dev, const char *name, int ext, size_t size, int constant, int global)
{
    (void)h, (void)host, (void)dev, (void)name, (void)ext, (void)size, (void)constant, (void)global;
}
unsigned __cudaPushCallConfiguration(dim3 grid, dim3 block, size_t smem, void *s)
{
    pushed.grid = grid, pushed.block = block, pushed.smem = smem, pushed.s = (cudaStream_t)s;
    return 0;
}
cudaError_t __cudaPopCallConfiguration(dim3 *grid, dim3 *block, size_t *smem, void *s)
{
    *grid = pushed.grid, *block = pushed.block, *smem = pushed.smem, *(cudaStream_t *)s = pushed.s;
    return cudaSuccess;
}
cudaError_t __cudaGetKernel(cudaKernel_t *k, const void *host)
{
    *k = (cudaKernel_t)host;
    return cudaSuccess;
}
cudaError_t __cudaLaunchKernel(cudaKernel_t k, dim3 grid, dim3 block, void **args, size_t smem, cudaStream_t s)
{
    (void)args, (void)smem;
    return launch((const void *)k, grid, block, 0, s);
}
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t *c, const void *f, void **args)
{
    (void)args;
    int programmatic = 0;
    for (unsigned i = 0; i < c->numAttrs; ++i)
        programmatic |= c->attrs[i].id == cudaLaunchAttributeProgrammaticStreamSerialization &&
                        c->attrs[i].val.programmaticStreamSerializationAllowed;
    return launch(f, c->gridDim, c->blockDim, programmatic, c->stream);
}
cudaError_t cudaFuncGetAttributes(struct cudaFuncAttributes *a, const void *f)
{
    (void)f;
    memset(a, 0, sizeof *a);
    a->numRegs = regs;
    a->maxDynamicSharedSizeBytes = 49152;
    return cudaSuccess;
}
cudaError_t cudaFuncSetAttribute(const void *f, enum cudaFuncAttribute at, int v)
{
    (void)f, (void)at, (void)v;
    return cudaSuccess;
}
cudaError_t cudaOccupancyMaxActiveClusters(int *n, const void *f, const cudaLaunchConfig_t *c)
{
    (void)f, (void)c;
    *n = clusters;
    return cudaSuccess;
}

/* ---- device and errors */
cudaError_t cudaGetDevice(int *d) { return *d = 0, cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int *v, enum cudaDeviceAttr a, int d)
{
    (void)d;
    *v = a == cudaDevAttrMultiProcessorCount ? 152 : a == cudaDevAttrMaxSharedMemoryPerBlockOptin ? 232448 : 0;
    return cudaSuccess;
}
cudaError_t cudaGetLastError(void)
{
    const cudaError_t e = last_error;
    last_error = cudaSuccess;
    return e;
}
const char *cudaGetErrorString(cudaError_t e) { return e == cudaSuccess ? "no error" : "an error of the stand-in"; }
static int encode(void) { return 0; } /* cuTensorMapEncodeTiled */
cudaError_t cudaGetDriverEntryPointByVersion(const char *name, void **f, unsigned v, unsigned long long flags,
                                             enum cudaDriverEntryPointQueryResult *q)
{
    (void)name, (void)v, (void)flags;
    *f = (void *)encode;
    *q = cudaDriverEntryPointSuccess;
    return cudaSuccess;
}

/* ---- memory */
cudaError_t cudaPointerGetAttributes(struct cudaPointerAttributes *a, const void *p)
{
    memset(a, 0, sizeof *a);
    a->type = cudaMemoryTypeDevice;
    a->devicePointer = (void *)p;
    return cudaSuccess;
}
cudaError_t cudaMemcpyAsync(void *d, const void *s, size_t n, enum cudaMemcpyKind k, cudaStream_t st)
{
    (void)k, (void)st;
    memmove(d, s, n);
    return cudaSuccess;
}
cudaError_t cudaMemcpy2DAsync(void *d, size_t dp, const void *s, size_t sp, size_t w, size_t h, enum cudaMemcpyKind k,
                              cudaStream_t st)
{
    (void)k, (void)st;
    for (size_t i = 0; i < h; ++i)
        memmove((char *)d + i * dp, (const char *)s + i * sp, w);
    return cudaSuccess;
}
cudaError_t cudaMemsetAsync(void *d, int v, size_t n, cudaStream_t st)
{
    (void)st;
    memset(d, v, n);
    return cudaSuccess;
}
cudaError_t cudaHostAlloc(void **p, size_t n, unsigned flags)
{
    (void)flags;
    return (*p = calloc(1, n)) ? cudaSuccess : result(cudaErrorMemoryAllocation);
}
cudaError_t cudaFreeHost(void *p) { return free(p), cudaSuccess; }
cudaError_t cudaGetSymbolAddress(void **p, const void *s) { return *p = (void *)s, cudaSuccess; }

/* ---- streams, events, graphs */
cudaError_t cudaStreamCreateWithFlags(cudaStream_t *s, unsigned flags)
{
    (void)flags;
    return (*s = (cudaStream_t)calloc(1, sizeof(struct stream))) ? cudaSuccess : result(cudaErrorMemoryAllocation);
}
cudaError_t cudaStreamDestroy(cudaStream_t s) { return free(s), cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t s)
{
    return of(s)->capturing ? result(cudaErrorStreamCaptureUnsupported) : cudaSuccess;
}
cudaError_t cudaStreamIsCapturing(cudaStream_t s, enum cudaStreamCaptureStatus *c)
{
    *c = of(s)->capturing ? cudaStreamCaptureStatusActive : cudaStreamCaptureStatusNone;
    return cudaSuccess;
}
cudaError_t cudaStreamBeginCapture(cudaStream_t s, enum cudaStreamCaptureMode m)
{
    (void)m;
    if (of(s)->capturing)
        return result(cudaErrorIllegalState);
    of(s)->capturing = 1;
    of(s)->g = calloc(1, sizeof(struct graph));
    return cudaSuccess;
}
cudaError_t cudaStreamEndCapture(cudaStream_t s, cudaGraph_t *g)
{
    *g = (cudaGraph_t)of(s)->g;
    of(s)->capturing = 0;
    of(s)->g = NULL;
    return cudaSuccess;
}
cudaError_t cudaGraphInstantiate(cudaGraphExec_t *e, cudaGraph_t g, unsigned long long flags)
{
    (void)flags;
    *e = malloc(sizeof(struct graph));
    memcpy(*e, g, sizeof(struct graph));
    return cudaSuccess;
}
cudaError_t cudaGraphDestroy(cudaGraph_t g) { return free(g), cudaSuccess; }
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t e) { return free(e), cudaSuccess; }
cudaError_t cudaGraphLaunch(cudaGraphExec_t e, cudaStream_t s)
{
    if (of(s)->capturing)
        return result(cudaErrorStreamCaptureUnsupported);
    put("graph\n");
    put(((struct graph *)e)->text);
    put("end\n");
    return cudaSuccess;
}
cudaError_t cudaEventCreate(cudaEvent_t *e) { return (*e = calloc(1, sizeof(struct event))) ? cudaSuccess : cudaErrorMemoryAllocation; }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t *e, unsigned f) { return (void)f, cudaEventCreate(e); }
cudaError_t cudaEventDestroy(cudaEvent_t e) { return free(e), cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t e, cudaStream_t s) { return ((struct event *)e)->captured = of(s)->capturing, cudaSuccess; }
cudaError_t cudaStreamWaitEvent(cudaStream_t s, cudaEvent_t e, unsigned f)
{
    (void)f;
    if (((struct event *)e)->captured && !of(s)->capturing)
        of(s)->capturing = 2;
    put("wait\n");
    return cudaSuccess;
}
cudaError_t cudaEventElapsedTime(float *ms, cudaEvent_t a, cudaEvent_t b) { return (void)a, (void)b, *ms = 0.f, cudaSuccess; }
