/* The parts of the CUDA runtime that the host side of libgdn_tree.so calls, for tests without a GPU: nothing runs, every
 * kernel launch is written to a log, and any other call can be made to fail.  A kernel's shared memory limit counts in the
 * context it was raised in.  Linked with the library's objects in place of
 * the runtime (test_host_launches.py). */
#define _GNU_SOURCE
#include <pthread.h>
#include <stddef.h>
#include <stdio.h>
#include <string.h>
#include <unistd.h>

enum { SUCCESS = 0, INVALID_VALUE = 1, UNKNOWN = 999 };

static struct { const void *host; const char *name; } kernels[256];
static int n_kernels;

static char log_text[1 << 14];   /* names of the launched kernels and of a few other calls, one per line */
static int calls;                /* calls other than launches so far */
static int fail_at = -1;         /* number of the call that fails */

static unsigned long long context;                                                  /* id of the current one */
static struct { const void *host; unsigned long long context; int bytes; } limits[256];   /* raised so far */
static int n_limits;

void fake_context(unsigned long long id) { context = id; }
void fake_reset(int fail_call) { log_text[0] = 0; calls = 0; fail_at = fail_call; }
const char *fake_log(void) { return log_text; }
int fake_calls(void) { return calls; }

static int call_result(void) { return calls++ == fail_at ? UNKNOWN : SUCCESS; }

static void note(const char *line)
{
    static pthread_mutex_t lock = PTHREAD_MUTEX_INITIALIZER;
    pthread_mutex_lock(&lock);
    const size_t n = strlen(log_text);
    snprintf(log_text + n, sizeof log_text - n, "%s\n", line);
    pthread_mutex_unlock(&lock);
}

static int launched(const void *host)
{
    const char *name = "?";
    for (int i = 0; i < n_kernels; ++i)
        if (kernels[i].host == host) name = kernels[i].name;
    note(name);
    return SUCCESS;
}

/* registration of kernels and variables, from the library's start-up code */
void **__cudaRegisterFatBinary(void *binary) { (void)binary; static void *handle; return &handle; }
void __cudaRegisterFatBinaryEnd(void **handle) { (void)handle; }
void __cudaUnregisterFatBinary(void **handle) { (void)handle; }
void __cudaRegisterVar(void **h, char *host, char *dev, const char *name, int ext, size_t size, int constant, int global)
{
    (void)h; (void)host; (void)dev; (void)name; (void)ext; (void)size; (void)constant; (void)global;
}
void __cudaRegisterFunction(void **h, const char *host, char *dev, const char *name, int limit, void *tid, void *bid, void *bdim,
                            void *gdim, int *size)
{
    (void)h; (void)dev; (void)limit; (void)tid; (void)bid; (void)bdim; (void)gdim; (void)size;
    if (n_kernels < 256) {
        kernels[n_kernels].host = host;
        kernels[n_kernels++].name = name;
    }
}

/* launches */
typedef struct { unsigned x, y, z; } dim3_t;
typedef struct { dim3_t grid, block; size_t smem; void *stream; void *attrs; unsigned n_attrs; } launch_config;
unsigned __cudaPushCallConfiguration(dim3_t grid, dim3_t block, size_t smem, void *stream)
{
    (void)grid; (void)block; (void)smem; (void)stream;
    return 0;
}
int __cudaPopCallConfiguration(dim3_t *grid, dim3_t *block, size_t *smem, void *stream)
{
    memset(grid, 0, sizeof *grid);
    memset(block, 0, sizeof *block);
    *smem = 0;
    memset(stream, 0, sizeof(void *));
    return SUCCESS;
}
int cudaLaunchKernel(const void *f, dim3_t grid, dim3_t block, void **args, size_t smem, void *stream)
{
    (void)grid; (void)block; (void)args; (void)smem; (void)stream;
    return launched(f);
}
int cudaLaunchKernelExC(const launch_config *cfg, const void *f, void **args)
{
    size_t limit = 48 << 10;
    (void)args;
    for (int i = 0; i < n_limits; ++i)
        if (limits[i].host == f && limits[i].context == context) limit = (size_t)limits[i].bytes;
    return cfg->smem > limit ? INVALID_VALUE : launched(f);
}
int cudaGetLastError(void) { return SUCCESS; }

/* everything else */
int cudaGetDevice(int *dev) { *dev = 0; return call_result(); }
int cudaDeviceGetAttribute(int *value, int attr, int dev) { (void)attr; (void)dev; *value = 148; return call_result(); }
int cudaFuncSetAttribute(const void *f, int attr, int value)
{
    if (attr == 8 && n_limits < 256) {   /* cudaFuncAttributeMaxDynamicSharedMemorySize */
        limits[n_limits].host = f;
        limits[n_limits].context = context;
        limits[n_limits++].bytes = value;
    }
    return call_result();
}
int cudaMemsetAsync(void *p, int v, size_t n, void *s) { (void)p; (void)v; (void)n; (void)s; return call_result(); }
int cudaMemcpyAsync(void *d, const void *p, size_t n, int k, void *s) { (void)d; (void)p; (void)n; (void)k; (void)s; return call_result(); }
int cudaGetSymbolAddress(void **p, const void *symbol) { *p = (void *)symbol; note("cudaGetSymbolAddress"); return call_result(); }
int cudaStreamCreateWithFlags(void **s, unsigned f) { (void)f; *s = NULL; note("cudaStreamCreate"); return call_result(); }
int cudaStreamSynchronize(void *s) { (void)s; return call_result(); }
int cudaStreamWaitEvent(void *s, void *e, unsigned f) { (void)s; (void)e; (void)f; return call_result(); }
int cudaEventCreateWithFlags(void **e, unsigned f) { (void)f; *e = NULL; return call_result(); }
int cudaEventRecord(void *e, void *s)
{
    char line[32];
    (void)e; (void)s;
    snprintf(line, sizeof line, "record:%d", (int)gettid());
    note(line);
    usleep(500);   /* another thread's turn, if it may have one */
    return call_result();
}

static int encode_tiled(void) { return call_result(); }   /* cuTensorMapEncodeTiled: arguments not looked at */
static int ctx_get_id(void *ctx, unsigned long long *id) { (void)ctx; *id = context; return SUCCESS; }   /* cuCtxGetId */
int cudaGetDriverEntryPoint(const char *name, void **f, unsigned long long flags, int *found)
{
    (void)flags;
    *f = strcmp(name, "cuTensorMapEncodeTiled") == 0 ? (void *)encode_tiled : strcmp(name, "cuCtxGetId") == 0 ? (void *)ctx_get_id : NULL;
    *found = *f ? 0 : 1;
    return call_result();
}
