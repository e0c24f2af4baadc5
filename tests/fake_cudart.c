/* A stand-in for the CUDA runtime, preloaded before libbasker_gb300.so, for tests of
 * the library's host code without a GPU: device memory is host memory, kernels do not
 * run (their names are kept), and a test makes an allocation or a status read fail.
 * The names and signatures are those of the CUDA runtime API. */
#define _GNU_SOURCE
#include <stdint.h>
#include <stdio.h>
#include <stdlib.h>
#include <string.h>
#include <sys/mman.h>

typedef struct { unsigned x, y, z; } dim3_t;
enum { OK = 0, OUT_OF_MEMORY = 2 };

/* ---- the test's controls */
static int64_t cap = INT64_MAX, held;       /* bytes of device memory: all there are, and allocated */
static int status_reads;                    /* status words read so far */
static struct { int at, word, value; } plant[16];   /* those to change: a 32-bit word, and what to put there */
static int nplants;
static size_t ints_bytes;                   /* size of the copy to replace, and the value its ints get */
static int ints_value, ints_times;
static char launched[1 << 16];              /* names of the kernels launched since the last question */

void fake_cap(int64_t bytes) { cap = bytes; }
int64_t fake_held(void) { return held; }

/* The next-but-`skip` status read has `value` in its 32-bit word `word`. */
void fake_status(int skip, int word, int value)
{
    plant[nplants].at = status_reads + skip;
    plant[nplants].word = word;
    plant[nplants].value = value;
    nplants = (nplants + 1) % 16;
}

/* The next `times` synchronous copies of `bytes` bytes to the host read as ints of `value`. */
void fake_ints(int64_t bytes, int value, int times)
{
    ints_bytes = (size_t)bytes;
    ints_value = value;
    ints_times = times;
}

const char *fake_launched(void)
{
    static char out[sizeof launched];
    memcpy(out, launched, sizeof out);
    launched[0] = 0;
    return out;
}

/* ---- memory */
struct block { void *p; int64_t bytes; };
enum { LARGE = 64 << 20 };                  /* from here on address space only, until it is written */
static struct block *blocks;
static size_t nblocks, room;

int cudaMalloc(void **p, size_t bytes)
{
    *p = NULL;
    if (held + (int64_t)bytes > cap) return OUT_OF_MEMORY;
    if (nblocks == room) blocks = realloc(blocks, (room = room ? 2 * room : 256) * sizeof *blocks);
    if (bytes >= LARGE) {
        *p = mmap(NULL, bytes, PROT_READ | PROT_WRITE, MAP_PRIVATE | MAP_ANONYMOUS | MAP_NORESERVE, -1, 0);
        if (*p == MAP_FAILED) *p = NULL;
    } else {
        *p = calloc(bytes ? bytes : 1, 1);
    }
    if (!*p) return OUT_OF_MEMORY;
    blocks[nblocks].p = *p;
    blocks[nblocks++].bytes = (int64_t)bytes;
    held += (int64_t)bytes;
    return OK;
}

int cudaFree(void *p)
{
    for (size_t i = 0; p && i < nblocks; i++)
        if (blocks[i].p == p) {
            const size_t bytes = (size_t)blocks[i].bytes;
            held -= blocks[i].bytes;
            blocks[i] = blocks[--nblocks];
            if (bytes >= LARGE) munmap(p, bytes);
            else free(p);
            break;
        }
    return OK;
}

int cudaMallocHost(void **p, size_t bytes) { *p = calloc(bytes ? bytes : 1, 1); return OK; }
int cudaFreeHost(void *p) { free(p); return OK; }

int cudaMemcpy(void *d, const void *s, size_t n, int kind)
{
    if (n) memmove(d, s, n);
    if (kind == 2 && ints_times > 0 && n == ints_bytes) {
        for (size_t i = 0; i < n / 4; i++) ((int32_t *)d)[i] = ints_value;
        ints_times--;
    }
    return OK;
}

int cudaMemcpyAsync(void *d, const void *s, size_t n, int kind, void *stream)
{
    (void)stream;
    if (n) memmove(d, s, n);
    if (kind == 2 && n == 40) {              /* device to host: the status word of a call */
        for (int i = 0; i < nplants; i++)
            if (plant[i].at == status_reads) ((int32_t *)d)[plant[i].word] = plant[i].value;
        status_reads++;
    }
    return OK;
}

int cudaMemset(void *d, int v, size_t n) { if (n) memset(d, v, n); return OK; }
int cudaMemsetAsync(void *d, int v, size_t n, void *stream) { (void)stream; return cudaMemset(d, v, n); }

/* ---- device, streams, events, graphs */
int cudaGetDevice(int *d) { *d = 0; return OK; }
int cudaSetDevice(int d) { (void)d; return OK; }
int cudaDeviceGetAttribute(int *v, int attr, int d) { (void)attr; (void)d; *v = 152; return OK; }
int cudaDeviceSynchronize(void) { return OK; }
int cudaGetLastError(void) { return OK; }
int cudaStreamCreateWithFlags(void **s, unsigned flags) { (void)flags; *s = &held; return OK; }
int cudaStreamDestroy(void *s) { (void)s; return OK; }
int cudaStreamSynchronize(void *s) { (void)s; return OK; }
int cudaStreamBeginCapture(void *s, int mode) { (void)s; (void)mode; return OK; }
int cudaStreamEndCapture(void *s, void **g) { (void)s; *g = &held; return OK; }
int cudaGraphInstantiate(void **e, void *g, unsigned long long flags) { (void)g; (void)flags; *e = &held; return OK; }
int cudaGraphLaunch(void *e, void *s) { (void)e; (void)s; return OK; }
int cudaGraphDestroy(void *g) { (void)g; return OK; }
int cudaGraphExecDestroy(void *e) { (void)e; return OK; }
int cudaEventCreate(void **e) { *e = &held; return OK; }
int cudaEventDestroy(void *e) { (void)e; return OK; }
int cudaEventRecord(void *e, void *s) { (void)e; (void)s; return OK; }
int cudaEventSynchronize(void *e) { (void)e; return OK; }
int cudaEventElapsedTime(float *ms, void *a, void *b) { (void)a; (void)b; *ms = 1.0f; return OK; }
int cudaGetSymbolAddress(void **p, const void *sym) { (void)sym; *p = &held; return OK; }

/* ---- kernels */
static struct { const void *fun; const char *name; } kernels[512];
static int nkernels;

void **__cudaRegisterFatBinary(void *image) { (void)image; return (void **)&held; }
void __cudaRegisterFatBinaryEnd(void **h) { (void)h; }
void __cudaUnregisterFatBinary(void **h) { (void)h; }
void __cudaRegisterVar(void **h, char *var, char *addr, const char *name, int ext, size_t size, int constant, int global)
{
    (void)h; (void)var; (void)addr; (void)name; (void)ext; (void)size; (void)constant; (void)global;
}
void __cudaRegisterFunction(void **h, const char *fun, char *dfun, const char *name, int limit, void *tid, void *bid,
                            void *bdim, void *gdim, int *wsize)
{
    (void)h; (void)dfun; (void)limit; (void)tid; (void)bid; (void)bdim; (void)gdim; (void)wsize;
    if (nkernels < 512) {
        kernels[nkernels].fun = fun;
        kernels[nkernels++].name = name;
    }
}

static int launch(const void *fun)
{
    const char *name = "?";
    for (int i = 0; i < nkernels; i++)
        if (kernels[i].fun == fun) name = kernels[i].name;
    const size_t at = strlen(launched);
    snprintf(launched + at, sizeof launched - at, "%s\n", name);
    return OK;
}

int __cudaGetKernel(const void **handle, const void *fun) { *handle = fun; return OK; }
static dim3_t cfg_grid, cfg_block;
static size_t cfg_smem;
static void *cfg_stream;
unsigned __cudaPushCallConfiguration(dim3_t grid, dim3_t block, size_t smem, void *stream)
{
    cfg_grid = grid; cfg_block = block; cfg_smem = smem; cfg_stream = stream;
    return 0;
}
int __cudaPopCallConfiguration(dim3_t *grid, dim3_t *block, size_t *smem, void *stream)
{
    *grid = cfg_grid; *block = cfg_block; *smem = cfg_smem; *(void **)stream = cfg_stream;
    return OK;
}
int __cudaLaunchKernel(const void *kernel, dim3_t grid, dim3_t block, void **args, size_t smem, void *stream)
{
    (void)grid; (void)block; (void)args; (void)smem; (void)stream;
    return launch(kernel);
}
int cudaLaunchKernelExC(const void *config, const void *fun, void **args) { (void)config; (void)args; return launch(fun); }
int cudaFuncSetAttribute(const void *fun, int attr, int v) { (void)fun; (void)attr; (void)v; return OK; }
int cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int *n, const void *fun, int threads, size_t smem, unsigned flags)
{
    (void)fun; (void)threads; (void)smem; (void)flags;
    *n = 4;
    return OK;
}
