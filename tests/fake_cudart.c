/* A stand-in for the CUDA runtime calls of the library, preloaded by
 * test_failed_calls.py: device memory is host memory, kernels do nothing, and a named
 * call can be made to fail, as the runtime fails it: it returns the error and keeps it
 * for cudaGetLastError. */
#include <stddef.h>
#include <stdlib.h>
#include <string.h>

typedef int err_t;
typedef struct { unsigned x, y, z; } dim3_t;

static err_t last_error;
static char fail_name[64];
static int fail_after = -1;
static err_t fail_code;
static size_t copy_bytes;
static unsigned char symbols[1 << 16];
static struct { void *p; size_t n; } blocks[64];
static unsigned nblocks, launches, last_grid, last_block;

/* The call `name` fails with `code` once, after `after` calls of it that succeed. */
void fake_fail(const char *name, int after, int code)
{
    strncpy(fail_name, name, sizeof fail_name - 1);
    fail_after = after;
    fail_code = code;
}
size_t fake_copy_bytes(void) { return copy_bytes; }
void *fake_symbols(void) { return symbols; }
/* The latest of the last 64 allocations that has n bytes. */
void *fake_block(size_t n)
{
    for (unsigned i = 1; i <= 64 && i <= nblocks; ++i)
        if (blocks[(nblocks - i) % 64].n == n) return blocks[(nblocks - i) % 64].p;
    return NULL;
}
unsigned fake_launches(void) { return launches; }
/* Grid and block size of the last launch by cudaLaunchKernelExC. */
unsigned fake_grid(void) { return last_grid; }
unsigned fake_block_size(void) { return last_block; }
int fake_pending(void) { return fail_after >= 0; }

static err_t outcome(const char *name)
{
    if (fail_after < 0 || strcmp(name, fail_name) != 0) return 0;
    if (fail_after-- > 0) return 0;
    last_error = fail_code;
    return fail_code;
}
#define OUTCOME(name) do { const err_t e_ = outcome(name); if (e_) return e_; } while (0)

/* every launch is one call named "launch" */
static err_t launch(void)
{
    OUTCOME("launch");
    ++launches;
    return 0;
}

static err_t allocate(void **p, size_t n)
{
    *p = aligned_alloc(256, (n + 255) / 256 * 256);
    if (!*p) return 2;
    memset(*p, 0, n);
    blocks[nblocks % 64].p = *p;
    blocks[nblocks++ % 64].n = n;
    return 0;
}

err_t cudaGetLastError(void)
{
    const err_t e = last_error;
    last_error = 0;
    return e;
}
err_t cudaGetDevice(int *d) { *d = 0; return 0; }
err_t cudaDeviceGetAttribute(int *v, int attr, int dev) { (void)dev; *v = attr == 16 ? 152 : 1; return 0; }
err_t cudaMalloc(void **p, size_t n) { OUTCOME("cudaMalloc"); return allocate(p, n); }
err_t cudaMallocHost(void **p, size_t n) { OUTCOME("cudaMallocHost"); return allocate(p, n); }
err_t cudaMallocAsync(void **p, size_t n, void *st) { (void)st; OUTCOME("cudaMallocAsync"); return allocate(p, n); }
err_t cudaFree(void *p) { free(p); return 0; }
err_t cudaFreeHost(void *p) { free(p); return 0; }
err_t cudaFreeAsync(void *p, void *st) { (void)st; free(p); return 0; }
err_t cudaMemset(void *p, int v, size_t n) { OUTCOME("cudaMemset"); memset(p, v, n); return 0; }
err_t cudaMemsetAsync(void *p, int v, size_t n, void *st)
{
    (void)st;
    OUTCOME("cudaMemsetAsync");
    memset(p, v, n);
    return 0;
}
err_t cudaMemcpy(void *d, const void *s, size_t n, int kind)
{
    (void)kind;
    OUTCOME("cudaMemcpy");
    copy_bytes = n;
    memcpy(d, s, n);
    return 0;
}
err_t cudaMemcpyAsync(void *d, const void *s, size_t n, int kind, void *st)
{
    (void)kind;
    (void)st;
    OUTCOME("cudaMemcpyAsync");
    memcpy(d, s, n);
    return 0;
}
err_t cudaDeviceSynchronize(void) { return 0; }
err_t cudaStreamSynchronize(void *st) { (void)st; OUTCOME("cudaStreamSynchronize"); return 0; }
err_t cudaStreamCreateWithFlags(void **st, unsigned f) { (void)f; *st = malloc(1); return 0; }
err_t cudaStreamDestroy(void *st) { free(st); return 0; }
err_t cudaFuncSetAttribute(const void *f, int attr, int v)
{
    (void)f;
    (void)attr;
    (void)v;
    OUTCOME("cudaFuncSetAttribute");
    return 0;
}
err_t cudaGetSymbolAddress(void **p, const void *sym) { (void)sym; *p = symbols; return 0; }
err_t cudaEventCreate(void **e) { *e = malloc(1); return 0; }
err_t cudaEventDestroy(void *e) { free(e); return 0; }
err_t cudaEventRecord(void *e, void *st) { (void)e; (void)st; return 0; }
err_t cudaEventSynchronize(void *e) { (void)e; return 0; }
err_t cudaEventElapsedTime(float *ms, void *a, void *b) { (void)a; (void)b; *ms = 1.f; return 0; }
err_t __cudaGetKernel(void **k, const void *f) { *k = (void *)f; return 0; }
err_t __cudaLaunchKernel(void *k, dim3_t g, dim3_t b, void **args, size_t smem, void *st)
{
    (void)k; (void)g; (void)b; (void)args; (void)smem; (void)st;
    return launch();
}
err_t cudaLaunchKernelExC(const void *cfg, const void *f, void **args)
{
    (void)f; (void)args;
    last_grid = ((const dim3_t *)cfg)[0].x;   /* the configuration begins with the two sizes */
    last_block = ((const dim3_t *)cfg)[1].x;
    return launch();
}
err_t cudaLaunchCooperativeKernel(const void *f, dim3_t g, dim3_t b, void **args, size_t smem, void *st)
{
    (void)f; (void)g; (void)b; (void)args; (void)smem; (void)st;
    return launch();
}
