/* A CUDA runtime without a device, preloaded in front of the real one by test_fake_runtime.py: "device" memory is
 * host memory, kernels do nothing, and the calls that the tests look at are written to a log.  Two devices. */
#include <stdio.h>
#include <stdlib.h>
#include <string.h>

static char g_log[1 << 16];
static size_t g_len;
static int g_device, g_capturing, g_fail_sync, g_fail_launch, g_fail_malloc;
static void note(const char *what, long a)
{
    if (g_len + 64 < sizeof(g_log)) g_len += (size_t)sprintf(g_log + g_len, "%s:%d:%ld\n", what, g_device, a);
}
const char *fake_log(void) { return g_log; }
void fake_clear(void) { g_len = 0; g_log[0] = 0; }
void fake_set(const char *what, int v)
{
    if (!strcmp(what, "capturing")) g_capturing = v;
    if (!strcmp(what, "fail_sync")) g_fail_sync = v;
    if (!strcmp(what, "fail_launch")) g_fail_launch = v;
    if (!strcmp(what, "fail_malloc")) g_fail_malloc = v;
}
typedef struct { unsigned grid[3], block[3]; size_t smem; void *stream; void *attrs; unsigned n_attrs; } config_t;

int cudaGetDevice(int *d) { *d = g_device; return 0; }
int cudaSetDevice(int d) { g_device = d; note("set_device", d); return 0; }
int cudaDeviceGetAttribute(int *v, int attr, int d) { (void)d; *v = attr == 97 ? 232448 : 148; return 0; } /* 97: opt-in shared memory per block */
int cudaDeviceSynchronize(void) { note("sync", 0); return g_fail_sync ? 999 : 0; }
int cudaGetLastError(void) { return 0; }
int cudaMalloc(void **p, size_t n) { if (g_fail_malloc) return 2; *p = calloc(1, n); note("malloc", (long)n); return 0; }
int cudaFree(void *p) { if (p) { note("free", 0); free(p); } return 0; }
int cudaMemcpy(void *d, const void *s, size_t n, int k) { (void)k; memcpy(d, s, n); return 0; }
int cudaMemcpyAsync(void *d, const void *s, size_t n, int k, void *st) { (void)k; (void)st; memcpy(d, s, n); return 0; }
int cudaMemset(void *d, int v, size_t n) { memset(d, v, n); return 0; }
int cudaMemsetAsync(void *d, int v, size_t n, void *st) { (void)st; memset(d, v, n); note("memset", (long)n); return 0; }
int cudaStreamSynchronize(void *st) { (void)st; return 0; }
int cudaStreamIsCapturing(void *st, int *v) { (void)st; *v = g_capturing; return 0; }
int cudaFuncSetAttribute(const void *f, int a, int v) { (void)f; (void)a; note("attribute", v); return 0; }
struct attributes { size_t a, b, c; int max_threads, regs; char rest[256]; };
int cudaFuncGetAttributes(struct attributes *at, const void *f) { (void)f; at->regs = 96; return 0; }
int cudaLaunchKernel(const void *f, unsigned long long g0, unsigned g1, unsigned long long b0, unsigned b1, void **args, size_t smem, void *st)
{
    (void)f; (void)g0; (void)g1; (void)b0; (void)b1; (void)args; (void)smem; (void)st;
    note("launch", 0);
    return g_fail_launch ? 719 : 0;
}
int cudaLaunchKernelExC(const config_t *c, const void *f, void **args)
{
    (void)f; (void)args;
    note("forward", (long)c->n_attrs); /* 1: may begin beside the launch before it */
    return g_fail_launch ? 719 : 0;
}
