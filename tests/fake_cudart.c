/* A stand-in for the CUDA runtime calls of nb_create and the builds, preloaded
 * before libcudart: two devices, memory that is never read, and kernels that do
 * not run.  It keeps cudaFuncSetAttribute's shared memory limit per (kernel,
 * device), as the runtime does, and counts launches that ask for more dynamic
 * shared memory than the limit of the device they go to (48 KB unless raised),
 * which the runtime would refuse. */
#include <stddef.h>
#include <stdint.h>
#include <stdlib.h>
#include <string.h>

typedef struct { unsigned grid[3], block[3]; size_t smem; void *stream; void *attrs; unsigned n; } cfg_t;

static int dev;
static struct { const void *f; int d, bytes; } lim[256];
static int nlim;
int fake_launches, fake_refused;

int cudaSetDevice(int d) { dev = d; return d < 2 ? 0 : 101; }
int cudaGetDevice(int *d) { *d = dev; return 0; }
int cudaDeviceGetAttribute(int *v, int a, int d) { (void)a; (void)d; *v = 152; return 0; }
int cudaMalloc(void **p, size_t n)
{
    static uintptr_t at = 1 << 30;
    *p = (void *)at;
    at += (n + 4095) / 4096 * 4096;
    return 0;
}
int cudaFree(void *p) { (void)p; return 0; }
int cudaMallocHost(void **p, size_t n) { *p = calloc(1, n); return 0; }
int cudaFreeHost(void *p) { free(p); return 0; }
int cudaMemsetAsync(void *p, int v, size_t n, void *s) { (void)p; (void)v; (void)n; (void)s; return 0; }
int cudaMemcpyAsync(void *d, const void *s, size_t n, int kind, void *st)
{
    (void)s; (void)st;
    if (kind == 2) memset(d, 0, n);
    return 0;
}
int cudaStreamSynchronize(void *s) { (void)s; return 0; }
int cudaGetLastError(void) { return fake_refused ? 1 : 0; }
int cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int *b, const void *f, int t, size_t m, unsigned g)
{
    (void)f; (void)t; (void)m; (void)g;
    *b = 2;
    return 0;
}
int cudaFuncSetAttribute(const void *f, int a, int v)
{
    if (a == 8 && nlim < 256) {   /* cudaFuncAttributeMaxDynamicSharedMemorySize */
        lim[nlim].f = f; lim[nlim].d = dev; lim[nlim++].bytes = v;
    }
    return 0;
}
static int launch(const void *f, size_t smem)
{
    size_t room = 48 << 10;
    for (int i = 0; i < nlim; i++)
        if (lim[i].f == f && lim[i].d == dev && (size_t)lim[i].bytes > room) room = lim[i].bytes;
    fake_launches++;
    if (smem <= room) return 0;
    fake_refused++;
    return 1;
}
int cudaLaunchKernelExC(const cfg_t *c, const void *f, void **a) { (void)a; return launch(f, c->smem); }
