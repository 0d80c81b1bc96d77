/* A runtime with two devices and no GPU, in place of libcudart for librbx: allocations and copies do
 * nothing, and a launch that asks for more than 48 KB of dynamic shared memory fails, as on a GPU,
 * unless the kernel was allowed that much on the current device. main() runs a job of every precision
 * on either device. */
#include <stdio.h>
#include <string.h>

#include "rbx.h"

typedef struct { unsigned x, y, z; } dim3_;

static int dev, last;
static struct { const void *f; int dev, bytes; } allowed[256];
static int n_allowed;
static struct { dim3_ g, b; size_t smem; void *s; } conf;

static int launch(const void *f, size_t smem)
{
    if (smem <= 48 * 1024) return 0;
    for (int i = 0; i < n_allowed; i++)
        if (allowed[i].f == f && allowed[i].dev == dev && (size_t)allowed[i].bytes >= smem) return 0;
    return last = 1;
}

int cudaFuncSetAttribute(const void *f, int attr, int value)
{
    if (attr == 8) {   /* cudaFuncAttributeMaxDynamicSharedMemorySize */
        if (n_allowed == 256) return 1;
        allowed[n_allowed].f = f;
        allowed[n_allowed].dev = dev;
        allowed[n_allowed++].bytes = value;
    }
    return 0;
}
unsigned __cudaPushCallConfiguration(dim3_ g, dim3_ b, size_t smem, void *s)
{
    conf.g = g; conf.b = b; conf.smem = smem; conf.s = s;
    return 0;
}
int __cudaPopCallConfiguration(dim3_ *g, dim3_ *b, size_t *smem, void *s)
{
    *g = conf.g; *b = conf.b; *smem = conf.smem; *(void **)s = conf.s;
    return 0;
}
int __cudaGetKernel(const void **k, const void *f) { *k = f; return 0; }
int __cudaLaunchKernel(const void *k, dim3_ g, dim3_ b, void **a, size_t smem, void *s) { return launch(k, smem); }
int cudaLaunchKernelExC(const void *config, const void *f, void **a) { return launch(f, *(const size_t *)((const char *)config + 24)); }
int cudaGetLastError(void) { int e = last; last = 0; return e; }
const char *cudaGetErrorString(int e) { return e ? "invalid argument" : "no error"; }
int cudaGetDevice(int *d) { *d = dev; return 0; }
int cudaSetDevice(int d) { dev = d; return 0; }
int cudaDeviceGetAttribute(int *v, int a, int d) { *v = 152; return 0; }
int cudaDeviceGetDefaultMemPool(void **p, int d) { *p = (void *)16; return 0; }
int cudaMemPoolSetAttribute(void *p, int a, void *v) { return 0; }
int cudaMallocAsync(void **p, size_t n, void *s) { *p = (void *)4096; return 0; }
int cudaFreeAsync(void *p, void *s) { return 0; }
int cudaMemsetAsync(void *p, int v, size_t n, void *s) { return 0; }
int cudaMemcpyAsync(void *to, const void *from, size_t n, int kind, void *s)
{
    if (kind == 2) {   /* to the host: zeros, but a mask of 1000 nodes */
        memset(to, 0, n);
        if (n == sizeof(int)) *(int *)to = 1000;
    }
    return 0;
}
int cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int *n, const void *f, int t, size_t m, unsigned fl) { *n = 2; return 0; }
int cudaStreamSynchronize(void *s) { return 0; }
int cudaStreamIsCapturing(void *s, int *status) { *status = 0; return 0; }
int cudaEventCreate(void **e) { *e = (void *)16; return 0; }
int cudaEventDestroy(void *e) { return 0; }
int cudaEventRecord(void *e, void *s) { return 0; }
int cudaEventElapsedTime(float *ms, void *a, void *b) { *ms = 1.f; return 0; }
int cudaGetSymbolAddress(void **p, const void *s) { *p = (void *)4096; return 0; }
static int encode(void) { return 0; }
int cudaGetDriverEntryPointByVersion(const char *n, void **f, unsigned v, unsigned long long fl, int *q)
{
    *f = (void *)encode;
    if (q) *q = 0;
    return 0;
}

int main(void)
{
    int bad = 0;
    char out[64];
    rbx_autotune(0);
    for (int d = 0; d < 2; d++)
        for (int precision = 0; precision < 3; precision++) {
            rbx_geometry g;
            rbx_job *j = NULL;
            memset(&g, 0, sizeof g);
            g.nx = g.ny = 64; g.dx = 1e-3; g.x0 = g.y0 = -31.5e-3; g.n_xducers = 48; g.ring_radius = 28e-3;
            g.mask_radius = 25e-3; g.c0 = 1500.0; g.ds = 5e-4; g.tau = 0.1; g.precision = precision;
            cudaSetDevice(d);
            int st[7] = {rbx_create(&j, NULL), rbx_set_geometry(j, &g, NULL), rbx_update_frequency(j, 3e5, 1e5, out, NULL),
                         rbx_forward(j, 3e5, (const float *)out, out), rbx_adjoint(j, 3e5, out, out, 0),
                         rbx_adjoint(j, 3e5, out, out, 1),
                         rbx_forward_noalloc((float *)out, (float *)out, (unsigned char *)out, (float *)out, 48, 1000, 3e5,
                                             1500.0, out, NULL, NULL, 0)};
            for (int k = 0; k < 7; k++)
                if (st[k]) printf("device %d precision %d call %d: status %d %s\n", d, precision, k, st[k], rbx_last_error(j)), bad = 1;
            rbx_destroy(j);
        }
    return bad;
}
