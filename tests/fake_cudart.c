/* The part of the CUDA runtime that an attribution without a context calls, for
 * two devices that exist only here: launches do nothing but check that a kernel
 * with more than 48 KB of dynamic shared memory was opted in on the current
 * device. */
#include <stddef.h>

enum { kFuncs = 64, kInvalidValue = 1 };
static int cur;
static const void *funcs[2][kFuncs];
static int limit[2][kFuncs], used[2], last_error, launches[2];
static _Alignas(256) char scratch[2][256];

void fake_set_device(int dev) { cur = dev; }
int fake_launches(int dev) { return launches[dev]; }

int cudaGetDevice(int *dev) { return *dev = cur, 0; }
int cudaDeviceGetAttribute(int *v, int attr, int dev) { return (void)attr, (void)dev, *v = 152, 0; }
int cudaGetSymbolAddress(void **p, const void *sym) { return (void)sym, *p = scratch[cur], 0; }
int cudaMemsetAsync(void *p, int v, size_t n, void *s) { return (void)p, (void)v, (void)n, (void)s, 0; }
int cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int *n, const void *f, int block, size_t smem, unsigned fl) {
  return (void)f, (void)block, (void)smem, (void)fl, *n = 1, 0;
}
int cudaFuncSetAttribute(const void *f, int attr, int value) {
  (void)attr;
  funcs[cur][used[cur]] = f;
  limit[cur][used[cur]++] = value;
  return 0;
}
int cudaGetLastError(void) {
  const int e = last_error;
  last_error = 0;
  return e;
}

static int launch(const void *f, size_t smem) {
  int opt = 48 << 10;
  for (int i = 0; i < used[cur]; ++i)
    if (funcs[cur][i] == f) opt = limit[cur][i];
  ++launches[cur];
  return smem > (size_t)opt ? (last_error = kInvalidValue) : 0;
}

typedef struct {
  unsigned x, y, z;
} dim3;
struct config {
  dim3 grid, block;
  size_t smem;
};
int __cudaGetKernel(const void **kernel, const void *f) { return *kernel = f, 0; }
int __cudaLaunchKernel(const void *kernel, dim3 grid, dim3 block, void **args, size_t smem, void *stream) {
  return (void)grid, (void)block, (void)args, (void)stream, launch(kernel, smem);
}
int cudaLaunchKernelExC(const struct config *c, const void *f, void **args) { return (void)args, launch(f, c->smem); }
