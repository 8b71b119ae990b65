/* Stand-in for the few CUDA runtime calls pwf_fbp makes, preloaded before
 * libcudart: two devices, each with its own shared-memory limits per kernel, and
 * launches that are checked against them and go nowhere. */
#include <stddef.h>

typedef struct { unsigned x, y, z; } dim3;
enum { OK = 0, INVALID_VALUE = 1, MAX_DYNAMIC_SHARED = 8, DEFAULT_LIMIT = 48 * 1024, KERNELS = 256 };

static int device = 0, launches = 0, last_error = OK, used = 0;
static struct { int device; const void *kernel; int bytes; } limits[KERNELS];

void fake_set_device(int d) { device = d; }
int fake_launches(void) { return launches; }

int cudaGetLastError(void) {
  int e = last_error;
  last_error = OK;
  return e;
}

int cudaFuncSetAttribute(const void *kernel, int attribute, int value) {
  if (attribute != MAX_DYNAMIC_SHARED || value < 0 || value > 227 * 1024 || used == KERNELS) return last_error = INVALID_VALUE;
  limits[used].device = device;
  limits[used].kernel = kernel;
  limits[used].bytes = value;
  used++;
  return OK;
}

int __cudaGetKernel(const void **handle, const void *kernel) {
  *handle = kernel;
  return OK;
}

int __cudaLaunchKernel(const void *kernel, dim3 grid, dim3 block, void **args, size_t shared, void *stream) {
  size_t limit = DEFAULT_LIMIT;
  (void)grid, (void)block, (void)args, (void)stream;
  for (int i = 0; i < used; i++)
    if (limits[i].device == device && limits[i].kernel == kernel) limit = (size_t)limits[i].bytes;
  if (shared > limit) return last_error = INVALID_VALUE;
  launches++;
  return OK;
}
