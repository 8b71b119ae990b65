// sincos_acc, and the library routine beside it, over an array of phases.
#include "passes.cuh"

__global__ void probe(const float* y, float* out, int n, int library) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  float s, c;
  if (library) sincosf(y[i], &s, &c);
  else pwf::sincos_acc(y[i], s, c);
  out[i] = s;
  out[n + i] = c;
}

extern "C" int probe_sincos(const float* y, float* out, int n, int library) {
  if (n < 1) return 1;
  probe<<<(n + 255) / 256, 256>>>(y, out, n, library);
  return (int)(cudaGetLastError() == cudaSuccess ? cudaDeviceSynchronize() : cudaErrorUnknown);
}
