// The tiles of the packed residual pass without the CTAs of bins 0 and nx/2
// (col_kernel_pk at length 64, 8 positions per tile), for a test of what a tile
// reads. tw holds room for the two twiddle tables, one after the other.
#include "device_tables.cuh"
#include "passes.cuh"

using namespace pwf;

__global__ void probe_tables(float2* fwd, float2* inv) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  fill_twiddles(fwd, 64, FWD, i);
  fill_twiddles(inv, 64, INV, i);
}

extern "C" int probe_packed_tiles(void* field, const void* yhat, const void* ix, const void* iy, void* tw, double* acc,
                                  int nproj, int nx) {
  constexpr int N = 64, C = 8;
  float2* fwd = static_cast<float2*>(tw);
  float2* inv = fwd + N;
  static_assert(twiddle_len(N, FWD) <= N && twiddle_len(N, INV) <= N, "a table fits N entries");
  if (nproj < 1 || nx < 2 * C || nx % (2 * C) != 0) return 1;
  PassArgs a{};
  a.B = nproj;
  a.ny = N;
  a.nx = nx;
  a.in = static_cast<const float2*>(field);
  a.out = static_cast<float2*>(field);
  a.tw_fwd = fwd;
  a.tw_inv = inv;
  a.yhat = static_cast<const float2*>(yhat);
  a.ix = static_cast<const float*>(ix);
  a.iy = static_cast<const float*>(iy);
  a.acc = acc;
  a.scale = 1.0f / (float)(N * nx);
  probe_tables<<<1, 64>>>(fwd, inv);
  const int tiles = nproj * (nx / 2 / C);
  col_kernel_pk<N, C, true><<<tiles, col2_threads(N, C), col_smem_bytes(N, C)>>>(a, nproj, tiles);
  return (int)(cudaGetLastError() == cudaSuccess ? cudaDeviceSynchronize() : cudaErrorUnknown);
}
