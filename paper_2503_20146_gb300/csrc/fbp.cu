// Filtered back projection of the retrieved fields (the tomographic step after
// PWF; Methods, "Reconstruction procedure": standard FBP with the Ram-Lak
// filter, applied to every detector row independently, then the factor
// lambda / p / (2 pi)). Parallel-beam, angles over [0, pi).
//
// k_fbp_tables writes the filter spectrum, the twiddles and the angles' cosines
// and sines (all in double precision) into the workspace; the filter and the
// back projection follow in one of two forms:
//   * tiles (from 32 detector rows on, see tile_form): the voxels (x, z) of every
//     slice meet the detector at the same place, so the lanes of a warp are
//     slices. fbp_filter_kernel<L, true> writes the filtered rows slice-minor,
//     [angle][block of slices][column][slice], and fbp_backproject_tiles runs
//     warp-uniform interpolation on them.
//   * direct (a few rows, where lanes over slices would idle):
//     fbp_filter_kernel<L, false> writes each row as records (q[o], q[o+1] -
//     q[o]), so that one 16-byte load gives both taps, and
//     fbp_backproject_kernel takes one thread per (x, 8 values of z) of one slice
//     (warps laid out as 8 x 4 voxel patches).
// In both, a filtered row sits in the middle of a row of 2 nx columns (detector
// pixel i at column i + nx/2, zeros around it), so that the back projection of
// any voxel of the nx x nx grid (|s| <= nx / sqrt(2) + 1) reads inside the row
// without bounds checks and gets zero outside the detector. The ramp kernel is
// real and even, so the complex field psi is filtered as it is.
#include <cuda_runtime.h>

#include <cmath>

#include "../../include/pwf.h"
#include "device_tables.cuh"
#include "passes.cuh"

namespace pwf {
namespace {

// The tile form from 32 rows and 64 tiles on. A tile takes about 1 us per angle
// whatever part of its lanes holds slices, so it needs rows to fill them and
// tiles to fill the GPU. Direct / tiles, us per call (angles, ny, nx): (180, 24,
// 1024) 3688 / 4801, (180, 32, 1024) 4939 / 4832, (180, 64, 1024) 9851 / 5172, (32,
// 64, 128) 78 / 68, (32, 24, 128) 58 / 66, (90, 40, 48; 9 tiles) 87 / 117.
bool tile_form(int ny, int nx) { return ny >= 32 && (long long)(nx / 16) * (nx / 16) * ((ny + 63) / 64) >= 64; }
// slices per block of the tile form: two per lane, or four from 65 rows on
int tile_slices(int ny) { return ny > 64 ? 128 : 64; }

// The angles of one call travel in the launch's arguments, in parts.
constexpr int ANGLE_PART = 256;
struct AnglePart {
  double rad[ANGLE_PART];
};

// Filter spectrum, twiddles and angle table. Ram-Lak kernel h(0) = 1/4, h(k) =
// -1/(pi^2 k^2) for odd k, placed circularly on length L = 2 nx; its DFT is
// real and even: H(m) = 1/4 + 2 sum_{odd k < nx} h(k) cos(2 pi k m / L), one warp
// per m; the inverse transform's 1/L is folded in. (On the host the L nx / 2
// cosines alone took 13 ms at nx = 1024.)
__global__ void k_fbp_tables(const __grid_constant__ AnglePart part, int first, int count, int L, float* ramp,
                             float2* twf, float2* twi, double2* cs) {
  const int idx = blockIdx.x * blockDim.x + threadIdx.x;
  if (idx < count) {
    double s, c;
    sincos(part.rad[idx], &s, &c);
    cs[first + idx] = make_double2(c, s);
  }
  if (first > 0) return;  // the other tables are written with the first part
  fill_twiddles(twf, L, FWD, idx);
  fill_twiddles(twi, L, INV, idx);
  const int m = idx >> 5, lane = idx & 31;
  if (m >= L) return;
  // lane's terms k = 2 lane + 1 + 64 i: the cosine advances by a fixed rotation
  double c, sn, rc, rs, h = 0.0;
  sincospi(2.0 * (double)(((2 * lane + 1) * (long)m) % L) / (double)L, &sn, &c);
  sincospi(2.0 * (double)((64 * (long)m) % L) / (double)L, &rs, &rc);
  for (int k = 2 * lane + 1; k < L / 2; k += 64) {
    h -= 2.0 / (M_PI * M_PI * (double)k * k) * c;
    const double t = c * rc - sn * rs;
    sn = fma(sn, rc, c * rs);
    c = t;
  }
  for (int o = 16; o > 0; o >>= 1) h += __shfl_xor_sync(0xffffffffu, h, o);
  if (lane == 0) ramp[m] = (float)((0.25 + h) / L);
}

// Dynamic shared memory above 48 KB has to be allowed for a kernel on each device
// that runs it (a process may call from several): pwf_fbp has no plan that would
// do it once, so every call does, with the same number each time (the most the
// kernel can ask for), whichever thread comes first. It costs nothing
// measurable: 8 x 1 x 512, two short kernels, 49.6 us with it or without.
template <class K>
cudaError_t allow_shared(K* kernel, size_t bytes) {
  return bytes <= 48 * 1024 ? cudaSuccess
                            : cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
}

// One detector row per TPF threads. The nx samples are zero-padded to L = 2 nx (so that the circular convolution of
// length L is the linear one), transformed with the Stockham runner of the PWF
// passes, multiplied by the ramp's spectrum and transformed back.
template <int L, bool TILES>
__global__ void __launch_bounds__(row_threads(L))
    fbp_filter_kernel(const float2* __restrict__ in, float2* __restrict__ out, const float* __restrict__ ramp,
                      const float2* __restrict__ tw_fwd, const float2* __restrict__ tw_inv, int n_angles, int ny, int slices) {
  constexpr int EPT = ept_for(L), TPF = tpf_for(L), ROWS = rows_for(L), nx = L / 2;
  constexpr int RS = first_radix<L, FWD>();
  constexpr int RK = last_radix<L, FWD>();
  extern __shared__ float2 smem[];
  const int rr = threadIdx.x / TPF, t = threadIdx.x - rr * TPF;
  // tile form: the rows of a CTA lie in one angle; direct form: consecutive rows
  // of the whole series. Rows past the end repeat the last row (every thread of
  // a warp must reach the warp barriers of the transform); what they compute is
  // not used.
  const int groups = (ny + ROWS - 1) / ROWS;
  const int angle = TILES ? blockIdx.x / groups : 0;
  const int y0 = TILES ? (blockIdx.x - angle * groups) * ROWS : 0;
  const long long first = TILES ? (long long)angle * ny + y0 : (long long)blockIdx.x * ROWS;
  const long long end = TILES ? (long long)angle * ny + ny : (long long)n_angles * ny;
  const long long row = first + rr < end ? first + rr : end - 1;
  const float2* src = in + (size_t)row * nx;
  const RowLayout<L, ROWS * TPF> sm{smem + rr * row_smem_len(L), 1 + rr};
  float2 v[EPT];
#pragma unroll
  for (int j = 0; j < EPT; j++) {
    const int i = slot_index<L, RS>(t, j);
    v[j] = i < nx ? src[i] : make_float2(0.f, 0.f);
  }
  fft_run<L, FWD>(v, sm, t, tw_fwd);
#pragma unroll
  for (int j = 0; j < EPT; j++) v[j] = cscale(v[j], __ldg(&ramp[slot_index<L, RK>(t, j)]));
  fft_run<L, INV>(v, sm, t, tw_inv);
  // the padded row (samples at columns nx/2 .. 3nx/2 - 1, zeros around) into
  // shared memory: the transform's buffer is free again
  float2* rowbuf = smem + rr * row_smem_len(L);
  sm.sync();
#pragma unroll
  for (int j = 0; j < EPT; j++) {
    const int i = slot_index<L, RS>(t, j);
    const int o = i + nx / 2;
    rowbuf[o < L ? o : o - L] = i < nx ? v[j] : make_float2(0.f, 0.f);
  }
  if constexpr (TILES) {
    // columns nx/4 .. 7nx/4 - 1 (all that a voxel of the grid can meet), two
    // rows at a time so that a store writes 16 bytes
    __syncthreads();
    constexpr int P = ROWS / 2;
    static_assert(ROWS % 2 == 0 && 64 % ROWS == 0, "the rows of a CTA lie in one block of slices");
    float4* dst = reinterpret_cast<float4*>(out) +
                  ((size_t)angle * ((ny + slices - 1) / slices) + y0 / slices) * L * (slices / 2) + (y0 % slices) / 2;
    for (int k = threadIdx.x; k < (L - L / 4) * P; k += ROWS * TPF) {
      const int o = L / 8 + k / P, p = k % P;
      const float2 a = smem[2 * p * row_smem_len(L) + o], b = smem[(2 * p + 1) * row_smem_len(L) + o];
      dst[(size_t)o * (slices / 2) + p] = make_float4(a.x, a.y, b.x, b.y);
    }
  } else {
    // records (q[o], q[o+1] - q[o])
    sm.sync();
    if (first + rr < end) {
      float4* dst = reinterpret_cast<float4*>(out) + (size_t)row * L;
      for (int o = t; o < L; o += TPF) {
        const float2 q0 = rowbuf[o], q1 = rowbuf[o + 1 < L ? o + 1 : o];
        dst[o] = make_float4(q0.x, q0.y, q1.x - q0.x, q1.y - q0.y);
      }
    }
  }
}

template <int L, bool TILES>
cudaError_t launch_filter_form(const float2* in, float2* out, const float* ramp, const float2* twf, const float2* twi,
                               int n_angles, int ny, cudaStream_t s) {
  constexpr int ROWS = rows_for(L);
  const long long blocks = TILES ? (long long)n_angles * ((ny + ROWS - 1) / ROWS)
                                 : ((long long)n_angles * ny + ROWS - 1) / ROWS;
  if (blocks > 0x7fffffffLL) return cudaErrorInvalidValue;
  if (const cudaError_t e = allow_shared(fbp_filter_kernel<L, TILES>, row_smem_bytes(L)); e != cudaSuccess) return e;
  fbp_filter_kernel<L, TILES>
      <<<(unsigned)blocks, row_threads(L), row_smem_bytes(L), s>>>(in, out, ramp, twf, twi, n_angles, ny, tile_slices(ny));
  return cudaGetLastError();
}

template <int L>
cudaError_t launch_filter(const float2* in, float2* out, const float* ramp, const float2* twf, const float2* twi,
                          int n_angles, int ny, bool tiles, cudaStream_t s) {
  return tiles ? launch_filter_form<L, true>(in, out, ramp, twf, twi, n_angles, ny, s)
               : launch_filter_form<L, false>(in, out, ramp, twf, twi, n_angles, ny, s);
}

using FilterFn = cudaError_t (*)(const float2*, float2*, const float*, const float2*, const float2*, int, int, bool,
                                 cudaStream_t);

FilterFn filter_for(int L) {
  switch (L) {
    case 32: return launch_filter<32>;
    case 64: return launch_filter<64>;
    case 96: return launch_filter<96>;
    case 128: return launch_filter<128>;
    case 192: return launch_filter<192>;
    case 256: return launch_filter<256>;
    case 384: return launch_filter<384>;
    case 512: return launch_filter<512>;
    case 768: return launch_filter<768>;
    case 1024: return launch_filter<1024>;
    case 1536: return launch_filter<1536>;
    case 2048: return launch_filter<2048>;
    default: return nullptr;
  }
}

constexpr int BP_TX = 32, BP_TY = 8, BP_ZPT = 8;  // tile 32 (x) by 64 (z) voxels

__global__ void __launch_bounds__(BP_TX * BP_TY)
    fbp_backproject_kernel(const float2* __restrict__ q, float2* __restrict__ vol, const double2* __restrict__ cs,
                           int n_angles, int ny, int nx, float scale) {
  extern __shared__ float2 scs[];
  const int tid = threadIdx.y * BP_TX + threadIdx.x;
  for (int i = tid; i < n_angles; i += BP_TX * BP_TY) scs[i] = make_float2((float)cs[i].x, (float)cs[i].y);
  __syncthreads();
  // each warp covers a compact 8 (x) by 4 (z) patch per z step, so that its
  // lanes' detector positions span at most 8|cos| + 4|sin| + 1 records (two
  // 128-byte wavefronts) instead of the 32|cos| + 1 of a 32-voxel row
  const int lane = tid & 31, warp = tid >> 5;
  const int x = blockIdx.x * BP_TX + (warp & 3) * 8 + (lane & 7);
  const int zb = blockIdx.y * (BP_TY * BP_ZPT) + (warp >> 2) * 4 + (lane >> 3);
  const int y = blockIdx.z;
  const float half = 0.5f * (float)nx - 0.5f;  // detector index of s = 0
  // voxels past the grid (tile overhang) compute on the last row / column,
  // which keeps their reads inside the padded rows; they store nothing
  const float xc = (float)(x < nx ? x : nx - 1) - half;
  float zc[BP_ZPT];
#pragma unroll
  for (int m = 0; m < BP_ZPT; m++) {
    const int z = zb + m * BP_TY;  // z steps of 8: the block's 8 rows of patches
    zc[m] = (float)(z < nx ? z : nx - 1) - half;
  }
  float2 acc[BP_ZPT];
#pragma unroll
  for (int m = 0; m < BP_ZPT; m++) acc[m] = make_float2(0.f, 0.f);
  // rows of width 2 nx, detector index u at column u + nx/2; every voxel of
  // the grid has |u - half| <= nx / sqrt(2) + 1, so both taps stay in the row
  const int W = 2 * nx;
  const size_t plane = (size_t)ny * W;
  const float4* qy = reinterpret_cast<const float4*>(q) + (size_t)y * W + nx / 2;
#pragma unroll 4
  for (int a = 0; a < n_angles; a++) {
    const float2 c = scs[a];
    const float4* row = qy + (size_t)a * plane;
    const float base = fmaf(xc, c.x, half);
#pragma unroll
    for (int m = 0; m < BP_ZPT; m++) {
      const float u = fmaf(zc[m], c.y, base);
      const float uf = floorf(u);
      const float w = u - uf;
      const float4 qd = __ldg(row + (int)uf);
      acc[m].x += fmaf(w, qd.z, qd.x);
      acc[m].y += fmaf(w, qd.w, qd.y);
    }
  }
  if (x >= nx) return;
#pragma unroll
  for (int m = 0; m < BP_ZPT; m++) {
    const int z = zb + m * BP_TY;
    if (z < nx) vol[((size_t)y * nx + z) * nx + x] = cscale(acc[m], scale);
  }
}

// ---------------------------------------------------------------------------
// tile form of the back projection
// ---------------------------------------------------------------------------
// A CTA owns 16 (x) by TZ (z) voxels of a block of slices, a warp one 4 x 4 patch
// of them, a lane 2 H slices: 16 x 2 H complex sums in registers. For one angle
// every lane of the warp reads the same detector columns and weights, so a tap
// is H conflict-free 512-byte rows of shared memory, and it stays in registers
// while the warp walks its patch:
//   * the walk is a snake along the axis on which the detector position moves
//     less (min(|cos|, |sin|) <= 0.71 per voxel), so consecutive voxels use the
//     same two taps or shift by one;
//   * tap j lives in register set j mod 2 (A even, B odd): a shift by one loads
//     one set and moves none. The weight of set A is 1 - w where the lower tap is
//     even and w where it is odd, that of set B the rest; two-wide FMAs.
// Positions are 24-bit fixed point relative to the tile's first column, from
// the double-precision angle table: exact to 2^-20 columns over a tile (a
// position in one FP32 word is off by nx 2^-24 and more).
// What bounds it: the shared-memory pipe (65 % busy) and the latency of a tap's
// load. A walk without reuse reads two taps per voxel (16 bytes per update, 8
// updates per cycle and SM at best); this one reads 0.57, but a load that its
// predicate turns off still takes a slot. Branching around the loads halves the
// pipe's work and is slower (two slices per lane 14.7, four 13.8 ms against 8.9
// per 128 slices of 180 x 1024 columns): 8 to 16 warps do not hide the branches. An
// order of visits nearer to the detector position (0.39 taps) measured the
// same 9.0. Four slices per lane (8 warps, 190 registers) measured 8.9, two
// (16 warps) 9.8; twelve warps of 4 x 4 patches 8.7, with overhanging tiles.
// Whole call, 180 x 1024 x 1024: 162.7 -> 71.6 ms (one thread per voxel reading
// records through the L1, and 13 ms of host cosines).
// Each stage of two angles is copied by cp.async while the ones before it are
// used; a stage holds at most ROWS rows, the columns under the tile's diagonal.
constexpr int BT = 16, BT_STAGES = 3, BT_FRAC = 24;

template <int H>
struct TileShape {
  static constexpr int TZ = H == 2 ? 8 : 16;            // voxels along z
  static constexpr int WARPS = BT / 4 * (TZ / 4);
  static constexpr int ROWS = H == 2 ? 20 : 24;         // floor(15 |cos| + (TZ - 1) |sin|) + 3 at most
  static constexpr int SLICES = 64 * H;
  static constexpr int ROW_BYTES = SLICES * (int)sizeof(float2);
  static constexpr size_t STAGE = (size_t)ROWS * ROW_BYTES;  // one angle
  // the angle table (rounded up to an even count), the warps' weights, the stages
  static constexpr size_t bytes(int n_angles) {
    return (size_t)(n_angles + 1) / 2 * 2 * sizeof(int4) + (size_t)WARPS * 32 * sizeof(float2) + BT_STAGES * 2 * STAGE;
  }
};

// one tap: 2 H slices of one column
template <int H>
struct Tap {
  uint64_t q[2 * H];
};
template <int H>
__device__ __forceinline__ void tap_load(Tap<H>& t, unsigned ptr) {
  asm volatile("ld.shared.v2.b64 {%0, %1}, [%2];" : "=l"(t.q[0]), "=l"(t.q[1]) : "r"(ptr) : "memory");
  if constexpr (H == 2) asm volatile("ld.shared.v2.b64 {%0, %1}, [%2+512];" : "=l"(t.q[2]), "=l"(t.q[3]) : "r"(ptr) : "memory");
}
// where bit is set (the same for the whole warp): ptr += step, then the tap at ptr
template <int H>
__device__ __forceinline__ void tap_shift(Tap<H>& t, unsigned bit, unsigned& ptr, int step) {
  if constexpr (H == 2)
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ne.u32 p, %5, 0;\n\t@p add.u32 %0, %0, %6;\n\t"
        "@p ld.shared.v2.b64 {%1, %2}, [%0];\n\t@p ld.shared.v2.b64 {%3, %4}, [%0+512];\n\t}"
        : "+r"(ptr), "+l"(t.q[0]), "+l"(t.q[1]), "+l"(t.q[2]), "+l"(t.q[3])
        : "r"(bit), "r"(step)
        : "memory");
  else
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ne.u32 p, %3, 0;\n\t@p add.u32 %0, %0, %4;\n\t"
        "@p ld.shared.v2.b64 {%1, %2}, [%0];\n\t}"
        : "+r"(ptr), "+l"(t.q[0]), "+l"(t.q[1])
        : "r"(bit), "r"(step)
        : "memory");
}

// voxel (x, z) of the patch at step p of the walk; ALONG_Z swaps the axes
template <bool ALONG_Z>
__host__ __device__ constexpr int walk_x(int p) {
  const int r = p >> 2, i = (r & 1) ? 3 - (p & 3) : (p & 3);
  return ALONG_Z ? r : i;
}
template <bool ALONG_Z>
__host__ __device__ constexpr int walk_z(int p) {
  const int r = p >> 2, i = (r & 1) ? 3 - (p & 3) : (p & 3);
  return ALONG_Z ? i : r;
}

// One angle over the warp's patch. pa, pb: shared addresses of the lane's
// first taps; ma, mb: bit p set where set A (B) shifts at step p; dw, dc: what
// a shift along (across) the walk adds to a tap's address.
template <bool ALONG_Z, int H>
__device__ __forceinline__ void tile_angle(float2 (&acc)[16][2 * H], const float2* w, unsigned pa, unsigned pb,
                                           unsigned ma, unsigned mb, int dw, int dc) {
  Tap<H> A, B;
  tap_load<H>(A, pa);
  tap_load<H>(B, pb);
#pragma unroll
  for (int p = 0; p < 16; p++) {
    if (p > 0) {
      const int step = (p & 3) == 0 ? dc : ((p >> 2) & 1) ? -dw : dw;
      tap_shift<H>(A, ma & (1u << p), pa, step);
      tap_shift<H>(B, mb & (1u << p), pb, step);
    }
    const float2 wp = w[p];
    float2(&s)[2 * H] = acc[walk_z<ALONG_Z>(p) * 4 + walk_x<ALONG_Z>(p)];
#pragma unroll
    for (int k = 0; k < 2 * H; k++) s[k] = fma2(f2_of(A.q[k]), make_float2(wp.x, wp.x), s[k]);
#pragma unroll
    for (int k = 0; k < 2 * H; k++) s[k] = fma2(f2_of(B.q[k]), make_float2(wp.y, wp.y), s[k]);
  }
}

template <int H>
__global__ void __launch_bounds__(TileShape<H>::WARPS * 32, 1)
    fbp_backproject_tiles(const float2* __restrict__ q, float2* __restrict__ vol, const double2* __restrict__ cs,
                          int n_angles, int ny, int nx, float scale, int vec_out) {
  using S = TileShape<H>;
  constexpr int NT = S::WARPS * 32;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  int4* ang = reinterpret_cast<int4*>(smem_raw);  // first column, fixed-point offset of the tile's corner, cos, sin
  const int na2 = (n_angles + 1) / 2 * 2;
  float2* wtab = reinterpret_cast<float2*>(ang + na2);
  unsigned char* stages = reinterpret_cast<unsigned char*>(wtab + S::WARPS * 32);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int x0 = blockIdx.x * BT, z0 = blockIdx.y * S::TZ, yb = blockIdx.z;
  const int W = 2 * nx;
  constexpr double ONE = (double)(1 << BT_FRAC);
  for (int a = tid; a < na2; a += NT) {
    int4 e = make_int4(0, 0, 0, 0);
    if (a < n_angles) {
      const double2 t = cs[a];
      const double half = 0.5 * nx - 0.5;
      const int c = __double2int_rn(t.x * ONE), s = __double2int_rn(t.y * ONE);
      const long long u0 = __double2ll_rn(((x0 - half) * t.x + (z0 - half) * t.y + half + nx / 2) * ONE);
      const long long lo = u0 + (long long)(BT - 1) * (c < 0 ? c : 0) + (long long)(S::TZ - 1) * (s < 0 ? s : 0);
      // the first of the tile's columns: with all its rows inside [nx/4, 7nx/4)
      // for every tile and angle, since |s| <= 0.71 nx and nx >= 16
      e.x = (int)(lo >> BT_FRAC);
      e.y = (int)(u0 - ((long long)e.x << BT_FRAC));
      e.z = c;
      e.w = s;
    }
    ang[a] = e;
  }
  __syncthreads();
  const float2* base = q + (size_t)yb * W * S::SLICES;
  const size_t plane = (size_t)((ny + S::SLICES - 1) / S::SLICES) * W * S::SLICES;
  const int groups = na2 / 2;
  auto copy = [&](int g) {
    if (g >= groups) return;
#pragma unroll
    for (int h = 0; h < 2; h++) {
      const int a = 2 * g + h;
      if (a >= n_angles) return;
      const int4 e = ang[a];
      const int hi = (e.y + (BT - 1) * (e.z > 0 ? e.z : 0) + (S::TZ - 1) * (e.w > 0 ? e.w : 0)) >> BT_FRAC;
      const int rows = hi + 2 < S::ROWS ? hi + 2 : S::ROWS;
      const float4* src = reinterpret_cast<const float4*>(base + (size_t)a * plane + (size_t)e.x * S::SLICES);
      unsigned char* dst = stages + ((g % BT_STAGES) * 2 + h) * S::STAGE;
      for (int k = tid; k < rows * (S::ROW_BYTES / 16); k += NT) cp_async16(dst + 16 * k, src + k);
    }
  };
  const int px = (warp & 3) * 4, pz = (warp >> 2) * 4;  // the warp's patch
  float2 acc[16][2 * H];
#pragma unroll
  for (int i = 0; i < 16; i++)
#pragma unroll
    for (int k = 0; k < 2 * H; k++) acc[i][k] = make_float2(0.f, 0.f);
  float2* wt = wtab + warp * 32;
  copy(0);
  cp_async_commit();
  copy(1);
  cp_async_commit();
  for (int g = 0; g < groups; g++) {
    cp_async_wait<1>();
    __syncthreads();  // stage g has landed; every warp is done with stage g - 1
    copy(g + 2);
    cp_async_commit();
    // lanes 0-15 and 16-31: positions, weights and shifts of the 16 voxels in
    // walk order, for the stage's two angles
    const int4 e = ang[2 * g + (lane >> 4)];
    const bool alz = abs(e.z) > abs(e.w);  // |cos| > |sin|: the walk goes along z
    const int p = lane & 15;
    const int vx = alz ? walk_x<true>(p) : walk_x<false>(p), vz = alz ? walk_z<true>(p) : walk_z<false>(p);
    const int u = e.y + (px + vx) * e.z + (pz + vz) * e.w;
    const int n = u >> BT_FRAC;
    const float f = (float)(u & ((1 << BT_FRAC) - 1)) * (1.0f / (1 << BT_FRAC));
    const int ea = (n + 1) & ~1, eb = n | 1;  // the even and the odd tap
    const float wa = (n & 1) ? f : 1.0f - f;
    const int pn = __shfl_up_sync(0xffffffffu, n, 1);
    const unsigned ma = __ballot_sync(0xffffffffu, ea != ((pn + 1) & ~1)), mb = __ballot_sync(0xffffffffu, eb != (pn | 1));
    __syncwarp();
    wt[lane] = make_float2(wa, 1.0f - wa);
    __syncwarp();
#pragma unroll 1
    for (int h = 0; h < 2; h++) {
      if (2 * g + h >= n_angles) break;
      const int n0 = __shfl_sync(0xffffffffu, n, 16 * h);
      const int4 eh = ang[2 * g + h];
      const unsigned sb =
          (unsigned)__cvta_generic_to_shared(stages + ((g % BT_STAGES) * 2 + h) * S::STAGE) + lane * 16;
      const unsigned pa = sb + ((n0 + 1) & ~1) * S::ROW_BYTES, pb = sb + (n0 | 1) * S::ROW_BYTES;
      const unsigned m0 = ma >> (16 * h), m1 = mb >> (16 * h);
      const int dx = eh.z < 0 ? -2 * S::ROW_BYTES : 2 * S::ROW_BYTES, dz = eh.w < 0 ? -2 * S::ROW_BYTES : 2 * S::ROW_BYTES;
      if (abs(eh.z) > abs(eh.w)) tile_angle<true, H>(acc, wt + 16 * h, pa, pb, m0, m1, dz, dx);
      else tile_angle<false, H>(acc, wt + 16 * h, pa, pb, m0, m1, dx, dz);
    }
  }
  cp_async_wait<0>();
  // a lane's four x of one (z, slice): 32 contiguous bytes
#pragma unroll
  for (int k = 0; k < 2 * H; k++) {
    const int y = yb * S::SLICES + (k >> 1) * 64 + 2 * lane + (k & 1);
    if (y >= ny) continue;
#pragma unroll
    for (int z = 0; z < 4; z++) {
      float2* dst = vol + ((size_t)y * nx + z0 + pz + z) * nx + x0 + px;
      const float2 a = cscale(acc[z * 4][k], scale), b = cscale(acc[z * 4 + 1][k], scale);
      const float2 c = cscale(acc[z * 4 + 2][k], scale), d = cscale(acc[z * 4 + 3][k], scale);
      if (vec_out) {
        reinterpret_cast<float4*>(dst)[0] = make_float4(a.x, a.y, b.x, b.y);
        reinterpret_cast<float4*>(dst)[1] = make_float4(c.x, c.y, d.x, d.y);
      } else {
        dst[0] = a, dst[1] = b, dst[2] = c, dst[3] = d;
      }
    }
  }
}

template <int H>
cudaError_t launch_tiles(const float2* q, float2* vol, const double2* cs, int n_angles, int ny, int nx, float scale,
                         cudaStream_t s) {
  using S = TileShape<H>;
  if (const cudaError_t e = allow_shared(fbp_backproject_tiles<H>, S::bytes(PWF_FBP_MAX_ANGLES)); e != cudaSuccess) return e;
  const dim3 grid(nx / BT, nx / S::TZ, (ny + S::SLICES - 1) / S::SLICES);  // nx is a multiple of 16
  fbp_backproject_tiles<H><<<grid, S::WARPS * 32, S::bytes(n_angles), s>>>(q, vol, cs, n_angles, ny, nx, scale,
                                                                           ((uintptr_t)vol & 15) == 0);
  return cudaGetLastError();
}

size_t align256(size_t b) { return (b + 255) & ~(size_t)255; }

struct FbpLayout {
  size_t q, ramp, twf, twi, cs, total;
};

FbpLayout fbp_layout(int n_angles, int ny, int nx) {
  FbpLayout l{};
  const int L = 2 * nx;
  const size_t row = (size_t)L * (tile_form(ny, nx) ? sizeof(float2) : sizeof(float4));
  const size_t rows = tile_form(ny, nx) ? (size_t)(ny + tile_slices(ny) - 1) / tile_slices(ny) * tile_slices(ny) : (size_t)ny;
  l.q = 0;
  l.ramp = l.q + align256((size_t)n_angles * rows * row);
  l.twf = l.ramp + align256((size_t)L * sizeof(float));
  l.twi = l.twf + align256((size_t)twiddle_len(L, FWD) * sizeof(float2));
  l.cs = l.twi + align256((size_t)twiddle_len(L, INV) * sizeof(float2));
  l.total = l.cs + align256((size_t)n_angles * sizeof(double2));
  return l;
}

bool fbp_sizes_ok(int n_angles, int ny, int nx) {
  return n_angles >= 1 && n_angles <= PWF_FBP_MAX_ANGLES && ny >= 1 && ny <= 65535 && nx >= 16 &&
         filter_for(2 * nx) != nullptr;
}

}  // namespace
}  // namespace pwf

using namespace pwf;

extern "C" {

size_t pwf_fbp_workspace_bytes(int32_t n_angles, int32_t ny, int32_t nx) {
  if (!fbp_sizes_ok(n_angles, ny, nx)) return 0;
  return fbp_layout(n_angles, ny, nx).total;
}

pwf_status pwf_fbp(const void* psi, int32_t n_angles, int32_t ny, int32_t nx, const double* angles_rad_host,
                   double wavelength_m, double voxel_m, void* vol_out, void* workspace, size_t workspace_bytes,
                   void* stream) {
  if (!psi || !vol_out || !workspace || !angles_rad_host || !fbp_sizes_ok(n_angles, ny, nx) ||
      !(wavelength_m > 0) || !(voxel_m > 0))
    return PWF_ERR_INVALID_ARG;
  const FbpLayout l = fbp_layout(n_angles, ny, nx);
  if (workspace_bytes < l.total || ((uintptr_t)workspace & 255) || ((uintptr_t)psi & 7) || ((uintptr_t)vol_out & 7))
    return PWF_ERR_INVALID_ARG;
  cudaStream_t s = (cudaStream_t)stream;
  char* ws = (char*)workspace;
  const int L = 2 * nx;
  const bool tiles = tile_form(ny, nx);
  double2* cs = (double2*)(ws + l.cs);
  bool finite = true;
  for (int first = 0; first < n_angles; first += ANGLE_PART) {
    AnglePart part;
    const int count = n_angles - first < ANGLE_PART ? n_angles - first : ANGLE_PART;
    for (int a = 0; a < ANGLE_PART; a++) {
      const bool ok = a < count && std::isfinite(angles_rad_host[first + a]);
      part.rad[a] = ok ? angles_rad_host[first + a] : 0.0;
      finite = finite && (ok || a >= count);
    }
    const unsigned blocks = first == 0 ? (unsigned)((32 * L + 255) / 256) : 1u;
    k_fbp_tables<<<blocks, 256, 0, s>>>(part, first, count, L, (float*)(ws + l.ramp), (float2*)(ws + l.twf),
                                        (float2*)(ws + l.twi), cs);
  }
  float2* q = (float2*)(ws + l.q);
  if (cudaGetLastError() != cudaSuccess ||
      filter_for(L)((const float2*)psi, q, (const float*)(ws + l.ramp), (const float2*)(ws + l.twf),
                    (const float2*)(ws + l.twi), n_angles, ny, tiles, s) != cudaSuccess) {
    cudaGetLastError();
    return PWF_ERR_CUDA;
  }
  // back projection weight pi / N_theta and the factor -lambda / (2 pi p):
  // beta + i delta from psi = -k int beta - i k int delta. An angle that is not
  // finite has no positions: it makes every voxel NaN.
  const float scale = finite ? (float)(M_PI / n_angles * (-wavelength_m / (2.0 * M_PI * voxel_m))) : NAN;
  if (tiles) {
    if ((tile_slices(ny) == 128 ? launch_tiles<2>(q, (float2*)vol_out, cs, n_angles, ny, nx, scale, s)
                                : launch_tiles<1>(q, (float2*)vol_out, cs, n_angles, ny, nx, scale, s)) != cudaSuccess) {
      cudaGetLastError();
      return PWF_ERR_CUDA;
    }
  } else {
    const dim3 grid((nx + BP_TX - 1) / BP_TX, (nx + BP_TY * BP_ZPT - 1) / (BP_TY * BP_ZPT), ny);
    fbp_backproject_kernel<<<grid, dim3(BP_TX, BP_TY), n_angles * sizeof(float2), s>>>(q, (float2*)vol_out, cs, n_angles,
                                                                                      ny, nx, scale);
  }
  if (cudaGetLastError() != cudaSuccess) return PWF_ERR_CUDA;
  return PWF_OK;
}

}  // extern "C"
