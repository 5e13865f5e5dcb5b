// Residual norm of the fine-level operator computed from caller buffers
// without any device allocation (mg_residual_norm_noalloc in mg.h).
//
// Some callers cannot allocate device memory when they need this norm: AMR
// codes and frameworks that reserve the GPU's memory up front in their own
// pool (a cudaMalloc outside the pool can fail on a device they have filled),
// and host code that must not block on the allocator, since cudaMalloc and
// cudaFree can wait for work in flight.  They still need the convergence
// measure of their own Phi, rho and boundary values, without building a
// hierarchy (whose arena is allocated).
//
// The per-block partial sums, the only scratch this computation needs, live
// in a file-scope __device__ array of fixed size.  Host code cannot use the
// array's name as a device address, so every call obtains the address with
// cudaGetSymbolAddress, with the caller's device current, and passes it to
// the kernels.  The lookup allocates nothing and is cheap; doing it on every
// call rather than caching it keeps the address right when the module is
// loaded again at another address (after cudaDeviceReset, or in another
// context of the same device).  The first call on a device also loads this
// file's kernels and the array.
#include <cmath>

#include "../../include/mg.h"
#include "exact_sum.cuh"
#include "mg_internal.h"

namespace gbmg {

void set_thread_error(const char* msg);        // mg_capi.cu
bool is_device_ptr(const void* p, int device);  // mg_capi.cu

namespace {

constexpr int kNoAllocMaxPartials = 4096;  // 32 KB of scratch on each device
constexpr int kNoAllocThreads = 256;

// One partial sum of squares per block of the first kernel.  Every call on a
// device uses the same array; each slot the second kernel reads is written by
// the first kernel of the same call, so nothing needs clearing between calls.
static __device__ __align__(256) double g_noalloc_partials[kNoAllocMaxPartials];

// 2 x in integer arithmetic (a zero or subnormal x gives 0, as exact_sum takes it).
__device__ __forceinline__ double twice(double x) {
  const unsigned long long b = bits_of(x);
  const unsigned e = (unsigned)(b >> 52) & 0x7ffu;
  if (e == 0) return 0.0;
  if (e == 0x7ffu) return x;
  if (e == 0x7feu) return double_of((b & 0x8000000000000000ull) | 0x7ff0000000000000ull);
  return double_of(b + (1ull << 52));
}

// Residual r^ = h^2 (Laplacian Phi - rho) of every active cell, with the
// modified stencil of Section 3 at level 0 (ghost at theta = 1/2 through the
// face value Phi_b, Fig. 5): r^ = sum_active Phi_j + 2 sum_ghost Phi_b
// - (6 + #ghost) Phi_i - h^2 rho_i.  Block sums of r^2 go to partials.
//
// A thread per cell ran about 12 FP64 operations for active and idle lanes
// alike, on a pipe that takes 16 cycles per warp instruction (504 us on a
// half-active 256^3 patch with face values, whose 688 MB take 102 us).  So a
// warp takes kTile cells of a row, lists the active ones and works with every
// lane in use, and the six terms are added in integer arithmetic
// (exact_sum.cuh), which leaves three FP64 instructions per active cell.
// What is left are chains of dependent loads (mask, list, neighbours' masks,
// values): eight blocks per SM at 32 registers and tiles of 256 cells hide
// them (172 us; with four blocks of 64 registers and 128 cells 247).
constexpr int kTile = 256;
constexpr int kBlocksPerSm = 8;

__global__ void __launch_bounds__(kNoAllocThreads, kBlocksPerSm)
noalloc_resnorm_kernel(const int8_t* __restrict__ mask, const double* __restrict__ phi,
                       const double* __restrict__ rho, const double* __restrict__ bx,
                       const double* __restrict__ by, const double* __restrict__ bz, int nx, int ny, int nz,
                       double h2, double* partials) {
  constexpr int kWarps = kNoAllocThreads / 32;
  __shared__ uint8_t active[kWarps][kTile];
  __shared__ double diag[8];  // 6 + #ghost
  if (threadIdx.x < 8) diag[threadIdx.x] = (double)(6 + (int)threadIdx.x);
  __syncthreads();
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const long long sy = nx, sz = (long long)nx * ny;
  const unsigned tiles = (unsigned)(nx + kTile - 1) / kTile;
  const unsigned n = tiles * (unsigned)ny * (unsigned)nz;
  double acc = 0.0;
  for (unsigned t = blockIdx.x * kWarps + w; t < n; t += gridDim.x * kWarps) {
    const unsigned row = t / tiles;
    const int k = (int)(row / (unsigned)ny), j = (int)(row - (unsigned)k * (unsigned)ny);
    const int i0 = (int)(t - row * tiles) * kTile;
    const long long r0 = (long long)row * nx;  // cell (0, j, k)
    const int8_t* __restrict__ m = mask + r0;
    int na = 0;
#pragma unroll
    for (int s = 0; s < kTile / 32; ++s) {
      const int i = i0 + 32 * s + lane;
      const bool act = i < nx && m[i] > 0;
      const unsigned all = __ballot_sync(0xffffffffu, act);
      if (act) active[w][na + __popc(all & ((1u << lane) - 1u))] = (uint8_t)(32 * s + lane);
      na += __popc(all);
    }
    __syncwarp();
    const bool row_in[4] = {j > 0, j + 1 < ny, k > 0, k + 1 < nz};
    const double* __restrict__ fx = bx ? bx + (long long)row * (nx + 1) : nullptr;
    const double* __restrict__ fy = by ? by + ((long long)k * (ny + 1) + j) * nx : nullptr;
    const double* __restrict__ fz = bz ? bz + r0 : nullptr;
    const double* __restrict__ p = phi + r0;
    for (int x = lane; x < na; x += 32) {
      const int i = i0 + active[w][x];
      const bool in[6] = {i > 0 && m[i - 1] > 0,         i + 1 < nx && m[i + 1] > 0,    row_in[0] && m[i - sy] > 0,
                          row_in[1] && m[i + sy] > 0,    row_in[2] && m[i - sz] > 0,    row_in[3] && m[i + sz] > 0};
      const long long off[6] = {-1, 1, -sy, sy, -sz, sz};
      const double* f[6] = {fx ? fx + i : nullptr, fx ? fx + i + 1 : nullptr, fy ? fy + i : nullptr,
                            fy ? fy + i + nx : nullptr, fz ? fz + i : nullptr, fz ? fz + i + sz : nullptr};
      double v[6];
      int ghosts = 0;
#pragma unroll
      for (int d = 0; d < 6; ++d) {
        v[d] = 0.0;
        if (in[d]) v[d] = p[i + off[d]];
        else if (f[d]) v[d] = twice(*f[d]);
        ghosts += !in[d];
      }
      const double r = fma(-diag[ghosts], p[i], exact_sum(v)) - h2 * rho[r0 + i];
      acc = fma(r, r, acc);
    }
    __syncwarp();
  }
  __shared__ double warp_sums[kWarps];
  for (int o = 16; o > 0; o >>= 1) acc += __shfl_down_sync(0xffffffffu, acc, o);
  if (lane == 0) warp_sums[w] = acc;
  __syncthreads();
  if (threadIdx.x < 32) {
    double v = threadIdx.x < kWarps ? warp_sums[threadIdx.x] : 0.0;
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    if (threadIdx.x == 0) partials[blockIdx.x] = v;
  }
}

// Sums the partials in a fixed order and writes ||r|| = sqrt(sum) / h^2.
__global__ void __launch_bounds__(kNoAllocThreads)
noalloc_finalize_kernel(const double* __restrict__ partials, int nblocks, double h2, double* out) {
  double acc = 0.0;
  for (int e = threadIdx.x; e < nblocks; e += blockDim.x) acc += partials[e];
  __shared__ double sm[kNoAllocThreads];
  sm[threadIdx.x] = acc;
  __syncthreads();
  for (int w = kNoAllocThreads / 2; w > 0; w >>= 1) {
    if ((int)threadIdx.x < w) sm[threadIdx.x] += sm[threadIdx.x + w];
    __syncthreads();
  }
  if (threadIdx.x == 0) out[0] = sqrt(sm[0]) / h2;
}

}  // namespace
}  // namespace gbmg

extern "C" mg_status mg_residual_norm_noalloc(const int8_t* mask, const double* phi, const double* rho,
                                              const double* bx, const double* by, const double* bz, int nx,
                                              int ny, int nz, double h, double* norm_out, void* cuda_stream) {
  using namespace gbmg;
  if (!mask || !phi || !rho || !norm_out) {
    set_thread_error("mg_residual_norm_noalloc: null mask, phi, rho or output");
    return MG_ERR_INVALID_ARG;
  }
  if (nx < 1 || ny < 1 || nz < 1 || nx > 2048 || ny > 2048 || nz > 2048) {
    set_thread_error("mg_residual_norm_noalloc: dimensions must be in 1..2048");
    return MG_ERR_INVALID_ARG;
  }
  if (!(h > 0) || !std::isfinite(h)) {
    set_thread_error("mg_residual_norm_noalloc: h must be finite and > 0");
    return MG_ERR_INVALID_ARG;
  }
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0) {
    set_thread_error("mg_residual_norm_noalloc: no usable current CUDA device");
    return MG_ERR_CUDA;
  }
  const void* const bufs[] = {mask, phi, rho, bx, by, bz, norm_out};
  for (const void* p : bufs)
    if (p && !is_device_ptr(p, dev)) {
      set_thread_error("mg_residual_norm_noalloc: a buffer is not device memory of the current GPU");
      return MG_ERR_INVALID_ARG;
    }
  void* scratch = nullptr;
  cudaError_t es = cudaGetSymbolAddress(&scratch, g_noalloc_partials);
  if (es != cudaSuccess || !scratch) {
    (void)cudaGetLastError();
    set_thread_error("mg_residual_norm_noalloc: cudaGetSymbolAddress of the scratch array failed");
    return MG_ERR_CUDA;
  }
  // a warp per tile of a row, at most the resident blocks
  const long long tiles = (long long)((nx + kTile - 1) / kTile) * ny * nz;
  long long blocks = (tiles + kNoAllocThreads / 32 - 1) / (kNoAllocThreads / 32);
  if (blocks > (long long)kBlocksPerSm * device_sms()) blocks = (long long)kBlocksPerSm * device_sms();
  if (blocks > kNoAllocMaxPartials) blocks = kNoAllocMaxPartials;
  cudaStream_t s = (cudaStream_t)cuda_stream;
  const double h2 = h * h;
  count_launch(2);
  noalloc_resnorm_kernel<<<(int)blocks, kNoAllocThreads, 0, s>>>(mask, phi, rho, bx, by, bz, nx, ny, nz, h2,
                                                                  (double*)scratch);
  noalloc_finalize_kernel<<<1, kNoAllocThreads, 0, s>>>((const double*)scratch, (int)blocks, h2, norm_out);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) {
    set_thread_error(cudaGetErrorString(e));
    return MG_ERR_CUDA;
  }
  return MG_OK;
}
