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
#include "row_tiles.h"

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
// warp takes kTile cells of a row, or of several short rows (row_tiles.h),
// lists the active ones and works with every lane in use, and the six terms are
// added in integer arithmetic (exact_sum.cuh), which leaves three FP64
// instructions per active cell.
// What is left are chains of dependent loads (mask, list, neighbours' masks,
// values): eight blocks per SM at 32 registers and tiles of 256 cells hide
// them (172 us; with four blocks of 64 registers and 128 cells 247).  ROWS: a
// tile has several rows, whose cells look up their own (half-active boxes, 512
// x 512 rows of 8 cells: 38 us, a tile per row 176, a thread per cell 100; 256
// x 256 rows of 48: 58, 56 and 153), as many as leave every resident warp a tile
// (32 x 32 rows of 32: 16.5 us, with full tiles of eight rows 21.7).
constexpr int kTile = 256;
constexpr int kBlocksPerSm = 8;

template <bool ROWS>
__global__ void __launch_bounds__(kNoAllocThreads, kBlocksPerSm)
noalloc_resnorm_kernel(const int8_t* __restrict__ mask, const double* __restrict__ phi,
                       const double* __restrict__ rho, const double* __restrict__ bx,
                       const double* __restrict__ by, const double* __restrict__ bz, RowTiles T, int ny, int nz,
                       double h2, double* partials) {
  constexpr int kWarps = kNoAllocThreads / 32;
  __shared__ uint8_t active[kWarps][kTile];
  __shared__ double diag[8];  // 6 + #ghost
  if (threadIdx.x < 8) diag[threadIdx.x] = (double)(6 + (int)threadIdx.x);
  __syncthreads();
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int nx = (int)T.nx;
  const long long sy = nx, sz = (long long)nx * ny;
  double acc = 0.0;
  for (unsigned t = blockIdx.x * kWarps + w; t < T.count; t += gridDim.x * kWarps) {
    unsigned row0, i0, cells;
    T.tile(t, &row0, &i0, &cells);
    const long long at0 = (long long)row0 * nx + i0;  // the tile's first cell
    int na = 0;
#pragma unroll
    for (int s = 0; s < kTile / 32; ++s) {
      if (32 * s >= (int)cells) break;
      const int c = 32 * s + lane;
      const bool act = c < (int)cells && mask[at0 + c] > 0;
      const unsigned all = __ballot_sync(0xffffffffu, act);
      if (act) active[w][na + __popc(all & ((1u << lane) - 1u))] = (uint8_t)c;
      na += __popc(all);
    }
    __syncwarp();
    const int k0 = (int)(row0 / (unsigned)ny), j0 = (int)(row0 - (unsigned)k0 * (unsigned)ny);
    for (int x = lane; x < na; x += 32) {
      const int c = active[w][x];
      unsigned row = row0;
      int i = (int)i0 + c, j = j0, k = k0;
      if (ROWS) {
        const unsigned dr = T.row_of((unsigned)c);
        row += dr;
        i = c - (int)dr * nx;
        k = (int)(row / (unsigned)ny);
        j = (int)(row - (unsigned)k * (unsigned)ny);
      }
      const int8_t* __restrict__ m = mask + (at0 + c);
      const double* __restrict__ p = phi + (at0 + c);
      const bool in[6] = {i > 0 && m[-1] > 0,      i + 1 < nx && m[1] > 0, j > 0 && m[-sy] > 0,
                          j + 1 < ny && m[sy] > 0, k > 0 && m[-sz] > 0,    k + 1 < nz && m[sz] > 0};
      const long long off[6] = {-1, 1, -sy, sy, -sz, sz};
      const long long fx = (long long)row * (nx + 1) + i, fy = (long long)(row + (unsigned)k) * nx + i, fz = at0 + c;
      const double* f[6] = {bx ? bx + fx : nullptr,      bx ? bx + fx + 1 : nullptr, by ? by + fy : nullptr,
                            by ? by + fy + nx : nullptr, bz ? bz + fz : nullptr,     bz ? bz + fz + sz : nullptr};
      double v[6];
      int ghosts = 0;
#pragma unroll
      for (int d = 0; d < 6; ++d) {
        v[d] = 0.0;
        if (in[d]) v[d] = p[off[d]];
        else if (f[d]) v[d] = twice(*f[d]);
        ghosts += !in[d];
      }
      const double r = fma(-diag[ghosts], p[0], exact_sum(v)) - h2 * rho[at0 + c];
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
  // a warp per tile, at most the resident blocks
  constexpr int kWarps = kNoAllocThreads / 32;
  const int resident = kBlocksPerSm * device_sms();
  const RowTiles T = row_tiles(nx, ny, nz, kTile, resident * kWarps);
  long long blocks = ((long long)T.count + kWarps - 1) / kWarps;
  if (blocks > resident) blocks = resident;
  if (blocks > kNoAllocMaxPartials) blocks = kNoAllocMaxPartials;
  cudaStream_t s = (cudaStream_t)cuda_stream;
  const double h2 = h * h;
  count_launch(2);
  if (T.per > 1)
    noalloc_resnorm_kernel<true><<<(int)blocks, kNoAllocThreads, 0, s>>>(mask, phi, rho, bx, by, bz, T, ny, nz, h2,
                                                                         (double*)scratch);
  else
    noalloc_resnorm_kernel<false><<<(int)blocks, kNoAllocThreads, 0, s>>>(mask, phi, rho, bx, by, bz, T, ny, nz, h2,
                                                                          (double*)scratch);
  noalloc_finalize_kernel<<<1, kNoAllocThreads, 0, s>>>((const double*)scratch, (int)blocks, h2, norm_out);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) {
    set_thread_error(cudaGetErrorString(e));
    return MG_ERR_CUDA;
  }
  return MG_OK;
}
