// Kernels of the learned initial guess's network: the 3x3x3 convolution as a
// tcgen05 implicit GEMM, its weight gradients, and the packing of weights.
//
// Convolution.  An output tile is 128 voxels by cout channels, accumulated in
// tensor memory (TMEM) in FP32 over K = 27 taps x cin input channels; up to
// four tiles (one box of voxels, one after another in it) are worked on
// together: an MMA with few columns waits for the one before it on the same
// accumulator (about 80 cycles at N = 16, of which 8 are work), so the tiles'
// MMAs of one tap follow each other.  Per 16 input channels one tcgen05.mma (kind::f16,
// BF16 x BF16 -> FP32, M = 128, N = cout) accumulates.  The A operand comes
// from the channels-last input by TMA copies of a 5-D view of it,
// (span channels, x, y, z, block of span channels), landing in shared memory
// in the K-major layout swizzled over rows of span channels; voxels outside
// the grid read 0 (the convolution's zero padding).  A row is as long as the
// channels and the widest swizzle allow: 64, 32 or 16 channels.  Two ways to
// stage it:
//  - halo rows (tiles that are whole rows of 128 voxels): one copy per 16
//    input channels of the box (130 x group + 2 x 3) around the group's rows;
//    each of the 27 taps is then a view of it, so the input is read 4.5 times
//    (group 4) instead of 27 times;
//  - tap tiles (other shapes): one copy per tap and channel chunk of the
//    group's box shifted by the tap.
// The B operand (the weights, packed [27][cin / 8][cout][8]) stays resident
// in shared memory for the whole launch when it fits (up to 72 KB), loaded
// once per CTA by one bulk copy; otherwise it is staged with each tap.  The
// pipeline depth is as many stages as fit in the shared-memory budget.
//
// Roles: warp 0's lane 0 issues the copies into the ring of stages, warp 1
// allocates TMEM and its lane 0 issues the MMAs (each stage is released by a
// tcgen05.commit when its MMAs have read it), warps 2-5 read the two
// accumulator buffers back (tcgen05.ld, one TMEM lane quarter per warp),
// add the bias, apply ReLU and the optional mask, and store BF16.  Tiles are
// distributed over persistent CTAs; the two accumulators let the next tile's
// MMAs run while the last one drains.  Every wait is bounded by time and by a
// shared abort flag: a wait that runs out sets the error word, every role
// leaves its loop, the copy and MMA threads wait (bounded) for their
// operations in flight, and TMEM is released.
#include <cudaTypedefs.h>

#include "async_copy.cuh"
#include "mg_internal.h"
#include "unet_internal.h"

namespace gbmg {

namespace {

constexpr unsigned long long kConvLimitNs = 1000000000ull;

struct ConvSmemHeader {
  unsigned long long full[kConvMaxStages];
  unsigned long long empty[kConvMaxStages];
  unsigned long long accf[2];
  unsigned long long acce[2];
  unsigned long long wbar;
  uint32_t tmem;
  int abort;
  int consumed;  // units the MMA thread has waited for (the copies still in flight at an abort are after it)
};

}  // namespace

// Shared-memory layout of one convolution launch: per pipeline unit the
// input bytes (a halo row box of 16 channels, or one tap's tile of kc
// chunks) and the weight bytes staged with it (0 when the layer's weights
// are resident: w_bytes, loaded once per CTA).
__host__ __device__ ConvLayout conv_layout(const ConvArgs& a) {
  ConvLayout l;
  const unsigned wall = 27u * (unsigned)a.cin * (unsigned)a.cout * 2u;
  l.w_load = a.wres ? wall : 0u;
  l.w_bytes = a.wres ? (wall + 1023u) / 1024u * 1024u : 0u;
  if (a.halo) {
    l.a_bytes = 3u * (unsigned)(a.group + 2) * 130u * 32u;
    l.b_bytes = 0;
    l.units = a.cin / 16;
  } else {
    l.a_bytes = (unsigned)a.group * (unsigned)a.kc * 2048u;
    l.b_bytes = a.wres ? 0u : (unsigned)a.kc * (unsigned)a.cout * 16u;
    l.units = 27 * (a.cin / (8 * a.kc));
  }
  // a swizzled copy's shared-memory destination must be aligned to its
  // pattern: the stages are laid out at a stride rounded up to 1024 bytes
  l.a_stride = (l.a_bytes + 1023u) / 1024u * 1024u;
  return l;
}

size_t conv_smem_bytes(const ConvArgs& a) {
  const ConvLayout l = conv_layout(a);
  return 1024 + (size_t)l.w_bytes + (size_t)a.stages * (l.a_stride + l.b_bytes);
}

// TMEM columns of a convolution CTA: two sets of `group` FP32 accumulators of
// cout columns, rounded up to the power of two the allocator takes.
__host__ __device__ uint32_t conv_tmem_cols(int group, int cout) {
  const int c = 2 * group * cout;
  return c <= 32 ? 32u : (c <= 64 ? 64u : (c <= 128 ? 128u : (c <= 256 ? 256u : 512u)));
}

namespace {

// Channels per shared-memory row and 8-channel chunks per unit: the widest
// row that divides the channels, and as many rows' blocks as make at most 64
// channels.
void conv_chunks(int cin, int* span, int* kc) {
  *span = cin % 64 == 0 ? 64 : (cin % 32 == 0 ? 32 : 16);
  const int blocks = cin / *span;
  int n = 64 / *span;
  while (blocks % n) --n;
  *kc = n * *span / 8;
}

int conv_groups(const ConvArgs& a) {
  return ((a.W + a.bx - 1) / a.bx) * ((a.H + a.by - 1) / a.by) * ((a.D + a.bz - 1) / a.bz);
}

}  // namespace

// The plan of a convolution.  Weights up to 72 KB stay resident.  Tiles that
// are whole rows of 128 voxels take the halo path (which needs resident
// weights).  As many tiles are worked on together, up to four, as leave about
// 100 groups, fit TMEM twice and leave three stages in shared memory (two of a
// halo path's).  With fewer groups SMs stand idle: on 128 rows of 128 voxels,
// 16 channels, a forward pass takes 51 us with every tile its own, 56 in fours;
// asking for 150 groups costs 56 -> 64 us on 512 rows.
void conv_plan(ConvArgs& a) {
  constexpr size_t kBudget = 225 * 1024;  // dynamic shared memory
  constexpr int kMaxCopySide = 256;       // of a TMA copy's box
  const unsigned wall = 27u * (unsigned)a.cin * (unsigned)a.cout * 2u;
  a.wres = wall <= 72u * 1024u ? 1 : 0;
  conv_chunks(a.cin, &a.span, &a.kc);
  conv_tile_box(a.W, a.H, a.D, kConvTileM, &a.bx, &a.by, &a.bz);
  a.halo = (a.bx == 128 && a.wres) ? 1 : 0;
  auto stages = [&]() {
    a.stages = 1;
    const ConvLayout l = conv_layout(a);
    const size_t per = l.a_stride + l.b_bytes, fixed = 1024 + (size_t)l.w_bytes;
    const size_t n = fixed < kBudget ? (kBudget - fixed) / per : 0;
    a.stages = n > (size_t)kConvMaxStages ? kConvMaxStages : (int)n;
  };
  for (a.group = 4; a.group >= 1; a.group /= 2) {
    if (2 * a.group * a.cout > 512 && a.group > 1) continue;
    if (a.halo) {
      if (a.group > a.H && a.group > 1) continue;
      a.span = 16;
      a.kc = 2;
      a.by = a.group;
      a.bz = 1;
    } else {
      conv_tile_box(a.W, a.H, a.D, kConvTileM * a.group, &a.bx, &a.by, &a.bz);
      if (a.group > 1 && (a.by > kMaxCopySide || a.bz > kMaxCopySide)) continue;  // a grid one or two voxels wide
    }
    stages();
    if (a.group == 1 || (a.stages >= (a.halo ? 2 : 3) && conv_groups(a) >= 100)) break;
  }
  if (a.stages < 2) a.stages = 2;
  a.ntx = (a.W + a.bx - 1) / a.bx;
  a.nty = (a.H + a.by - 1) / a.by;
  a.ntz = (a.D + a.bz - 1) / a.bz;
}

namespace {

__global__ void __launch_bounds__(kConvThreads, 1)
    conv_kernel(const __grid_constant__ CUtensorMap map, ConvArgs a) {
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  ConvSmemHeader& S = *reinterpret_cast<ConvSmemHeader*>(smem_raw);
  const ConvLayout lay = conv_layout(a);
  unsigned char* wres = smem_raw + 1024;  // resident weights (when lay.w_bytes > 0)
  unsigned char* stage_a = wres + lay.w_bytes;
  unsigned char* stage_b = stage_a + a.stages * lay.a_stride;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int ntiles = a.ntx * a.nty * a.ntz;
  const int units = lay.units;
  const int upt = a.cin / (8 * a.kc);
  const int NS = a.stages;
  const uint32_t acc_cols = (uint32_t)a.cout;
  const uint32_t tcols = conv_tmem_cols(a.group, a.cout);
  const int G = a.group;
  __shared__ float bias_s[256];
  if (a.bias)
    for (int i = threadIdx.x; i < a.cout; i += kConvThreads) bias_s[i] = a.bias[i];
  if (threadIdx.x == 0) {
    for (int i = 0; i < NS; ++i) {
      mbar_init(&S.full[i], 1);
      mbar_init(&S.empty[i], 1);
    }
    for (int i = 0; i < 2; ++i) {
      mbar_init(&S.accf[i], 1);
      mbar_init(&S.acce[i], 128);
    }
    mbar_init(&S.wbar, 1);
    S.abort = 0;
    S.consumed = 0;
    mbar_init_fence();
  }
  if (warp == 1) tmem_alloc(&S.tmem, tcols);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = S.tmem;
  volatile int* abort = &S.abort;

  if (warp == 0) {
    if (lane == 0) {
      // ---- copies ----
      if (lay.w_bytes) {  // the whole layer's weights, once per CTA
        mbar_expect_tx(&S.wbar, lay.w_load);
        bulk_load(wres, a.w, lay.w_load, &S.wbar);
      }
      int it = 0, st = 0;
      uint32_t ph = 1;  // parity of the wait for an empty stage: the first pass over the ring does not wait
      const bool stall = a.debug_stall && blockIdx.x == 0;
      const int blocks = a.kc * 8 / a.span;
      bool stop = false;
      // waits for the next stage and arms it; false at an abort
      auto acquire = [&]() {
        if (it >= NS && !mbar_wait_bounded(&S.empty[st], ph, kConvLimitNs, abort)) {
          atomicExch(a.err, 1);
          *abort = 1;
          return false;
        }
        if (stall && it >= NS) return false;  // stop issuing: the MMA thread's wait runs out
        fence_proxy_async();
        mbar_expect_tx(&S.full[st], lay.a_bytes + lay.b_bytes);
        return true;
      };
      auto advance = [&]() {
        ++it;
        if (++st == NS) {
          st = 0;
          ph ^= 1u;
        }
      };
      for (int t = blockIdx.x; t < ntiles && !stop && !*abort; t += gridDim.x) {
        const int tx = t % a.ntx, r = t / a.ntx, ty = r % a.nty, tz = r / a.nty;
        const int x0 = tx * a.bx, y0 = ty * a.by, z0 = tz * a.bz;
        if (a.halo) {
          for (int u = 0; u < units && !stop; ++u) {
            if ((stop = !acquire())) break;
            // the group's rows of 128 output voxels with a one-voxel halo in
            // x, y and z, 16 input channels: every tap is a view of it
            tma_load_5d(stage_a + st * lay.a_stride, &map, 0, x0 - 1, y0 - 1, z0 - 1, u, &S.full[st]);
            advance();
          }
        } else {
          const __nv_bfloat16* w = a.w;
#pragma unroll 1
          for (int dz = -1; dz < 2 && !stop; ++dz)
#pragma unroll 1
            for (int dy = -1; dy < 2 && !stop; ++dy)
#pragma unroll 1
              for (int dx = -1; dx < 2 && !stop; ++dx)
#pragma unroll 1
                for (int q = 0; q < upt; ++q) {
                  if ((stop = !acquire())) break;
                  tma_load_5d(stage_a + st * lay.a_stride, &map, 0, x0 + dx, y0 + dy, z0 + dz, q * blocks, &S.full[st]);
                  if (lay.b_bytes) bulk_load(stage_b + st * lay.b_bytes, w, lay.b_bytes, &S.full[st]);
                  w += (size_t)a.kc * a.cout * 8;
                  advance();
                }
        }
      }
      // at an abort, let the copies still in flight land before the CTA exits
      if (*abort) {
        __threadfence_block();
        for (int j = S.consumed; j < it; ++j) mbar_wait_bounded(&S.full[j % NS], (j / NS) & 1, kConvLimitNs);
        if (lay.w_bytes) mbar_wait_bounded(&S.wbar, 0, kConvLimitNs);
      }
    }
  } else if (warp == 1) {
    if (lane == 0) {
      // ---- MMAs ----
      // One thread issues them all, so whatever it computes per MMA bounds
      // the kernel (divisions per tap and whole descriptors: 2800 cycles per
      // tile of a 16 -> 16 layer): the taps of a group of four are unrolled
      // and descriptors advance by additions to their lower word.
      const uint32_t idesc = idesc_bf16_f32(kConvTileM, a.cout);
      const uint32_t wchunk = (uint32_t)a.cout * 16u;  // bytes of one 8-channel chunk of one tap's weights
      const uint32_t wtap = (uint32_t)(a.cin / 8) * wchunk >> 4;  // one tap's weights, in descriptor units of 16 bytes
      const int ksteps = a.kc / 2;
      // a tile's 128 rows of a block are 256 * span bytes, the tiles' of one
      // block follow each other; 16 channels on are 32 bytes within the rows,
      // or the next block
      const uint32_t tstep = 16u * (uint32_t)a.span;
      const uint32_t bstep = a.span == 16 ? (uint32_t)G * 256u : 2u;
      const uint64_t adesc = smem_desc_swizzled(stage_a, 2 * a.span);
      const uint64_t wdesc = smem_desc_kmajor(lay.w_bytes ? wres : stage_b, wchunk, 128);
      const uint32_t ahi = (uint32_t)(adesc >> 32), bhi = (uint32_t)(wdesc >> 32);
      const uint32_t arow = (uint32_t)(G + 2) * 260u;  // halo path: one plane of the box
      int it = 0, st = 0, tc = 0;
      uint32_t ph = 0;
      bool issued = false;
      if (lay.w_bytes && !mbar_wait_bounded(&S.wbar, 0, kConvLimitNs, abort)) {
        atomicExch(a.err, 1);
        *abort = 1;
      }
      for (int t = blockIdx.x; t < ntiles && !*abort; t += gridDim.x, ++tc) {
        const int b = tc & 1, n = tc >> 1;
        if (n > 0 && !mbar_wait_bounded(&S.acce[b], (n - 1) & 1, kConvLimitNs, abort)) {
          atomicExch(a.err, 1);
          *abort = 1;
          break;
        }
        tc_fence_after();
        const uint32_t d = tmem + (uint32_t)(b * G) * acc_cols;
        uint32_t wlo = (uint32_t)wdesc;  // resident weights: the unit's, in copy order
        bool ok = true;
        for (int u = 0; u < units; ++u) {
          if (!mbar_wait_bounded(&S.full[st], ph, kConvLimitNs, abort)) {
            atomicExch(a.err, 1);
            *abort = 1;
            ok = false;
            break;
          }
          S.consumed = it + 1;
          tc_fence_after();
          const uint32_t alo = (uint32_t)adesc + (uint32_t)st * (lay.a_stride >> 4);
          if (a.halo) {
            // channels 16u .. 16u + 15 of the 27 taps: a tile's 128 rows
            // start (dz, tile + dy, dx) rows of 32 bytes into the halo box
            uint32_t blo = wlo + (uint32_t)(2 * u) * (wchunk >> 4);
            uint32_t acc = u > 0 ? 1u : 0u;
            uint32_t plane = alo;
#pragma unroll 1
            for (int dz = 0; dz < 3; ++dz, plane += arow) {
              if (G == 4) {
#pragma unroll
                for (int dy = 0; dy < 3; ++dy)
#pragma unroll
                  for (int dx = 0; dx < 3; ++dx) {
#pragma unroll
                    for (int g = 0; g < 4; ++g)
                      tc_mma_f16_words(d + (uint32_t)g * acc_cols, plane + (uint32_t)((g + dy) * 260 + dx * 2), ahi, blo,
                                       bhi, idesc, acc);
                    acc = 1u;
                    blo += wtap;
                  }
              } else {
#pragma unroll 1
                for (int dy = 0; dy < 3; ++dy)
#pragma unroll 1
                  for (int dx = 0; dx < 3; ++dx) {
#pragma unroll 1
                    for (int g = 0; g < G; ++g)
                      tc_mma_f16_words(d + (uint32_t)g * acc_cols, plane + (uint32_t)((g + dy) * 260 + dx * 2), ahi, blo,
                                       bhi, idesc, acc);
                    acc = 1u;
                    blo += wtap;
                  }
              }
            }
          } else {
            uint32_t blo = lay.w_bytes ? wlo : (uint32_t)wdesc + (uint32_t)st * (lay.b_bytes >> 4);
#pragma unroll 1
            for (int ks = 0; ks < ksteps; ++ks) {
              const uint32_t al = alo + (uint32_t)ks * bstep;
              const uint32_t acc = (u > 0 || ks > 0) ? 1u : 0u;
              tc_mma_f16_words(d, al, ahi, blo, bhi, idesc, acc);
              if (G > 1) tc_mma_f16_words(d + acc_cols, al + tstep, ahi, blo, bhi, idesc, acc);
              if (G > 2) {
                tc_mma_f16_words(d + 2 * acc_cols, al + 2 * tstep, ahi, blo, bhi, idesc, acc);
                tc_mma_f16_words(d + 3 * acc_cols, al + 3 * tstep, ahi, blo, bhi, idesc, acc);
              }
              blo += 2u * wchunk >> 4;
            }
            wlo += (uint32_t)a.kc * (wchunk >> 4);
          }
          tc_commit(&S.empty[st]);
          issued = true;
          ++it;
          if (++st == NS) {
            st = 0;
            ph ^= 1u;
          }
        }
        if (!ok) break;
        tc_commit(&S.accf[b]);
      }
      // at an abort, wait for the MMAs in flight before TMEM is released
      if (*abort && issued) {
        for (int j = (it > NS ? it - NS : 0); j < it; ++j)
          mbar_wait_bounded(&S.empty[j % NS], (j / NS) & 1, kConvLimitNs);
      }
    }
  } else {
    // ---- epilogue: warps 2..5 own TMEM lane quarters 2, 3, 0, 1 ----
    const int q = warp & 3;
    const int lbx = __ffs(a.bx) - 1, lby = __ffs(a.by) - 1;
    int tc = 0;
    for (int t = blockIdx.x; t < ntiles; t += gridDim.x, ++tc) {
      const int b = tc & 1, n = tc >> 1;
      // lane 0 waits and the warp follows its verdict, so that the
      // warp-collective TMEM loads below run in every lane or in none
      int ok = 1;
      if (lane == 0) ok = mbar_wait_bounded(&S.accf[b], n & 1, kConvLimitNs, abort) ? 1 : 0;
      ok = __shfl_sync(0xffffffffu, ok, 0);
      if (!ok) {
        if (lane == 0) {
          if (!*abort) atomicExch(a.err, 1);
          *abort = 1;
        }
        break;
      }
      __syncwarp();
      tc_fence_after();
      const int tx = t % a.ntx, r = t / a.ntx, ty = r % a.nty, tz = r / a.nty;
      for (int gc = 0; gc < G * a.cout; gc += 16) {
        const int g = gc / a.cout, c0 = gc - g * a.cout;
        const int m = g * kConvTileM + 32 * q + lane;  // the boxes' sides are powers of two
        const int mx = m & (a.bx - 1), mr = m >> lbx;
        const int x = tx * a.bx + mx, y = ty * a.by + (mr & (a.by - 1)), z = tz * a.bz + (mr >> lby);
        const bool in = x < a.W && y < a.H && z < a.D;
        const size_t v = ((size_t)z * a.H + y) * a.W + x;
        float val[16];
        tmem_ld16(tmem + ((uint32_t)(32 * q) << 16) + (uint32_t)(b * G) * acc_cols + (uint32_t)gc, val);
        if (!in) continue;
#pragma unroll
        for (int i = 0; i < 16; ++i) {
          float f = val[i];
          if (a.bias) f += bias_s[c0 + i];
          if (a.relu) f = fmaxf(f, 0.0f);
          val[i] = f;
        }
        if (a.mask) {  // 16 channels of a voxel: 32 aligned bytes
          const uint4* mk = reinterpret_cast<const uint4*>(a.mask + v * a.mask_stride + a.mask_off + c0);
          const uint4 m0 = mk[0], m1 = mk[1];
          const uint32_t mw[8] = {m0.x, m0.y, m0.z, m0.w, m1.x, m1.y, m1.z, m1.w};
#pragma unroll
          for (int i = 0; i < 16; ++i) {
            // BF16 > 0: the value's bits as an FP32's upper half
            const uint32_t hb = (i & 1) ? mw[i >> 1] & 0xffff0000u : mw[i >> 1] << 16;
            if (!(__uint_as_float(hb) > 0.0f)) val[i] = 0.0f;
          }
        }
        if (a.out_f32) {
          float* o = a.out_f32 + v * a.cout + c0;
#pragma unroll
          for (int i = 0; i < 16; ++i) o[i] = val[i];
        }
        __align__(16) __nv_bfloat16 h[16];
#pragma unroll
        for (int i = 0; i < 16; ++i) h[i] = __float2bfloat16_rn(val[i]);
        uint4* dst = reinterpret_cast<uint4*>(a.out + v * a.out_stride + a.out_off + c0);
        dst[0] = reinterpret_cast<const uint4*>(h)[0];
        dst[1] = reinterpret_cast<const uint4*>(h)[1];
      }
      tc_fence_before();
      mbar_arrive(&S.acce[b]);
    }
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (warp == 1) tmem_dealloc(tmem, tcols);
}

__global__ void pack_weights_kernel(const float* __restrict__ w, int cout, int cin, int cin_pad, int backward,
                                    __nv_bfloat16* __restrict__ out) {
  const long long n = 27LL * cout * cin_pad;
  for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < n; e += (long long)gridDim.x * blockDim.x) {
    // forward: e enumerates [tap][cin_pad / 8][cout][8]
    // backward: [tap][cout / 8][cin_pad][8] (rows = forward input channels)
    const int j = (int)(e % 8);
    long long r = e / 8;
    int tap, kc, row;
    if (!backward) {
      row = (int)(r % cout);
      r /= cout;
      kc = (int)(r % (cin_pad / 8));
      tap = (int)(r / (cin_pad / 8));
      const int o = row, i = kc * 8 + j;
      out[e] = __float2bfloat16_rn(i < cin ? w[((size_t)o * cin + i) * 27 + tap] : 0.0f);
    } else {
      row = (int)(r % cin_pad);
      r /= cin_pad;
      kc = (int)(r % (cout / 8));
      tap = (int)(r / (cout / 8));
      const int i = row, o = kc * 8 + j;
      out[e] = __float2bfloat16_rn(i < cin ? w[((size_t)o * cin + i) * 27 + (26 - tap)] : 0.0f);
    }
  }
}

}  // namespace

cudaError_t init_conv_kernel(size_t smem_bytes) {
  return cudaFuncSetAttribute(conv_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem_bytes);
}

// Powers of two with bx * by * bz = voxels exactly (the copy of a box must
// deliver the rows the MMAs and the barrier's byte count expect; rows beyond
// the grid read 0 and are not stored).
void conv_tile_box(int W, int H, int D, int voxels, int* bx, int* by, int* bz) {
  auto pow2_at_most = [](int n, int cap) {
    int p = 1;
    while (2 * p <= n && 2 * p <= cap) p *= 2;
    return p;
  };
  *bx = pow2_at_most(W, 128);
  *by = pow2_at_most(H, voxels / *bx);
  *bz = voxels / (*bx * *by);
  (void)D;
}

namespace {
PFN_cuTensorMapEncodeTiled_v12000 conv_encode_fn() {
  static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
  if (!fn) {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) == cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = (PFN_cuTensorMapEncodeTiled_v12000)p;
  }
  return fn;
}
}  // namespace

bool make_conv_input_map(CUtensorMap* map, const __nv_bfloat16* x, int W, int H, int D, int cin, int span, int bx,
                         int by, int bz, int blocks) {
  PFN_cuTensorMapEncodeTiled_v12000 fn = conv_encode_fn();
  if (!fn) return false;
  const cuuint64_t dims[5] = {(cuuint64_t)span, (cuuint64_t)W, (cuuint64_t)H, (cuuint64_t)D, (cuuint64_t)(cin / span)};
  const cuuint64_t strides[4] = {(cuuint64_t)cin * 2, (cuuint64_t)W * cin * 2, (cuuint64_t)H * W * cin * 2,
                                 (cuuint64_t)span * 2};
  const cuuint32_t box[5] = {(cuuint32_t)span, (cuuint32_t)bx, (cuuint32_t)by, (cuuint32_t)bz, (cuuint32_t)blocks};
  const CUtensorMapSwizzle sw = span == 64   ? CU_TENSOR_MAP_SWIZZLE_128B
                                : span == 32 ? CU_TENSOR_MAP_SWIZZLE_64B
                                             : CU_TENSOR_MAP_SWIZZLE_32B;
  const cuuint32_t estr[5] = {1, 1, 1, 1, 1};
  return fn(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 5, (void*)x, dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
            sw, CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) ==
         CUDA_SUCCESS;
}

bool make_conv_map(CUtensorMap* map, const __nv_bfloat16* x, const ConvArgs& a) {
  if (a.halo) return make_conv_input_map(map, x, a.W, a.H, a.D, a.cin, 16, 130, a.group + 2, 3, 1);
  return make_conv_input_map(map, x, a.W, a.H, a.D, a.cin, a.span, a.bx, a.by, a.bz, a.kc * 8 / a.span);
}

int conv_grid(const ConvArgs& a, size_t smem_bytes) {
  int per_sm = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, conv_kernel, kConvThreads, smem_bytes) != cudaSuccess ||
      per_sm < 1) {
    (void)cudaGetLastError();
    per_sm = 1;
  }
  const int by_tmem = (int)(512 / conv_tmem_cols(a.group, a.cout));
  if (per_sm > by_tmem) per_sm = by_tmem;
  const int tiles = a.ntx * a.nty * a.ntz;
  const int g = per_sm * device_sms();
  return tiles < g ? tiles : g;
}

cudaError_t launch_conv(const CUtensorMap& map, const ConvArgs& a, int grid, cudaStream_t s) {
  count_launch();
  conv_kernel<<<grid, kConvThreads, conv_smem_bytes(a), s>>>(map, a);
  return cudaGetLastError();
}

cudaError_t launch_pack_weights(const float* w, int cout, int cin, int cin_pad, bool backward, __nv_bfloat16* out,
                                cudaStream_t s) {
  const long long n = 27LL * cout * cin_pad;
  long long blocks = (n + 255) / 256;
  if (blocks > 4096) blocks = 4096;
  count_launch();
  pack_weights_kernel<<<(int)blocks, 256, 0, s>>>(w, cout, cin, cin_pad, backward ? 1 : 0, out);
  return cudaGetLastError();
}

}  // namespace gbmg

// ---------------------------------------------------------------------------
// Element-wise kernels of the network (channels-last BF16 tensors)
// ---------------------------------------------------------------------------

namespace gbmg {

namespace {

// x[c][z][y][x] (FP32, natural layout, c < 3) -> X0[v][16] BF16 (channels 3..15 zero)
__global__ void input_to_bf16_kernel(const float* __restrict__ x, long long V, __nv_bfloat16* __restrict__ out) {
  for (long long v = blockIdx.x * (long long)blockDim.x + threadIdx.x; v < V; v += (long long)gridDim.x * blockDim.x) {
    __align__(16) __nv_bfloat16 h[16];
#pragma unroll
    for (int c = 0; c < 16; ++c) h[c] = __float2bfloat16_rn(c < 3 ? x[c * V + v] : 0.0f);
    uint4* d = reinterpret_cast<uint4*>(out + v * 16);
    d[0] = reinterpret_cast<const uint4*>(h)[0];
    d[1] = reinterpret_cast<const uint4*>(h)[1];
  }
}

// The kernels below take 8 channels (16 bytes) of a voxel per thread; those on
// two grid levels take a row (y, z) per block round, so a thread's place costs
// one 32-bit division (with a 64-bit division per channel they took 2 to 7
// times the time of their bytes).
__device__ __forceinline__ void unpack8(const uint4& r, float* f) {
  const uint32_t w[4] = {r.x, r.y, r.z, r.w};
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    f[2 * i] = __uint_as_float(w[i] << 16);
    f[2 * i + 1] = __uint_as_float(w[i] & 0xffff0000u);
  }
}

__device__ __forceinline__ uint4 pack8(const float* f) {
  __align__(16) __nv_bfloat16 o[8];
#pragma unroll
  for (int i = 0; i < 8; ++i) o[i] = __float2bfloat16_rn(f[i]);
  return *reinterpret_cast<const uint4*>(o);
}

__device__ __forceinline__ uint4 load8(const __nv_bfloat16* p) { return *reinterpret_cast<const uint4*>(p); }

// Sum over the 8 children (2x, 2y, 2z) .. of 8 channels at channel offset
// `ch` of a tensor of twice the size, in the order z, y, x.
__device__ __forceinline__ void child_sum8(const __nv_bfloat16* __restrict__ src, int stride, int ch, int W, int H, int x,
                                           int y, int z, float* acc) {
  uint4 r[8];
#pragma unroll
  for (int k = 0; k < 8; ++k) {
    const long long vs = ((long long)(2 * z + (k >> 2)) * (2 * H) + (2 * y + ((k >> 1) & 1))) * (2 * W) + (2 * x + (k & 1));
    r[k] = load8(src + vs * stride + ch);
  }
#pragma unroll
  for (int i = 0; i < 8; ++i) acc[i] = 0.0f;
#pragma unroll
  for (int k = 0; k < 8; ++k) {
    float f[8];
    unpack8(r[k], f);
#pragma unroll
    for (int i = 0; i < 8; ++i) acc[i] += f[i];
  }
}

// 2x2x2 mean of src (level size 2W x 2H x 2D, channel stride ss, offset so)
// into dst (W x H x D, c channels, stride ds, offset do)
__global__ void avg_pool_kernel(const __nv_bfloat16* __restrict__ src, int ss, int so, int W, int H, int D, int c,
                                __nv_bfloat16* __restrict__ dst, int ds, int dofs) {
  const int G = c / 8;
  for (int row = blockIdx.x; row < H * D; row += gridDim.x) {
    const int z = row / H, y = row - z * H;
    for (int e = threadIdx.x; e < W * G; e += blockDim.x) {
      const int x = e / G, g = e - x * G;
      float acc[8];
      child_sum8(src, ss, so + 8 * g, W, H, x, y, z, acc);
#pragma unroll
      for (int i = 0; i < 8; ++i) acc[i] *= 0.125f;
      *reinterpret_cast<uint4*>(dst + ((long long)row * W + x) * ds + dofs + 8 * g) = pack8(acc);
    }
  }
}

// nearest-neighbour upsampling by 2 of src (W x H x D, c channels, stride ss,
// offset so) into dst (2W x 2H x 2D, stride ds, offset do); a block round per
// output row
__global__ void upsample_kernel(const __nv_bfloat16* __restrict__ src, int ss, int so, int W, int H, int D, int c,
                                __nv_bfloat16* __restrict__ dst, int ds, int dofs) {
  const int G = c / 8;
  for (int row = blockIdx.x; row < 4 * H * D; row += gridDim.x) {
    const int z = row / (2 * H), y = row - z * (2 * H);
    const __nv_bfloat16* s = src + ((long long)(z >> 1) * H + (y >> 1)) * W * ss + so;
    __nv_bfloat16* o = dst + (long long)row * (2 * W) * ds + dofs;
    for (int e = threadIdx.x; e < W * G; e += blockDim.x) {
      const int x = e / G, g = e - x * G;
      const uint4 v = load8(s + (long long)x * ss + 8 * g);
      *reinterpret_cast<uint4*>(o + (long long)(2 * x) * ds + 8 * g) = v;
      *reinterpret_cast<uint4*>(o + (long long)(2 * x + 1) * ds + 8 * g) = v;
    }
  }
}

// the head: pred[v] = (b + sum_i w[i] u[v][i]) * (active ? 1 : 0), FP32;
// active from the input's mask channel (channel 1 of X0 > 0)
__global__ void head_kernel(const __nv_bfloat16* __restrict__ u, int c, const float* __restrict__ w,
                            const float* __restrict__ b, const __nv_bfloat16* __restrict__ x0, long long V,
                            float* __restrict__ pred) {
  __shared__ float ws[128];
  for (int i = threadIdx.x; i < c; i += blockDim.x) ws[i] = w[i];
  __syncthreads();
  for (long long v = blockIdx.x * (long long)blockDim.x + threadIdx.x; v < V; v += (long long)gridDim.x * blockDim.x) {
    const uint32_t m = *reinterpret_cast<const uint32_t*>(x0 + v * 16);  // channels 0 and 1
    float acc = b[0];
    for (int i = 0; i < c; i += 8) {
      float f[8];
      unpack8(load8(u + v * c + i), f);
#pragma unroll
      for (int k = 0; k < 8; ++k) acc = fmaf(ws[i + k], f[k], acc);
    }
    pred[v] = __uint_as_float(m & 0xffff0000u) > 0.0f ? acc : 0.0f;
  }
}

// channels [off, off + c) of a channels-last tensor -> FP32 natural [c][V]
__global__ void tensor_to_natural_kernel(const __nv_bfloat16* __restrict__ t, int stride, int off, int c, long long V,
                                         float* __restrict__ out) {
  const long long n = (long long)c * V;
  for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < n; e += (long long)gridDim.x * blockDim.x) {
    const int ch = (int)(e / V);
    const long long v = e - (long long)ch * V;
    out[e] = __bfloat162float(t[v * stride + off + ch]);
  }
}

int ew_grid(long long n) {
  long long b = (n + 255) / 256;
  const long long cap = 32LL * device_sms();
  if (b > cap) b = cap;
  return b < 1 ? 1 : (int)b;
}

// blocks of a kernel that takes a row per block round
int row_grid(long long rows) {
  const long long cap = 16LL * device_sms();
  return rows > cap ? (int)cap : (rows < 1 ? 1 : (int)rows);
}

}  // namespace

cudaError_t launch_input_to_bf16(const float* x, long long V, __nv_bfloat16* out, cudaStream_t s) {
  count_launch();
  input_to_bf16_kernel<<<ew_grid(V), 256, 0, s>>>(x, V, out);
  return cudaGetLastError();
}

cudaError_t launch_avg_pool(const __nv_bfloat16* src, int ss, int so, int W, int H, int D, int c, __nv_bfloat16* dst,
                            int ds, int dofs, cudaStream_t s) {
  count_launch();
  avg_pool_kernel<<<row_grid((long long)H * D), 256, 0, s>>>(src, ss, so, W, H, D, c, dst, ds, dofs);
  return cudaGetLastError();
}

cudaError_t launch_upsample(const __nv_bfloat16* src, int ss, int so, int W, int H, int D, int c, __nv_bfloat16* dst,
                            int ds, int dofs, cudaStream_t s) {
  count_launch();
  upsample_kernel<<<row_grid(4LL * H * D), 256, 0, s>>>(src, ss, so, W, H, D, c, dst, ds, dofs);
  return cudaGetLastError();
}

cudaError_t launch_head(const __nv_bfloat16* u, int c, const float* w, const float* b, const __nv_bfloat16* x0,
                        long long V, float* pred, cudaStream_t s) {
  count_launch();
  head_kernel<<<ew_grid(V), 256, 0, s>>>(u, c, w, b, x0, V, pred);
  return cudaGetLastError();
}

cudaError_t launch_tensor_to_natural(const __nv_bfloat16* t, int stride, int off, int c, long long V, float* out,
                                     cudaStream_t s) {
  count_launch();
  tensor_to_natural_kernel<<<ew_grid((long long)c * V), 256, 0, s>>>(t, stride, off, c, V, out);
  return cudaGetLastError();
}

}  // namespace gbmg

// ---------------------------------------------------------------------------
// Backward pass: weight gradients on the tensor cores, and the element-wise
// and reduction kernels
// ---------------------------------------------------------------------------
//
// Weight gradient of a convolution: dW[o][i][tap] = sum over voxels v of
// g[v][o] x[v + offset(tap)][i], with g the gradient of the pre-activation
// and x the layer's input (zero outside the grid).  As a GEMM: rows (tap, i)
// of the tap-major row space (27 x cin rows), columns o, K = the voxels, in
// tiles of 128.  Both operands are MN-major as the channels-last tensors lie in
// shared memory after a TMA copy: rows (voxels) of span channels, swizzled.
// The FP32 accumulators stay in TMEM over the CTA's range of tiles and are
// written once as its partial sums; a second kernel adds the partials in a
// fixed order.
//
// What bounds it is L2 (every tap reads the input again: 1.8 GB for the
// 16 -> 16 layer at 128^3) and the one thread that issues the copies (16
// copies of 16-byte rows with a division each took 570 us for that layer).
//  - Tap tiles (grids narrower than 128): a CTA takes 128 rows: 128 / span
//    copies per tile, one per (tap, block of span channels), from a table.
//  - Halo rows (a tile is one row of 128 voxels): one copy per tile and 16
//    channels of the box (130 x 3 x 3) around it, 9 reads of the input
//    instead of 27.  The nine (dz, dy) rows of the box are 130 rows of 32
//    bytes apart, so for each dx one operand of M = 128 takes eight of them as
//    its blocks of 16 channels; the ninth row's three dx, 32 bytes apart, are
//    a fourth operand (its other five blocks read what follows and are not
//    used).  A CTA takes the four operands of one block of 16 channels, or two
//    of them (dx 0 and 1, or dx 2 and the ninth row) while that leaves every
//    CTA an SM of its own.
// The split over ranges of tiles follows the tap tiles' count of CTAs on both
// paths: the tensor cores truncate as they accumulate, so sums over other
// ranges would differ by more (6e-5) than the gradients' own precision.

namespace gbmg {

namespace {

constexpr int kWgStages = 3;
constexpr unsigned kWgHaloBytes = 9u * 130u * 32u;

struct WgSmemHeader {
  unsigned long long full[kWgStages];
  unsigned long long empty[kWgStages];
  unsigned long long accf;
  uint32_t tmem;
  int abort;
  int consumed;
  int4 box[8];  // tap tiles: dx, dy, dz and channel block of every copy
};

// bytes of one stage's input (a multiple of 1024; on the halo path with room
// for the unused blocks' reads) and gradient
__host__ __device__ unsigned wg_a_bytes(const WgradArgs& a) {
  return a.halo ? (kWgHaloBytes + 8u * 32u + 1023u) / 1024u * 1024u : 128u * 256u;
}
__host__ __device__ unsigned wg_b_bytes(const WgradArgs& a) { return (unsigned)a.cout * 256u; }

__host__ __device__ uint32_t wg_tmem_cols(const WgradArgs& a) {
  const int c = a.cout * (a.halo ? 4 / a.halves : 1);
  return c <= 32 ? 32u : (c <= 64 ? 64u : (c <= 128 ? 128u : (c <= 256 ? 256u : 512u)));
}

__global__ void __launch_bounds__(kConvThreads, 1)
    wgrad_kernel(const __grid_constant__ CUtensorMap map_x, const __grid_constant__ CUtensorMap map_g, WgradArgs a) {
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  WgSmemHeader& S = *reinterpret_cast<WgSmemHeader*>(smem_raw);
  const unsigned a_bytes = wg_a_bytes(a), b_bytes = wg_b_bytes(a);
  constexpr int NS = kWgStages;
  unsigned char* stage_a = smem_raw + 1024;
  unsigned char* stage_b = stage_a + NS * a_bytes;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int mb = blockIdx.x % a.nmblk, sp = blockIdx.x / a.nmblk;
  const int T = a.ntx * a.nty * a.ntz;
  const int t_lo = (int)((long long)T * sp / a.nsplit), t_hi = (int)((long long)T * (sp + 1) / a.nsplit);
  const uint32_t tcols = wg_tmem_cols(a);
  const int copies = a.halo ? 1 : 128 / a.span;  // input copies per stage
  // halo path: the CTA's 16 channels and its first and number of operands
  const int hu = mb / a.halves, op0 = a.halves == 2 ? 2 * (mb & 1) : 0, nop = 4 / a.halves;
  if (threadIdx.x == 0) {
    for (int i = 0; i < NS; ++i) {
      mbar_init(&S.full[i], 1);
      mbar_init(&S.empty[i], 1);
    }
    mbar_init(&S.accf, 1);
    S.abort = 0;
    S.consumed = 0;
    mbar_init_fence();
  }
  if (!a.halo && threadIdx.x >= 32 && threadIdx.x < 40) {
    const int blocks = a.cin / a.span;
    int R = mb * copies + (int)threadIdx.x - 32;
    if (R >= 27 * blocks) R = 27 * blocks - 1;  // padding rows: any valid block (their sums are not used)
    const int tap = R / blocks;
    S.box[threadIdx.x - 32] = make_int4(tap % 3 - 1, (tap / 3) % 3 - 1, tap / 9 - 1, R % blocks);
  }
  if (a.halo && warp >= 2) {
    // the rows after a halo box are read into unused accumulator rows: finite
    for (int s = 0; s < NS; ++s)
      for (unsigned o = kWgHaloBytes + 4u * (threadIdx.x - 64); o < a_bytes; o += 4u * 128u)
        *reinterpret_cast<uint32_t*>(stage_a + s * a_bytes + o) = 0u;
  }
  if (warp == 1) tmem_alloc(&S.tmem, tcols);
  tc_fence_before();
  fence_proxy_async();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = S.tmem;
  volatile int* abort = &S.abort;
  if (warp == 0) {
    if (lane == 0) {
      const unsigned x_bytes = a.halo ? kWgHaloBytes : a_bytes;
      int it = 0, st = 0;
      uint32_t ph = 1;
      bool stop = false;
      for (int t = t_lo; t < t_hi && !stop; ++t) {
        const int tx = t % a.ntx, r = t / a.ntx, ty = r % a.nty, tz = r / a.nty;
        const int x0 = tx * a.bx, y0 = ty * a.by, z0 = tz * a.bz;
        if (it >= NS && !mbar_wait_bounded(&S.empty[st], ph, kConvLimitNs, abort)) {
          atomicExch(a.err, 1);
          *abort = 1;
          stop = true;
          break;
        }
        mbar_expect_tx(&S.full[st], x_bytes + b_bytes);
        unsigned char* A = stage_a + st * a_bytes;
        if (a.halo) {
          tma_load_5d(A, &map_x, 0, x0 - 1, y0 - 1, z0 - 1, hu, &S.full[st]);
        } else {
#pragma unroll 1
          for (int g = 0; g < copies; ++g) {
            const int4 c = S.box[g];
            tma_load_5d(A + g * 256 * a.span, &map_x, 0, x0 + c.x, y0 + c.y, z0 + c.z, c.w, &S.full[st]);
          }
        }
        tma_load_5d(stage_b + st * b_bytes, &map_g, 0, x0, y0, z0, 0, &S.full[st]);
        ++it;
        if (++st == NS) {
          st = 0;
          ph ^= 1u;
        }
      }
      if (*abort) {
        for (int j = S.consumed; j < it; ++j) mbar_wait_bounded(&S.full[j % NS], (j / NS) & 1, kConvLimitNs);
      }
    }
  } else if (warp == 1) {
    if (lane == 0) {
      const uint32_t idesc = idesc_bf16_f32(kConvTileM, a.cout, true);
      // input: eight blocks of 16 channels 130 rows apart (halo), or blocks
      // of span channels one after another; gradient: blocks of gspan channels
      const uint32_t xs = 2u * (uint32_t)(a.halo ? 16 : a.span), gs = 2u * (uint32_t)a.gspan;
      const uint64_t adesc = smem_desc_mn_swizzled(stage_a, xs, a.halo ? 130u * 32u : 128u * xs);
      const uint64_t adesc9 = smem_desc_mn_swizzled(stage_a, 32u, 32u);  // the ninth row's taps, one row apart
      const uint64_t bdesc = smem_desc_mn_swizzled(stage_b, gs, 128u * gs);
      const uint32_t ahi = (uint32_t)(adesc >> 32), ahi9 = (uint32_t)(adesc9 >> 32), bhi = (uint32_t)(bdesc >> 32);
      int it = 0, st = 0;
      uint32_t ph = 0;
      bool issued = false;
      for (int t = t_lo; t < t_hi && !*abort; ++t) {
        if (!mbar_wait_bounded(&S.full[st], ph, kConvLimitNs, abort)) {
          atomicExch(a.err, 1);
          *abort = 1;
          break;
        }
        S.consumed = it + 1;
        tc_fence_after();
        const uint32_t alo = (uint32_t)adesc + (uint32_t)st * (a_bytes >> 4);
        const uint32_t blo = (uint32_t)bdesc + (uint32_t)st * (b_bytes >> 4);
        const uint32_t acc0 = t > t_lo ? 1u : 0u;
        if (a.halo) {
          // operand dx (0 .. 2) starts dx rows on, operand 3 at the ninth row;
          // 16 voxels are 32 units of 16 bytes
          const uint32_t ninth = (uint32_t)adesc9 + (uint32_t)st * (a_bytes >> 4) + 8u * 130u * 2u;
          if (nop == 4) {
#pragma unroll
            for (int ks = 0; ks < 8; ++ks) {
              const uint32_t b = blo + (uint32_t)ks * gs;
              const uint32_t acc = ks > 0 ? 1u : acc0;
              tc_mma_f16_words(tmem, alo + (uint32_t)(ks * 32), ahi, b, bhi, idesc, acc);
              tc_mma_f16_words(tmem + (uint32_t)a.cout, alo + (uint32_t)(ks * 32 + 2), ahi, b, bhi, idesc, acc);
              tc_mma_f16_words(tmem + 2u * (uint32_t)a.cout, alo + (uint32_t)(ks * 32 + 4), ahi, b, bhi, idesc, acc);
              tc_mma_f16_words(tmem + 3u * (uint32_t)a.cout, ninth + (uint32_t)(ks * 32), ahi9, b, bhi, idesc, acc);
            }
          } else {
            const uint32_t a0 = alo + 2u * (uint32_t)op0;
            const uint32_t a1 = op0 == 2 ? ninth : alo + 2u;
            const uint32_t a1hi = op0 == 2 ? ahi9 : ahi;
#pragma unroll
            for (int ks = 0; ks < 8; ++ks) {
              const uint32_t b = blo + (uint32_t)ks * gs;
              const uint32_t acc = ks > 0 ? 1u : acc0;
              tc_mma_f16_words(tmem, a0 + (uint32_t)(ks * 32), ahi, b, bhi, idesc, acc);
              tc_mma_f16_words(tmem + (uint32_t)a.cout, a1 + (uint32_t)(ks * 32), a1hi, b, bhi, idesc, acc);
            }
          }
        } else {
#pragma unroll
          for (int ks = 0; ks < 8; ++ks)
            tc_mma_f16_words(tmem, alo + (uint32_t)ks * xs, ahi, blo + (uint32_t)ks * gs, bhi, idesc, ks > 0 ? 1u : acc0);
        }
        tc_commit(&S.empty[st]);
        issued = true;
        ++it;
        if (++st == NS) {
          st = 0;
          ph ^= 1u;
        }
      }
      if (!*abort) tc_commit(&S.accf);
      else if (issued)
        for (int j = (it > NS ? it - NS : 0); j < it; ++j)
          mbar_wait_bounded(&S.empty[j % NS], (j / NS) & 1, kConvLimitNs);
    }
  } else {
    const int q = warp & 3;
    int ok = 1;
    if (lane == 0) ok = mbar_wait_bounded(&S.accf, 0, 4 * kConvLimitNs, abort) ? 1 : 0;
    ok = __shfl_sync(0xffffffffu, ok, 0);
    if (ok) {
      __syncwarp();
      tc_fence_after();
      const int m = 32 * q + lane;
      const int nacc = a.halo ? nop : 1;
      for (int j = 0; j < nacc; ++j) {
        int row = mb * 128 + m;
        bool use = true;
        if (a.halo) {  // operand dx: block m / 16 is (dz, dy); operand 3: the ninth's dx
          const int k = op0 + j, blk = m >> 4;
          const int tap = k < 3 ? 3 * blk + k : 24 + blk;
          row = tap * a.cin + 16 * hu + (m & 15);
          use = k < 3 || blk < 3;
        }
        float* dst = a.partial + ((size_t)sp * a.rows + row) * a.cout;
        for (int c0 = 0; c0 < a.cout; c0 += 16) {
          float v[16];
          tmem_ld16(tmem + ((uint32_t)(32 * q) << 16) + (uint32_t)(j * a.cout + c0), v);
          if (!use) continue;
          float4* o = reinterpret_cast<float4*>(dst + c0);
#pragma unroll
          for (int i = 0; i < 4; ++i) o[i] = make_float4(v[4 * i], v[4 * i + 1], v[4 * i + 2], v[4 * i + 3]);
        }
      }
    } else if (lane == 0) {
      if (!*abort) atomicExch(a.err, 1);
      *abort = 1;
    }
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (warp == 1) tmem_dealloc(tmem, tcols);
}

// dW[o][i][tap] = sum over splits of partial[split][tap * cin_pad + i][o], in
// split order; i < cin (the real input channels); neighbouring threads take
// neighbouring o, the partials' fastest index.
__global__ void wgrad_reduce_kernel(const float* __restrict__ partial, int nsplit, int rows, int cin_pad, int cin,
                                    int cout, float* __restrict__ dw) {
  const int n = 27 * cin * cout;
  for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < n; e += gridDim.x * blockDim.x) {
    const int r = e / cout, o = e - r * cout;
    const int tap = r / cin, i = r - tap * cin;
    const float* p = partial + ((size_t)tap * cin_pad + i) * cout + o;
    float acc = 0.0f;
#pragma unroll 8
    for (int s = 0; s < nsplit; ++s) acc += p[(size_t)s * rows * cout];
    dw[((size_t)o * cin + i) * 27 + tap] = acc;
  }
}

// A block's threads of the per-channel sums below: every thread keeps one
// group of 8 channels, `lanes` voxels at a time.
struct ChannelLanes {
  int G, lanes, g, l;
  bool on;
};
__device__ __forceinline__ ChannelLanes channel_lanes(int c) {
  ChannelLanes x;
  x.G = c / 8;
  x.lanes = blockDim.x / x.G;
  x.l = threadIdx.x / x.G;
  x.g = threadIdx.x - x.l * x.G;
  x.on = x.l < x.lanes;
  return x;
}
// The threads' 8 sums each into out[c], in a fixed order.
__device__ __forceinline__ void channel_reduce(const ChannelLanes& x, const float* acc, int c, float (*sh)[9], float* out) {
#pragma unroll
  for (int i = 0; i < 8; ++i) sh[threadIdx.x][i] = acc[i];
  __syncthreads();
  for (int k = threadIdx.x; k < c; k += blockDim.x) {
    float s = 0.0f;
    for (int l = 0; l < x.lanes; ++l) s += sh[l * x.G + (k >> 3)][k & 7];
    out[k] = s;
  }
}

// Per-block partial sums over voxels of g[v][o] (bias gradient), one row of
// partials per block; then a fixed-order reduction.
__global__ void __launch_bounds__(256) channel_sum_kernel(const __nv_bfloat16* __restrict__ g, int c, long long V,
                                                          float* __restrict__ part) {
  __shared__ float sh[256][9];
  const ChannelLanes x = channel_lanes(c);
  float acc[8] = {0, 0, 0, 0, 0, 0, 0, 0};
  if (x.on) {
    const long long step = (long long)gridDim.x * x.lanes;
#pragma unroll 4
    for (long long v = (long long)blockIdx.x * x.lanes + x.l; v < V; v += step) {
      float f[8];
      unpack8(load8(g + v * c + 8 * x.g), f);
#pragma unroll
      for (int i = 0; i < 8; ++i) acc[i] += f[i];
    }
  }
  channel_reduce(x, acc, c, sh, part + (size_t)blockIdx.x * c);
}

// out[k] = sum of part[r][k] over the rows: 32 columns per block, 8 rows at a
// time.
__global__ void __launch_bounds__(256) partial_rows_sum_kernel(const float* __restrict__ part, int nrows, int c,
                                                               float* __restrict__ out) {
  __shared__ float sh[8][32];
  const int k = blockIdx.x * 32 + (threadIdx.x & 31), l = threadIdx.x >> 5;
  float acc = 0.0f;
  if (k < c) {
#pragma unroll 8
    for (int r = l; r < nrows; r += 8) acc += part[(size_t)r * c + k];
  }
  sh[l][threadIdx.x & 31] = acc;
  __syncthreads();
  if (l == 0 && k < c) {
    float s = 0.0f;
#pragma unroll
    for (int i = 0; i < 8; ++i) s += sh[i][threadIdx.x];
    out[k] = s;
  }
}

// Head backward.  g_pred (FP32, dL/dpred), act = input channel 1 > 0:
// gz[v][i] = (top[v][i] > 0) w[i] g act (BF16), and per-block partial sums
// of g act top[v][i] (head weights) and g act (head bias).
__global__ void __launch_bounds__(256)
    head_backward_kernel(const float* __restrict__ gp, const __nv_bfloat16* __restrict__ x0,
                         const __nv_bfloat16* __restrict__ top, int c, const float* __restrict__ w, long long V,
                         __nv_bfloat16* __restrict__ gz, float* __restrict__ part) {
  __shared__ float sh[256][9];
  __shared__ float bias[256];
  const ChannelLanes x = channel_lanes(c);
  float acc[8] = {0, 0, 0, 0, 0, 0, 0, 0}, acc_b = 0.0f;
  if (x.on) {
    float wv[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) wv[i] = w[8 * x.g + i];
    const long long step = (long long)gridDim.x * x.lanes;
#pragma unroll 2
    for (long long v = (long long)blockIdx.x * x.lanes + x.l; v < V; v += step) {
      const uint32_t m = *reinterpret_cast<const uint32_t*>(x0 + v * 16);  // channels 0 and 1
      const float g = __uint_as_float(m & 0xffff0000u) > 0.0f ? gp[v] : 0.0f;
      acc_b += g;
      float t[8], o[8];
      unpack8(load8(top + v * c + 8 * x.g), t);
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        acc[i] += g * t[i];
        o[i] = t[i] > 0.0f ? wv[i] * g : 0.0f;
      }
      *reinterpret_cast<uint4*>(gz + v * c + 8 * x.g) = pack8(o);
    }
  }
  bias[threadIdx.x] = x.on && x.g == 0 ? acc_b : 0.0f;
  channel_reduce(x, acc, c, sh, part + (size_t)blockIdx.x * (c + 1));
  if (threadIdx.x == 0) {
    float s = 0.0f;
    for (int l = 0; l < x.lanes; ++l) s += bias[l * x.G];
    part[(size_t)blockIdx.x * (c + 1) + c] = s;
  }
}

// Gradient through nearest upsampling: dst[v][i] = sum over the 8 children of
// src[child][so + i] (src at twice the size), FP32 sum rounded to BF16.
__global__ void upsample_backward_kernel(const __nv_bfloat16* __restrict__ src, int ss, int so, int W, int H, int D,
                                         int c, __nv_bfloat16* __restrict__ dst) {
  const int G = c / 8;
  for (int row = blockIdx.x; row < H * D; row += gridDim.x) {
    const int z = row / H, y = row - z * H;
    for (int e = threadIdx.x; e < W * G; e += blockDim.x) {
      const int x = e / G, g = e - x * G;
      float acc[8];
      child_sum8(src, ss, so + 8 * g, W, H, x, y, z, acc);
      *reinterpret_cast<uint4*>(dst + ((long long)row * W + x) * c + 8 * g) = pack8(acc);
    }
  }
}

// Gradient of a down level's second convolution output that feeds both the
// concatenation (skip, already masked) and the pooling of the level below:
// gz[v][i] = skip[v][i] + (act[v][i] > 0) gpool[parent][i] / 8.
__global__ void skip_pool_combine_kernel(const __nv_bfloat16* __restrict__ skip, int ss,
                                         const __nv_bfloat16* __restrict__ act, int as,
                                         const __nv_bfloat16* __restrict__ gpool, int W, int H, int D, int c,
                                         __nv_bfloat16* __restrict__ gz) {
  const int G = c / 8;
  for (int row = blockIdx.x; row < H * D; row += gridDim.x) {
    const int z = row / H, y = row - z * H;
    const long long prow = ((long long)(z >> 1) * (H / 2) + (y >> 1)) * (W / 2);
    for (int e = threadIdx.x; e < W * G; e += blockDim.x) {
      const int x = e / G, g = e - x * G;
      const long long v = (long long)row * W + x;
      float a[8], p[8], k[8];
      unpack8(load8(act + v * as + 8 * g), a);
      unpack8(load8(gpool + (prow + (x >> 1)) * c + 8 * g), p);
      unpack8(load8(skip + v * ss + 8 * g), k);
#pragma unroll
      for (int i = 0; i < 8; ++i) k[i] += a[i] > 0.0f ? 0.125f * p[i] : 0.0f;
      *reinterpret_cast<uint4*>(gz + v * c + 8 * g) = pack8(k);
    }
  }
}

// Loss and its gradient (relative squared error over the active cells):
// per-block partials of sum act y^2 and sum act (p - y)^2 ...
__global__ void loss_partials_kernel(const float* __restrict__ p, const float* __restrict__ y,
                                     const __nv_bfloat16* __restrict__ x0, long long V, double* __restrict__ part) {
  double den = 0.0, num = 0.0;
  for (long long v = blockIdx.x * (long long)blockDim.x + threadIdx.x; v < V; v += (long long)gridDim.x * blockDim.x) {
    if (!(__bfloat162float(x0[v * 16 + 1]) > 0.0f)) continue;
    const double yy = y[v], d = (double)p[v] - yy;
    den += yy * yy;
    num += d * d;
  }
  __shared__ double sd[256], sn[256];
  sd[threadIdx.x] = den;
  sn[threadIdx.x] = num;
  __syncthreads();
  for (int w = blockDim.x / 2; w > 0; w >>= 1) {
    if ((int)threadIdx.x < w) {
      sd[threadIdx.x] += sd[threadIdx.x + w];
      sn[threadIdx.x] += sn[threadIdx.x + w];
    }
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    part[2 * blockIdx.x] = sd[0];
    part[2 * blockIdx.x + 1] = sn[0];
  }
}

// ... summed in a fixed order: out[0] = den, out[1] = num
__global__ void loss_finalize_kernel(const double* __restrict__ part, int nblocks, double* __restrict__ out) {
  if (threadIdx.x == 0 && blockIdx.x == 0) {
    double d = 0.0, n = 0.0;
    for (int b = 0; b < nblocks; ++b) {
      d += part[2 * b];
      n += part[2 * b + 1];
    }
    out[0] = d;
    out[1] = n;
  }
}

// g[v] = 2 act (p - y) / den
__global__ void loss_grad_kernel(const float* __restrict__ p, const float* __restrict__ y,
                                 const __nv_bfloat16* __restrict__ x0, long long V, const double* __restrict__ sums,
                                 float* __restrict__ g) {
  const double den = sums[0];
  for (long long v = blockIdx.x * (long long)blockDim.x + threadIdx.x; v < V; v += (long long)gridDim.x * blockDim.x) {
    const bool act = __bfloat162float(x0[v * 16 + 1]) > 0.0f;
    g[v] = act && den > 0.0 ? (float)(2.0 * ((double)p[v] - (double)y[v]) / den) : 0.0f;
  }
}

// Adam (Kingma & Ba, Algorithm 1) on the flat FP32 parameters; bc1 = 1 -
// beta1^t, bc2 = 1 - beta2^t.
__global__ void adam_kernel(float* __restrict__ p, const float* __restrict__ g, float* __restrict__ m,
                            float* __restrict__ v, long long n, float lr, float b1, float b2, float eps, float bc1,
                            float bc2) {
  for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < n; e += (long long)gridDim.x * blockDim.x) {
    const float gg = g[e];
    const float mm = b1 * m[e] + (1.0f - b1) * gg;
    const float vv = b2 * v[e] + (1.0f - b2) * gg * gg;
    m[e] = mm;
    v[e] = vv;
    p[e] -= lr * (mm / bc1) / (sqrtf(vv / bc2) + eps);
  }
}

}  // namespace

size_t wgrad_smem_bytes(const WgradArgs& a) {
  return 1024 + (size_t)kWgStages * (wg_a_bytes(a) + wg_b_bytes(a));
}

void wgrad_plan(WgradArgs& a) {
  auto span_of = [](int c) { return c % 64 == 0 ? 64 : (c % 32 == 0 ? 32 : 16); };
  conv_tile_box(a.W, a.H, a.D, kConvTileM, &a.bx, &a.by, &a.bz);
  a.ntx = (a.W + a.bx - 1) / a.bx;
  a.nty = (a.H + a.by - 1) / a.by;
  a.ntz = (a.D + a.bz - 1) / a.bz;
  a.gspan = span_of(a.cout);
  a.halo = a.bx == 128 ? 1 : 0;
  a.span = a.halo ? 16 : span_of(a.cin);
  const int blocks = (27 * a.cin + 127) / 128;
  a.rows = a.halo ? 27 * a.cin : blocks * 128;
  const int T = a.ntx * a.nty * a.ntz;
  int ns = 2 * device_sms() / blocks;
  if (ns < 1) ns = 1;
  a.nsplit = ns > T ? T : ns;
  a.halves = a.halo && a.cin / 16 * 2 * a.nsplit <= device_sms() ? 2 : 1;
  a.nmblk = a.halo ? a.halves * (a.cin / 16) : blocks;
}

bool make_wgrad_maps(CUtensorMap* mx, CUtensorMap* mg, const __nv_bfloat16* x, const __nv_bfloat16* g,
                     const WgradArgs& a) {
  const bool okx = a.halo ? make_conv_input_map(mx, x, a.W, a.H, a.D, a.cin, 16, 130, 3, 3, 1)
                          : make_conv_input_map(mx, x, a.W, a.H, a.D, a.cin, a.span, a.bx, a.by, a.bz, 1);
  return okx && make_conv_input_map(mg, g, a.W, a.H, a.D, a.cout, a.gspan, a.bx, a.by, a.bz, a.cout / a.gspan);
}

cudaError_t init_wgrad_kernel(size_t smem_bytes) {
  return cudaFuncSetAttribute(wgrad_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem_bytes);
}

cudaError_t launch_wgrad(const CUtensorMap& mx, const CUtensorMap& mg, const WgradArgs& a, cudaStream_t s) {
  count_launch();
  wgrad_kernel<<<a.nmblk * a.nsplit, kConvThreads, wgrad_smem_bytes(a), s>>>(mx, mg, a);
  return cudaGetLastError();
}

cudaError_t launch_wgrad_reduce(const float* partial, int nsplit, int rows, int cin_pad, int cin, int cout, float* dw,
                                cudaStream_t s) {
  count_launch();
  wgrad_reduce_kernel<<<ew_grid((long long)cout * cin * 27), 256, 0, s>>>(partial, nsplit, rows, cin_pad, cin, cout, dw);
  return cudaGetLastError();
}

cudaError_t launch_bias_grad(const __nv_bfloat16* g, int c, long long V, float* part, int nblocks, float* db,
                             cudaStream_t s) {
  count_launch(2);
  channel_sum_kernel<<<nblocks, 256, 0, s>>>(g, c, V, part);
  partial_rows_sum_kernel<<<(c + 31) / 32, 256, 0, s>>>(part, nblocks, c, db);
  return cudaGetLastError();
}

cudaError_t launch_head_backward(const float* gp, const __nv_bfloat16* x0, const __nv_bfloat16* top, int c,
                                 const float* w, long long V, __nv_bfloat16* gz, float* part, int nblocks, float* dwb,
                                 cudaStream_t s) {
  count_launch(2);
  head_backward_kernel<<<nblocks, 256, 0, s>>>(gp, x0, top, c, w, V, gz, part);
  partial_rows_sum_kernel<<<(c + 32) / 32, 256, 0, s>>>(part, nblocks, c + 1, dwb);
  return cudaGetLastError();
}

cudaError_t launch_upsample_backward(const __nv_bfloat16* src, int ss, int so, int W, int H, int D, int c,
                                     __nv_bfloat16* dst, cudaStream_t s) {
  count_launch();
  upsample_backward_kernel<<<row_grid((long long)H * D), 256, 0, s>>>(src, ss, so, W, H, D, c, dst);
  return cudaGetLastError();
}

cudaError_t launch_skip_pool_combine(const __nv_bfloat16* skip, int ss, const __nv_bfloat16* act, int as,
                                     const __nv_bfloat16* gpool, int W, int H, int D, int c, __nv_bfloat16* gz,
                                     cudaStream_t s) {
  count_launch();
  skip_pool_combine_kernel<<<row_grid((long long)H * D), 256, 0, s>>>(skip, ss, act, as, gpool, W, H, D, c, gz);
  return cudaGetLastError();
}

cudaError_t launch_loss(const float* p, const float* y, const __nv_bfloat16* x0, long long V, double* part, int nblocks,
                        double* sums, float* g, cudaStream_t s) {
  count_launch(3);
  loss_partials_kernel<<<nblocks, 256, 0, s>>>(p, y, x0, V, part);
  loss_finalize_kernel<<<1, 32, 0, s>>>(part, nblocks, sums);
  loss_grad_kernel<<<ew_grid(V), 256, 0, s>>>(p, y, x0, V, sums, g);
  return cudaGetLastError();
}

cudaError_t launch_adam(float* p, const float* g, float* m, float* v, long long n, float lr, float b1, float b2,
                        float eps, float bc1, float bc2, cudaStream_t s) {
  count_launch();
  adam_kernel<<<ew_grid(n), 256, 0, s>>>(p, g, m, v, n, lr, b1, b2, eps, bc1, bc2);
  return cudaGetLastError();
}

}  // namespace gbmg

// ---------------------------------------------------------------------------
// The network's input channels from one patch's data (device buffers in the
// C ABI's natural layout), and the scale that maps its output back to Phi
// ---------------------------------------------------------------------------

namespace gbmg {

namespace {

struct CellFaces {
  int n;        // ghost faces
  double sum;   // sum of their Dirichlet values
  double sq;    // sum of their squares
};

__device__ __forceinline__ CellFaces ghost_faces(const int8_t* __restrict__ mask, const double* __restrict__ bx,
                                                 const double* __restrict__ by, const double* __restrict__ bz, int nx,
                                                 int ny, int nz, long long v) {
  const int i = (int)(v % nx), j = (int)((v / nx) % ny), k = (int)(v / ((long long)nx * ny));
  const long long sy = nx, sz = (long long)nx * ny;
  const bool in[6] = {i > 0, i + 1 < nx, j > 0, j + 1 < ny, k > 0, k + 1 < nz};
  const long long off[6] = {-1, 1, -sy, sy, -sz, sz};
  const long long nx1 = nx + 1, ny1 = ny + 1;
  const long long fi[6] = {((long long)k * ny + j) * nx1 + i, ((long long)k * ny + j) * nx1 + i + 1,
                           ((long long)k * ny1 + j) * nx + i, ((long long)k * ny1 + j + 1) * nx + i,
                           ((long long)k * ny + j) * nx + i, ((long long)(k + 1) * ny + j) * nx + i};
  const double* fb[6] = {bx, bx, by, by, bz, bz};
  CellFaces r = {0, 0.0, 0.0};
  for (int d = 0; d < 6; ++d) {
    if (in[d] && mask[v + off[d]] > 0) continue;
    const double f = fb[d] ? fb[d][fi[d]] : 0.0;
    r.n += 1;
    r.sum += f;
    r.sq += f * f;
  }
  return r;
}

// per-block partial sums: [0] sum of src^2 over active cells, [1] active
// cells, [2] sum of ghost-face values squared, [3] ghost faces
__global__ void features_partials_kernel(const int8_t* __restrict__ mask, const double* __restrict__ rho,
                                         const double* __restrict__ bx, const double* __restrict__ by,
                                         const double* __restrict__ bz, int nx, int ny, int nz, double h2n2,
                                         double* __restrict__ part) {
  const long long V = (long long)nx * ny * nz;
  double a[4] = {0.0, 0.0, 0.0, 0.0};
  for (long long v = blockIdx.x * (long long)blockDim.x + threadIdx.x; v < V; v += (long long)gridDim.x * blockDim.x) {
    if (mask[v] <= 0) continue;
    const double src = h2n2 * rho[v];
    a[0] += src * src;
    a[1] += 1.0;
    const CellFaces f = ghost_faces(mask, bx, by, bz, nx, ny, nz, v);
    a[2] += f.sq;
    a[3] += f.n;
  }
  __shared__ double sh[4][256];
  for (int q = 0; q < 4; ++q) sh[q][threadIdx.x] = a[q];
  __syncthreads();
  for (int w = blockDim.x / 2; w > 0; w >>= 1) {
    if ((int)threadIdx.x < w)
      for (int q = 0; q < 4; ++q) sh[q][threadIdx.x] += sh[q][threadIdx.x + w];
    __syncthreads();
  }
  if (threadIdx.x < 4) part[4 * blockIdx.x + threadIdx.x] = sh[threadIdx.x][0];
}

// s = sqrt(mean src^2 + mean face^2) (1 when that is not positive), in a
// fixed order over the blocks
__global__ void features_scale_kernel(const double* __restrict__ part, int nblocks, double* __restrict__ s_out) {
  if (threadIdx.x || blockIdx.x) return;
  double a[4] = {0.0, 0.0, 0.0, 0.0};
  for (int b = 0; b < nblocks; ++b)
    for (int q = 0; q < 4; ++q) a[q] += part[4 * b + q];
  const double ms = (a[1] > 0 ? a[0] / a[1] : 0.0) + (a[3] > 0 ? a[2] / a[3] : 0.0);
  const double s = sqrt(ms);
  *s_out = s > 0.0 ? s : 1.0;
}

// xin[0] = src / s on active cells; xin[1] = +1 active, -1 inactive; xin[2] =
// mean ghost-face value / s where the cell has ghost faces
__global__ void features_write_kernel(const int8_t* __restrict__ mask, const double* __restrict__ rho,
                                      const double* __restrict__ bx, const double* __restrict__ by,
                                      const double* __restrict__ bz, int nx, int ny, int nz, double h2n2,
                                      const double* __restrict__ s_dev, float* __restrict__ xin) {
  const long long V = (long long)nx * ny * nz;
  const double s = *s_dev;
  for (long long v = blockIdx.x * (long long)blockDim.x + threadIdx.x; v < V; v += (long long)gridDim.x * blockDim.x) {
    const bool act = mask[v] > 0;
    double f0 = 0.0, f2 = 0.0;
    if (act) {
      f0 = h2n2 * rho[v] / s;
      const CellFaces f = ghost_faces(mask, bx, by, bz, nx, ny, nz, v);
      if (f.n) f2 = f.sum / f.n / s;
    }
    xin[v] = (float)f0;
    xin[V + v] = act ? 1.0f : -1.0f;
    xin[2 * V + v] = (float)f2;
  }
}

// phi[v] = s pred[v] (FP64)
__global__ void scale_prediction_kernel(const float* __restrict__ pred, long long V, const double* __restrict__ s_dev,
                                        double* __restrict__ phi) {
  const double s = *s_dev;
  for (long long v = blockIdx.x * (long long)blockDim.x + threadIdx.x; v < V; v += (long long)gridDim.x * blockDim.x)
    phi[v] = s * (double)pred[v];
}

// y[v] = phi[v] / s (the training target of a solved patch)
__global__ void scale_target_kernel(const double* __restrict__ phi, long long V, const double* __restrict__ s_dev,
                                    float* __restrict__ y) {
  const double s = *s_dev;
  for (long long v = blockIdx.x * (long long)blockDim.x + threadIdx.x; v < V; v += (long long)gridDim.x * blockDim.x)
    y[v] = (float)(phi[v] / s);
}

}  // namespace

cudaError_t launch_features(const int8_t* mask, const double* rho, const double* bx, const double* by,
                            const double* bz, int nx, int ny, int nz, double h, double* part, int nblocks,
                            double* s_dev, float* xin, cudaStream_t s) {
  const int n = nx > ny ? (nx > nz ? nx : nz) : (ny > nz ? ny : nz);
  const double h2n2 = h * h * (double)n * (double)n;
  count_launch(3);
  features_partials_kernel<<<nblocks, 256, 0, s>>>(mask, rho, bx, by, bz, nx, ny, nz, h2n2, part);
  features_scale_kernel<<<1, 32, 0, s>>>(part, nblocks, s_dev);
  features_write_kernel<<<ew_grid((long long)nx * ny * nz), 256, 0, s>>>(mask, rho, bx, by, bz, nx, ny, nz, h2n2, s_dev,
                                                                        xin);
  return cudaGetLastError();
}

cudaError_t launch_scale_prediction(const float* pred, long long V, const double* s_dev, double* phi, cudaStream_t s) {
  count_launch();
  scale_prediction_kernel<<<ew_grid(V), 256, 0, s>>>(pred, V, s_dev, phi);
  return cudaGetLastError();
}

cudaError_t launch_scale_target(const double* phi, long long V, const double* s_dev, float* y, cudaStream_t s) {
  count_launch();
  scale_target_kernel<<<ew_grid(V), 256, 0, s>>>(phi, V, s_dev, y);
  return cudaGetLastError();
}

}  // namespace gbmg
