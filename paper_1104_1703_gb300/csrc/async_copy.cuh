// Inline-PTX wrappers for the Blackwell (sm_103a) asynchronous data path
// shared by the temporal-blocked smoothing pass (kernels_pass.cu) and the
// learned-guess network's convolutions (kernels_unet.cu): mbarriers, TMA
// tile copies (cp.async.bulk.tensor), plain bulk copies (cp.async.bulk), the
// global timer for bounded waits, and the tcgen05 tensor-core instructions
// with their tensor-memory (TMEM) accumulators.
#pragma once

#include <cuda.h>

#include <cstdint>

namespace gbmg {
namespace {

__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(unsigned long long* bar, unsigned count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}

// Makes the barrier inits visible to the async proxy (TMA, tensor cores).
__device__ __forceinline__ void mbar_init_fence() {
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}

__device__ __forceinline__ void mbar_expect_tx(unsigned long long* bar, unsigned bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes)
               : "memory");
}

__device__ __forceinline__ void mbar_arrive(unsigned long long* bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}

__device__ __forceinline__ bool mbar_try_wait(unsigned long long* bar, unsigned parity) {
  unsigned ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(smem_u32(bar)), "r"(parity)
      : "memory");
  return ok != 0;
}

__device__ __forceinline__ unsigned long long global_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

// Waits until the barrier completes the phase of `parity`; false if that has
// not happened within `limit_ns`, or as soon as *abort becomes nonzero (when
// abort is non-null).
__device__ __forceinline__ bool mbar_wait_bounded(unsigned long long* bar, unsigned parity,
                                                  unsigned long long limit_ns, const volatile int* abort = nullptr) {
  if (mbar_try_wait(bar, parity)) return true;
  const unsigned long long t0 = global_ns();
  for (;;) {
    if (mbar_try_wait(bar, parity)) return true;
    if (abort && *abort) return false;
    if (global_ns() - t0 > limit_ns) return false;
  }
}

// Orders this thread's earlier generic-proxy shared-memory accesses before
// its later async-proxy ones (a TMA copy into a buffer that was just read).
__device__ __forceinline__ void fence_proxy_async() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }

__device__ __forceinline__ void tma_load_3d(void* dst, const CUtensorMap* map, int x, int y, int z,
                                            unsigned long long* bar) {
  asm volatile(
      "cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], [%5];"
      ::"r"(smem_u32(dst)), "l"((unsigned long long)map), "r"(x), "r"(y), "r"(z), "r"(smem_u32(bar))
      : "memory");
}

__device__ __forceinline__ void tma_load_5d(void* dst, const CUtensorMap* map, int c0, int c1, int c2, int c3, int c4,
                                            unsigned long long* bar) {
  asm volatile(
      "cp.async.bulk.tensor.5d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4, %5, %6}], "
      "[%7];" ::"r"(smem_u32(dst)),
      "l"((unsigned long long)map), "r"(c0), "r"(c1), "r"(c2), "r"(c3), "r"(c4), "r"(smem_u32(bar))
      : "memory");
}

// Contiguous copy of `bytes` (a multiple of 16; both addresses 16-byte
// aligned) from global to shared memory, completed on `bar`.
__device__ __forceinline__ void bulk_load(void* dst, const void* src, unsigned bytes, unsigned long long* bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                   smem_u32(dst)),
               "l"((unsigned long long)src), "r"(bytes), "r"(smem_u32(bar))
               : "memory");
}

// ---- tcgen05 (fifth-generation tensor cores, accumulators in TMEM) ----
//
// The .sync.aligned forms want the warp's lanes converged: a caller whose
// lanes have just parted (one issuing lane, rows outside the grid) does not
// have to join them itself, each of these waits for the whole warp first.

// Allocates `ncols` TMEM columns (a power of two >= 32) for this CTA; the
// whole warp executes it and the TMEM address lands in *dst (shared memory).
__device__ __forceinline__ void tmem_alloc(uint32_t* dst, uint32_t ncols) {
  __syncwarp();
  asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(dst)), "r"(ncols)
               : "memory");
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}

__device__ __forceinline__ void tmem_dealloc(uint32_t taddr, uint32_t ncols) {
  __syncwarp();
  asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols) : "memory");
}

__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

// D[tmem] (+)= A[smem] * B[smem]^T, kind::f16 (both operands BF16 here), one
// CTA; `accumulate` = 0 overwrites D.  The descriptors come as words: offsets
// within shared memory only change the lower one.
__device__ __forceinline__ void tc_mma_f16_words(uint32_t d_tmem, uint32_t a_lo, uint32_t a_hi, uint32_t b_lo,
                                                 uint32_t b_hi, uint32_t idesc, uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t.reg .b64 a, b;\n\t"
      "setp.ne.b32 p, %6, 0;\n\t"
      "mov.b64 a, {%1, %2};\n\t"
      "mov.b64 b, {%3, %4};\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], a, b, %5, p;\n\t}" ::"r"(d_tmem),
      "r"(a_lo), "r"(a_hi), "r"(b_lo), "r"(b_hi), "r"(idesc), "r"(accumulate)
      : "memory");
}

// Arrives once on `bar` when every tcgen05 operation this thread issued
// before it has completed (so their shared-memory operands may be reused and
// their accumulators read).
__device__ __forceinline__ void tc_commit(unsigned long long* bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(bar))
               : "memory");
}

// 16 consecutive 32-bit columns of this warp's 32 TMEM lanes (one lane per
// thread) into registers.
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, float* v) {
  uint32_t r[16];
  __syncwarp();
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, "
      "%15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
        "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(taddr));
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
  for (int i = 0; i < 16; ++i) v[i] = __uint_as_float(r[i]);
}

// Shared-memory matrix descriptor of a tcgen05 operand in the canonical
// K-major layout without swizzle: 8-row x 16-byte core matrices stored as
// 128 contiguous bytes; `lbo` is the byte distance between core matrices
// adjacent along K, `sbo` between core matrices adjacent along M (or N).
__device__ __forceinline__ uint64_t smem_desc_kmajor(const void* base, uint32_t lbo, uint32_t sbo) {
  const uint64_t a = smem_u32(base);
  return ((a >> 4) & 0x3fffull) | (((uint64_t)(lbo >> 4) & 0x3fffull) << 16) |
         (((uint64_t)(sbo >> 4) & 0x3fffull) << 32) | (1ull << 46);
}

// The same for a K-major operand in a swizzled layout, as a TMA copy with
// that swizzle leaves it: rows of `span` bytes (32, 64 or 128) one after
// another, 8 rows a group of `8 * span` bytes.  The pattern's address bits are
// the absolute ones, so `base` may be any row of a buffer that is aligned to
// the pattern (8 * span bytes) and any 32-byte step along K within the rows.
__device__ __forceinline__ uint64_t smem_desc_swizzled(const void* base, uint32_t span) {
  const uint64_t a = smem_u32(base);
  const uint64_t type = span == 128 ? 2ull : (span == 64 ? 4ull : 6ull);
  return ((a >> 4) & 0x3fffull) | (1ull << 16) | (((uint64_t)(8u * span >> 4) & 0x3fffull) << 32) | (1ull << 46) |
         (type << 61);
}

// Shared-memory matrix descriptor of an MN-major operand in a swizzled layout:
// rows (K) of `span` bytes of M or N elements, 8 rows a group, groups one after another along K; `next` is the byte
// distance between blocks of span bytes adjacent along M (or N).  (Here the
// first offset field is the M or N distance and the second the K distance.)
__device__ __forceinline__ uint64_t smem_desc_mn_swizzled(const void* base, uint32_t span, uint32_t next) {
  const uint64_t a = smem_u32(base);
  const uint64_t type = span == 128 ? 2ull : (span == 64 ? 4ull : 6ull);
  return ((a >> 4) & 0x3fffull) | (((uint64_t)(next >> 4) & 0x3fffull) << 16) |
         (((uint64_t)(8u * span >> 4) & 0x3fffull) << 32) | (1ull << 46) | (type << 61);
}

// Instruction descriptor of kind::f16 with BF16 A and B, FP32 accumulator,
// tile M x N; operands K-major unless mn_major (then both MN-major).
__host__ __device__ constexpr uint32_t idesc_bf16_f32(int M, int N, bool mn_major = false) {
  return (1u << 4) | (1u << 7) | (1u << 10) | (mn_major ? (1u << 15) | (1u << 16) : 0u) |
         ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}

}  // namespace
}  // namespace gbmg
