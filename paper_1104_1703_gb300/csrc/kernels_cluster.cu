// The coarse levels of a multigrid iteration as one launch of one
// thread-block cluster, out of distributed shared memory (Guillet & Teyssier,
// arXiv:1104.1703, Section 2 recipe on levels m .. deepest).
//
// What bounds these levels: 10^2 to 10^5 unknowns are too few to fill the
// GPU, so a launch per step costs its latency (1.65 to 2.0 us per half-sweep of
// a 64^3 or 32^3 level in a replayed graph, whatever it holds), and one CTA alone
// is bound by its SM's FP64 rate (2 operations per clock) on a 16^3 level.  Here
// the levels live in the shared memory of up to 16 SMs for the whole visit: a
// half-sweep with its exchange takes 0.32 (FP32) to 0.6 us (FP64).
//
// Split.  A level is cut into slabs of z-planes, one per CTA; the cut of the
// coarsest distributed level decides (so that the fullest CTA holds as few
// unknowns as the shared memory allows) and every finer cut is its double, so
// the children of a CTA's cells are its own.  The levels below (the tail)
// belong to CTA 0 alone, which runs them with block barriers while the others
// wait (0.06 to 0.1 us per half-sweep in FP32, 0.27 to 0.45 in FP64): a level is
// distributed only when one SM would take longer.  Per level a CTA holds
//  - its correction dPhi, dense, both colours, with one halo row in y, one
//    padding slot per row and one halo plane on each side in z;
//  - its unknowns as records in list order: a 16-bit offset (bit 15: the
//    side of the non-shared x-neighbour), b, in second order 1/D and the red
//    ones' D, and where the children and the coarse corners are.
// All but dPhi and b is fixed by the mask: the host lays every CTA's arrays
// out, cl_build_kernel writes its headers and records once, and a launch
// copies them in with one bulk copy before it waits for the previous kernel.
//
// Exchange.  A CTA that updates a cell of its first or last plane also sends
// it to the neighbour's halo plane with st.async, which counts its bytes on
// the neighbour's mbarrier of that side and step.  The receiver knows how
// many to expect, so after a half-sweep it waits for its neighbours' data
// alone: a cluster-wide barrier takes about 1000 cycles on 16 CTAs, more than
// the half-sweep (300).  A CTA without records in that plane sends a 4-byte
// token, so every step exchanges a message each way with each neighbour.
// Consecutive steps use different mbarriers (red, black, prolongation), and a
// CTA sends its next message on one only after a step in between, whose
// answer says that the neighbour is done with the earlier one; the records
// that read a halo plane are the ones that answer, so no halo value is
// overwritten unread.  Cluster barriers remain where the tail begins and
// ends; they also keep the ascent's stores out of the descent's reads.
//
// The residual of a red unknown overwrites the unknown's own dPhi: after it
// the recipe corrects only black unknowns and the next red half-sweep
// overwrites every red one unread (the launcher requires n_pre, n_post >= 1).
// The next level's right-hand side then sums its four red children, whose
// slots hold 0 where they are no unknowns.
//
// Each step's code stands once in the kernel, in one loop over steps: a
// launch runs it from a cold instruction cache, and a second copy of a step
// cost 2 to 3 us when it was first reached.  256 threads: what every warp
// runs alike (headers, exchange, barriers) is issued by two warps per
// scheduler instead of four.
//
// The arithmetic per unknown, and its order, are those of the list kernels
// and of the one-CTA bottom cycle: the results are the same bits.
#include <cmath>
#include <cstring>

#include "async_copy.cuh"
#include "cluster_internal.h"
#include "cycle_device.cuh"

namespace gbmg {

namespace {

constexpr int kClThreads = 256;
constexpr int kClBatch = 16;  // global loads in flight per thread where a level comes in or goes out
constexpr int kClHoist = 2;  // records per colour and thread kept in registers over a level's sweeps
constexpr unsigned long long kClLimitNs = 1000000000ull;  // a wait that runs out ends the launch with NaN
constexpr size_t kClMapBytes = 16 * 1024;  // a coarsest solve's map up to this size is staged in shared memory

// child records: the in-plane offset of slot I of row 2J, the index of plane
// 2K in its owner's slab, the owner, and whether plane 2K + 1 is the next
// CTA's first one
constexpr int kChildPlane = 15, kChildRank = 23;
constexpr uint32_t kChildNext = 1u << 31;
// corner records of the prolongation: element offset of the parent slot and
// the directions of the far corners
constexpr uint32_t kParOff = (1u << 27) - 1, kParX = 1u << 27, kParY = 1u << 28, kParZ = 1u << 29, kParOdd = 1u << 30,
                   kParCol = 1u << 31;

// What one CTA holds of one level, in 16-byte groups (one shared-memory load
// each), at the start of its shared memory.  Offsets are bytes there.
struct __align__(16) ClHeader {
  uint32_t phi[2], b[2];
  uint32_t off[2], id[2];
  uint32_t n[2];
  uint32_t Ps, pl;              // row pitch and plane size of dPhi, bytes
  uint32_t rx_lo[2], rx_hi[2];  // bytes a step receives from the lower / upper neighbour, per colour
  // bit 0 / 1: a lower / upper neighbour; 2 + colour, 4 + colour: no records
  // of that colour in the plane next to it, a token goes instead
  uint32_t flags;
  uint32_t lo_end, hi_begin;    // records below / from these element offsets are in the first / last plane
  uint32_t dg;
  uint32_t lo[2], hi[2];        // from an element's offset to its copy's in the neighbour's halo (mod 2^32)
  uint32_t child[2], par, phi_bytes;
  uint32_t gat[2], pad[2];      // FP64 form: the records' offsets in the global arrays
};
static_assert(sizeof(ClHeader) == 128, "eight groups of 16 bytes");

__device__ __forceinline__ uint32_t map_rank(uint32_t addr, int rank) {
  uint32_t r;
  asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
  return r;
}
__device__ __forceinline__ void st_async(uint32_t addr, float v, uint32_t bar) {
  asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.f32 [%0], %1, [%2];" ::"r"(addr), "f"(v),
               "r"(bar)
               : "memory");
}
__device__ __forceinline__ void st_async(uint32_t addr, double v, uint32_t bar) {
  asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.f64 [%0], %1, [%2];" ::"r"(addr), "d"(v),
               "r"(bar)
               : "memory");
}
__device__ __forceinline__ void st_async_token(uint32_t addr, uint32_t bar) {
  asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.u32 [%0], %1, [%2];" ::"r"(addr), "r"(0u),
               "r"(bar)
               : "memory");
}
__device__ __forceinline__ void ld_cluster(uint32_t addr, float& v) {
  asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(v) : "r"(addr) : "memory");
}
__device__ __forceinline__ void ld_cluster(uint32_t addr, double& v) {
  asm volatile("ld.shared::cluster.f64 %0, [%1];" : "=d"(v) : "r"(addr) : "memory");
}
__device__ __forceinline__ void cl_arrive() {
  __syncwarp();  // the aligned forms want converged warps
  asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
}
__device__ __forceinline__ void cl_wait() {
  __syncwarp();
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ bool try_wait_cluster(uint32_t bar, unsigned parity) {
  unsigned ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(bar), "r"(parity)
      : "memory");
  return ok != 0;
}

// Waits after a first try failed; gives up after kClLimitNs, or once another
// wait of the CTA has.
__device__ __noinline__ void wait_slow(uint32_t bar, unsigned parity, int* abort_flag) {
  unsigned long long t0 = 0;
  for (unsigned n = 0; !try_wait_cluster(bar, parity); ++n) {
    if (n < 64) continue;
    if (*(volatile int*)abort_flag) return;
    if (t0 == 0) t0 = global_ns();
    if (global_ns() - t0 > kClLimitNs) {
      *(volatile int*)abort_flag = 1;
      return;
    }
  }
}

struct ClBuildLevel {
  Geom g;
  const void* invd[2];
  const void* diag;  // of the red colour
  const uint32_t* list[2];
  const uint32_t* pstart[2];
  int z[kClMaxRanks + 1];  // first plane of every CTA (then nz)
};
struct ClBuildArgs {
  ClHeader H[kClMaxRanks][kClMaxLevels];
  ClBuildLevel L[kClMaxLevels];
  uint32_t fine_phi[kClMaxRanks];  // colour 0 of level tail - 1 in every CTA
  uint32_t blob[kClMaxRanks];
  int nlev, tail, ranks;
  uint32_t stride;
  unsigned char* out;
};

// The headers and records of CTA blockIdx.x into its blob; blockIdx.y
// strides over its records.
template <int KIND, typename T>
__global__ void __launch_bounds__(256) cl_build_kernel(const __grid_constant__ ClBuildArgs a) {
  const int r = blockIdx.x;
  const uint32_t t0 = blockIdx.y * blockDim.x + threadIdx.x, nt = gridDim.y * blockDim.x;
  unsigned char* out = a.out + (size_t)r * a.stride;
  if (blockIdx.y == 0) {
    for (uint32_t w = threadIdx.x; w < sizeof(ClHeader) / 4 * a.nlev; w += blockDim.x)
      reinterpret_cast<uint32_t*>(out)[w] = reinterpret_cast<const uint32_t*>(&a.H[r][0])[w];
    if (threadIdx.x < (unsigned)kClMaxRanks)
      reinterpret_cast<uint32_t*>(out + sizeof(ClHeader) * a.nlev)[threadIdx.x] = a.fine_phi[threadIdx.x];
  }
  for (int l = 0; l < a.nlev; ++l) {
    const ClBuildLevel& L = a.L[l];
    const ClHeader& h = a.H[r][l];
    const int z0 = L.z[r];
    const int Ps = (int)(h.Ps / sizeof(T)), pl = (int)(h.pl / sizeof(T));
    for (int c = 0; c < 2; ++c) {
      const uint32_t first = h.n[c] ? L.pstart[c][z0] : 0u;
      for (uint32_t i = t0; i < h.n[c]; i += nt) {
        const uint32_t e = L.list[c][first + i];
        const uint32_t at = e & kListAt;
        const bool ok = entry_ok(L.g, at, 13);
        int q, j, k;
        L.g.slot_of(ok ? at : (uint32_t)L.g.off0, &q, &j, &k);
        const uint32_t o = ok ? (uint32_t)((k - z0 + 1) * pl + (j + 1) * Ps + q) : 0u;
        reinterpret_cast<uint16_t*>(out + h.off[c])[i] = (uint16_t)(o | ((e & kListPlusX) ? 0x8000u : 0u));
        if (KIND == 1) {
          reinterpret_cast<T*>(out + h.id[c])[i] = ok ? static_cast<const T*>(L.invd[c])[at] : T(0);
          if (c == 0) reinterpret_cast<T*>(out + h.dg)[i] = ok ? static_cast<const T*>(L.diag)[at] : T(0);
        }
        if (sizeof(T) == 8) reinterpret_cast<uint32_t*>(out + h.gat[c])[i] = ok ? at : (uint32_t)L.g.off0;
        if (l > 0) {  // the four red children: slot I of rows 2j, 2j + 1 of planes 2k, 2k + 1
          const ClBuildLevel& F = a.L[l - 1];
          const int fPs = (int)(a.H[0][l - 1].Ps / sizeof(T));
          const int I = 2 * q + ((c ^ j ^ k) & 1);
          int owner = r;
          if (l >= a.tail) {
            owner = 0;
            while (owner + 1 < a.ranks && F.z[owner + 1] <= 2 * k) ++owner;
          }
          const bool next = 2 * k + 1 < F.g.nz && F.z[owner + 1] == 2 * k + 1;
          reinterpret_cast<uint32_t*>(out + h.child[c])[i] =
              (uint32_t)((2 * j + 1) * fPs + I) | ((uint32_t)(2 * k - F.z[owner] + 1) << kChildPlane) |
              ((uint32_t)owner << kChildRank) | (next ? kChildNext : 0u);
        }
        if (c == 1 && l + 1 < a.nlev) {  // the eight coarse corners (p2_sum's)
          const ClHeader& hc = a.H[0][l + 1];
          const int cPs = (int)(hc.Ps / sizeof(T)), cpl = (int)(hc.pl / sizeof(T));
          const int zc0 = l + 1 >= a.tail ? 0 : a.L[l + 1].z[r];
          const int ix = 2 * q + ((1 ^ j ^ k) & 1);
          const int Yn = j >> 1, Zn = k >> 1;
          reinterpret_cast<uint32_t*>(out + h.par)[i] =
              (uint32_t)((Zn - zc0 + 1) * cpl + (Yn + 1) * cPs + (q >> 1)) | ((ix & 1) ? kParX : 0u) |
              ((j & 1) ? kParY : 0u) | ((k & 1) ? kParZ : 0u) | ((q & 1) ? kParOdd : 0u) |
              (((q + Yn + Zn) & 1) ? kParCol : 0u);
        }
      }
    }
  }
}

template <typename T>
struct ClArgs {
  const unsigned char* blobs;
  uint32_t stride;
  uint32_t blob[kClMaxRanks], phi_end[kClMaxRanks];  // per CTA: bytes copied in; end of its dPhi arrays
  const uint32_t* list[2];    // the unknowns of the launch's level 0,
  uint32_t first[kClMaxRanks][2];  // every CTA's first one,
  T* phi[2];                  // correction and right-hand side
  const T* rhs[2];
  int nlev, tail, ranks;
  int n_pre, n_post, coarse_sweeps, n_cycles;
  const T* cmat;  // the coarsest solve's map, or nullptr
  uint32_t cmat_n[2];
  uint32_t map_off, map_bytes;  // CTA 0's shared-memory copy of it (0 bytes: none)
  int* err;
  struct {  // the deeper levels' fields (FP64 form: the level API exposes them)
    T* phi[2];
    T* rhs[2];
  } deep[kClMaxLevels];
};

// Sweeps of a level of the tail, which CTA 0 runs alone: nothing is sent, one
// record per colour and thread, all that stays fixed in registers.  Its own loop,
// because the deepest level often takes 2 * coarse_sweeps half-sweeps here (no
// map above kCoarseMatMax unknowns): in the loop of the distributed levels, which
// holds two records and the sends, each cost 0.2 to 0.3 us more (FP64: every
// idle slot's instructions take the FP64 pipe), 15 to 30 us per visit.  V-cycles
// (launch per step; that loop; this one): 161 x 200 x 143 with holes, first order,
// 346 unknowns deepest, FP64 401, 419, 398 us, FP32 132, 142, 123; 96 x 80 x 100,
// 68 unknowns, FP64 181, 169, 139.  (One warp for levels of at most 64 unknowns
// per colour, two records per thread: 163 in the last.)
template <int KIND, typename T>
__device__ __forceinline__ void cl_tail_sweeps(T* const (&phi)[2], const uint16_t* const (&off)[2],
                                               const T* const (&b)[2], const T* const (&id)[2], const uint32_t (&n)[2],
                                               int Ps, int pl, int sweeps) {
  const uint32_t x = threadIdx.x;
  bool has[2];
  T* self[2];
  const T* other[2];
  int dx[2];
  T bb[2], ii[2];
#pragma unroll
  for (int c = 0; c < 2; ++c) {
    has[c] = x < n[c];
    const uint32_t e = has[c] ? off[c][x] : 0u;
#ifdef MG_CHECKED
    has[c] = has[c] && (e & 0x7fffu) != 0;  // an entry that failed its bounds check
#endif
    self[c] = phi[c] + (e & 0x7fffu);
    other[c] = phi[c ^ 1] + (e & 0x7fffu);
    dx[c] = (e & 0x8000u) ? 1 : -1;
    bb[c] = has[c] ? b[c][x] : T(0);
    ii[c] = KIND == 1 ? (has[c] ? id[c][x] : T(0)) : T(1) / T(6);
  }
#pragma unroll 1
  for (int s = 0; s < sweeps; ++s)
#pragma unroll
    for (int c = 0; c < 2; ++c) {
      if (has[c]) {
        const T* p = other[c];
        const T sum = ((p[0] + p[dx[c]]) + (p[-Ps] + p[Ps])) + (p[-pl] + p[pl]);
        *self[c] = (sum - bb[c]) * ii[c];
      }
      __syncthreads();
    }
}

template <int KIND, typename T>
__global__ void __launch_bounds__(kClThreads, 1) cluster_cycle_kernel(const __grid_constant__ ClArgs<T> a) {
  extern __shared__ __align__(128) unsigned char smem[];
  // [side * 3 + step]: messages from the lower / upper neighbour, step 0 / 1 a
  // red / black half-sweep, 2 the prolongation; 6: the bulk copy
  __shared__ unsigned long long bars[7];
  __shared__ uint32_t token;
  __shared__ T xmap[2 * kCoarseMatMax];  // inputs of the coarsest solve's map
  __shared__ int abort_flag;
  constexpr int W = (int)sizeof(T);
  constexpr bool kGat = sizeof(T) == 8;
  unsigned rank_u;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(rank_u));
  const int rank = (int)rank_u;
  const uint32_t tid = threadIdx.x;
  if (tid == 0) {
    for (int i = 0; i < 7; ++i) mbar_init(&bars[i], 1);
    abort_flag = 0;
    mbar_init_fence();
    const uint32_t map_bytes = rank == 0 ? a.map_bytes : 0u;
    mbar_expect_tx(&bars[6], a.blob[rank] + map_bytes);
    bulk_load(smem, a.blobs + (size_t)rank * a.stride, a.blob[rank], &bars[6]);
    if (map_bytes) bulk_load(smem + a.map_off, a.cmat, map_bytes, &bars[6]);
  }
  for (uint32_t o = a.blob[rank] + 16 * tid; o < a.phi_end[rank]; o += 16 * kClThreads)
    *reinterpret_cast<uint4*>(smem + o) = make_uint4(0, 0, 0, 0);
  __syncthreads();
  const bool copied = mbar_wait_bounded(&bars[6], 0, kClLimitNs);
  if (__syncthreads_or(!copied)) {  // no headers: this CTA takes part with no records
    for (uint32_t o = 4 * tid; o < sizeof(ClHeader) * a.nlev; o += 4 * kClThreads)
      *reinterpret_cast<uint32_t*>(smem + o) = 0;
    abort_flag = 1;
    __syncthreads();
  }
  cl_arrive();  // every CTA's barriers and dPhi are set up before any data is sent
  const ClHeader* const H = reinterpret_cast<const ClHeader*>(smem);
  const uint32_t* const fine_phi = reinterpret_cast<const uint32_t*>(smem + sizeof(ClHeader) * a.nlev);
  const uint32_t base = smem_u32(smem), bar0 = smem_u32(bars);
  const int lo_rank = rank > 0 ? rank - 1 : 0, hi_rank = rank + 1 < a.ranks ? rank + 1 : rank;
  const uint32_t lo_base = map_rank(base, lo_rank), hi_base = map_rank(base, hi_rank);
  const uint32_t lo_bar = map_rank(bar0, lo_rank) + 24, hi_bar = map_rank(bar0, hi_rank);  // its side towards this CTA
  auto arr = [&](uint32_t o) { return reinterpret_cast<T*>(smem + o); };
  auto u16 = [&](uint32_t o) { return reinterpret_cast<const uint16_t*>(smem + o); };
  auto u32 = [&](uint32_t o) { return reinterpret_cast<const uint32_t*>(smem + o); };
  if (!kGat)  // level 0's unknowns keep their offset in the global arrays in the place of b until b is known
#pragma unroll 1
    for (int c = 0; c < 2; ++c) {
      const uint32_t n = H[0].n[c], bc = H[0].b[c];
      const uint32_t* list = a.list[c] + a.first[rank][c];
#pragma unroll 1
      for (uint32_t i0 = tid; i0 < n; i0 += kClBatch * kClThreads) {
        uint32_t e[kClBatch];
#pragma unroll
        for (int u = 0; u < kClBatch; ++u) e[u] = i0 + u * kClThreads < n ? list[i0 + u * kClThreads] : 0u;
#pragma unroll
        for (int u = 0; u < kClBatch; ++u)
          if (i0 + u * kClThreads < n)
            *reinterpret_cast<uint32_t*>(smem + bc + (i0 + u * kClThreads) * W) = e[u] & kListAt;
      }
    }
  pdl_wait();
#pragma unroll 1
  for (int c = 0; c < 2; ++c) {
    const uint32_t n = H[0].n[c];
    T* b = arr(H[0].b[c]);
    const uint32_t* gat = kGat ? u32(H[0].gat[c]) : reinterpret_cast<const uint32_t*>(b);
    T* phi = arr(H[0].phi[c]);
    const uint16_t* off = u16(H[0].off[c]);
    const T* rhs = a.rhs[c];
#pragma unroll 1
    for (uint32_t i0 = tid; i0 < n; i0 += kClBatch * kClThreads) {
      T v[kClBatch];
#pragma unroll
      for (int u = 0; u < kClBatch; ++u) v[u] = i0 + u * kClThreads < n ? rhs[gat[i0 + u * kClThreads]] : T(0);
      if (a.n_cycles > 1)  // a later visit of a W-cycle starts from the last one's result
        for (uint32_t i = i0; i < n && i < i0 + kClBatch * kClThreads; i += kClThreads)
          phi[off[i] & 0x7fffu] = a.phi[c][gat[i]];
#pragma unroll
      for (int u = 0; u < kClBatch; ++u)
        if (i0 + u * kClThreads < n) b[i0 + u * kClThreads] = v[u];
    }
  }
  cl_wait();
  __syncthreads();

  uint32_t parity = 0;  // bit side * 3 + step: the parity of the next wait
  // What a step of colour c exchanges at a level: bytes to receive per side,
  // and whether a token goes out per side.
  struct Exchange {
    uint32_t rx[2];
    uint32_t token;
  };
  auto exchange = [&](const ClHeader& h, int c) {
    return Exchange{{h.rx_lo[c], h.rx_hi[c]}, ((h.flags >> (2 + c)) & 1u) | (((h.flags >> (4 + c)) & 1u) << 1)};
  };
  // Every thread's stores of this CTA, and the neighbours' messages of this
  // step, are in place after it (tail levels exchange none).
  auto settle = [&](const Exchange& x, int step) {
    if (tid == 0) {
      if (x.rx[0]) mbar_expect_tx(&bars[step], x.rx[0]);
      if (x.rx[1]) mbar_expect_tx(&bars[3 + step], x.rx[1]);
      if (x.token & 1u) st_async_token(map_rank(smem_u32(&token), lo_rank), lo_bar + 8u * step);
      if (x.token & 2u) st_async_token(map_rank(smem_u32(&token), hi_rank), hi_bar + 8u * step);
    }
    __syncthreads();
#pragma unroll
    for (int side = 0; side < 2; ++side) {
      if (!x.rx[side]) continue;
      const uint32_t bit = 1u << (3 * side + step);
      const unsigned p = (parity & bit) ? 1u : 0u;
      if (!try_wait_cluster(bar0 + 8u * (3 * side + step), p))
        wait_slow(bar0 + 8u * (3 * side + step), p, &abort_flag);
      parity ^= bit;
    }
  };

  if (a.n_cycles > 1) {  // the neighbours' copies of the correction that the level starts from
#pragma unroll 1
    for (int c = 0; c < 2; ++c) {
      const ClHeader& h = H[0];
      const uint16_t* off = u16(h.off[c]);
      for (uint32_t i = tid; i < h.n[c]; i += kClThreads) {
        const uint32_t at = off[i] & 0x7fffu, o = h.phi[c] + at * W;
        if ((h.flags & 1u) && at < h.lo_end) st_async(lo_base + o + h.lo[c], *arr(o), lo_bar + 8u * c);
        if ((h.flags & 2u) && at >= h.hi_begin) st_async(hi_base + o + h.hi[c], *arr(o), hi_bar + 8u * c);
      }
      settle(exchange(h, c), c);
    }
  }

  // mg(i) = {smooth; residual and R1; N_cycles times mg(i + 1); P2; smooth},
  // mg(last) the coarsest solve.  owe: 4 bits per level, the visits of the
  // next level it still owes (the same in every thread of a CTA, and in every
  // CTA above the tail).
  const int last = a.nlev - 1;
  uint32_t owe = 0;
  int i = 0, sweeps = last == 0 ? a.coarse_sweeps : a.n_pre;
  bool down = true;
#pragma unroll 1
  for (;;) {
    const ClHeader& h = H[i];
    const uint32_t n[2] = {h.n[0], h.n[1]};
    const uint32_t phi[2] = {h.phi[0], h.phi[1]}, hb[2] = {h.b[0], h.b[1]};
    const uint32_t hoff[2] = {h.off[0], h.off[1]}, hid[2] = {h.id[0], h.id[1]};
    const int Ps = (int)h.Ps / W, pl = (int)h.pl / W;
    if (down && i == last && a.cmat && i >= a.tail && n[0] == a.cmat_n[0] && n[1] == a.cmat_n[1]) {
      // the coarsest solve by its precomputed map (bottom_coarse_map's
      // product: eight threads per row)
      const uint32_t nr = n[0], nt = nr + n[1], ncol = nt + n[1];
      for (uint32_t j = tid; j < ncol; j += kClThreads)
        xmap[j] = j < nr ? arr(hb[0])[j] : (j < nt ? arr(hb[1])[j - nr] : arr(phi[1])[u16(hoff[1])[j - nt] & 0x7fffu]);
      __syncthreads();
      constexpr int kParts = 8;
      const uint32_t p = tid % kParts;
      const T* M = a.map_bytes ? arr(a.map_off) : a.cmat;
#pragma unroll 1
      for (uint32_t r0 = 0; r0 < nt; r0 += kClThreads / kParts) {
        const uint32_t row_i = r0 + tid / kParts;
        T acc0 = T(0), acc1 = T(0);
        if (row_i < nt) {
          const T* row = M + (size_t)row_i * ncol;
          uint32_t j = p;
#pragma unroll 1
          for (; j + kParts < ncol; j += 2 * kParts) {
            acc0 = fma(row[j], xmap[j], acc0);
            acc1 = fma(row[j + kParts], xmap[j + kParts], acc1);
          }
          if (j < ncol) acc0 = fma(row[j], xmap[j], acc0);
        }
        T acc = acc0 + acc1;
#pragma unroll
        for (int o = kParts / 2; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
        if (row_i < nt && p == 0) {
          const int c = row_i < nr ? 0 : 1;
          arr(phi[c])[u16(hoff[c])[c ? row_i - nr : row_i] & 0x7fffu] = acc;
        }
      }
      __syncthreads();
    } else if (i >= a.tail) {
      T* const f[2] = {arr(phi[0]), arr(phi[1])};
      const uint16_t* const off[2] = {u16(hoff[0]), u16(hoff[1])};
      const T* const b[2] = {arr(hb[0]), arr(hb[1])};
      const T* const id[2] = {arr(hid[0]), arr(hid[1])};
      cl_tail_sweeps<KIND, T>(f, off, b, id, n, Ps, pl, sweeps);
    } else {
      const Exchange ex[2] = {exchange(h, 0), exchange(h, 1)};
      const uint32_t lo_end = (h.flags & 1u) ? h.lo_end : 0u, hi_begin = (h.flags & 2u) ? h.hi_begin : 0xffffffffu;
      const uint32_t lo_to[2] = {lo_base + h.lo[0], lo_base + h.lo[1]}, hi_to[2] = {hi_base + h.hi[0], hi_base + h.hi[1]};
      if (n[0] <= (uint32_t)(kClHoist * kClThreads) && n[1] <= (uint32_t)(kClHoist * kClThreads)) {
        // what stays fixed over the sweeps in registers, so a half-sweep is
        // six loads per record, the update, its store and the exchange
        uint32_t at[2][kClHoist];  // element offset; bit 15: x-neighbour, 16: present, 17 / 18: goes to the lower / upper CTA
        T bb[2][kClHoist], ii[2][kClHoist];
#pragma unroll
        for (int c = 0; c < 2; ++c)
#pragma unroll
          for (int k = 0; k < kClHoist; ++k) {
            const uint32_t x = tid + k * kClThreads;
            bool has = x < n[c];
            uint32_t e = has ? u16(hoff[c])[x] : 0u;
#ifdef MG_CHECKED
            has = has && (e & 0x7fffu) != 0;  // an entry that failed its bounds check
#endif
            bb[c][k] = has ? arr(hb[c])[x] : T(0);
            ii[c][k] = KIND == 1 ? (has ? arr(hid[c])[x] : T(0)) : T(1) / T(6);
            const uint32_t o = e & 0x7fffu;
            at[c][k] = e | (has ? 1u << 16 : 0u) | (has && o < lo_end ? 1u << 17 : 0u) | (has && o >= hi_begin ? 1u << 18 : 0u);
          }
#pragma unroll 1
        for (int s = 0; s < sweeps; ++s) {
#pragma unroll
          for (int c = 0; c < 2; ++c) {
            T v[kClHoist];
#pragma unroll
            for (int k = 0; k < kClHoist; ++k) {
              if (!(at[c][k] & (1u << 16))) continue;
              const T* p = arr(phi[c ^ 1]) + (at[c][k] & 0x7fffu);
              const T sum = ((p[0] + p[(at[c][k] & 0x8000u) ? 1 : -1]) + (p[-Ps] + p[Ps])) + (p[-pl] + p[pl]);
              v[k] = (sum - bb[c][k]) * ii[c][k];
            }
#pragma unroll
            for (int k = 0; k < kClHoist; ++k) {
              if (!(at[c][k] & (1u << 16))) continue;
              const uint32_t o = phi[c] + (at[c][k] & 0x7fffu) * W;
              *arr(o) = v[k];
              if (at[c][k] & (1u << 17)) st_async(lo_to[c] + o, v[k], lo_bar + 8u * c);
              if (at[c][k] & (1u << 18)) st_async(hi_to[c] + o, v[k], hi_bar + 8u * c);
            }
            settle(ex[c], c);
          }
        }
      } else {
#pragma unroll 1
        for (int half = 0; half < 2 * sweeps; ++half) {
          const int c = half & 1;
          const uint32_t nc = c ? n[1] : n[0];
          const uint16_t* off = u16(c ? hoff[1] : hoff[0]);
          const T* b = arr(c ? hb[1] : hb[0]);
          const T* id = arr(c ? hid[1] : hid[0]);
          const T* o = arr(c ? phi[0] : phi[1]);
          const uint32_t self = c ? phi[1] : phi[0];
          const uint32_t lt = c ? lo_to[1] : lo_to[0], ht = c ? hi_to[1] : hi_to[0];
          // four records per thread are loaded before any is stored
          constexpr int U = 4;
#pragma unroll 1
          for (uint32_t i0 = tid; i0 < nc; i0 += U * kClThreads) {
            uint32_t e[U];
            T v[U];
#pragma unroll
            for (int u = 0; u < U; ++u) {
              const uint32_t x = i0 + u * kClThreads < nc ? i0 + u * kClThreads : i0;
              e[u] = off[x];
              const T* p = o + (e[u] & 0x7fffu);
#ifdef MG_CHECKED
              if ((e[u] & 0x7fffu) == 0) p += Ps + pl;
#endif
              const T s = ((p[0] + p[(e[u] & 0x8000u) ? 1 : -1]) + (p[-Ps] + p[Ps])) + (p[-pl] + p[pl]);
              v[u] = (s - b[x]) * (KIND == 1 ? id[x] : T(1) / T(6));
            }
#pragma unroll
            for (int u = 0; u < U; ++u) {
              const uint32_t x = e[u] & 0x7fffu, q = self + x * W;
              if (u && i0 + u * kClThreads >= nc) break;
#ifdef MG_CHECKED
              if (x == 0) continue;
#endif
              *arr(q) = v[u];
              if (x < lo_end) st_async(lt + q, v[u], lo_bar + 8u * c);
              if (x >= hi_begin) st_async(ht + q, v[u], hi_bar + 8u * c);
            }
          }
          settle(c ? ex[1] : ex[0], c);
        }
      }
    }
    if (down && i < last) {
      // residuals of the red unknowns into their own slots
      {
        const uint16_t* off = u16(hoff[0]);
        const T* b = arr(hb[0]);
        const T* dg = arr(h.dg);
        const T* o = arr(phi[1]);
        T* self = arr(phi[0]);
#pragma unroll 1
        for (uint32_t x = tid; x < n[0]; x += kClThreads) {
          const uint32_t e = off[x], at = e & 0x7fffu;
#ifdef MG_CHECKED
          if (at == 0) continue;
#endif
          const T* p = o + at;
          const T s = ((p[0] + p[(e & 0x8000u) ? 1 : -1]) + (p[-Ps] + p[Ps])) + (p[-pl] + p[pl]);
          self[at] = fma(-(KIND == 1 ? dg[x] : T(6)), self[at], s) - b[x];
        }
      }
      // The tail reads the other CTAs' residuals, and they read its
      // correction: a barrier before it begins.  A fresh visit of the next
      // level in a W-cycle starts from 0: the zeroed halo planes must not be
      // overtaken by the neighbours' data.
      const ClHeader& g = H[i + 1];
      const bool rezero = a.n_cycles > 1 && (i + 1 < a.tail || rank == 0);
      const bool meet = i + 1 == a.tail || (i + 1 < a.tail && a.n_cycles > 1);
#pragma unroll 1
      for (int pass = 0; pass < 2; ++pass) {
        if (rezero && (pass == 0) == (i + 1 < a.tail))
          for (uint32_t o = 16 * tid; o < 2 * g.phi_bytes; o += 16 * kClThreads)
            *reinterpret_cast<uint4*>(smem + g.phi[0] + o) = make_uint4(0, 0, 0, 0);
        if (pass == 0 && meet) {
          cl_arrive();
          cl_wait();
        }
      }
      __syncthreads();
      if (i + 1 == a.tail && rank != 0) {
        cl_arrive();  // CTA 0 runs the tail
        cl_wait();
        ++i;
      } else {
        // R1: b of the next level's unknowns from their red children
        const uint32_t fPs = h.Ps, fpl = h.pl;
        const bool far = i + 1 == a.tail;  // other CTAs' residuals
        const uint32_t near = map_rank(base + phi[0], rank);
#pragma unroll 1
        for (int c = 0; c < 2; ++c) {
          const uint32_t* child = u32(g.child[c]);
          T* b = arr(g.b[c]);
#pragma unroll 1
          for (uint32_t x = tid; x < g.n[c]; x += kClThreads) {
            const uint32_t w = child[x];
            const uint32_t in = (w & ((1u << kChildPlane) - 1u)) * W;
            const int owner = (int)((w >> kChildRank) & 31u);
            const uint32_t p = (far ? map_rank(base + fine_phi[owner], owner) : near) + in + ((w >> kChildPlane) & 255u) * fpl;
            const uint32_t p2 = (w & kChildNext) ? map_rank(base + fine_phi[owner + 1], owner + 1) + in + fpl : p + fpl;
            T r0, r1, r2, r3;
            ld_cluster(p, r0);
            ld_cluster(p + fPs, r1);
            ld_cluster(p2, r2);
            ld_cluster(p2 + fPs, r3);
            b[x] = T(-0.5) * (((r0 + r1) + r2) + r3);
          }
        }
        __syncthreads();
        owe = (owe & ~(15u << (4 * i))) | ((uint32_t)a.n_cycles << (4 * i));
        ++i;
        sweeps = i == last ? a.coarse_sweeps : a.n_pre;
        continue;
      }
    } else if (down && last < a.tail) {
      cl_arrive();  // the deepest level is a distributed one: no CTA ascends before all have descended
      cl_wait();
    }
    // up: level i is done
    --i;
    if (i < 0) break;
    if (rank == 0 || i + 1 != a.tail) {
      owe -= 1u << (4 * i);
      if ((owe >> (4 * i)) & 15u) {
        ++i;  // visit it again, from its current correction
        down = true;
        sweeps = i == last ? a.coarse_sweeps : a.n_pre;
        continue;
      }
      if (i + 1 == a.tail) {
        cl_arrive();  // the others wait for the tail
        cl_wait();
      }
    }
    // P2 of level i + 1 into level i's black unknowns (a red half-sweep follows)
    {
      const ClHeader &f = H[i], &g = H[i + 1];
      const uint32_t* par = u32(f.par);
      const uint16_t* off = u16(f.off[1]);
      const uint32_t cb = map_rank(base, i + 1 >= a.tail ? 0 : rank);
      const uint32_t cPs = g.Ps, cpl = g.pl;
      const uint32_t c0 = cb + g.phi[0], c1 = cb + g.phi[1];
      const uint32_t lo_end = (f.flags & 1u) ? f.lo_end : 0u, hi_begin = (f.flags & 2u) ? f.hi_begin : 0xffffffffu;
      const uint32_t nf = f.n[1], fphi = f.phi[1], lt = lo_base + f.lo[1], ht = hi_base + f.hi[1];
#pragma unroll 1
      for (uint32_t x = tid; x < nf; x += kClThreads) {
        const uint32_t w = par[x], at = off[x] & 0x7fffu;
#ifdef MG_CHECKED
        if (at == 0) continue;
#endif
        const uint32_t sn = (w & kParOff) * W;
        const int odd = (w & kParOdd) ? 1 : 0;
        const uint32_t sf = sn + (uint32_t)(((w & kParX) ? odd : odd - 1) * W);
        const uint32_t dY = (w & kParY) ? cPs : 0u - cPs, dZ = (w & kParZ) ? cpl : 0u - cpl;
        const uint32_t cp = (w & kParCol) ? c1 : c0, cq = (w & kParCol) ? c0 : c1;
        T e0, e1a, e1b, e1c, e2a, e2b, e2c, e3;
        ld_cluster(cp + sn, e0);
        ld_cluster(cq + sf, e1a);
        ld_cluster(cq + sn + dY, e1b);
        ld_cluster(cq + sn + dZ, e1c);
        ld_cluster(cp + sn + dY + dZ, e2a);
        ld_cluster(cp + sf + dZ, e2b);
        ld_cluster(cp + sf + dY, e2c);
        ld_cluster(cq + sf + dY + dZ, e3);
        const T e1 = (e1a + e1b) + e1c, e2 = (e2a + e2b) + e2c;
        const T p2 = fma(T(3), e2, fma(T(27), e0, T(9) * e1)) + e3;
        const uint32_t o = fphi + at * W;
        const T v = fma(p2, T(1) / T(64), *arr(o));
        *arr(o) = v;
        if (at < lo_end) st_async(lt + o, v, lo_bar + 16u);
        if (at >= hi_begin) st_async(ht + o, v, hi_bar + 16u);
      }
      settle(exchange(f, 1), 2);
    }
    down = false;
    sweeps = a.n_post;
  }
  cl_arrive();  // no CTA leaves while another may read its shared memory
  // Results to the global arrays: level 0's correction, which the finer level
  // prolongs, and in the FP64 form the deeper levels' fields.
  const bool bad = *(volatile int*)&abort_flag != 0;
  if (bad && tid == 0) atomicExch(a.err, 1);
#pragma unroll 1
  for (int l = 0; l < (kGat ? a.nlev : 1); ++l)
#pragma unroll 1
    for (int c = 0; c < 2; ++c) {
      const ClHeader& h = H[l];
      const T* phi = arr(h.phi[c]);
      const T* b = arr(h.b[c]);
      const uint16_t* off = u16(h.off[c]);
      const uint32_t* to = kGat ? u32(h.gat[c]) : a.list[c] + a.first[rank][c];
      T* out = l == 0 ? a.phi[c] : a.deep[l].phi[c];
      T* out_b = a.deep[l].rhs[c];
      const uint32_t nl = h.n[c];
#pragma unroll 1
      for (uint32_t i0 = tid; i0 < nl; i0 += kClBatch * kClThreads) {
        uint32_t g[kClBatch];
#pragma unroll
        for (int u = 0; u < kClBatch; ++u) g[u] = i0 + u * kClThreads < nl ? to[i0 + u * kClThreads] & kListAt : 0u;
#pragma unroll
        for (int u = 0; u < kClBatch; ++u) {
          const uint32_t x = i0 + u * kClThreads;
          if (x >= nl) break;
          const uint32_t at = off[x] & 0x7fffu;
#ifdef MG_CHECKED
          if (at == 0) continue;
#endif
          out[g[u]] = bad ? T(NAN) : phi[at];
          if (l > 0) out_b[g[u]] = b[x];
        }
      }
    }
  cl_wait();
}

long long level_slots(const Geom& g) { return (long long)g.hx * g.ny * g.nz; }

// Most unknowns of one colour that a CTA takes of a distributed level; a level
// above it runs as one launch per step on all SMs.  Measured per V-cycle of the
// whole hierarchy (12 in one graph), with that level in the cluster and without:
//  - FP64, bound by the FP64 pipe of 16 SMs: 427 to 512 per CTA gain (150 x 15 x
//    15 72.7 -> 68.5 us, 256 x 8 x 8 67.0 -> 64.7), 550 to 1152 lose (29 x 22 x
//    31 61.7 -> 69.0, 32^3 of a ball 65.7 -> 73.2, all of 32^3 82.5 -> 94.4, 24^3
//    69.1 -> 90.6);
//  - FP64 levels that the one-CTA bottom takes otherwise (small_level): 20^3, 800
//    per CTA, 148 -> 76; 3 x 32 x 32, 1024, 94 -> 89;
//  - FP32: up to 2048 per CTA gain (24^3, 1152, 48.9 -> 45.3; 32^3, 1024, 51.3 ->
//    47.0; 8 x 8 x 256, 2048, 45.4 -> 44.2), from 2250 on they lose (15 x 150 x
//    15 49.7 -> 51.5, 64^3 of a union, 3307, 136.9 -> 143.9, 36^3, 5184, 55.7 ->
//    71.2).
uint32_t cl_max_unknowns(const LevelDev& D, int prec) {
  if (prec == kFP32) return 2048u;
  return small_level(D.g) ? 1280u : 512u;
}
// The tail's levels: one record per colour and thread of its one CTA.
bool cl_tail_level(const LevelDev& D, int order) {
  return D.hcount[order * 2] <= (uint32_t)kClThreads && D.hcount[order * 2 + 1] <= (uint32_t)kClThreads;
}

template <typename T>
struct ClFields {
  T* const* phi;
  T* const* rhs;
};
ClFields<double> cl_fields(const LevelDev& L, double) { return {L.phi, L.rhs}; }
ClFields<float> cl_fields(const LevelDev& L, float) { return {L.phi32, L.rhs32}; }

size_t al16(size_t x) { return (x + 15) & ~(size_t)15; }

uint32_t cl_count(const LevelDev& D, int order, int c, int z0, int z1) {
  return D.hpstart[order][c][z1] - D.hpstart[order][c][z0];
}

int cl_plane(const LevelDev* levels, const ClPlan& p, int i, int r) {
  const int nz = levels[p.first + i].g.nz;
  if (i >= p.tail) return r > 0 ? nz : 0;
  if (r >= p.ranks) return nz;
  const int z = p.cut[r] << (p.tail - 1 - i);
  return z < nz ? z : nz;
}

// CTA r's layout: the headers of its levels (but for what depends on its
// neighbours), its copied bytes, the end of dPhi and its total.  `most`: the
// most records of one colour at a distributed level.
struct ClCta {
  ClHeader H[kClMaxLevels];
  uint32_t blob, phi_end, total, most;
};
bool cl_cta(const LevelDev* levels, const ClPlan& p, int order, int prec, int r, ClCta& o) {
  const uint32_t W = prec == kFP64 ? 8 : 4;
  std::memset(&o, 0, sizeof(o));
  size_t end = sizeof(ClHeader) * p.nlev + sizeof(uint32_t) * kClMaxRanks;
  auto take = [&](size_t bytes) {
    const size_t at = end;
    end += al16(bytes);
    return (uint32_t)at;
  };
  for (int i = 0; i < p.nlev; ++i) {
    const LevelDev& D = levels[p.first + i];
    ClHeader& h = o.H[i];
    const int z0 = cl_plane(levels, p, i, r), z1 = cl_plane(levels, p, i, r + 1);
    h.Ps = (uint32_t)(D.g.hx + 1) * W;
    h.pl = (uint32_t)(D.g.ny + 2) * h.Ps;
    h.lo_end = 2 * (h.pl / W);
    h.hi_begin = (uint32_t)(z1 - z0) * (h.pl / W);
    if ((size_t)(z1 - z0 + 2) * (h.pl / W) > 0x7fff || z1 - z0 > 250) return false;  // 15-bit offsets, 8-bit planes
    h.phi_bytes = z1 > z0 ? (uint32_t)al16((size_t)(z1 - z0 + 2) * h.pl) : 0u;
    for (int c = 0; c < 2; ++c) {
      h.n[c] = z1 > z0 ? cl_count(D, order, c, z0, z1) : 0u;
      if (i < p.tail && h.n[c] > o.most) o.most = h.n[c];
      h.off[c] = take(2 * (size_t)h.n[c]);
      if (order == 2) h.id[c] = take((size_t)W * h.n[c]);
      if (i > 0) h.child[c] = take(4 * (size_t)h.n[c]);
      if (prec == kFP64) h.gat[c] = take(4 * (size_t)h.n[c]);
    }
    if (order == 2) h.dg = take((size_t)W * h.n[0]);
    if (i + 1 < p.nlev) h.par = take(4 * (size_t)h.n[1]);
  }
  o.blob = (uint32_t)end;
  end += 16;  // the corner (-1, -1, -1) of the first array reads one element before it
  for (int i = 0; i < p.nlev; ++i)
    for (int c = 0; c < 2; ++c) o.H[i].phi[c] = take(o.H[i].phi_bytes);
  o.phi_end = (uint32_t)end;
  for (int i = 0; i < p.nlev; ++i)
    for (int c = 0; c < 2; ++c) o.H[i].b[c] = take((size_t)W * o.H[i].n[c]);
  o.total = (uint32_t)end;
  return end <= kClSmemBytes;
}

// The plan of a launch from level m: which levels are distributed, and the
// cut that leaves the fullest CTA the fewest records of one colour among the
// cuts whose CTAs all fit their shared memory.
bool cl_plan_from(const LevelDev* levels, int m, int deepest, int order, int prec, ClPlan& p) {
  p = ClPlan();
  p.nlev = deepest - m + 1;
  if (m < 1 || p.nlev < 1 || p.nlev > kClMaxLevels) return false;
  p.first = m;
  // the tail: from its first level on all are small (a coarser level never has
  // more unknowns, but it can have more of one colour)
  p.tail = p.nlev;
  while (p.tail > 0 && cl_tail_level(levels[m + p.tail - 1], order)) --p.tail;
  if (p.tail == 0) return false;  // one CTA: the bottom cycle's case
  const int nzc = levels[m + p.tail - 1].g.nz;
  if (nzc < 2) return false;
  p.ranks = nzc >= 16 ? 16 : (nzc >= 8 ? 8 : (nzc >= 4 ? 4 : 2));
  // an upper bound of a CTA's bytes: per record and per plane of a level,
  // and CTA 0's tail
  const size_t W = prec == kFP64 ? 8 : 4;
  struct Lite {
    const uint32_t* ps[2];
    int nz, dbl;
    size_t per[2], plane;
  } lite[kClMaxLevels];
  size_t fixed = p.nlev * (sizeof(ClHeader) + 13 * 16) + 256, tail_bytes = 0;
  uint64_t total = 0;
  for (int i = 0; i < p.nlev; ++i) {
    const LevelDev& D = levels[m + i];
    Lite& t = lite[i];
    t.nz = D.g.nz;
    t.dbl = p.tail - 1 - i;
    t.plane = 2 * W * (size_t)(D.g.ny + 2) * (D.g.hx + 1);
    for (int c = 0; c < 2; ++c) {
      t.ps[c] = D.hpstart[order][c];
      if (!t.ps[c]) return false;
      t.per[c] = 2 + W + (order == 2 ? W : 0) + (order == 2 && c == 0 ? W : 0) + (i > 0 ? 4 : 0) +
                 (c == 1 && i + 1 < p.nlev ? 4 : 0) + (prec == kFP64 ? 4 : 0);
      if (i >= p.tail) tail_bytes += t.per[c] * t.ps[c][t.nz];
      else if (i == 0) total = total > t.ps[c][t.nz] ? total : t.ps[c][t.nz];
    }
    if (i >= p.tail) tail_bytes += t.plane * (t.nz + 2);
  }
  const uint32_t cap = cl_max_unknowns(levels[m], prec);
  if (total > (uint64_t)cap * p.ranks) return false;
  auto fits = [&](int r, int zc0, int zc1, uint32_t most) {
    size_t bytes = fixed + (r == 0 ? tail_bytes : 0);
    for (int i = 0; i < p.tail; ++i) {
      const Lite& t = lite[i];
      const int z0 = zc0 << t.dbl, z1 = zc1 == nzc || (zc1 << t.dbl) > t.nz ? t.nz : zc1 << t.dbl;
      if ((size_t)(z1 - z0 + 2) * t.plane > 0x7fff * 2 * W || z1 - z0 > 250) return false;
      bytes += t.plane * (z1 - z0 + 2);
      for (int c = 0; c < 2; ++c) {
        const uint32_t n = t.ps[c][z1] - t.ps[c][z0];
        if (n > most) return false;
        bytes += t.per[c] * n;
      }
    }
    return bytes <= kClSmemBytes;
  };
  // greedy fill: each CTA takes planes while it stays within `most` records
  // and its shared memory, and leaves one plane for every CTA after it
  auto fill = [&](uint32_t most) {
    int z = 0;
    for (int r = 0; r < p.ranks; ++r) {
      p.cut[r] = z;
      const int zmax = nzc - (p.ranks - 1 - r);
      int z1 = z;
      while (z1 < zmax && fits(r, z, z1 + 1, most)) ++z1;
      if (z1 == z) return false;
      z = z1;
    }
    return z == nzc;
  };
  uint32_t lo = (uint32_t)(total / p.ranks), hi = cap;
  if (!fill(hi)) return false;
  for (int t = 0; t < 6 && hi > lo + lo / 16 + 8; ++t) {  // fill(hi) holds
    const uint32_t mid = lo + (hi - lo) / 3;
    if (fill(mid)) hi = mid;
    else lo = mid;
  }
  if (!fill(hi)) return false;
  ClCta cta;
  p.smem = 0;
  p.stride = 0;
  for (int r = 0; r < p.ranks; ++r) {
    if (!cl_cta(levels, p, order, prec, r, cta)) return false;
    p.blob[r] = cta.blob;
    p.phi_end[r] = cta.phi_end;
    p.stride = p.stride > cta.blob ? p.stride : cta.blob;
    p.smem = p.smem > cta.total ? p.smem : cta.total;
    if (r == 0) p.total0 = cta.total;
    for (int c = 0; c < 2; ++c) p.top_first[r][c] = levels[m].hpstart[order][c][cl_plane(levels, p, 0, r)];
  }
  p.stride = (p.stride + 127u) & ~127u;
  return true;
}

// The build's arguments: every CTA's headers, completed with what its
// neighbours' layouts fix.
void cl_build_args(const LevelDev* levels, const ClPlan& p, int order, int prec, ClBuildArgs& b) {
  const uint32_t W = prec == kFP64 ? 8 : 4;
  static thread_local ClCta cta[kClMaxRanks];
  std::memset(&b, 0, sizeof(b));
  for (int r = 0; r < p.ranks; ++r) cl_cta(levels, p, order, prec, r, cta[r]);
  for (int i = 0; i < p.nlev; ++i) {
    const LevelDev& D = levels[p.first + i];
    ClBuildLevel& L = b.L[i];
    L.g = D.g;
    for (int c = 0; c < 2; ++c) {
      L.invd[c] = prec == kFP64 ? (const void*)D.invd[c] : (const void*)D.invd32[c];
      L.list[c] = D.list[order][c];
      L.pstart[c] = D.pstart[order][c];
    }
    L.diag = prec == kFP64 ? (const void*)D.diag[0] : (const void*)D.diag32[0];
    for (int r = 0; r <= kClMaxRanks; ++r) L.z[r] = cl_plane(levels, p, i, r);
    for (int r = 0; r < p.ranks; ++r) {
      ClHeader& h = cta[r].H[i];
      const int z0 = L.z[r], z1 = L.z[r + 1];
      if (i >= p.tail) {  // the others read CTA 0's correction
        if (r > 0)
          for (int c = 0; c < 2; ++c) h.phi[c] = cta[0].H[i].phi[c];
        continue;
      }
      const bool lo = r > 0, hi = r + 1 < p.ranks;
      h.flags = (lo ? 1u : 0u) | (hi ? 2u : 0u);
      for (int c = 0; c < 2; ++c) {
        if (lo) {
          const uint32_t from = cl_count(D, order, c, z0 - 1, z0) * W;
          h.rx_lo[c] = from ? from : 4u;
          if (cl_count(D, order, c, z0, z0 + 1) == 0) h.flags |= 4u << c;
          h.lo[c] = cta[r - 1].H[i].phi[c] - h.phi[c] + (uint32_t)(z0 - L.z[r - 1]) * h.pl;
        }
        if (hi) {
          const uint32_t from = cl_count(D, order, c, z1, z1 + 1) * W;
          h.rx_hi[c] = from ? from : 4u;
          if (cl_count(D, order, c, z1 - 1, z1) == 0) h.flags |= 16u << c;
          h.hi[c] = cta[r + 1].H[i].phi[c] - h.phi[c] - (uint32_t)(z1 - z0) * h.pl;
        }
      }
    }
  }
  for (int r = 0; r < p.ranks; ++r) {
    std::memcpy(b.H[r], cta[r].H, sizeof(b.H[r]));
    b.fine_phi[r] = cta[r].H[p.tail - 1].phi[0];
    b.blob[r] = p.blob[r];
  }
  b.nlev = p.nlev;
  b.tail = p.tail;
  b.ranks = p.ranks;
  b.stride = p.stride;
}

template <int KIND, typename T>
cudaError_t cl_attributes(bool* fits) {
  cudaError_t e = cudaFuncSetAttribute(cluster_cycle_kernel<KIND, T>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)kClSmemBytes);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(cluster_cycle_kernel<KIND, T>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(kClMaxRanks);
  cfg.blockDim = dim3(kClThreads);
  cfg.dynamicSmemBytes = kClSmemBytes;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = kClMaxRanks;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  int n = 0;
  e = cudaOccupancyMaxActiveClusters(&n, cluster_cycle_kernel<KIND, T>, &cfg);
  if (e != cudaSuccess || n < 1) {
    (void)cudaGetLastError();
    *fits = false;
  }
  return cudaSuccess;
}

template <typename T>
cudaError_t cluster_t(const LevelDev* levels, const ClPlan& p, int order, int n_pre, int n_post, int coarse_sweeps,
                      int n_cycles, const void* blobs, const T* cmat, const uint32_t* cmat_n, int* err,
                      cudaStream_t s) {
  ClArgs<T> a;
  std::memset(&a, 0, sizeof(a));
  const LevelDev& D = levels[p.first];
  const ClFields<T> f = cl_fields(D, T());
  a.blobs = static_cast<const unsigned char*>(blobs);
  a.stride = p.stride;
  for (int r = 0; r < p.ranks; ++r) {
    a.blob[r] = p.blob[r];
    a.phi_end[r] = p.phi_end[r];
    for (int c = 0; c < 2; ++c) a.first[r][c] = p.top_first[r][c];
  }
  for (int c = 0; c < 2; ++c) {
    a.list[c] = D.list[order][c];
    a.phi[c] = f.phi[c];
    a.rhs[c] = f.rhs[c];
  }
  a.nlev = p.nlev;
  a.tail = p.tail;
  a.ranks = p.ranks;
  a.n_pre = n_pre;
  a.n_post = n_post;
  a.coarse_sweeps = coarse_sweeps;
  a.n_cycles = n_cycles;
  size_t smem = p.smem;
  if (cmat && cmat_n) {
    a.cmat = cmat;
    a.cmat_n[0] = cmat_n[0];
    a.cmat_n[1] = cmat_n[1];
    const size_t nt = (size_t)cmat_n[0] + cmat_n[1];
    const size_t bytes = al16(nt * (nt + cmat_n[1]) * sizeof(T));
    if (bytes <= kClMapBytes && p.total0 + bytes <= kClSmemBytes) {
      a.map_off = p.total0;
      a.map_bytes = (uint32_t)bytes;
      if (p.total0 + bytes > smem) smem = p.total0 + bytes;
    }
  }
  a.err = err;
  for (int i = 1; i < p.nlev; ++i) {
    const ClFields<T> g = cl_fields(levels[p.first + i], T());
    for (int c = 0; c < 2; ++c) {
      a.deep[i].phi[c] = g.phi[c];
      a.deep[i].rhs[c] = g.rhs[c];
    }
  }
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(p.ranks);
  cfg.blockDim = dim3(kClThreads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = p.ranks;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 2;
  count_launch();
  return order == 1 ? cudaLaunchKernelEx(&cfg, cluster_cycle_kernel<2, T>, a)
                    : cudaLaunchKernelEx(&cfg, cluster_cycle_kernel<1, T>, a);
}

}  // namespace

cudaError_t init_cluster_kernels(bool* usable) {
  *usable = true;
  cudaError_t e = cl_attributes<1, double>(usable);
  if (e == cudaSuccess) e = cl_attributes<2, double>(usable);
  if (e == cudaSuccess) e = cl_attributes<1, float>(usable);
  if (e == cudaSuccess) e = cl_attributes<2, float>(usable);
  return e;
}

bool cluster_level(const Geom& g) { return level_slots(g) <= kMidSlots && g.nz <= 512; }

size_t cluster_blob_bound(const LevelDev* levels, int nlev, int prec) {
  // per record 1/D, half a D, offset, children, half the corners and the
  // global offset; a CTA's blob is sized for the fullest one, which holds at
  // most four times the average of a box filled evenly
  const size_t W = prec == kFP64 ? 8 : 4;
  size_t bytes = 0;
  for (int l = 1; l < nlev; ++l)
    if (cluster_level(levels[l].g)) bytes += 2 * (size_t)level_slots(levels[l].g) * (W + W / 2 + 2 + 4 + 2 + 4);
  bytes = 4 * bytes + kClMaxRanks * (kClMaxLevels * (sizeof(ClHeader) + 10 * 16) + 256);
  const size_t full = (size_t)kClMaxRanks * kClSmemBytes;
  return bytes < full ? bytes : full;
}

ClPlan cluster_plan(const LevelDev* levels, int deepest, int order, int prec, size_t blob_bound) {
  ClPlan p;
  for (int m = 1; m <= deepest; ++m) {
    if (cl_plan_from(levels, m, deepest, order, prec, p) && (size_t)p.stride * p.ranks <= blob_bound) return p;
    if (small_level(levels[m].g)) break;  // the one-CTA bottom takes everything from here on
  }
  return ClPlan();
}

cudaError_t launch_cluster_build(const LevelDev* levels, const ClPlan& plan, int order, int prec, void* blobs,
                                 cudaStream_t s) {
  static thread_local ClBuildArgs b;
  cl_build_args(levels, plan, order, prec, b);
  b.out = static_cast<unsigned char*>(blobs);
  const dim3 grid(plan.ranks, 8);
  count_launch();
  if (prec == kFP64) {
    if (order == 2) cl_build_kernel<1, double><<<grid, 256, 0, s>>>(b);
    else cl_build_kernel<2, double><<<grid, 256, 0, s>>>(b);
  } else {
    if (order == 2) cl_build_kernel<1, float><<<grid, 256, 0, s>>>(b);
    else cl_build_kernel<2, float><<<grid, 256, 0, s>>>(b);
  }
  return cudaGetLastError();
}

cudaError_t launch_cluster_cycle(const LevelDev* levels, const ClPlan& plan, int order, int n_pre, int n_post,
                                 int coarse_sweeps, int n_cycles, int prec, const void* blobs, const void* cmat,
                                 const uint32_t* cmat_n, int* err, cudaStream_t s) {
  return prec == kFP32 ? cluster_t<float>(levels, plan, order, n_pre, n_post, coarse_sweeps, n_cycles, blobs,
                                          static_cast<const float*>(cmat), cmat_n, err, s)
                       : cluster_t<double>(levels, plan, order, n_pre, n_post, coarse_sweeps, n_cycles, blobs,
                                           static_cast<const double*>(cmat), cmat_n, err, s);
}

}  // namespace gbmg
