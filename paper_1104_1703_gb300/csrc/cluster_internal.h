// The coarse levels' cluster cycle (kernels_cluster.cu): its plan, kept per
// order by the hierarchy, and the entry points.
#pragma once

#include "mg_internal.h"

namespace gbmg {

constexpr int kClMaxLevels = 8;
constexpr int kClMaxRanks = 16;              // CTAs of the cluster
constexpr size_t kClSmemBytes = 224 * 1024;  // dynamic shared memory per CTA

// A launch over levels first .. first + nlev - 1 of one order; levels from
// `tail` on (relative to first) are CTA 0's alone.
struct ClPlan {
  int first = 0;  // 0: no launch
  int nlev = 0, tail = 0, ranks = 0;
  int cut[kClMaxRanks + 1] = {};  // first plane of every CTA at the coarsest distributed level
  uint32_t blob[kClMaxRanks] = {}, phi_end[kClMaxRanks] = {};  // per CTA: bytes of headers and records; end of dPhi
  uint32_t top_first[kClMaxRanks][2] = {};  // its first list entry of the first level, per colour
  uint32_t stride = 0;  // bytes between the CTAs' blobs
  uint32_t smem = 0;    // dynamic shared memory of the fullest CTA,
  uint32_t total0 = 0;  // and of CTA 0
};

// Usable on the current device: it runs the largest cluster.
cudaError_t init_cluster_kernels(bool* usable);
// Levels whose lists keep the plane starts the plan needs.
bool cluster_level(const Geom& g);
// Bytes of the record blobs of one order, at most (host, before the mask is known).
size_t cluster_blob_bound(const LevelDev* levels, int nlev, int prec);
// The plan of the first level from which everything down to `deepest` fits.
ClPlan cluster_plan(const LevelDev* levels, int deepest, int order, int prec, size_t blob_bound);
// Builds the CTAs' headers and records (after the lists).
cudaError_t launch_cluster_build(const LevelDev* levels, const ClPlan& plan, int order, int prec, void* blobs,
                                 cudaStream_t s);
// One multigrid iteration with n_cycles coarse iterations per level on levels
// plan.first .. deepest.  err: set when a wait for a neighbour ran out (the
// result is then NaN).
cudaError_t launch_cluster_cycle(const LevelDev* levels, const ClPlan& plan, int order, int n_pre, int n_post,
                                 int coarse_sweeps, int n_cycles, int prec, const void* blobs, const void* cmat,
                                 const uint32_t* cmat_n, int* err, cudaStream_t s);

}  // namespace gbmg
