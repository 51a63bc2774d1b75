// Launching k_step_rows (rows.h).  One translation unit per storage type
// instantiates the kernels, so that they compile in parallel.
#pragma once
#include <algorithm>
#include <mutex>

#include "polfed_internal.h"
#include "rows.h"

namespace polfed {

// Per-kernel, per-device launch configuration, filled once under its mutex.
struct LaunchCache {
  static constexpr int kDevices = 64;
  std::mutex mu;
  struct {
    bool set = false;
    int nsm = 0, maxdyn = 0;
  } d[kDevices];
};

template <class NT, int LPR, bool J2, StepMode MODE>
int launch_rows_t(const StepRun& run, int max_group, int64_t items, bool cooperative, int max_teams,
                         cudaStream_t s) {
  auto kern = k_step_rows<NT, LPR, J2, MODE>;
  static LaunchCache cache;  // the batched runner's worker threads launch concurrently
  int dev = 0;
  PF_CUDA(cudaGetDevice(&dev));
  if (dev < 0 || dev >= LaunchCache::kDevices) return fail(POLFED_EINVAL, "device ordinal beyond the launch cache");
  {
    std::lock_guard<std::mutex> lk(cache.mu);
    auto& c = cache.d[dev];
    if (!c.set) {
      int optin = 0;
      PF_CUDA(cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev));
      cudaFuncAttributes fa;
      PF_CUDA(cudaFuncGetAttributes(&fa, kern));
      c.maxdyn = optin - (int)fa.sharedSizeBytes;
      PF_CUDA(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, c.maxdyn));
      PF_CUDA(cudaDeviceGetAttribute(&c.nsm, cudaDevAttrMultiProcessorCount, dev));
      c.set = true;
    }
  }
  const int nsm = cache.d[dev].nsm;
  int tile = ((max_group + 1) * 16 * LPR + 15) & ~15;
  const int rowd = std::is_same<NT, RF64>::value ? (tile / (16 * LPR)) * (int)sizeof(double) : 0;
  const int per_team = tile + 2 * (int)sizeof(WorkItem<NT>) + rowd;
  int teams = std::min(max_teams, cache.d[dev].maxdyn / per_team);
  if (teams < 1) return fail(POLFED_EINVAL, "slice tile does not fit in shared memory");
  // one CTA per SM; as many teams as there are work items for them
  // (moments: as many CTAs as the buffer of their sums holds)
  const int grid = (int)std::min<int64_t>(MODE == kMoments ? std::min(nsm, kMaxMomentCtas) : nsm, items);
  teams = (int)std::min<int64_t>(teams, (items + grid - 1) / grid);
  StepRun r = run;
  void* args[] = {(void*)&r, (void*)&tile};
  if (cooperative)
    PF_CUDA(cudaLaunchCooperativeKernel((const void*)kern, dim3(grid), dim3(kTeam * teams), args, (size_t)per_team * teams, s));
  else
    PF_CUDA(cudaLaunchKernel((const void*)kern, dim3(grid), dim3(kTeam * teams), args, (size_t)per_team * teams, s));
  return grid;
}

// One StepMode of one storage type over lanes per row and J2.
template <class NT, StepMode MODE>
int launch_rows_mode(const StepRun& run, int lpr, bool j2, int max_group, int64_t items, bool cooperative, int max_teams,
                     cudaStream_t s) {
#define PF_L(L_)                                                                                         \
  case L_:                                                                                               \
    return j2 ? launch_rows_t<NT, L_, true, MODE>(run, max_group, items, cooperative, max_teams, s)      \
              : launch_rows_t<NT, L_, false, MODE>(run, max_group, items, cooperative, max_teams, s);
  switch (lpr) { PF_L(1) PF_L(2) PF_L(4) PF_L(8) }
#undef PF_L
  return fail(POLFED_EINVAL, "unsupported lanes-per-row");
}

}  // namespace polfed
