// FP64 instances of the step kernel.
#include "launch_rows.h"

namespace polfed {

int launch_rows_f64(const StepRun& run, int lpr, bool j2, StepMode mode, int max_group, int64_t items, bool cooperative,
                    int max_teams, cudaStream_t s) {
  switch (mode) {
    case kFilter: return launch_rows_mode<RF64, kFilter>(run, lpr, j2, max_group, items, cooperative, max_teams, s);
    case kDirect: return launch_rows_mode<RF64, kDirect>(run, lpr, j2, max_group, items, cooperative, max_teams, s);
    case kMoments: return launch_rows_mode<RF64, kMoments>(run, lpr, j2, max_group, items, cooperative, max_teams, s);
    default: return fail(POLFED_EINVAL, "per-column coefficients need FP32 storage");
  }
}

}  // namespace polfed
