// Two-column strip kernels with the cluster path's split residual (D64), for
// batches of stages that would also fit a cluster (a translation unit of its
// own: they compile beside the other kernels).
#include "nmpc_core.cuh"
#include "nmpc_strip_d64.h"

namespace nmpc_dev {
#include "nmpc_patch.cuh"
}  // namespace nmpc_dev

using nmpc_dev::k_strip2;

StripKernel strip_d64_kernel(int n_lo, bool rbn, bool full_width) {
  if (n_lo <= 1) {
    if (full_width) return rbn ? k_strip2<1, true, true, true> : k_strip2<1, false, true, true>;
    return rbn ? k_strip2<1, true, true, false> : k_strip2<1, false, true, false>;
  }
  if (full_width) return rbn ? k_strip2<2, true, true, true> : k_strip2<2, false, true, true>;
  return rbn ? k_strip2<2, true, true, false> : k_strip2<2, false, true, false>;
}
