// Two-column strip kernels with the cluster path's split residual (D64), for
// batches of stages that would also fit a cluster (a translation unit of its
// own: they compile beside the other kernels).
#include "nmpc_core.cuh"
#include "nmpc_strip_d64.h"

namespace nmpc_dev {
#include "nmpc_patch.cuh"
}  // namespace nmpc_dev

namespace {
template <int n_lo, bool FW, bool AL>
StripKernel pass_of(bool rbn, bool resid) {
  if (resid) return nmpc_dev::k_strip2<n_lo, false, true, FW, AL, true>;
  return rbn ? nmpc_dev::k_strip2<n_lo, true, true, FW, AL> : nmpc_dev::k_strip2<n_lo, false, true, FW, AL>;
}
template <int n_lo>
StripKernel shape_of(bool rbn, bool full_width, bool aligned, bool resid) {
  if (full_width)
    return aligned ? pass_of<n_lo, true, true>(rbn, resid) : pass_of<n_lo, true, false>(rbn, resid);
  return aligned ? pass_of<n_lo, false, true>(rbn, resid) : pass_of<n_lo, false, false>(rbn, resid);
}
}  // namespace

StripKernel strip_d64_kernel(int n_lo, bool rbn, bool full_width, bool aligned, bool resid) {
  return n_lo <= 1 ? shape_of<1>(rbn, full_width, aligned, resid)
                   : shape_of<2>(rbn, full_width, aligned, resid);
}
