// The two-column strip kernels of nmpc_strip_d64.cu.
#pragma once

namespace nmpc_dev {
struct IterArgs;
}

using StripKernel = void (*)(nmpc_dev::IterArgs, int, int);

// n_lo 1 or 2; rbn: red-black half 1; full_width: grids of at most 64 columns;
// aligned: even grid widths and array offsets (16-byte column pairs); resid: the
// float64 residual alone (rbn is not read then).
StripKernel strip_d64_kernel(int n_lo, bool rbn, bool full_width, bool aligned, bool resid);
