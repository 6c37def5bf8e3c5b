// The two-column strip kernels of nmpc_strip_d64.cu.
#pragma once

namespace nmpc_dev {
struct IterArgs;
}

using StripKernel = void (*)(nmpc_dev::IterArgs, int, int);

// n_lo 1 or 2; rbn: red-black half 1; full_width: grids of at most 64 columns.
StripKernel strip_d64_kernel(int n_lo, bool rbn, bool full_width);

// The actuator patches of those strips: PATCH_D64_ITEMS per CTA of 128 threads.
constexpr int PATCH_D64_ITEMS = 8;
StripKernel patch_d64_kernel(int n_lo);
