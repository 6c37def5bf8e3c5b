// Whole-instance solves of 1D instances (nmpc_line_inst.cu): host interface.
#pragma once

#include <cuda_runtime.h>

#include <vector>

namespace nmpc_dev {
struct IterArgs;
struct InstDev;
}  // namespace nmpc_dev

// One launch: the instances list[first .. first + n - 1] (cells per lane cpl),
// each on a cluster of csize CTAs of `warps` warps.
struct LineInstLaunch {
  int cpl, csize, warps, first, n;
  int rows, nu;  // most stages of a CTA, most controls of an instance
  size_t smem;
};

// The launches that solve the 1D instances `which` of a handle, longest work
// first, and the instance list they index; empty where an instance does not
// fit (the caller then iterates with one launch per iteration).
std::vector<LineInstLaunch> line_inst_plan(const std::vector<nmpc_dev::InstDev>& inst,
                                           const std::vector<int>& which, int num_sms,
                                           int max_smem, std::vector<int>* list);
cudaError_t line_inst_configure(int max_smem);

// Enqueue the launches: complete solves from S^0 in the iterate buffers 0
// (k_init_control has run); the returned iterates and their status words are
// written, *retry is set where an instance has to be solved by iterating (see
// the kernel).
cudaError_t line_inst_solve(const std::vector<LineInstLaunch>& plan, const nmpc_dev::IterArgs& A,
                            const int* list_d, int* retry, cudaStream_t st);
