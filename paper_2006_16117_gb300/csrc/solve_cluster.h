// Cluster-based block Thomas solve (solve_cluster.cu).
#pragma once

#include <vector>

#include "internal.h"

namespace sim {

// z_job = (A - σB)^{-1} q_job for the active jobs (vector slots in_slot ->
// out_slot).  Jobs of the same shift that are adjacent in `active` share one
// pass over the factors.  Returns false (nothing launched) when the block size
// does not fit the kernel's shared memory (T above about 2,800 in complex128).
bool block_solve_cluster(const Pencil& P, int precision, const JobSpace& js, const std::vector<int>& active,
                         int in_slot, int out_slot, const double2* d_sigma, void* const* d_factor_ptrs,
                         cudaStream_t st);

// Throws if a block solve on this job space has recorded a failed wait (an mbarrier
// poll limit) in host.err, and clears it.  For the host to call once it has waited
// for the stream: what such a solve left behind is no solution.
void block_solve_check(JobHost& host);

}  // namespace sim
