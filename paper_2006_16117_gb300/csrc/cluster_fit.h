// What the current device can hold: thread-block clusters of a shape, and its SMs.
#pragma once

#include <stddef.h>

namespace sim {

// How many clusters of `size` CTAs (`threads` threads and `smem` bytes of dynamic
// shared memory each) of a kernel the current device holds at once; 0 if it cannot
// place one (sizes beyond 8 are up to the device).  Also lifts the kernel's limits on
// cluster size and dynamic shared memory on that device, so a launch of a shape
// that fits needs no attributes of its own.  The answer depends on the device, the
// kernel and the shape only and is kept.
int clusters_that_fit(const void* kernel, int size, int threads, size_t smem);

// Multiprocessors of the GPU (one machine's are alike).
int sm_count();

}  // namespace sim
