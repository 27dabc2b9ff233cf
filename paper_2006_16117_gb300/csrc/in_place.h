// Which of the caller's vectors a kernel may use where they lie.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace sim {

// Vector p (complex128) with attributes `at`, for a kernel on device `dev`: memory of
// that device or managed memory, on a 16-byte boundary.  Another device's memory is
// not: a copy reaches it through unified addressing, a kernel only where peer
// access is on.
inline bool usable_in_place(const cudaPointerAttributes& at, int dev, const void* p) {
    const bool here = (at.type == cudaMemoryTypeDevice && at.device == dev) || at.type == cudaMemoryTypeManaged;
    return here && (reinterpret_cast<uintptr_t>(p) & 15) == 0;
}

}  // namespace sim
