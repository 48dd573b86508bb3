// Where a field's planes may go (host code).
#pragma once

#include <cstdint>
#include <driver_types.h>

namespace hrm {

// Whether a kernel on `device` may store whole doubles at dst, whose attributes are
// `a` (got: cudaPointerGetAttributes succeeded): plain memory of that device. What
// a copy alone can reach or may have to stage -- memory of another device, host or
// managed memory, an address that is no multiple of 8 -- is left to the copy.
inline bool kernel_target(const double* dst, bool got, const cudaPointerAttributes& a, int device) {
  return got && a.type == cudaMemoryTypeDevice && a.device == device && a.devicePointer == dst &&
         (uintptr_t)dst % sizeof(double) == 0;
}

}  // namespace hrm
