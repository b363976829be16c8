// The rule by which a host array may be accessed by a kernel, apart from the driver query that supplies its inputs.
#pragma once

#include <cstdint>

namespace ccr {

// Does one page-locked allocation, seen by the device under its host address, hold all of [p, p + bytes)?  [start, start + size) is
// the allocation or registration that the driver reports around p, `device` the address it reports for p on the device.
inline bool pinned_range_holds(bool host_memory, bool managed, uint64_t device, uint64_t start, uint64_t size, uint64_t p, uint64_t bytes) {
  return host_memory && !managed && device == p && start != 0 && start <= p && bytes <= size && p - start <= size - bytes;
}

}  // namespace ccr
