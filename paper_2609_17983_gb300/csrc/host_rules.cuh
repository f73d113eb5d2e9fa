// host_rules.cuh -- rules of the host side that need no CUDA header, so that a test
// can compile them alone.
#pragma once

#include <cstddef>
#include <cstdint>

namespace kvr {

// What the driver knows of a host address: page-locked and not managed, the
// device's address of it, the allocation or registration that it lies in, and
// whether the device may write there.
struct HostRange {
  bool page_locked = false, writable = false;
  uintptr_t device = 0, start = 0;
  size_t size = 0;
};

// Whether a kernel may store all of [p, p + bytes): a buffer that begins in
// page-locked memory may end outside it (a registration covers what the caller
// asked for, and no more), or in a neighbour with an address of its own.
inline bool device_stores_fit(uintptr_t p, size_t bytes, const HostRange &r) {
  return r.page_locked && r.writable && r.device == p && p >= r.start && p - r.start <= r.size &&
         bytes <= r.size - (p - r.start);
}

}  // namespace kvr
