// host_rules.cuh -- rules of the host side that need no CUDA header, so that a test
// can compile them alone.
#pragma once

#include <cstddef>
#include <cstdint>
#include <mutex>

namespace kvr {

// What is set or found out once per device (a kernel's shared memory limit, the
// clusters that fit): with(device, f) runs f on that device's value, one thread at
// a time; f answers from it, or sets the device up and remembers that it did.
constexpr int MAX_DEVICES = 64;  // of those beyond, nothing is remembered
template <class T>
class PerDevice {
 public:
  template <class F>
  auto with(int device, F f) {
    std::lock_guard<std::mutex> lock(mu_);
    T fresh{};
    return f(device >= 0 && device < MAX_DEVICES ? value_[device] : fresh);
  }

 private:
  std::mutex mu_;
  T value_[MAX_DEVICES]{};
};

// raise(bytes) when this device's setting is lower; the first error (0: none).  A
// setting is never lowered, so a launch of another thread keeps what it asked for.
template <class Raise>
int raise_to(PerDevice<size_t> &setting, int device, size_t bytes, Raise raise) {
  return setting.with(device, [&](size_t &have) -> int {
    if (have >= bytes) return 0;
    const int e = (int)raise(bytes);
    if (!e) have = bytes;
    return e;
  });
}

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
