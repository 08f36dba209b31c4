// Whether a kernel may read a host buffer in place.  Plain C++, so that the rule can be tried without a device.
#pragma once
#include <stddef.h>
#include <stdint.h>

namespace paac {

// What the driver says about one host address: pinned and visible to the device, where the device sees it, and the one
// allocation or registration it belongs to.
struct HostRange { bool pinned; uintptr_t device, start; size_t size; };

// The device's view of `bytes` bytes from p on, or nullptr where any of them may not be readable there (the caller then
// copies, which the driver checks).  Both ends being pinned is not enough: a program may have registered pieces of a larger
// array.  So all bytes have to lie in the range of p itself.  Ranges are given in the device's addresses; they are the
// host's wherever this library runs, and a buffer for which they are not is copied too.
template <class Query> const uint8_t* host_view(const uint8_t* p, size_t bytes, Query query) {
  HostRange r{};
  const uintptr_t at = reinterpret_cast<uintptr_t>(p);
  if (!query(p, r) || !r.pinned || r.device != at || at < r.start) return nullptr;
  const uintptr_t before = at - r.start;
  return before <= r.size && bytes <= r.size - before ? p : nullptr;
}

}  // namespace paac
