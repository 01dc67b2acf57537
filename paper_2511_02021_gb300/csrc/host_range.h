// Which host buffers a kernel may read or write in place (host code only).
#pragma once
#include <cstddef>
#include <cstdint>

namespace icon {

// the page-locked allocation or registration that holds an address: where it begins, its bytes,
// and the device's address for the one asked about; size 0 for memory the device has no mapping of
struct HostRange {
  uintptr_t dev = 0, start = 0;
  size_t size = 0;
};

// the device's address of `bytes` bytes of host memory at p if page-locked ranges cover all of
// them, one after the other without a gap and at successive device addresses, else 0. The two ends
// alone say nothing: where the device uses the host's addresses, a buffer registered at its
// ends only, with pageable memory between, has ends as far apart as a whole one's.
template <class Query>
uintptr_t mapped_address(uintptr_t p, size_t bytes, Query query) {
  const uintptr_t end = p + bytes;
  uintptr_t first = 0;
  for (uintptr_t a = p; a < end;) {
    const HostRange r = query(a);
    if (r.size == 0 || !r.dev || a < r.start || a - r.start >= r.size) return 0;
    if (a == p) first = r.dev;
    else if (r.dev - first != a - p) return 0;
    a = r.start + r.size;
  }
  return first;
}

}  // namespace icon
