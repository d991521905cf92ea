// Which host buffers the device may read and write itself (plain C++, no CUDA headers: also compiled by a CPU test).
#pragma once

#include <stddef.h>
#include <stdint.h>

namespace kvattn {

// What the driver says about a host address.
struct HostAddress {
  bool pinned;            // page-locked and mapped for the device
  uintptr_t device;       // its address on the device
  uintptr_t range_start;  // the one allocation or registration that it belongs to, in device addresses
  size_t range_bytes;
};

// The device address of a buffer that starts there, 0 unless all of the buffer lies in that one range.  (Looking at the
// buffer's first and last byte is not enough: under unified addressing two registrations with a gap between them look like
// one, and a kernel's access to the gap would fault.)
inline uintptr_t device_view(const HostAddress& a, size_t bytes) {
  if (!a.pinned || a.device == 0 || (a.device & 3) != 0) return 0;
  if (a.device < a.range_start || a.device - a.range_start > a.range_bytes) return 0;
  return bytes <= a.range_bytes - (a.device - a.range_start) ? a.device : 0;
}

}  // namespace kvattn
