// Whether the upload kernel may read a caller's buffer (host-only rule).
#pragma once
#include <cstddef>
#include <cstdint>

namespace fo {

// What the runtime knows about the memory a pointer lies in.
struct MemoryRange {
  bool device;      // device memory (not host, not managed)
  int device_id;    // whose
  uintptr_t base;   // the allocation's first byte and its length; length 0 if unknown
  size_t length;
};

// All of [p, p + bytes) lies in one device allocation of the server's device,
// which is also the calling thread's, at a multiple of `align`.  Anything else
// goes to the runtime's copies, which take host, managed and peer memory and
// return an error for a buffer that ends too early, where a kernel would fault.
inline bool upload_kernel_may_read(const MemoryRange& m, uintptr_t p, size_t bytes, size_t align, int server_device,
                                   int current_device) {
  return m.device && m.device_id == server_device && current_device == server_device && p % align == 0 &&
         p >= m.base && p - m.base <= m.length && bytes <= m.length - (p - m.base);
}

}  // namespace fo
