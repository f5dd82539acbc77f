// Test shim: the library's host rule for the upload kernel compiled on its own
// (no CUDA).  Built by tests/test_upload_rule.py.
#include "fo_upload.hpp"

extern "C" int shim_may_read(int device, int device_id, uint64_t base, uint64_t length, uint64_t p, uint64_t bytes,
                             uint64_t align, int server_device, int current_device) {
  const fo::MemoryRange m{device != 0, device_id, uintptr_t(base), size_t(length)};
  return fo::upload_kernel_may_read(m, uintptr_t(p), size_t(bytes), size_t(align), server_device, current_device);
}
