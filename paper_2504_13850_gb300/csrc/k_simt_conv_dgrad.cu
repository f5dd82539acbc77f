// CUDA-core convolution kernels: input gradient.
#include "simt_conv_kernels.cuh"

namespace fo {
namespace simt {

void launch_dgrad(const Geo& g, const void* a, int dta, const void* b, int dtb, void* c, int dtc, bool acc,
                  cudaStream_t st, const void* mask) {
  launch_any<DGRAD>(g, a, dta, b, dtb, nullptr, c, dtc, false, acc, st, mask);
}

}  // namespace simt
}  // namespace fo
