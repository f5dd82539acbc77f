// CUDA-core convolution kernels: weight gradient.
#include "simt_conv_kernels.cuh"

namespace fo {
namespace simt {

void launch_wgrad(const Geo& g, const void* a, int dta, const void* b, int dtb, void* c, cudaStream_t st) {
  launch_any<WGRAD>(g, a, dta, b, dtb, nullptr, c, kF32, false, false, st);
}

}  // namespace simt
}  // namespace fo
