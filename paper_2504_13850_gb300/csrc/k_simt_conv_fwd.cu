// CUDA-core convolution kernels: forward.
#include "simt_conv_kernels.cuh"

namespace fo {
namespace simt {

void launch_fwd(const Geo& g, const void* a, int dta, const void* b, int dtb, const float* bias, void* c, int dtc,
                bool relu, cudaStream_t st) {
  launch_any<FWD>(g, a, dta, b, dtb, bias, c, dtc, relu, false, st);
}

}  // namespace simt
}  // namespace fo
