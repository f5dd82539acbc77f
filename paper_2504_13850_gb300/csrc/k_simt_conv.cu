// CUDA-core convolutions (simt_conv_kernels.cuh): problem geometry, tile
// choice, K splits of the weight gradient and their sum, and the entry points.
#include "simt_conv_kernels.cuh"

namespace fo {
namespace simt {

namespace {

Geo make_geo(const ConvShape& s, int mode) {
  Geo g{s.N, s.H, s.W, s.Ci, s.Co, s.k, s.stride, s.pad, s.Ho, s.Wo, 0, 0, 0, 1, 0};
  const int pix_out = s.N * s.Ho * s.Wo, pix_in = s.N * s.H * s.W;   // within kIndexSlack of 2^31 (checked at creation)
  if (mode == FWD) {
    g.M = pix_out; g.Ncol = s.Co; g.K = s.k * s.k * s.Ci;
  } else if (mode == DGRAD) {
    g.M = pix_in; g.Ncol = s.Ci; g.K = s.k * s.k * s.Co;
  } else {
    g.M = s.Co; g.Ncol = s.k * s.k * s.Ci; g.K = pix_out;
  }
  g.kper = g.K;
  return g;
}

// Sums the `splits` partial outputs [splits][n]: eight lanes per output take
// every eighth split, and their sums are added in lane order (a fixed order).
__global__ void __launch_bounds__(256) sum_splits_k(const float* __restrict__ part, int splits, int64_t n,
                                                    float* __restrict__ out) {
  pdl_wait();
  pdl_trigger();
  __shared__ float red[8][32];
  const int e = threadIdx.x % 32, l = threadIdx.x / 32;
  for (int64_t i0 = int64_t(blockIdx.x) * 32; i0 < n; i0 += int64_t(gridDim.x) * 32) {
    float t = 0.f;
    if (i0 + e < n)
#pragma unroll 4
      for (int z = l; z < splits; z += 8) t += part[int64_t(z) * n + i0 + e];
    red[l][e] = t;
    __syncthreads();
    if (l == 0 && i0 + e < n) {
      float o = 0.f;
#pragma unroll
      for (int z = 0; z < 8; ++z) o += red[z][e];
      out[i0 + e] = o;
    }
    __syncthreads();
  }
}

int sm_count() {
  static int sms = 0;
  if (!sms) {
    int dev = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (sms <= 0) sms = 148;
  }
  return sms;
}

}  // namespace

TileShape tile_of(const Geo& g, int mode) {
  auto blocks = [&](int bm, int bn) { return int64_t(ceil_div(g.M, bm)) * ceil_div(g.Ncol, bn); };
  if (g.Ncol <= 32) return {128, 32};
  if (mode == WGRAD) return g.Ncol % 128 == 0 && g.M % 128 == 0 ? TileShape{128, 128} : TileShape{64, 64};   // K is split
  if (blocks(128, 128) >= sm_count()) return {128, 128};
  if (blocks(64, 64) >= sm_count()) return {64, 64};
  return {32, 64};
}

}  // namespace simt

using namespace simt;

void conv_fwd_simt(const ConvShape& s, const void* x, int dt_x, const void* w, int dt_w,
                   const float* bias, void* y, int dt_y, bool relu, cudaStream_t st) {
  launch_fwd(make_geo(s, FWD), x, dt_x, w, dt_w, bias, y, dt_y, relu, st);
}

void conv_dgrad_simt(const ConvShape& s, const void* dy, int dt_dy, const void* w, int dt_w,
                     void* dx, int dt_dx, bool accumulate, const void* mask, cudaStream_t st) {
  launch_dgrad(make_geo(s, DGRAD), dy, dt_dy, w, dt_w, dx, dt_dx, accumulate, st, mask);
}

// The weight gradient's K (output pixels) is long and its output small:
// split K so the grid covers about two blocks per SM, into fp32 partials that
// a second pass sums in a fixed order (deterministic).
int simt_wgrad_splits(const ConvShape& s) {
  const Geo g = make_geo(s, WGRAD);
  const TileShape t = tile_of(g, WGRAD);
  const int64_t blocks = int64_t(ceil_div(g.Ncol, t.bn)) * ceil_div(g.M, t.bm);
  int64_t sp = (2 * sm_count() + blocks - 1) / blocks;
  sp = std::min<int64_t>(sp, std::max<int64_t>(1, g.K / 128));   // at least four 32-deep k-tiles per split
  return int(std::max<int64_t>(1, sp));
}

int64_t simt_wgrad_scratch_floats(const ConvShape& s) {
  const int sp = simt_wgrad_splits(s);
  const Geo g = make_geo(s, WGRAD);
  return sp > 1 ? int64_t(sp) * g.M * g.Ncol : 0;
}

void conv_wgrad_simt(const ConvShape& s, const void* dy, int dt_dy, const void* x, int dt_x,
                     float* dw, float* scratch, cudaStream_t st) {
  Geo g = make_geo(s, WGRAD);
  const int sp = scratch ? simt_wgrad_splits(s) : 1;
  if (sp <= 1) {
    launch_wgrad(g, dy, dt_dy, x, dt_x, dw, st);
    return;
  }
  g.kper = (g.K + sp - 1) / sp;
  g.kper = (g.kper + 31) / 32 * 32;
  const int real = int(ceil_div(g.K, g.kper));
  launch_wgrad(g, dy, dt_dy, x, dt_x, scratch, st);
  const int64_t n = int64_t(g.M) * g.Ncol;
  launch_k(sum_splits_k, int(std::min<int64_t>(ceil_div(n, 32), 8 * sm_count())), 256, 0, st, scratch, real, n, dw);
}

}  // namespace fo
